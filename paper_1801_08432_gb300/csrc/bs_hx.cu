// Fused on-the-fly y = H x over k interleaved vectors (sm_103a).
//
// One CTA owns one destination proton row ip' of one basis block (sector pair
// s' = (s_p', s_n')) and a tile of its neutron columns jn'; every thread owns
// one column (its k values).  The thread sums, in a fixed order,
//   pp: sum over pp jumps into ip' (diagonal and SPE included) c * x[ip, jn']
//   nn: sum over nn jumps into jn' (diagonal and SPE included) c * x[ip', jn]
//   pn: for every source block s linked to s' (a proton one-body class
//       s_p -> s_p' and the matching neutron class s_n -> s_n'),
//       sum over proton jumps (ip, a, phi_p) into ip'
//         phi_p * sum over neutron jumps (jn, b, phi_n) into jn'
//           phi_n * W_pn[a][b] * x_s[ip, jn]
// and writes y once.  This is the paper's factorization (pn = proton one-body
// jump x neutron one-body jump, Sec. on jumps and Table jumps) applied as a
// gather: each y element has one owner, so there are no atomics and the
// result is bit-reproducible.  In a W-truncated basis (Sec. "Truncation of
// the many-body space") a like-particle move may change an SD's W and so its
// sector: those moves come from other blocks through like-particle links,
// and the pn links already join any pair of blocks.
#include <cuda_runtime.h>

#include <type_traits>

#include "bs_internal.h"

namespace bs {

namespace {

template <typename T, int K>
struct Acc {
    T v[K];
};

// load k contiguous values (16-byte vectors where the width allows)
template <typename T, int K>
__device__ __forceinline__ void ldk(const T *__restrict__ p, T (&r)[K])
{
    if constexpr (sizeof(T) * K >= 16) {
        constexpr int W = 16 / sizeof(T);
#pragma unroll
        for (int c = 0; c < K; c += W) {
            if constexpr (sizeof(T) == 4) {
                float4 q = __ldg(reinterpret_cast<const float4 *>(p + c));
                r[c] = q.x; r[c + 1] = q.y; r[c + 2] = q.z; r[c + 3] = q.w;
            } else {
                double2 q = __ldg(reinterpret_cast<const double2 *>(p + c));
                r[c] = q.x; r[c + 1] = q.y;
            }
        }
    } else if constexpr (sizeof(T) == 4 && K == 2) {
        float2 q = __ldg(reinterpret_cast<const float2 *>(p));
        r[0] = q.x; r[1] = q.y;
    } else {
#pragma unroll
        for (int c = 0; c < K; ++c) r[c] = __ldg(p + c);
    }
}

template <typename T, int K>
__device__ __forceinline__ void stk(T *__restrict__ p, const T (&r)[K])
{
    if constexpr (sizeof(T) * K >= 16) {
        constexpr int W = 16 / sizeof(T);
#pragma unroll
        for (int c = 0; c < K; c += W) {
            if constexpr (sizeof(T) == 4) *reinterpret_cast<float4 *>(p + c) = make_float4(r[c], r[c + 1], r[c + 2], r[c + 3]);
            else *reinterpret_cast<double2 *>(p + c) = make_double2(r[c], r[c + 1]);
        }
    } else if constexpr (sizeof(T) == 4 && K == 2) {
        *reinterpret_cast<float2 *>(p) = make_float2(r[0], r[1]);
    } else {
#pragma unroll
        for (int c = 0; c < K; ++c) p[c] = r[c];
    }
}

struct HxArgs {
    const DevTask *tasks;
    const DevBlock *blocks;
    const int64_t *pp_ptr, *nn_ptr, *n1_ptr;
    const int32_t *pp_src, *nn_src;
    const uint32_t *n1_ent;
    const RowJump *jumps;
    const int64_t *jump_ptr;
    const DevLLink *llinks;
    const int64_t *ppx_ptr, *nnx_ptr;
    const int32_t *ppx_src, *nnx_src;
};

// A CTA's warps beyond the tile's columns form further groups (G in all): group
// g takes every G-th like-particle entry and proton jump, and the
// groups' sums meet in shared memory, in the order of the groups.  A thread's
// chain of dependent loads (list pointer, entry, element) is what bounds the
// kernel on small bases and narrow sectors, where the extra warps cost
// nothing.
template <typename T, int K, int NT>
__global__ void __launch_bounds__(NT) hx_fused_kernel(HxArgs A, const T *__restrict__ pp_coef,
                                                      const T *__restrict__ nn_coef, const T *__restrict__ wpn,
                                                      const T *__restrict__ ppx_coef, const T *__restrict__ nnx_coef,
                                                      const T *__restrict__ x, T *__restrict__ y)
{
    __shared__ __align__(16) T part[NT > 128 ? NT - 32 : 96][K];
    const DevTask t = A.tasks[blockIdx.x];
    const DevBlock D = A.blocks[t.block];
    const int cw = (min(128, D.nN - t.col0) + 31) / 32;          // warps of a group
    const int G = NT / 32 / cw, g = (int)(threadIdx.x >> 5) / cw;
    const int lc = (int)threadIdx.x - g * cw * 32;               // column in the tile
    const int col = t.col0 + lc;
    const bool live = g < G && col < D.nN;
    T acc[K];
#pragma unroll
    for (int c = 0; c < K; ++c) acc[c] = T(0);
    T xv[K];
    if (live) {
        // pp (same block): rows ip of x, column col
        {
            const int gr = D.p_start + t.row;
            const int64_t e1 = A.pp_ptr[gr + 1];
            const T *xc = x + (D.off + col) * K;
#pragma unroll 4
            for (int64_t e = A.pp_ptr[gr] + g; e < e1; e += G) {
                const T c = pp_coef[e];
                ldk<T, K>(xc + (int64_t)A.pp_src[e] * D.nN * K, xv);
#pragma unroll
                for (int q = 0; q < K; ++q) acc[q] = fma(c, xv[q], acc[q]);
            }
        }
        // nn (same block): row ip', columns jn
        {
            const int gn = D.n_start + col;
            const int64_t e1 = A.nn_ptr[gn + 1];
            const T *xr = x + (D.off + (int64_t)t.row * D.nN) * K;
#pragma unroll 4
            for (int64_t e = A.nn_ptr[gn] + g; e < e1; e += G) {
                const T c = nn_coef[e];
                ldk<T, K>(xr + (int64_t)A.nn_src[e] * K, xv);
#pragma unroll
                for (int q = 0; q < K; ++q) acc[q] = fma(c, xv[q], acc[q]);
            }
        }
        // like-particle moves from other blocks (W-truncated bases): pp moves from
        // the block of another proton sector with this neutron sector (same
        // column), nn moves from the block of another neutron sector with this
        // proton sector (same row)
        for (int L = D.llink_begin + g; L < D.llink_end; L += G) {
            const DevLLink lk = A.llinks[L];
            const DevBlock S = A.blocks[lk.src_block];
            if (lk.species == 0) {
                const int64_t e1 = A.ppx_ptr[lk.ptr_off + t.row + 1];
                const T *xc = x + (S.off + col) * K;
                for (int64_t e = A.ppx_ptr[lk.ptr_off + t.row]; e < e1; ++e) {
                    const T c = ppx_coef[e];
                    ldk<T, K>(xc + (int64_t)A.ppx_src[e] * S.nN * K, xv);
#pragma unroll
                    for (int q = 0; q < K; ++q) acc[q] = fma(c, xv[q], acc[q]);
                }
            } else {
                const int64_t e1 = A.nnx_ptr[lk.ptr_off + col + 1];
                const T *xr = x + (S.off + (int64_t)t.row * S.nN) * K;
                for (int64_t e = A.nnx_ptr[lk.ptr_off + col]; e < e1; ++e) {
                    const T c = nnx_coef[e];
                    ldk<T, K>(xr + (int64_t)A.nnx_src[e] * K, xv);
#pragma unroll
                    for (int q = 0; q < K; ++q) acc[q] = fma(c, xv[q], acc[q]);
                }
            }
        }
        // pn: the row's proton one-body jumps from every linked block, in one list, each times the column's neutron
        // one-body jumps of that link.  The next jump's record and list bounds are on the way while this one runs: link by
        // link, with its block and two pointers to read before any jump, sd 4p4n k = 4 took 34 us (27 now), pf 5p4n
        // 4p-4h (269 blocks) 2.53 ms (2.07).
        int64_t j = A.jump_ptr[t.list] + g;
        const int64_t j1 = A.jump_ptr[t.list + 1];
        RowJump nj{};
        int64_t nb0 = 0, ne0 = 0;
        auto fetch = [&]() {
            nj = A.jumps[j];
            nb0 = A.n1_ptr[nj.nptr + col];
            ne0 = A.n1_ptr[nj.nptr + col + 1];
        };
        if (j < j1) fetch();
        while (j < j1) {
            const RowJump J = nj;
            const int64_t v0 = nb0, v1 = ne0;
            j += G;
            if (j < j1) fetch();
            const T *xr = x + J.xoff * K;
            const T *Wa = wpn + (J.w & 0x7FFFFFFFu);
            T part[K];
#pragma unroll
            for (int q = 0; q < K; ++q) part[q] = T(0);
#pragma unroll 2
            for (int64_t v = v0; v < v1; ++v) {
                const uint32_t en = A.n1_ent[v];
                T w = __ldg(Wa + ((en >> 16) & 0x7FFFu));
                if (en >> 31) w = -w;
                ldk<T, K>(xr + (int64_t)(en & 0xFFFFu) * K, xv);
#pragma unroll
                for (int q = 0; q < K; ++q) part[q] = fma(w, xv[q], part[q]);
            }
            if (J.w >> 31) {
#pragma unroll
                for (int q = 0; q < K; ++q) acc[q] -= part[q];
            } else {
#pragma unroll
                for (int q = 0; q < K; ++q) acc[q] += part[q];
            }
        }
    }
    if (G > 1) {   // CTA-uniform
        if (live && g > 0) {
#pragma unroll
            for (int q = 0; q < K; ++q) part[(g - 1) * cw * 32 + lc][q] = acc[q];
        }
        __syncthreads();
        if (live && g == 0) {
            for (int h = 1; h < G; ++h)
#pragma unroll
                for (int q = 0; q < K; ++q) acc[q] += part[(h - 1) * cw * 32 + lc][q];
        }
    }
    if (live && g == 0) stk<T, K>(y + (D.off + (int64_t)t.row * D.nN + col) * K, acc);
}

template <typename T, int K>
cudaError_t launch(const Device &Dv, const DevCoefs<T> &C, const T *x, T *y, cudaStream_t s)
{
    HxArgs A{Dv.tasks, Dv.blocks, Dv.pp_ptr, Dv.nn_ptr, Dv.n1_ptr,
             Dv.pp_src, Dv.nn_src, Dv.n1_ent, Dv.jumps, Dv.jump_ptr, Dv.llinks, Dv.ppx_ptr, Dv.nnx_ptr, Dv.ppx_src, Dv.nnx_src};
    auto run = [&](auto nt) {
        constexpr int NT = decltype(nt)::value;
        hx_fused_kernel<T, K, NT><<<Dv.ntasks, NT, 0, s>>>(A, C.pp_coef, C.nn_coef, C.wpn, C.ppx_coef, C.nnx_coef, x, y);
    };
    // Threads by the number of CTAs: with few, more groups shorten each thread's chain of loads; with many, they only
    // take registers.  us at 128 / 256 / 512 threads: sd 2p2n (66 CTAs) FP64 k = 1 15 / 11 / 9; sd 4p4n (495) FP32
    // k = 1 46 / 29 / 21, k = 4 52 / 31 / 27, k = 8 62 / 43 / 39, FP64 k = 4 183 / 148 / 152, k = 8 298 / 245 / -;
    // pf 3p3n (2,200) FP32 k = 1 110 / 95 / 92, k = 2 111 / 105 / 106, k = 4 128 / 124 / 130, k = 8 218 / 211 / 209, FP64
    // k = 1 383 / 332 / 321, k = 4 938 / 824 / 857; pf 4p3n (7,000) FP32 k = 1 384 / 382 / 402, k = 2 398 / 416 / 474,
    // k = 4 501 / 549 / 592; pf 6p2n (35,000) FP32 k = 1 734 / 827 / 995, k = 4 896 / 1210 / 1455.
    constexpr bool wide = K * sizeof(T) == 64;
    if (Dv.ntasks < 1000 && !wide) run(std::integral_constant<int, 512>{});
    else if (Dv.ntasks < 2500) run(std::integral_constant<int, 256>{});
    else run(std::integral_constant<int, 128>{});
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_hx_row(const bs_ctx *c, const void *x, void *y, int k, bs_dtype dt, cudaStream_t s, int variant,
                          bool &used);

cudaError_t launch_hx_pipe(const bs_ctx *c, const void *x, void *y, int k, bs_dtype dt, cudaStream_t s, int v,
                           bool &used);
cudaError_t launch_hx_core(const bs_ctx *c, const void *x, void *y, int k, bs_dtype dt, cudaStream_t s, int v,
                           bool &used, cudaEvent_t t0, cudaEvent_t t1);

// modes of bs_set_kernel the default rule names
constexpr int kPairMode = 16, kCoreMode = 20;

static int kslot(int k)
{
    return k == 1 ? 0 : k == 2 ? 1 : k == 4 ? 2 : 3;
}

// Kernel choice: mode 1 = tiled kernel; mode 2 + v = row kernel variant v;
// mode 2 + R + v = pipelined kernel variant v (R = number of row variants);
// then the core-grouped modes; mode 0 = the mode the autotuner picked for
// (k, dtype), else one chosen by the size of the basis.  A variant that does
// not fit the basis falls back to the tiled kernel.
int launch_hx(const bs_ctx *c, const void *x, void *y, int k, bs_dtype dt, void *stream, std::string &err)
{
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaSetDevice(c->device);
    bool used = false;
    int mode = c->hx_mode;
    // bs_time_kernel: events around the dominant kernel of this product
    const bool timing = c->tev_used < (int)c->tev.size() / 2;
    cudaEvent_t t0 = timing ? c->tev[2 * (size_t)c->tev_used] : nullptr;
    cudaEvent_t t1 = timing ? c->tev[2 * (size_t)c->tev_used + 1] : nullptr;
    bool core_used = false;
    if (timing && e == cudaSuccess) e = cudaEventRecord(t0, s);
    const int R = row_variants();
    if (mode == 0) mode = c->tuned[dt == BS_F64 ? 0 : 1][kslot(k)];
    if (mode == 0 && e == cudaSuccess) {
        const int64_t dim = c->basis.dim;
        // Columns of the widest neutron sector, proton rows (the CTAs of the row and pipelined kernels), and CTAs
        // that fill the chip (one per SM).
        const int nN = c->dev.max_nN, rows = c->dev.nrtasks, chip = c->tab.grid;
        if (dt == BS_F64 || c->dev.trunc) {
            // The first pipelined variant, else the first row variant, else the tiled kernel; small bases the tiled
            // kernel, but where the pipelined one (k >= 2) has a full chip of rows and wide sectors to work on.
            // FP64, us, tiled / row / pipelined at k = 1, 2, 4, 8:
            //   sd 2p2n 9 / 37 / -, 11 / 39 / 28, 15 / 51 / 37, 21 / 71 / 60;  sd 4p4n (495 rows, 81 columns) 64 / 95 / -,
            //   93 / 117 / 126, 152 / 178 / 150, 244 / 561 / 334;  sd 3p5n (220, 119) 50 / 53 / -, 74 / 66 / 64,
            //   115 / 101 / 88, 201 / 286 / 172;  pf 2p3n (190, 145) 60 / 68 / -, 89 / 85 / 75, 131 / 132 / 113, 254 / 340 / 222;
            //   sd 5p5n (69,784 states) 146 / 127 / -, 223 / 213 / 230, 375 / 341 / 308, 620 / 1047 / 597.
            if (dim < 50000 && !(k > 1 && rows >= chip && nN >= 96)) {
                mode = 1;
            } else {
                e = launch_hx_pipe(c, x, y, k, dt, s, 0, used);
                if (!used) mode = 2;
            }
        } else {
            // FP32, not tuned; us per product by the tiled / row / pair-core kernels at k = 1 and 2:
            //   sd 4p4n 21 / 69 / 52, 25 / 71 / 54;  pf 2p4n (190 rows, 565 columns) 72 / 91 / 109, 87 / 106 / 121;
            //   pf 3p3n 94 / 170 / 101, 111 / 179 / 107;  pf 2p5n (20 proton cores) 237 / 213 / 268, 339 / 290 / -;
            //   pf 4p3n 384 / 714 / 316, 398 / 761 / 353;  pf 4p4n 1835 / 1779 / 580, 2096 / 2232 / 721;
            //   pf 6p2n (sectors of 30 columns) 736 / 4956 / -, 724 / 4975 / -;
            // by the tiled / pipelined / core-grouped (20) / pair-core kernels at k = 4 and 8:
            //   sd 4p4n 27 / 50 / 83 / 67, 39 / 72 / 86 / 89;  pf 2p4n 111 / 97 / 70 / 166, 185 / 177 / 91 / 180;
            //   pf 3p3n 127 / 152 / 167 / 162, 210 / 238 / 185 / 228;  pf 4p3n 500 / 741 / 929 / 689, 943 / 1166 / 1001 / 1084;
            //   pf 3p4n (190 proton cores) 648 / 437 / 239 / 276, 1188 / 788 / 330 / 451;
            //   pf 4p4n (1,140) 2781 / 2107 / 1231 / 1140, 5454 / 3915 / 1582 / 2008;  pf 6p2n 888 / 5798 / 9786 / 6620.
            // So: the tiled kernel for narrow sectors (the wide kernels give a thread a column) and small bases, but from
            // k = 4 on not where a full chip of rows is 256 columns wide; pairs of cores (a CTA each) where the proton
            // cores fill the chip, at k = 4 three times; the core-grouped kernel else.
            const int cores = c->dev.pr[k == 1 ? 2 : k == 2 ? 1 : 0].nitems;
            if (nN < 64 || (dim < 100000 && (k < 4 || nN < 256 || rows < chip))) mode = 1;
            else if (k < 4) mode = cores >= chip ? kPairMode : 2;
            else if (k == 4) mode = nN < 256 ? 1 : cores >= 3 * chip ? kPairMode : kCoreMode;
            else mode = kCoreMode;
            if (mode == kPairMode || mode == kCoreMode) {
                // a form that does not fit this basis: the next one
                for (int m : {mode, (int)kCoreMode, 13})
                    if (e == cudaSuccess && !used) e = launch_hx_core(c, x, y, k, dt, s, m - 2 - R - pipe_variants(), used, t0, t1);
                core_used = used;
                if (!used) {
                    e = e == cudaSuccess ? launch_hx_pipe(c, x, y, k, dt, s, 0, used) : e;
                    if (!used) mode = 2;
                }
            }
        }
    }
    const int P = pipe_variants();
    if (e == cudaSuccess && !used && mode >= 2 + R + P) {
        e = launch_hx_core(c, x, y, k, dt, s, mode - 2 - R - P, used, t0, t1);
        core_used = used;
    }
    if (e == cudaSuccess && !used && mode >= 2 + R && mode < 2 + R + P)
        e = launch_hx_pipe(c, x, y, k, dt, s, mode - 2 - R, used);
    if (e == cudaSuccess && !used && mode >= 2 && mode < 2 + R) e = launch_hx_row(c, x, y, k, dt, s, mode - 2, used);
    if (e == cudaSuccess && !used) {
        if (dt == BS_F64) {
            const double *xi = (const double *)x;
            double *yo = (double *)y;
            switch (k) {
            case 1: e = launch<double, 1>(c->dev, c->dev.c64, xi, yo, s); break;
            case 2: e = launch<double, 2>(c->dev, c->dev.c64, xi, yo, s); break;
            case 4: e = launch<double, 4>(c->dev, c->dev.c64, xi, yo, s); break;
            default: e = launch<double, 8>(c->dev, c->dev.c64, xi, yo, s); break;
            }
        } else {
            const float *xi = (const float *)x;
            float *yo = (float *)y;
            switch (k) {
            case 1: e = launch<float, 1>(c->dev, c->dev.c32, xi, yo, s); break;
            case 2: e = launch<float, 2>(c->dev, c->dev.c32, xi, yo, s); break;
            case 4: e = launch<float, 4>(c->dev, c->dev.c32, xi, yo, s); break;
            default: e = launch<float, 8>(c->dev, c->dev.c32, xi, yo, s); break;
            }
        }
    }
    if (timing && e == cudaSuccess) {
        if (!core_used) e = cudaEventRecord(t1, s);
        ++c->tev_used;
    }
    if (e != cudaSuccess) {
        err = std::string("hx launch: ") + cudaGetErrorString(e);
        return BS_ECUDA;
    }
    return BS_OK;
}

}  // namespace bs
