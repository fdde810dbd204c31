// Adjoint of y = H(theta) x (sm_103a).
//
// H is real symmetric, so the input adjoint is gx = H gy (the forward
// kernels).  H is linear in theta = (SPEs, TBMEs) through the decoupling of
// Eq. (hamdef) / Eq. (xpndef), so
//   d/dtheta_t (gy . H x) = sum over jumps of (dc_jump / dtheta_t) gy[dst] . x[src].
// The kernels here reduce gy . x over the jumps into two-body transition
// densities rho(ij,kl), one small matrix per pair key (2m, parity); the host
// contracts them with dW/dtheta.  Through the cores left by the pair kl (and
// ij) each is a Gram matrix,
//   rho(ij,kl) = sum_cores (sign gy[core + ij]) . (sign x[core + kl]),
// with the cores (Z-1 protons, N-1 neutrons) for pn, (N-2 neutrons, any
// proton SD) for nn and (Z-2 protons, any neutron SD) for pp: see
// adj_gram.  Spaces its tables do not cover (more than 32 states per
// species), and vectors that leave its range, take the kernels before it: one value per pp and nn jump, split
// into two-body moves on the host, and the pn densities by atomics per pair
// of jumps.  Products of FP32 vectors are formed in FP32.  adj_gram sums a
// unit's columns in double-float, normalized every 8 to 15 columns of a
// thread (each time within 135 2^-48 of the sum of magnitudes; the products
// themselves are rounded by 2^-24).  Everything else is FP64, collected with
// FP64 atomics (the order of those additions, and so the last bits, may
// differ from run to run).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <new>
#include <type_traits>

#include "bs_internal.h"

namespace bs {

namespace {

template <typename T, int K>
__device__ __forceinline__ double dotk(const T *__restrict__ a, const T *__restrict__ b)
{
    double s = 0.0;
    if constexpr (sizeof(T) == 4) {
        float f = 0.f;   // K <= 8 products of FP32 values
#pragma unroll
        for (int q = 0; q < K; ++q) f = fmaf(a[q], b[q], f);
        s = (double)f;
    } else {
#pragma unroll
        for (int q = 0; q < K; ++q) s = fma(a[q], b[q], s);
    }
    return s;
}

__device__ __forceinline__ double block_sum(double v, double *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    return t;   // valid in thread 0
}

// pp: G[e] = gy[row ip'] . x[row ip_e] over the block's columns and k vectors
template <typename T, int K>
__global__ void adj_pp(const RowTask *tasks, const DevBlock *blocks, const int64_t *pp_ptr, const int32_t *pp_src,
                       const T *__restrict__ x, const T *__restrict__ gy, double *__restrict__ G)
{
    __shared__ double red[32];
    const RowTask t = tasks[blockIdx.x];
    const DevBlock D = blocks[t.block];
    const int g = D.p_start + t.row;
    const T *gr = gy + (D.off + (int64_t)t.row * D.nN) * K;
    for (int64_t e = pp_ptr[g]; e < pp_ptr[g + 1]; ++e) {
        const T *xr = x + (D.off + (int64_t)pp_src[e] * D.nN) * K;
        double s = 0.0;
        for (int c = threadIdx.x; c < D.nN; c += blockDim.x) s += dotk<T, K>(gr + (int64_t)c * K, xr + (int64_t)c * K);
        s = block_sum(s, red);
        if (threadIdx.x == 0) G[e] = s;
    }
}

// nn: G[e] = sum over the block's rows ip of gy[ip, jn'] . x[ip, jn_e]; one CTA per (block, column jn')
template <typename T, int K>
__global__ void adj_nn(const DevBlock *blocks, const int *col_block, const int *col_local, const int64_t *nn_ptr,
                       const int32_t *nn_src, const T *__restrict__ x, const T *__restrict__ gy,
                       double *__restrict__ G)
{
    __shared__ double red[32];
    const DevBlock D = blocks[col_block[blockIdx.x]];
    const int jc = col_local[blockIdx.x];
    const int g = D.n_start + jc;
    for (int64_t e = nn_ptr[g]; e < nn_ptr[g + 1]; ++e) {
        const int js = nn_src[e];
        double s = 0.0;
        for (int r = threadIdx.x; r < D.nP; r += blockDim.x) {
            const int64_t base = D.off + (int64_t)r * D.nN;
            s += dotk<T, K>(gy + (base + jc) * K, x + (base + js) * K);
        }
        s = block_sum(s, red);
        if (threadIdx.x == 0) G[e] = s;
    }
}

// pn: rho[w_off + a nb + b] += phi_u sum_{jn'} sum_{v: b_v = b} phi_v gy[ip', jn'] . x_s[ip_u, jn_v]
template <typename T, int K>
__global__ void adj_pn(const RowTask *tasks, const DevBlock *blocks, const DevLink *links, const int64_t *p1_ptr,
                       const uint32_t *p1_ent, const int64_t *n1_ptr, const uint32_t *n1_ent,
                       const T *__restrict__ x, const T *__restrict__ gy, double *__restrict__ rho)
{
    extern __shared__ double acc[];   // [nb]
    const RowTask t = tasks[blockIdx.x];
    const DevBlock D = blocks[t.block];
    const T *gr = gy + (D.off + (int64_t)t.row * D.nN) * K;
    for (int L = D.link_begin; L < D.link_end; ++L) {
        const DevLink lk = links[L];
        const int64_t pb = p1_ptr[lk.p_ptr_off + t.row], pe = p1_ptr[lk.p_ptr_off + t.row + 1];
        if (pb == pe) continue;
        const DevBlock S = blocks[lk.src_block];
        for (int64_t u = pb; u < pe; ++u) {
            for (int b = threadIdx.x; b < lk.nb; b += blockDim.x) acc[b] = 0.0;
            __syncthreads();
            const uint32_t ep = p1_ent[u];
            const T *xr = x + (S.off + (int64_t)(ep & 0xFFFFu) * S.nN) * K;
            for (int c = threadIdx.x; c < D.nN; c += blockDim.x) {
                const T *gc = gr + (int64_t)c * K;
                for (int64_t v = n1_ptr[lk.n_ptr_off + c]; v < n1_ptr[lk.n_ptr_off + c + 1]; ++v) {
                    const uint32_t en = n1_ent[v];
                    const double d = dotk<T, K>(gc, xr + (int64_t)(en & 0xFFFFu) * K);
                    atomicAdd(&acc[(en >> 16) & 0x7FFFu], (en >> 31) ? -d : d);
                }
            }
            __syncthreads();
            const double sp = (ep >> 31) ? -1.0 : 1.0;
            const int64_t row0 = lk.w_off + (int64_t)((ep >> 16) & 0x7FFFu) * lk.nb;
            for (int b = threadIdx.x; b < lk.nb; b += blockDim.x)
                if (acc[b] != 0.0) atomicAdd(&rho[row0 + b], sp * acc[b]);
            __syncthreads();
        }
    }
}

inline int sgn_below(uint64_t m, int s) { return (__builtin_popcountll(m & ((1ULL << s) - 1ULL)) & 1) ? -1 : 1; }

// sign of a+_i a+_j a_l a_k on X (k<l occupied, i<j empty after removal)
int move_sign(uint64_t X, int i, int j, int k, int l)
{
    int s = sgn_below(X, k);
    uint64_t m = X & ~(1ULL << k);
    s *= sgn_below(m, l);
    m &= ~(1ULL << l);
    s *= sgn_below(m, j);
    m |= 1ULL << j;
    s *= sgn_below(m, i);
    return s;
}

// Splits the per-jump overlaps G of one species (destination-CSR like the
// pp/nn lists) into two-body move densities rho2[p*npairs+q] and the
// one-body number densities rho1[s].
void split_like(const Basis &B, const Interaction &I, int spc, const LikeJumps &Lj, const std::vector<double> &G,
                std::vector<double> &rho2, std::vector<double> &rho1)
{
    const Species &S = B.sp[spc];
    const int ns = (int)B.st.size();
    for (int64_t g = 0; g < (int64_t)S.bits.size(); ++g) {
        const uint64_t dst = S.bits[(size_t)g];
        const int64_t s0 = S.sec[(size_t)S.sec_of_sd[(size_t)g]].start;
        for (int64_t e = Lj.ptr[(size_t)g]; e < Lj.ptr[(size_t)g + 1]; ++e) {
            const double v = G[(size_t)e];
            if (v == 0.0) continue;
            const uint64_t src = S.bits[(size_t)(s0 + Lj.src[(size_t)e])];
            const uint64_t diff = src ^ dst;
            const int nd = __builtin_popcountll(diff);
            if (nd == 0) {
                for (int a = 0; a < ns; ++a) {
                    if (!(src >> a & 1)) continue;
                    rho1[a] += v;
                    for (int b = a + 1; b < ns; ++b)
                        if (src >> b & 1) {
                            const int p = I.pair_id[(size_t)a * ns + b];
                            rho2[(size_t)p * I.npairs + p] += v;
                        }
                }
            } else if (nd == 2) {
                const int k = __builtin_ctzll(src & diff), i = __builtin_ctzll(dst & diff);
                for (int x = 0; x < ns; ++x) {
                    if (x == k || !(src >> x & 1)) continue;
                    const int kk = std::min(k, x), ll = std::max(k, x), ii = std::min(i, x), jj = std::max(i, x);
                    const int q = I.pair_id[(size_t)kk * ns + ll], p = I.pair_id[(size_t)ii * ns + jj];
                    rho2[(size_t)p * I.npairs + q] += v * move_sign(src, ii, jj, kk, ll);
                }
            } else if (nd == 4) {
                const uint64_t out = src & diff, in = dst & diff;
                const int k = __builtin_ctzll(out), l = 63 - __builtin_clzll(out);
                const int i = __builtin_ctzll(in), j = 63 - __builtin_clzll(in);
                const int q = I.pair_id[(size_t)k * ns + l], p = I.pair_id[(size_t)i * ns + j];
                rho2[(size_t)p * I.npairs + q] += v * move_sign(src, i, j, k, l);
            }
        }
    }
}

template <typename T, int K>
int launch_adj(bs_ctx *c, const T *x, const T *gy, cudaStream_t s, std::vector<int> &cb, std::vector<int> &cl)
{
    const Device &D = c->dev;
    const AdjPlan::Moves *M = c->adj.have_moves ? c->adj.moves : nullptr;
    adj_pp<T, K><<<D.nrtasks, 128, 0, s>>>(D.rtasks, D.blocks, M ? M[0].ptr : D.pp_ptr, M ? M[0].src : D.pp_src, x, gy, c->adj_gpp);
    if (!cb.empty()) {
        int *dcb = nullptr, *dcl = nullptr;
        cudaError_t me = cudaMallocAsync((void **)&dcb, cb.size() * sizeof(int), s);
        if (me == cudaSuccess && (me = cudaMallocAsync((void **)&dcl, cl.size() * sizeof(int), s)) != cudaSuccess) cudaFreeAsync(dcb, s);
        if (me != cudaSuccess) {
            (void)cudaGetLastError();
            c->err = std::string("adjoint: ") + cudaGetErrorString(me);
            return BS_ENOMEM;
        }
        cudaMemcpyAsync(dcb, cb.data(), cb.size() * sizeof(int), cudaMemcpyHostToDevice, s);
        cudaMemcpyAsync(dcl, cl.data(), cl.size() * sizeof(int), cudaMemcpyHostToDevice, s);
        adj_nn<T, K><<<(int)cb.size(), 128, 0, s>>>(D.blocks, dcb, dcl, M ? M[1].ptr : D.nn_ptr, M ? M[1].src : D.nn_src, x, gy,
                                                           c->adj_gnn);
        cudaFreeAsync(dcb, s);
        cudaFreeAsync(dcl, s);
    }
    adj_pn<T, K><<<D.nrtasks, 128, (size_t)std::max(1, D.max_nb) * sizeof(double), s>>>(
        D.rtasks, D.blocks, D.links, D.p1_ptr, D.p1_ent, D.n1_ptr, D.n1_ent, x, gy, c->adj_rho);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        c->err = std::string("adjoint launch: ") + cudaGetErrorString(e);
        return BS_ECUDA;
    }
    return BS_OK;
}

// ---------------------------------------------------------------- Gram matrices
constexpr int kGramThreads = 256;
constexpr int kGramTile = 64;          // at most 64 x 64 pairs: 16 x 16 threads of 4 x 4

struct GramArgs {
    const GramUnit *units;
    const GramRow *rows;
    const int *range;                  // batch b: units range[b] .. range[b + 1] - 1
    int nbatch;
    int *next;                         // batches claimed beyond the grid's first ones (zero before the launch)
    const uint16_t *colpos;            // neutron cores (bs_pair.cpp)
    const uint32_t *nsign;
    int ncn;
};

// Two partial sums: FP64, or double-float for FP32 vectors (the FP32 pipe adds
// two terms to hi + lo in 7 packed operations; one FP64 add takes as long as 60).
template <typename T>
struct GramSum;
template <>
struct GramSum<double> {
    double v[2] = {0.0, 0.0};
    __device__ __forceinline__ void add(double f0, double f1)
    {
        v[0] += f0;
        v[1] += f1;
    }
    // K = 1: one fused multiply-add each
    __device__ __forceinline__ void add_prod(double a0, double a1, double b)
    {
        v[0] = fma(a0, b, v[0]);
        v[1] = fma(a1, b, v[1]);
    }
    using Part = double;
    __device__ __forceinline__ double part(int i) const { return v[i]; }
    __device__ __forceinline__ void normalize() {}
    static __device__ __forceinline__ double value(double a) { return a; }
};
template <>
struct GramSum<float> {
    float2 hi = {0.0f, 0.0f}, lo = {0.0f, 0.0f};
    __device__ __forceinline__ void add(float f0, float f1)
    {
        // two-sums; x - y as fma(y, -1, x), the same rounding
        const float2 m = make_float2(-1.0f, -1.0f), f = make_float2(f0, f1);
        const float2 t = __fadd2_rn(hi, f), b = __ffma2_rn(hi, m, t);
        const float2 e = __ffma2_rn(__ffma2_rn(b, m, t), m, hi), g = __ffma2_rn(b, m, f);
        lo = __fadd2_rn(lo, __fadd2_rn(e, g));
        hi = t;
    }
    __device__ __forceinline__ void add_prod(float a0, float a1, float b) { add(__fmul_rn(a0, b), __fmul_rn(a1, b)); }
    // lo back below the last bit of hi: the remainders that add collects are rounded to lo's last bit
    __device__ __forceinline__ void normalize()
    {
        const float2 m = make_float2(-1.0f, -1.0f), t = __fadd2_rn(hi, lo);
        lo = __ffma2_rn(__ffma2_rn(hi, m, t), m, lo);
        hi = t;
    }
    using Part = float2;   // hi, lo
    __device__ __forceinline__ float2 part(int i) const { return i ? make_float2(hi.y, lo.y) : make_float2(hi.x, lo.x); }
    static __device__ __forceinline__ float2 join(float2 a, float2 b)
    {
        const float t = a.x + b.x, z = t - a.x;
        return make_float2(t, a.y + b.y + ((a.x - (t - z)) + (b.x - z)));
    }
    static __device__ __forceinline__ float2 normal(float2 a)
    {
        const float t = a.x + a.y;
        return make_float2(t, a.y - (t - a.x));
    }
    static __device__ __forceinline__ double value(float2 a) { return (double)a.x + (double)a.y; }
};

// K values of a staged element, in 16-byte accesses where it is that wide
template <typename T, int K>
__device__ __forceinline__ void gget(const T *p, T (&v)[K])
{
    if constexpr (K * sizeof(T) >= 16) {
#pragma unroll
        for (int q = 0; q < K; q += 16 / (int)sizeof(T)) *reinterpret_cast<int4 *>(v + q) = *reinterpret_cast<const int4 *>(p + q);
    } else {
#pragma unroll
        for (int q = 0; q < K; ++q) v[q] = p[q];
    }
}
template <typename T, int K>
__device__ __forceinline__ void gput(T *p, const T (&v)[K])
{
    if constexpr (K * sizeof(T) >= 16) {
#pragma unroll
        for (int q = 0; q < K; q += 16 / (int)sizeof(T)) *reinterpret_cast<int4 *>(p + q) = *reinterpret_cast<const int4 *>(v + q);
    } else {
#pragma unroll
        for (int q = 0; q < K; ++q) p[q] = v[q];
    }
}

// rho(ij,kl) += sum over a unit's columns (pn: neutron cores of one group;
// pp: neutron SDs; nn: proton SDs) of gy[ij] . x[kl], for the pairs ij, kl
// that the unit's core leaves free.  A CTA stages the two
// [pairs][columns][K] tiles in shared memory, each element once and with its
// sign, and every element meets all the pairs of the other tile: a thread
// keeps 4 x 4 or 4 x 3 pairs in registers, whichever leaves fewer threads
// without work, and slices of the CTA take every S-th column where one set of
// threads covers the pairs several times.  A unit's sums are added to the
// matrix tile in shared memory (FP64), which goes to memory when the CTA's
// units (ordered by tile, claimed in batches from a counter) leave it.  FP32
// operations bound it (K multiply-adds and 7 adds per pair and column) or
// FP64 ones.  48Cr k = 4: 26.7 ms for pn alone with an FP64 shared-memory
// atomic per pair of jumps, 2.3 ms with every pair of the key in fixed
// threads, 2.1 ms this way (0.44 of the FP32 pipe; many small units).
template <typename T>
__host__ __device__ constexpr int gram_lg(int e) { return e == 4 ? 6 : e == 8 ? 5 : e == 16 ? 4 : e == 32 ? 3 : 2; }   // 2^lg columns of 128 pairs fit
template <typename T, int K>
__host__ __device__ constexpr int gram_pad() { return K * (int)sizeof(T) < 16 ? K : 16 / (int)sizeof(T); }   // neighbouring pairs' elements in other banks
template <typename T, int K>
__host__ __device__ constexpr int gram_tile_elems() { return 2 * kGramTile * ((1 << gram_lg<T>(K * (int)sizeof(T))) * K + gram_pad<T, K>()); }
template <typename T, int K>
constexpr size_t gram_smem() { return (size_t)kGramTile * kGramTile * 8 + (size_t)gram_tile_elems<T, K>() * sizeof(T); }

template <typename T, int K>
__global__ void __launch_bounds__(kGramThreads, 2) adj_gram(GramArgs A, const T *__restrict__ x, const T *__restrict__ gy,
                                                            double *__restrict__ rho)
{
    constexpr int E = K * (int)sizeof(T);                 // bytes of an element
    constexpr int LG = gram_lg<T>(E), PAD = gram_pad<T, K>();
    extern __shared__ __align__(16) unsigned char gsm[];
    double *mat = reinterpret_cast<double *>(gsm);        // the tile's sums, [kl][ij]
    T *tiles = reinterpret_cast<T *>(mat + kGramTile * kGramTile);   // gy's pairs, then x's
    __shared__ int claim;
    // per pair of the two tiles (gy's, then x's): first element, l | sign << 8 (-1: none), place in the matrix tile
    __shared__ int64_t roff[2 * kGramTile];
    __shared__ int rl[2 * kGramTile], rp[2 * kGramTile];
    constexpr int NB = E <= 16 ? 8 : 128 / E;             // elements a thread has on the way at a time
    const int tid = threadIdx.x;
    int out = -1, np = 0, ta = 0, tb = 0;                 // the matrix tile the sums belong to
    int64_t out_at = 0;
    auto leave = [&]() {   // (every thread, between barriers)
        for (int i = tid; i < kGramTile * kGramTile; i += kGramThreads) {
            const int a = i % kGramTile, b = i / kGramTile;
            const double v = mat[i];
            if (out >= 0 && a < ta && b < tb && v != 0.0) atomicAdd(rho + out_at + (int64_t)b * np + a, v);
            mat[i] = 0.0;
        }
    };
    auto unit = [&](const GramUnit &U, auto rbc) {
        constexpr int RB = decltype(rbc)::value;
        const int ga = (U.na + 3) / 4, gb = (U.nb + RB - 1) / RB;
        const int na = 4 * ga, nall = na + RB * gb;   // staged rows: every thread has 4 and RB, absent ones zero
        int lg = LG;   // few pairs leave room for more columns at a time
        while (nall << (lg + 1 - LG) <= 2 * kGramTile) ++lg;
        const int CH = 1 << lg, LD = CH * K + PAD;
        const T *sg = tiles, *sx = tiles + na * LD;
        const int nt = ga * gb, S = kGramThreads / nt;
        const int slice = tid / nt, t = tid % nt, ia = t % ga, ib = t / ga;
        if (tid < 2 * kGramTile) rl[tid] = -1;
        __syncthreads();
        for (int r = tid; r < U.na + U.nb; r += kGramThreads) {
            const bool isx = r >= U.na;
            const GramRow R = A.rows[isx ? U.b0 + r - U.na : U.a0 + r];
            const int slot = isx ? na + r - U.na : r;
            roff[slot] = R.off;
            rl[slot] = R.l | R.sign << 8;
            rp[slot] = isx ? R.pos - U.pb : R.pos - U.pa;
        }
        __syncthreads();
        GramSum<T> acc[2][RB];
        int n = 0;   // columns since the sums were normalized
        for (int c0 = 0; c0 < U.ncol; c0 += CH) {
            if (c0) __syncthreads();
            // columns first, then elements: NB dependent pairs of loads in flight
            const int total = nall * CH;
            for (int n0 = tid; n0 < total; n0 += NB * kGramThreads) {
                int64_t at[NB];
                bool neg[NB];
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    const int n = n0 + j * kGramThreads, slot = n >> lg, col = c0 + (n & (CH - 1));
                    at[j] = -1;
                    neg[j] = false;
                    if (n < total && col < U.ncol) {
                        const int r = rl[slot];
                        if (r >= 0) {
                            at[j] = roff[slot];
                            neg[j] = r >> 8;
                            if (U.core0 >= 0) {   // pn: the column of core + l, and the sign of a+_l on the core
                                const int l = r & 255;
                                const int p = __ldg(A.colpos + (size_t)l * A.ncn + U.core0 + col);
                                neg[j] = neg[j] != (bool)(__ldg(A.nsign + U.core0 + col) >> l & 1u);
                                at[j] = p == 0xFFFF ? -1 : at[j] + p;
                            } else {
                                at[j] += (int64_t)col * U.stride;
                            }
                        }
                    }
                }
                alignas(16) T v[NB][K];
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    const int slot = (n0 + j * kGramThreads) >> lg;
#pragma unroll
                    for (int q = 0; q < K; ++q) v[j][q] = T(0);
                    if (at[j] >= 0) {
                        const T *s = (slot >= na ? x : gy) + at[j] * K;
                        if constexpr (E >= 16) {
#pragma unroll
                            for (int q = 0; q < K; q += 16 / (int)sizeof(T))
                                *reinterpret_cast<int4 *>(v[j] + q) = __ldg(reinterpret_cast<const int4 *>(s + q));
                        } else {
#pragma unroll
                            for (int q = 0; q < K; ++q) v[j][q] = __ldg(s + q);
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    const int n = n0 + j * kGramThreads, slot = n >> lg, c = n & (CH - 1);
                    if (n >= total) continue;
#pragma unroll
                    for (int q = 0; q < K; ++q) v[j][q] = neg[j] ? -v[j][q] : v[j][q];
                    gput<T, K>(tiles + slot * LD + c * K, v[j]);
                }
            }
            __syncthreads();
            const int cn = min(CH, U.ncol - c0);
            if (slice < S) {
                for (int cb = slice; cb < cn; cb += 8 * S) {
                    const int ce = min(cn, cb + 8 * S);
                    for (int c = cb; c < ce; c += S, ++n) {
                        alignas(16) T a[4][K], b[RB][K];
#pragma unroll
                        for (int p = 0; p < 4; ++p) gget<T, K>(sg + (ia + ga * p) * LD + c * K, a[p]);
#pragma unroll
                        for (int q = 0; q < RB; ++q) gget<T, K>(sx + (ib + gb * q) * LD + c * K, b[q]);
#pragma unroll
                        for (int p = 0; p < 2; ++p)
#pragma unroll
                            for (int q = 0; q < RB; ++q) {
                                if constexpr (K == 1) {
                                    acc[p][q].add_prod(a[2 * p][0], a[2 * p + 1][0], b[q][0]);
                                } else {
                                    T f0 = a[2 * p][0] * b[q][0], f1 = a[2 * p + 1][0] * b[q][0];
#pragma unroll
                                    for (int k = 1; k < K; ++k) {
                                        f0 = fma(a[2 * p][k], b[q][k], f0);
                                        f1 = fma(a[2 * p + 1][k], b[q][k], f1);
                                    }
                                    acc[p][q].add(f0, f1);
                                }
                            }
                    }
                    if (n >= 8) {   // (not tested column by column: that costs 45 us of 48Cr k = 4)
                        n = 0;
#pragma unroll
                        for (int p = 0; p < 2; ++p)
#pragma unroll
                            for (int q = 0; q < RB; ++q) acc[p][q].normalize();
                    }
                }
            }
        }
        // slices meet in the tiles' place, [pair of the thread][slice][thread], and are added in order
        using Part = typename GramSum<T>::Part;
        Part *part = reinterpret_cast<Part *>(tiles);
        static_assert(sizeof(Part) * 16 * kGramThreads <= sizeof(T) * gram_tile_elems<T, K>(), "slices' sums do not fit");
        if (S > 1) {
            __syncthreads();
            if (slice < S) {
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int q = 0; q < RB; ++q) part[(p * RB + q) * kGramThreads + tid] = acc[p / 2][q].part(p & 1);
            }
            __syncthreads();
            for (int n = tid; n < 4 * RB * nt; n += kGramThreads) {
                const int pq = n / nt, th = n % nt;
                const int a = th % ga + ga * (pq / RB), b = th / ga + gb * (pq % RB);
                if (a >= U.na || b >= U.nb) continue;
                Part v = part[pq * kGramThreads + th];
                if constexpr (std::is_same<T, double>::value) {
                    for (int sl = 1; sl < S; ++sl) v += part[pq * kGramThreads + sl * nt + th];
                } else {
                    for (int s0 = 1; s0 < S; s0 += 8) {   // eight loads under way (one by one: 130 us more at 48Cr k = 4)
                        Part w[8];
#pragma unroll
                        for (int h = 0; h < 8; ++h) w[h] = s0 + h < S ? part[pq * kGramThreads + (s0 + h) * nt + th] : Part{};
#pragma unroll
                        for (int h = 0; h < 8; ++h) v = GramSum<T>::join(v, w[h]);
                        v = GramSum<T>::normal(v);
                    }
                }
                mat[rp[na + b] * kGramTile + rp[a]] += GramSum<T>::value(v);
            }
        } else if (slice < S) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < RB; ++q) {
                    const int a = ia + ga * p, b = ib + gb * q;
                    if (a < U.na && b < U.nb) mat[rp[na + b] * kGramTile + rp[a]] += GramSum<T>::value(acc[p / 2][q].part(p & 1));
                }
        }
        __syncthreads();   // tiles, records and sums are free for the next unit
    };
    leave();   // zeros
    __syncthreads();
    for (int batch = blockIdx.x; batch < A.nbatch;) {
        for (int u = A.range[batch]; u < A.range[batch + 1]; ++u) {
            const GramUnit U = A.units[u];
            if (U.tile != out) {
                leave();
                out = U.tile;
                out_at = U.out;
                np = U.np;
                ta = U.ta;
                tb = U.tb;
                __syncthreads();
            }
            // 4 x 4 or 4 x 3 pairs a thread: the less work per thread and column
            const int ga = (U.na + 3) / 4, t4 = ga * ((U.nb + 3) / 4), t3 = ga * ((U.nb + 2) / 3);
            const int s4 = kGramThreads / t4, s3 = t3 <= kGramThreads ? kGramThreads / t3 : 0;
            if (s3 > 0 && 3 * s4 <= 4 * s3 && 3 * ((U.ncol + s3 - 1) / s3) < 4 * ((U.ncol + s4 - 1) / s4)) unit(U, std::integral_constant<int, 3>{});
            else unit(U, std::integral_constant<int, 4>{});
        }
        // the next batch: a counter shared by the CTAs
        if (tid == 0) claim = (int)gridDim.x + atomicAdd(A.next, 1);
        __syncthreads();
        batch = claim;
        __syncthreads();
    }
    leave();
}

// Overlaps per SD: pd[g] = gy . x over the other species' SDs of proton SD g, one warp each.
template <typename T, int K>
__global__ void adj_pdiag(const RowTask *tasks, int n, const DevBlock *blocks, const T *__restrict__ x, const T *__restrict__ gy,
                          double *__restrict__ pd)
{
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (w >= n) return;
    const RowTask t = tasks[w];
    const DevBlock D = blocks[t.block];
    const int64_t base = (D.off + (int64_t)t.row * D.nN) * K;
    double s = 0.0;
    for (int c = lane; c < D.nN; c += 32) s += dotk<T, K>(gy + base + (int64_t)c * K, x + base + (int64_t)c * K);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) pd[D.p_start + t.row] = s;
}

// nd[g] likewise for neutron SDs: a CTA takes 128 columns and 32 rows of a block.
constexpr int kNdRows = 32;
template <typename T, int K>
__global__ void adj_ndiag(const int4 *tasks, const DevBlock *blocks, const T *__restrict__ x, const T *__restrict__ gy,
                          double *__restrict__ nd)
{
    const int4 t = tasks[blockIdx.x];   // block, first row, first column
    const DevBlock D = blocks[t.x];
    const int c = t.z + (int)threadIdx.x;
    if (c >= D.nN) return;
    double s = 0.0;
    for (int r = t.y; r < min(D.nP, t.y + kNdRows); ++r) {
        const int64_t at = (D.off + (int64_t)r * D.nN + c) * K;
        s += dotk<T, K>(gy + at, x + at);
    }
    atomicAdd(nd + D.n_start + c, s);
}

template <typename T, int K>
cudaError_t launch_gram(bs_ctx *c, const T *x, const T *gy, cudaStream_t s)
{
    const AdjPlan &P = c->adj;
    const Device &D = c->dev;
    GramArgs A{P.units, P.rows, P.range, P.nbatch, reinterpret_cast<int *>(P.out + P.nout), P.colpos, P.nsign, P.ncn};
    if (P.nbatch > 0) {
        constexpr size_t smem = gram_smem<T, K>();
        const cudaError_t e = cudaFuncSetAttribute(adj_gram<T, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        adj_gram<T, K><<<std::min(P.nbatch, P.nctas), kGramThreads, smem, s>>>(A, x, gy, P.out);
    }
    adj_pdiag<T, K><<<(D.nrtasks + 3) / 4, 128, 0, s>>>(D.rtasks, D.nrtasks, D.blocks, x, gy, P.out + P.pd);
    if (P.nnd > 0) adj_ndiag<T, K><<<P.nnd, 128, 0, s>>>(P.ndtasks, D.blocks, x, gy, P.out + P.nd);
    return cudaGetLastError();
}

// (N-2)-cores of one species: for every pair key the pairs each core leaves free, with the SD they lead to.
struct Core2 {
    uint64_t bits;
    std::vector<std::pair<int, int64_t>> at;   // position in the key's pair list, global SD
    int key;
};

void core2_lists(const Basis &B, const Interaction &I, int spc, std::vector<Core2> &out)
{
    const Species &S = B.sp[spc];
    const int ns = (int)B.st.size();
    if (S.nparticles < 2) return;
    std::vector<uint64_t> cores;
    for (uint64_t r : S.bits)
        for (int a = 0; a < ns; ++a)
            if (r >> a & 1)
                for (int b = a + 1; b < ns; ++b)
                    if (r >> b & 1) cores.push_back(r & ~(1ULL << a) & ~(1ULL << b));
    std::sort(cores.begin(), cores.end());
    cores.erase(std::unique(cores.begin(), cores.end()), cores.end());
    for (size_t key = 0; key < I.pairs_by_key.size(); ++key)
        for (uint64_t c : cores) {
            Core2 q{c, {}, (int)key};
            const std::vector<int> &v = I.pairs_by_key[key];
            for (size_t t = 0; t < v.size(); ++t) {
                const uint64_t m = (1ULL << I.pair_i[(size_t)v[t]]) | (1ULL << I.pair_j[(size_t)v[t]]);
                if (c & m) continue;
                auto it = S.index.find(c | m);
                if (it != S.index.end()) q.at.push_back({(int)t, it->second});
            }
            if (!q.at.empty()) out.push_back(std::move(q));
        }
}

template <typename V>
cudaError_t put_plan(AdjPlan &P, V *&d, const std::vector<V> &h)
{
    cudaError_t e = cudaMalloc((void **)&d, std::max<size_t>(1, h.size()) * sizeof(V));
    if (e != cudaSuccess) return e;
    P.owned.push_back(d);
    return h.empty() ? cudaSuccess : cudaMemcpy(d, h.data(), h.size() * sizeof(V), cudaMemcpyHostToDevice);
}

// No plan: for want of memory the kernels by jumps run until the next load.
int plan_failed(bs_ctx *c, cudaError_t e)
{
    (void)cudaGetLastError();
    release_adj(c->adj);
    c->adj.tried = true;
    if (e == cudaErrorMemoryAllocation) return BS_OK;
    c->err = std::string("adjoint tables: ") + cudaGetErrorString(e);
    return BS_ECUDA;
}

// Units of the Gram matrices, once per loaded interaction; P.on stays false (with no error) where they do not apply.
int build_plan(bs_ctx *c)
{
    AdjPlan &P = c->adj;
    const Basis &B = c->basis;
    const Interaction &I = c->inter;
    PairTables own;   // spaces too wide for the pair-core product have no tables of it yet
    P.tried = true;
    const int ns = (int)B.st.size();
    if (B.trunc || ns > 32 || B.dim >= (int64_t)1 << 31) return BS_OK;
    if (!c->tab.pair.on && B.Z > 0 && B.N > 0) build_pair_tables(B, I, own, -1);
    const PairTables &R = c->tab.pair.on ? c->tab.pair : own;
    if (!R.on && B.Z > 0 && B.N > 0) return BS_OK;
    cudaError_t e;
    P.ncn = R.ncn;
    if ((e = put_plan(P, P.colpos, R.colpos)) != cudaSuccess || (e = put_plan(P, P.nsign, R.nsign)) != cudaSuccess) {
        return plan_failed(c, e);
    }
    struct U { GramUnit u; double cost; };
    std::vector<U> units;
    std::vector<GramRow> rows;
    std::map<std::pair<int64_t, int>, int> tile_of;
    // one unit per pair of 64-pair tiles; [r0, r0 + n) the records, positions ascending
    auto add = [&](int64_t out, int np, int r0, int n, int ncol, int64_t stride, int core0) {
        for (int ja = 0; ja < np; ja += kGramTile)
            for (int jb = 0; jb < np; jb += kGramTile) {
                GramUnit u = {};
                u.out = out + (int64_t)jb * np + ja;
                u.np = np;
                u.pa = ja;
                u.pb = jb;
                u.ta = std::min(kGramTile, np - ja);
                u.tb = std::min(kGramTile, np - jb);
                u.a0 = u.b0 = -1;
                for (int r = r0; r < r0 + n; ++r) {
                    const int p = rows[(size_t)r].pos;
                    if (p >= ja && p < ja + u.ta) { if (u.a0 < 0) u.a0 = r; ++u.na; }
                    if (p >= jb && p < jb + u.tb) { if (u.b0 < 0) u.b0 = r; ++u.nb; }
                }
                if (!u.na || !u.nb) continue;
                u.ncol = ncol;
                u.stride = stride;
                u.core0 = core0;
                u.tile = tile_of.emplace(std::make_pair(u.out, np), (int)tile_of.size()).first->second;
                // in cycles: a unit's and 2048 staged elements' latency, per column of a thread 16 sums
                const int cols = 2048 / ((u.na + 3) / 4 * 4 + (u.nb + 3) / 4 * 4), slices = 256 / (((u.na + 3) / 4) * ((u.nb + 3) / 4));
                units.push_back(U{u, 1500.0 * (1 + (ncol + cols - 1) / cols) + 376.0 * ((ncol + slices - 1) / slices)});
            }
    };
    int64_t nout = 0;
    // pn: the matrices of the pair tables
    P.pn_size = B.Z > 0 && B.N > 0 ? (int64_t)R.w.size() : 0;
    nout = P.pn_size;
    if (P.pn_size)
        for (const PairCore &pc : R.cores)
            for (int g = 0; g < pc.ngrp; ++g) {
                const PairGroup &G = R.grps[(size_t)(pc.grp0 + g)];
                const int r0 = (int)rows.size();
                for (int r = 0; r < G.nrec; ++r) {
                    const PairRec &q = R.recs[(size_t)(pc.rec0 + G.rec0 + r)];
                    rows.push_back(GramRow{(int64_t)q.xoff, (int)(q.wj & 0xFFFFu), (uint8_t)(q.wj >> 16 & 255u), (uint8_t)(q.srec >> 31), 0});
                }
                add(G.woff, G.np, r0, G.nrec, G.ncore, 1, G.core0);
            }
    // like particles: pair-key matrices shared by both species
    P.like_off.clear();
    for (const std::vector<int> &v : I.pairs_by_key) {
        P.like_off.push_back(nout);
        nout += (int64_t)v.size() * (int64_t)v.size();
    }
    for (int spc = 0; spc < 2; ++spc) {
        const Species &S = B.sp[spc];
        std::vector<Core2> cores;
        core2_lists(B, I, spc, cores);
        for (const Core2 &q : cores) {
            const int sec = S.sec_of_sd[(size_t)q.at[0].second];   // all of a core's SDs for one key share it
            int blk = -1;
            if (spc == 0) blk = B.block_of_psec[(size_t)sec];
            else
                for (size_t b = 0; b < B.blocks.size(); ++b)
                    if (B.blocks[b].ns == sec) blk = (int)b;
            if (blk < 0) continue;
            const Block &K = B.blocks[(size_t)blk];
            const std::vector<int> &v = I.pairs_by_key[(size_t)q.key];
            const int r0 = (int)rows.size();
            for (const auto &e : q.at) {
                const int k = I.pair_i[(size_t)v[(size_t)e.first]], l = I.pair_j[(size_t)v[(size_t)e.first]];
                const uint64_t m = S.bits[(size_t)e.second];
                const bool neg = (sgn_below(m, k) < 0) != (sgn_below(m & ~(1ULL << k), l) < 0);
                const int64_t loc = e.second - S.sec[(size_t)sec].start;
                rows.push_back(GramRow{K.off + loc * (spc == 0 ? K.nN : 1), e.first, 0, (uint8_t)neg, 0});
            }
            add(P.like_off[(size_t)q.key], (int)v.size(), r0, (int)q.at.size(), (int)(spc == 0 ? K.nN : K.nP), spc == 0 ? 1 : K.nN, -1);
        }
    }
    P.pd = nout;
    nout += (int64_t)B.sp[0].bits.size();
    P.nd = nout;
    nout += (int64_t)B.sp[1].bits.size();
    P.nout = nout;
    // by matrix, then in batches of about equal cost, eight for each CTA (two per SM)
    std::stable_sort(units.begin(), units.end(), [](const U &a, const U &b) { return a.u.tile < b.u.tile; });
    int nsm = 152;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) (void)cudaGetLastError();
    double total = 0.0;
    for (const U &u : units) total += u.cost;
    P.nctas = nsm * 2;
    const int parts = (int)std::min<size_t>((size_t)P.nctas * 8, units.size());
    std::vector<int> range(1, 0);
    std::vector<GramUnit> gu;
    double run = 0.0;
    for (const U &u : units) {
        if (!gu.empty() && (int)range.size() < parts && run + 0.5 * u.cost >= total * (double)range.size() / parts) range.push_back((int)gu.size());
        run += u.cost;
        gu.push_back(u.u);
    }
    range.push_back((int)gu.size());
    P.nbatch = gu.empty() ? 0 : (int)range.size() - 1;
    std::vector<int4> nt;
    for (size_t b = 0; b < B.blocks.size(); ++b)
        for (int64_t r = 0; r < B.blocks[b].nP; r += kNdRows)
            for (int64_t q = 0; q < B.blocks[b].nN; q += 128) nt.push_back(make_int4((int)b, (int)r, (int)q, 0));
    P.nnd = (int)nt.size();
    // where every pn density belongs in the W_pn layout
    P.pn_to_w.assign((size_t)P.pn_size, -1);
    if (P.pn_size) {
        std::map<std::pair<int, int>, std::vector<std::pair<int, int>>> pairs;
        for (int i = 0; i < ns; ++i)
            for (int j = 0; j < ns; ++j)
                pairs[{B.st[(size_t)i].twom + B.st[(size_t)j].twom, B.st[(size_t)i].par ^ B.st[(size_t)j].par}].push_back({i, j});
        int64_t w = 0;   // the matrices in the order of the keys, as build_pair_tables lays them out
        for (const auto &kv : pairs)
            for (const auto &kl : kv.second)
                for (const auto &ij : kv.second) {
                    const int op = ij.first * ns + kl.first, on = ij.second * ns + kl.second;
                    const int g = I.ops.group_of_op[(size_t)op], h = g < 0 ? -1 : I.conj_group[(size_t)g];
                    if (h >= 0 && I.ops.group_of_op[(size_t)on] == h)
                        P.pn_to_w[(size_t)w] = I.wpn_off[(size_t)g] + (int64_t)I.ops.local_of_op[(size_t)op] * (int64_t)I.ops.ops[(size_t)h].size() +
                                               I.ops.local_of_op[(size_t)on];
                    ++w;
                }
    }
    if ((e = put_plan(P, P.units, gu)) != cudaSuccess || (e = put_plan(P, P.rows, rows)) != cudaSuccess ||
        (e = put_plan(P, P.range, range)) != cudaSuccess || (e = put_plan(P, P.ndtasks, nt)) != cudaSuccess ||
        (e = put_plan(P, P.out, std::vector<double>((size_t)nout + 1, 0.0))) != cudaSuccess ||
        (e = cudaMallocHost((void **)&P.host, (size_t)nout * sizeof(double))) != cudaSuccess) {
        return plan_failed(c, e);
    }
    P.on = true;
    return BS_OK;
}

// gtheta from the Gram matrices; nothing is added where they are not all finite
int gram_backward(bs_ctx *c, const void *x, const void *gy, double *gtheta, int k, bs_dtype dt, cudaStream_t s, bool &finite)
{
    AdjPlan &P = c->adj;
    const Interaction &I = c->inter;
    const Basis &B = c->basis;
    cudaError_t e = cudaMemsetAsync(P.out, 0, (size_t)(P.nout + 1) * sizeof(double), s);
    if (e == cudaSuccess) {
        if (dt == BS_F64) {
            const double *xi = (const double *)x, *gi = (const double *)gy;
            e = k == 1 ? launch_gram<double, 1>(c, xi, gi, s) : k == 2 ? launch_gram<double, 2>(c, xi, gi, s)
              : k == 4 ? launch_gram<double, 4>(c, xi, gi, s) : launch_gram<double, 8>(c, xi, gi, s);
        } else {
            const float *xi = (const float *)x, *gi = (const float *)gy;
            e = k == 1 ? launch_gram<float, 1>(c, xi, gi, s) : k == 2 ? launch_gram<float, 2>(c, xi, gi, s)
              : k == 4 ? launch_gram<float, 4>(c, xi, gi, s) : launch_gram<float, 8>(c, xi, gi, s);
        }
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(P.host, P.out, (size_t)P.nout * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        c->err = std::string("adjoint: ") + cudaGetErrorString(e);
        return BS_ECUDA;
    }
    finite = std::all_of(P.host, P.host + P.nout, [](double v) { return std::isfinite(v); });
    if (!finite) return BS_OK;
    const int ns = (int)B.st.size(), no = (int)c->spe_in.size();
    std::vector<double> n1((size_t)ns, 0.0);
    for (int spc = 0; spc < 2; ++spc) {
        const double *d = P.host + (spc == 0 ? P.pd : P.nd);
        for (size_t g = 0; g < B.sp[spc].bits.size(); ++g)
            for (uint64_t m = B.sp[spc].bits[g]; m; m &= m - 1) n1[(size_t)__builtin_ctzll(m)] += d[g];
    }
    for (int st = 0; st < ns; ++st) gtheta[B.st[(size_t)st].orb] += n1[(size_t)st];
    std::vector<double> rho2((size_t)I.npairs * I.npairs, 0.0), rho(I.Wpn.size(), 0.0);
    for (size_t key = 0; key < I.pairs_by_key.size(); ++key) {
        const std::vector<int> &v = I.pairs_by_key[key];
        const double *m = P.host + P.like_off[key];
        for (size_t b = 0; b < v.size(); ++b)   // row kl, column ij
            for (size_t a = 0; a < v.size(); ++a) rho2[(size_t)v[a] * I.npairs + (size_t)v[b]] = m[b * v.size() + a];
    }
    for (int64_t i = 0; i < P.pn_size; ++i)
        if (P.pn_to_w[(size_t)i] >= 0) rho[(size_t)P.pn_to_w[(size_t)i]] = P.host[i];
    for (const WTerm &t : c->dWpp) gtheta[no + t.t] += rho2[(size_t)t.at] * t.c;
    for (const WTerm &t : c->dWpn) gtheta[no + t.t] += rho[(size_t)t.at] * t.c;
    return BS_OK;
}

}  // namespace

void release_adj(AdjPlan &P)
{
    for (void *p : P.owned) cudaFree(p);
    if (P.host) cudaFreeHost(P.host);
    P = AdjPlan();
}

int run_backward(bs_ctx *c, const void *x, const void *gy, void *gx, double *gtheta, int k, bs_dtype dt,
                 void *stream)
{
    cudaStream_t s = (cudaStream_t)stream;
    int rc = launch_hx(c, gy, gx, k, dt, stream, c->err);   // gx = H gy (H symmetric)
    if (rc || !gtheta) return rc;
    if (!c->have_dW) {
        build_interaction_derivatives(c->basis, c->inter, c->tbme_in, c->dWpp, c->dWpn);
        c->have_dW = true;
    }
    if (!c->adj.tried) {
        try {
            rc = build_plan(c);
        } catch (const std::bad_alloc &) {
            rc = plan_failed(c, cudaErrorMemoryAllocation);
        }
        if (rc) return rc;
    }
    if (c->adj.on) {
        // A sum of FP32 products beyond 3.4e38 leaves double-float's range, and an infinite element meets the zeros that
        // stand for occupied states: such vectors take the kernels by jumps, whose sums are FP64 over the jumps alone.
        bool finite = false;
        rc = gram_backward(c, x, gy, gtheta, k, dt, s, finite);
        if (rc || finite) return rc;
    }
    const Tables &T = c->tab;
    const Interaction &I = c->inter;
    cudaError_t e;
    // The products' lists hold no move whose matrix element is zero; its density counts all the same.
    if (!c->adj_gpp) {
        bool zeros = false;
        for (const std::vector<int> &v : I.pairs_by_key)
            for (int p : v)
                for (int q : v) zeros = zeros || I.Wpp[(size_t)p * I.npairs + q] == 0.0;
        for (int spc = 0; zeros && spc < 2; ++spc) {
            AdjPlan::Moves &m = c->adj.moves[spc];
            like_moves(c->basis, I, spc, m.list);
            if ((e = put_plan(c->adj, m.ptr, m.list.ptr)) != cudaSuccess || (e = put_plan(c->adj, m.src, m.list.src)) != cudaSuccess) {
                (void)cudaGetLastError();
                c->err = std::string("adjoint: ") + cudaGetErrorString(e);
                return e == cudaErrorMemoryAllocation ? BS_ENOMEM : BS_ECUDA;
            }
        }
        c->adj.have_moves = zeros;
    }
    const LikeJumps &pp = c->adj.have_moves ? c->adj.moves[0].list : T.pp, &nn = c->adj.have_moves ? c->adj.moves[1].list : T.nn;
    if (!c->adj_gpp) {
        if ((e = cudaMalloc(&c->adj_gpp, std::max<size_t>(1, pp.src.size()) * sizeof(double))) != cudaSuccess ||
            (e = cudaMalloc(&c->adj_gnn, std::max<size_t>(1, nn.src.size()) * sizeof(double))) != cudaSuccess ||
            (e = cudaMalloc(&c->adj_rho, std::max<size_t>(1, I.Wpn.size()) * sizeof(double))) != cudaSuccess) {
            c->err = std::string("adjoint: ") + cudaGetErrorString(e);
            (void)cudaGetLastError();
            cudaFree(c->adj_gpp);   // all or none
            cudaFree(c->adj_gnn);
            c->adj_gpp = c->adj_gnn = c->adj_rho = nullptr;
            return BS_ENOMEM;
        }
    }
    cudaMemsetAsync(c->adj_gpp, 0, std::max<size_t>(1, pp.src.size()) * sizeof(double), s);
    cudaMemsetAsync(c->adj_gnn, 0, std::max<size_t>(1, nn.src.size()) * sizeof(double), s);
    cudaMemsetAsync(c->adj_rho, 0, std::max<size_t>(1, I.Wpn.size()) * sizeof(double), s);
    // one CTA per (block, neutron column) for the nn densities
    std::vector<int> cb, cl;
    for (size_t b = 0; b < c->basis.blocks.size(); ++b)
        for (int64_t j = 0; j < c->basis.blocks[b].nN; ++j) { cb.push_back((int)b); cl.push_back((int)j); }
    if (dt == BS_F64) {
        const double *xi = (const double *)x, *gi = (const double *)gy;
        switch (k) {
        case 1: rc = launch_adj<double, 1>(c, xi, gi, s, cb, cl); break;
        case 2: rc = launch_adj<double, 2>(c, xi, gi, s, cb, cl); break;
        case 4: rc = launch_adj<double, 4>(c, xi, gi, s, cb, cl); break;
        default: rc = launch_adj<double, 8>(c, xi, gi, s, cb, cl); break;
        }
    } else {
        const float *xi = (const float *)x, *gi = (const float *)gy;
        switch (k) {
        case 1: rc = launch_adj<float, 1>(c, xi, gi, s, cb, cl); break;
        case 2: rc = launch_adj<float, 2>(c, xi, gi, s, cb, cl); break;
        case 4: rc = launch_adj<float, 4>(c, xi, gi, s, cb, cl); break;
        default: rc = launch_adj<float, 8>(c, xi, gi, s, cb, cl); break;
        }
    }
    if (rc) return rc;
    std::vector<double> gpp(pp.src.size()), gnn(nn.src.size()), rho(I.Wpn.size());
    cudaMemcpyAsync(gpp.data(), c->adj_gpp, gpp.size() * sizeof(double), cudaMemcpyDeviceToHost, s);
    cudaMemcpyAsync(gnn.data(), c->adj_gnn, gnn.size() * sizeof(double), cudaMemcpyDeviceToHost, s);
    cudaMemcpyAsync(rho.data(), c->adj_rho, rho.size() * sizeof(double), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) {
        c->err = std::string("adjoint: ") + cudaGetErrorString(e);
        return BS_ECUDA;
    }
    const int ns = (int)c->basis.st.size();
    std::vector<double> rho2((size_t)I.npairs * I.npairs, 0.0), rho1p(ns, 0.0), rho1n(ns, 0.0);
    split_like(c->basis, I, 0, pp, gpp, rho2, rho1p);
    split_like(c->basis, I, 1, nn, gnn, rho2, rho1n);
    const int no = (int)c->spe_in.size();
    for (int st = 0; st < ns; ++st) gtheta[c->basis.st[(size_t)st].orb] += rho1p[st] + rho1n[st];
    for (const WTerm &t : c->dWpp) gtheta[no + t.t] += rho2[(size_t)t.at] * t.c;
    for (const WTerm &t : c->dWpn) gtheta[no + t.t] += rho[(size_t)t.at] * t.c;
    return BS_OK;
}

}  // namespace bs
