// pn term of y = H x by pairs of cores (sm_103a): for one proton core cp and
// one group of neutron cores cn of equal (2M, parity),
//   G[ij][cn] = sum_kl W[ij][kl] X[kl][cn],  X[kl][cn] = sign x[cp+k, cn+l],
// a dense matrix product with one W for all of them (bs_pair.cpp), whose
// result is added to the rows cp + i of y at column cn + j.  Against the
// (Z-1)-core kernel, which gathers an element of x once per neutron jump for
// at most four rows, an element is gathered once per (proton, neutron)
// particle pair it holds and feeds every pair ij: 14 times fewer gathers at
// pf 4p4n.  What bounds it is instruction issue (at k = 2 half the slots busy;
// a sixth of the instructions are the packed multiply-adds, the others signs,
// weights, stage hand-overs and the adds to y).  pf 4p4n, pn term: 0.46, 0.54,
// 0.75, 1.46 ms at k = 1, 2, 4, 8; the row kernel's whole product took 1.78
// and 2.14 ms at k = 1, 2 (0.58 and 0.72 now), the (Z-1)-core kernel takes
// 0.84 and 1.03 ms at k = 4, 8, so k = 8 stays there.  The price is the
// multiply-adds with states the neutron core occupies (their x is zero):
// ((ns - N + 1) / ns)^2 of them are of use, 0.72 at pf 4p4n.
//
// One CTA per SM and item: a proton core with all its rows and CP of the K
// components.  The item's output rows Y live in shared memory.  Four producer warps gather X (cp.async, zeros for occupied
// states) and W into a ring of stages of KC pairs kl; sixteen consumer warps
// in four groups share it: group g owns the rows of a fixed subset of the
// proton states i, its warp w the cores 32 w .. 32 w + 31, one core per lane,
// with up to 16 rows x CP components of G in registers.  A finished tile is
// added to the group's own rows of Y, so groups never touch the same element
// and one group's adds run under the others' multiply-adds.  Inside a group
// the adds go in rounds: rows whose neutron state j has the same place among
// the states of its (2m, parity) meet a column once, so no two threads add
// to one element in a round.  No atomics, a fixed order of additions.  Waits
// are bounded: on expiry the CTA records BS_ETIMEOUT, stops waiting and runs
// to its end (its rows are then garbage, as the status says).
#include <cuda_runtime.h>

#include <algorithm>

#include "bs_internal.h"
#include "bs_tma.cuh"

namespace bs {

using namespace tma;

namespace {

constexpr int kCons = 512, kProd = 128;   // threads: one producer warp and four consumer warps on each scheduler
// registers a thread: 640 x 96 at launch = 512 x 112 + 128 x 32
constexpr int kConsRegs = 112, kProdRegs = 32;
static_assert(kCons * kConsRegs + kProd * kProdRegs <= (kCons + kProd) * 96, "register split above the launch's registers");

struct PairArgs {
    const PairItem *items;
    const PairTile *tiles;
    const PairRec *recs;
    const PairRec *rows;
    const PairRow *store;
    const uint16_t *colpos;
    const uint32_t *nsign;
    const float *w;
    int *err;
    int ncn;
    int S;                // ring stages
    int cols;             // output columns held (largest item)
    int max_rec, max_rows, max_tiles;
    int64_t part_stride;
};

template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void *src, bool ok)
{
    const int n = ok ? BYTES : 0;   // 0: the destination is filled with zeros, nothing is read
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(BYTES), "r"(n) : "memory");
}
// arrives on the barrier once this thread's copies so far have landed
__device__ __forceinline__ void cp_arrive(uint32_t bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_group(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }

__device__ __forceinline__ float sgn(float v, uint32_t s) { return __uint_as_float(__float_as_uint(v) ^ s); }

// Stage geometry: KC pairs kl, X [KC][128][CP] then W [KC][4 groups x 16 rows].
template <int CP>
struct Geo {
    static constexpr int KC = CP == 4 ? 4 : 8;
    static constexpr int XW = kPairCores * CP, WW = 4 * kPairRows;
    static constexpr int floats = KC * (XW + WW);
};

// CP components of an output column: read into (or, PUT, written from) o.
template <int CP, bool PUT>
__device__ __forceinline__ void ycol(float *y, float (&o)[CP])
{
    if constexpr (CP == 4) {
        if constexpr (PUT) {
            *reinterpret_cast<float4 *>(y) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
            const float4 v = *reinterpret_cast<const float4 *>(y);
            o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
        }
    } else if constexpr (CP == 2) {
        if constexpr (PUT) {
            *reinterpret_cast<float2 *>(y) = make_float2(o[0], o[1]);
        } else {
            const float2 v = *reinterpret_cast<const float2 *>(y);
            o[0] = v.x; o[1] = v.y;
        }
    } else {
        if constexpr (PUT) *y = o[0];
        else o[0] = *y;
    }
}

// One tile of a consumer warp: TR rows (an even number, >= the group's rows).
template <int CP, int TR>
__device__ __forceinline__ void pair_tile(const PairArgs &A, const PairTile &T, const PairRec *recs, const PairRec *rows,
                                          float *Y, const float *ring, uint32_t full0, uint32_t empty0, int &slot,
                                          uint32_t &phase, bool &dead, int grp, int cg, int lane)
{
    using G = Geo<CP>;
    const int core = cg * 32 + lane;
    const bool live = cg * 32 < T.ncore;   // warp-uniform
    const uint32_t mask = core < T.ncore ? __ldg(A.nsign + T.core0 + core) : 0u;
    float2 acc[TR / 2][CP];
#pragma unroll
    for (int p = 0; p < TR / 2; ++p)
#pragma unroll
        for (int c = 0; c < CP; ++c) acc[p][c] = make_float2(0.0f, 0.0f);
    const int nrec = T.nrec;
    const PairRec *kr = recs + T.rec0;
    for (int k0 = 0; k0 < nrec; k0 += G::KC, kr += G::KC) {
        if (!dead && __any_sync(0xffffffffu, bar_wait(full0 + 8u * slot, phase))) dead = true;
        if (live) {
            const float *X = ring + (size_t)slot * G::floats + core * CP;
            const float *W = ring + (size_t)slot * G::floats + G::KC * G::XW + grp * kPairRows;
            auto step = [&](int kk) {
                const uint32_t sr = kr[kk].srec;
                const uint32_t s = ((mask << (sr & 31u)) ^ sr) & 0x80000000u;
                float xs[CP];
                if constexpr (CP == 4) {
                    const float4 q = *reinterpret_cast<const float4 *>(X + kk * G::XW);
                    xs[0] = q.x; xs[1] = q.y; xs[2] = q.z; xs[3] = q.w;
                } else if constexpr (CP == 2) {
                    const float2 q = *reinterpret_cast<const float2 *>(X + kk * G::XW);
                    xs[0] = q.x; xs[1] = q.y;
                } else {
                    xs[0] = X[kk * G::XW];
                }
#pragma unroll
                for (int c = 0; c < CP; ++c) xs[c] = sgn(xs[c], s);
                float w[TR];
#pragma unroll
                for (int p = 0; p + 4 <= TR; p += 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(W + kk * G::WW + p);
                    w[p] = v.x; w[p + 1] = v.y; w[p + 2] = v.z; w[p + 3] = v.w;
                }
                if constexpr (TR % 4 == 2) {
                    const float2 v = *reinterpret_cast<const float2 *>(W + kk * G::WW + TR - 2);
                    w[TR - 2] = v.x; w[TR - 1] = v.y;
                }
                // packed by rows: two fused multiply-adds per instruction, the weights as loaded
#pragma unroll
                for (int p = 0; p < TR / 2; ++p)
#pragma unroll
                    for (int c = 0; c < CP; ++c)
                        acc[p][c] = __ffma2_rn(make_float2(w[2 * p], w[2 * p + 1]), make_float2(xs[c], xs[c]), acc[p][c]);
            };
            if (k0 + G::KC <= nrec) {
#pragma unroll 2
                for (int kk = 0; kk < G::KC; ++kk) step(kk);
            } else {
                for (int kk = 0; kk < nrec - k0; ++kk) step(kk);
            }
        }
        __syncwarp();
        if (lane == 0) bar_arrive(empty0 + 8u * slot);
        if (++slot == A.S) {
            slot = 0;
            phase ^= 1u;
        }
    }
    // add to Y: the rows are in the order of their rounds, a round's first row waits for the
    // group's other warps (the first of all: for their last tile)
    const int n = T.nrow[grp];
    const uint32_t first = T.first[grp];
    if (!live) {
        for (int b = __popc(first); b > 0; --b) bar_group(1 + grp);
        return;
    }
    const PairRec *rr = rows + T.row0[grp];
    const uint16_t *cp = A.colpos + T.core0 + core;
    // columns, fetched eight rows ahead
    constexpr int AH = 8;
    uint32_t at[TR];
    auto fetch = [&](int r) {
        at[r] = 0xFFFFu;
        if (r < n && core < T.ncore) at[r] = __ldg(cp + ((rr[r].wj >> 16) & 255u) * (uint32_t)A.ncn);
    };
#pragma unroll
    for (int r = 0; r < (TR < AH ? TR : AH); ++r) fetch(r);
#pragma unroll
    for (int r = 0; r < TR; ++r) {
        if (r + AH < TR) fetch(r + AH);
        if (first >> r & 1u) bar_group(1 + grp);
        if (r < n && at[r] != 0xFFFFu) {
            float *y = Y + (rr[r].yoff + at[r]) * CP;
            const uint32_t sg = (mask << (rr[r].srec & 31u)) & 0x80000000u;
            float o[CP];
            ycol<CP, false>(y, o);
#pragma unroll
            for (int c = 0; c < CP; ++c) o[c] += sgn((r & 1) ? acc[r / 2][c].y : acc[r / 2][c].x, sg);
            ycol<CP, true>(y, o);
        }
    }
}

template <int CP, int K>
__global__ void __launch_bounds__(kCons + kProd, 1) hx_pair_kernel(PairArgs A, const float *__restrict__ xv, float *__restrict__ part)
{
    using G = Geo<CP>;
    extern __shared__ __align__(128) unsigned char smem[];
    float *Y = reinterpret_cast<float *>(smem);
    float *ring = Y + (((size_t)A.cols * CP + 31) / 32) * 32;
    PairRec *recs = reinterpret_cast<PairRec *>(ring + (size_t)A.S * G::floats);
    PairRec *rows = recs + A.max_rec;
    PairTile *tiles = reinterpret_cast<PairTile *>(rows + A.max_rows);
    uint64_t *bars = reinterpret_cast<uint64_t *>(tiles + A.max_tiles);
    const uint32_t full0 = su32(bars), empty0 = su32(bars + A.S);
    const int ch = (int)blockIdx.x % (K / CP);
    const PairItem it = A.items[blockIdx.x / (K / CP)];
    if (threadIdx.x == 0) {
        for (int s = 0; s < A.S; ++s) {
            bar_init(full0 + 8u * s, 32);
            bar_init(empty0 + 8u * s, kCons / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    {
        constexpr int NT = kCons + kProd;
        auto copy = [](void *d, const void *s, int n16) {
            for (int n = threadIdx.x; n < n16; n += NT) reinterpret_cast<int4 *>(d)[n] = __ldg(reinterpret_cast<const int4 *>(s) + n);
        };
        copy(recs, A.recs + it.rec0, it.nrec);
        copy(rows, A.rows + it.row0, it.nrow);
        copy(tiles, A.tiles + it.tile0, it.ntile * (int)(sizeof(PairTile) / 16));
        const int n4 = (it.cols * CP + 3) / 4;
        for (int n = threadIdx.x; n < n4; n += NT) reinterpret_cast<float4 *>(Y)[n] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp >= kCons / 32) {
        // ---------------- producers: warp pw fills every fourth stage, so that four of the
        // dependent loads (column, then element) are under way at a time
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kProdRegs));
        const int pw = warp - kCons / 32;
        const float *x = xv + ch * CP;
        int t = 0, k0 = 0, slot = pw, round = 0;
        bool dead = false;
        auto advance = [&]() {
            k0 += G::KC;
            if (k0 >= tiles[t].nrec) {
                k0 = 0;
                ++t;
            }
        };
        for (; slot >= A.S; slot -= A.S) ++round;
        for (int n = 0; n < pw && t < it.ntile; ++n) advance();
        while (t < it.ntile) {
            const PairTile &T = tiles[t];
            if (round > 0 && !dead && bar_wait(empty0 + 8u * slot, (uint32_t)(round - 1) & 1u)) {
                dead = true;
                atomicExch(A.err, BS_ETIMEOUT);
            }
            float *X = ring + (size_t)slot * G::floats;
            const int nq = (T.ncore + 31) / 32, kn = min(G::KC, T.nrec - k0);
            const PairRec *kr = recs + T.rec0 + k0;
            // X: four pairs at a time
#pragma unroll 1
            for (int h = 0; h < kn; h += 4) {
                int col[4][4];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    if (h + a >= kn) break;
                    const uint16_t *cp = A.colpos + ((kr[h + a].wj >> 16) & 255u) * (uint32_t)A.ncn + T.core0 + lane;
#pragma unroll
                    for (int q = 0; q < 4; ++q) col[a][q] = q * 32 + lane < T.ncore ? (int)__ldg(cp + q * 32) : 0xFFFF;
                }
                const uint32_t xd = su32(X + h * G::XW) + (uint32_t)(lane * 4 * CP);
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    if (h + a >= kn) break;
                    const uint32_t xo = kr[h + a].xoff;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q >= nq) break;
                        const bool ok = col[a][q] != 0xFFFF;
                        cp_async<4 * CP>(xd + (uint32_t)((a * G::XW + q * 32 * CP) * 4),
                                         x + (size_t)(ok ? xo + (uint32_t)col[a][q] : 0u) * K, ok);
                    }
                }
            }
            // W: this lane's two row slots
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int g = 2 * h + (lane >> 4), r = lane & 15;
                if (r >= T.nrow[g]) continue;
                const float *w = A.w + T.woff + (rows[T.row0[g] + r].wj & 0xFFFFu);
                const uint32_t wd = su32(X + G::KC * G::XW) + (uint32_t)(4 * (lane + 32 * h));
                for (int kk = 0; kk < kn; ++kk)
                    cp_async<4>(wd + (uint32_t)(kk * G::WW * 4), w + (kr[kk].wj & 0xFFFFu) * (uint32_t)T.np, true);
            }
            cp_arrive(full0 + 8u * slot);
            slot += 4;
            while (slot >= A.S) {
                slot -= A.S;
                ++round;
            }
            for (int n = 0; n < 4 && t < it.ntile; ++n) advance();
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else {
        // ---------------- consumers; the four warps of a group take the four column slices in an
        // order that differs by group, so that narrow tiles leave no scheduler without work
        const int grp = warp >> 2, cg = (warp + grp) & 3;
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kConsRegs));
        int slot = 0;
        uint32_t phase = 0;
        bool dead = false;
        for (int t = 0; t < it.ntile; ++t) {
            const PairTile &T = tiles[t];
#define BS_TILE(R) pair_tile<CP, R>(A, T, recs, rows, Y, ring, full0, empty0, slot, phase, dead, grp, cg, lane)
            switch ((T.nrow[grp] + 1) >> 1) {
            case 0: case 1: BS_TILE(2); break;
            case 2: BS_TILE(4); break;
            case 3: BS_TILE(6); break;
            case 4: BS_TILE(8); break;
            case 5: BS_TILE(10); break;
            case 6: BS_TILE(12); break;
            case 7: BS_TILE(14); break;
            default: BS_TILE(16); break;
            }
#undef BS_TILE
        }
        if (dead && lane == 0) atomicExch(A.err, BS_ETIMEOUT);
    }
    __syncthreads();
    // the finished rows, with the sign of a+_i on the proton core
    for (int r = warp; r < it.nstore; r += (kCons + kProd) / 32) {
        const PairRow R = A.store[it.store0 + r];
        const uint32_t s = R.sign ? 0x80000000u : 0u;
        const float *y = Y + (size_t)R.ycol * CP;
        float *o = part + (int64_t)R.part * A.part_stride + R.elem * K + ch * CP;
        for (int c = lane; c < R.n; c += 32) {
            if constexpr (CP == 4) {
                const float4 v = *reinterpret_cast<const float4 *>(y + 4 * (size_t)c);
                *reinterpret_cast<float4 *>(o + (size_t)c * K) = make_float4(sgn(v.x, s), sgn(v.y, s), sgn(v.z, s), sgn(v.w, s));
            } else if constexpr (CP == 2) {
                const float2 v = *reinterpret_cast<const float2 *>(y + 2 * (size_t)c);
                *reinterpret_cast<float2 *>(o + (size_t)c * K) = make_float2(sgn(v.x, s), sgn(v.y, s));
            } else {
                o[(size_t)c * K] = sgn(y[c], s);
            }
        }
    }
}

constexpr size_t kSmemMax = 227 * 1024;
constexpr int kMaxStages = 8, kMinStages = 3;

size_t pair_smem(int cp, int cols, int max_rec, int max_rows, int max_tiles, int S)
{
    const size_t stage = cp == 4 ? Geo<4>::floats : cp == 2 ? Geo<2>::floats : Geo<1>::floats;
    return (((size_t)cols * cp + 31) / 32) * 32 * 4 + S * stage * 4 + (size_t)(max_rec + max_rows) * sizeof(PairRec) +
           (size_t)max_tiles * sizeof(PairTile) + 16 * (size_t)S;
}

template <int CP, int K>
cudaError_t launch_pair_t(const bs_ctx *ctx, const float *x, float *part, cudaStream_t s, bool &used)
{
    const Device &D = ctx->dev;
    const Device::PairDev &P = D.pr[CP == 4 ? 0 : CP == 2 ? 1 : 2];
    int S = kMaxStages;
    while (S > kMinStages && pair_smem(CP, P.cols, P.max_rec, P.max_rows, P.max_tiles, S) > kSmemMax) --S;
    const size_t smem = pair_smem(CP, P.cols, P.max_rec, P.max_rows, P.max_tiles, S);
    used = P.nitems > 0 && smem <= kSmemMax;
    if (!used || !x) return cudaSuccess;   // x == nullptr: only whether it fits
    auto kern = hx_pair_kernel<CP, K>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // the register split counts on the launch's 96 a thread: any other build of the kernel is not run
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
    if ((used = fa.numRegs == 96) == false) return cudaSuccess;
    PairArgs A{P.items, P.tiles, D.pr_recs, P.rows, P.store, D.pr_colpos, D.pr_nsign, D.pr_w, D.err, D.pr_ncn, S,
               P.cols, P.max_rec, P.max_rows, P.max_tiles, (int64_t)ctx->basis.dim * K};
    kern<<<P.nitems * (K / CP), kCons + kProd, smem, s>>>(A, x, part);
    return cudaGetLastError();
}

}  // namespace

// Most output columns an item may have when cp components are taken at a time
// (its rows repeat at most its records; 64 tiles assumed).
int pair_cap_cols(int cp, int max_rec)
{
    const size_t fixed = pair_smem(cp, 0, max_rec, max_rec, 64, kMinStages + 1) + 256;
    return fixed >= kSmemMax ? 0 : (int)((kSmemMax - fixed) / (4 * (size_t)cp));
}

// The pn term into the partial vectors 0 .. Z - 1 (FP32, k = 1, 2, 4, 8); x == nullptr only checks whether it applies.
cudaError_t launch_hx_pair(const bs_ctx *c, const float *x, float *part, int k, cudaStream_t s, bool &used)
{
    switch (k) {
    case 1: return launch_pair_t<1, 1>(c, x, part, s, used);
    case 2: return launch_pair_t<2, 2>(c, x, part, s, used);
    case 4: return launch_pair_t<4, 4>(c, x, part, s, used);
    default: return launch_pair_t<4, 8>(c, x, part, s, used);
    }
}

}  // namespace bs
