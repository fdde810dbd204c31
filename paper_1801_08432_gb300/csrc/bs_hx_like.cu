// Like-particle terms of y = H x for k = 1, 2 (sm_103a), as two sparse
// products with uniform lists:
//   nn:  y[r, q]  = sum_s Hnn[q, s] x[r, s]   over the neutron SDs s,
//   pp:  y[r, q] += sum_s Hpp[r, s] x[s, q]   over the proton SDs s, plus the
//                                              partial vectors of the pn term.
// One species' matrix is the same for every SD of the other, so a CTA stages
// a panel of x in shared memory, all SDs of one sector of the acting
// species by 256 bytes of the other's (64 / K SDs of K components, 32 / K
// for more than 840 SDs), and a warp owns a whole output row of the panel:
// its 32 lanes hold the row's columns, so the list entry (source, coefficient)
// is the same for all lanes and the source row is read without bank
// conflicts, 2 wavefronts per 64 multiply-adds.  Shared-memory wavefronts
// bound it (3.3 per entry at pf 4p4n k = 2: 0.5 the entry's own broadcast
// read, 0.8 the staging; L1 85 % busy in the nn kernel).
// Against lists per lane (a lane gathers its own column's sources) this reads
// no padding and no conflicts, and an entry costs 8 bytes per 64
// multiply-adds instead of 8 bytes per lane: 0.19 ms for both terms at pf
// 4p4n k = 2 against 0.60 ms by the tiled kernel without its pn term.  (At
// k = 4, 8 the core-grouped kernels take these terms.)
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "bs_internal.h"

namespace bs {

// The matrix of one species, sources numbered inside the sector, in order.
void build_like_lists(const LikeJumps &L, LikeLists &O)
{
    O = LikeLists();
    O.ptr = L.ptr;
    std::vector<std::pair<int32_t, float>> v;
    for (size_t g = 0; g + 1 < L.ptr.size(); ++g) {
        v.clear();
        for (int64_t e = L.ptr[g]; e < L.ptr[g + 1]; ++e) v.push_back({L.src[(size_t)e], (float)L.coef[(size_t)e]});
        std::sort(v.begin(), v.end());
        for (const auto &e : v) O.ent.push_back(LikeEnt{e.first, e.second});
    }
}

// Panels of every block: pos SDs of the other species each, the widest matrices first.
void build_like_panels(const Basis &B, int spc, int pos, std::vector<LikePanel> &O, int &max_n)
{
    O.clear();
    max_n = 0;
    for (const Block &K : B.blocks) {
        LikePanel p = {};
        p.off = K.off;
        p.nN = (int)K.nN;
        p.n = (int)(spc == 0 ? K.nP : K.nN);
        p.row0 = B.sp[spc].sec[(size_t)(spc == 0 ? K.ps : K.ns)].start;
        max_n = std::max(max_n, p.n);
        const int64_t other = spc == 0 ? K.nN : K.nP;
        for (int64_t c = 0; c < other; c += pos) {
            p.pos0 = (int)c;
            p.npos = (int)std::min<int64_t>(pos, other - c);
            O.push_back(p);
        }
    }
    std::stable_sort(O.begin(), O.end(), [](const LikePanel &a, const LikePanel &b) { return a.n > b.n; });
}

namespace {

struct LikeArgs {
    const LikePanel *panels;
    const int64_t *ptr;
    const LikeEnt *ent;
    const float *part;     // pp: partial vectors to add, nz of them
    int nz;
    int64_t pstride;
};

// PW floats of a panel row (64 or 32); NN: the acting species is the neutrons.
template <int K, int PW, bool NN>
__global__ void __launch_bounds__(1024) hx_like_kernel(LikeArgs A, const float *__restrict__ x, float *__restrict__ y)
{
    constexpr int V = PW / 32;            // floats per lane
    constexpr int LD = PW + V;            // row stride: staging rows of consecutive SDs meet other banks
    extern __shared__ __align__(16) float sm[];
    const LikePanel P = A.panels[blockIdx.x];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    LikeEnt *buf = reinterpret_cast<LikeEnt *>(sm) + warp * 32;   // this warp's list entries
    float *X = sm + (blockDim.x >> 5) * 64;
    if constexpr (NN) {
        // (position r, SDs q): runs of consecutive q
        const int run = P.n * K;
        for (int r = warp; r < P.npos; r += nw) {
            const float *s = x + (P.off + (int64_t)(P.pos0 + r) * P.nN) * K;
            for (int f = lane; f < run; f += 32) X[f / K * LD + r * K + f % K] = __ldg(s + f);
        }
    } else {
        const int w = P.npos * K;
        for (int g = warp; g < P.n; g += nw) {
            const float *s = x + (P.off + (int64_t)g * P.nN + P.pos0) * K;
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (lane + 32 * v < w) X[g * LD + lane + 32 * v] = __ldg(s + lane + 32 * v);
        }
    }
    __syncthreads();
    const float *Xl = X + lane * V;
    int g = warp + nw * (int)blockIdx.y;   // grid.y CTAs share a panel's rows
    int64_t e0 = 0, e1 = 0;
    LikeEnt nx{0, 0.0f};              // this lane's entry of the next batch
    if (g < P.n) {
        e0 = A.ptr[P.row0 + g];
        e1 = A.ptr[P.row0 + g + 1];
        if (e0 + lane < e1) nx = A.ent[e0 + lane];
    }
    while (g < P.n) {
        float2 acc = make_float2(0.0f, 0.0f);
        const int gd = g;
        bool more = true;
        while (more) {
            const int cnt = (int)min((int64_t)32, e1 - e0);
            __syncwarp();
            buf[lane] = nx;
            __syncwarp();
            // the next batch: of this row, or the first of the warp's next row
            e0 += 32;
            if (e0 >= e1) {
                more = false;
                g += nw * (int)gridDim.y;
                if (g < P.n) {
                    e0 = A.ptr[P.row0 + g];
                    e1 = A.ptr[P.row0 + g + 1];
                }
            }
            if (g < P.n && e0 + lane < e1) nx = A.ent[e0 + lane];
            // entries in pairs: two per broadcast read
            auto one = [&](int src, float c) {
                if constexpr (V == 2) {
                    const float2 v = *reinterpret_cast<const float2 *>(Xl + src * LD);
                    acc = __ffma2_rn(make_float2(c, c), v, acc);
                } else {
                    acc.x = fmaf(c, Xl[src * LD], acc.x);
                }
            };
            const int4 *b2 = reinterpret_cast<const int4 *>(buf);
            int j = 0;
#pragma unroll 4
            for (; j + 2 <= cnt; j += 2) {
                const int4 q = b2[j >> 1];
                one(q.x, __int_as_float(q.y));
                one(q.z, __int_as_float(q.w));
            }
            if (j < cnt) one(buf[j].src, buf[j].coef);
        }
        // store: nn writes its rows, pp adds them and the partial vectors
#pragma unroll
        for (int v = 0; v < V; v += (K > 1 ? V : 1)) {
            const int f = lane * V + v, c = f / K;
            if (c >= P.npos) continue;
            constexpr bool two = V == 2 && K > 1;
            if constexpr (NN) {
                float *o = y + (P.off + (int64_t)(P.pos0 + c) * P.nN + gd) * K + f % K;
                if constexpr (two) *reinterpret_cast<float2 *>(o) = acc;
                else *o = v ? acc.y : acc.x;
            } else {
                const int64_t at = (P.off + (int64_t)gd * P.nN + P.pos0) * K + f;
                if constexpr (two) {
                    float2 s = *reinterpret_cast<const float2 *>(y + at);
                    s.x += acc.x;
                    s.y += acc.y;
                    for (int t = 0; t < A.nz; ++t) {
                        const float2 p = __ldg(reinterpret_cast<const float2 *>(A.part + t * A.pstride + at));
                        s.x += p.x;
                        s.y += p.y;
                    }
                    *reinterpret_cast<float2 *>(y + at) = s;
                } else {
                    float s = y[at] + (v ? acc.y : acc.x);
                    for (int t = 0; t < A.nz; ++t) s += __ldg(A.part + t * A.pstride + at);
                    y[at] = s;
                }
            }
        }
    }
}

constexpr size_t kLikeSmem = 227 * 1024;

size_t like_smem(int max_n, int pw, int threads)
{
    return (size_t)(threads / 32) * 256 + (size_t)max_n * (size_t)(pw + pw / 32) * 4;
}

// wide panels leave one CTA on an SM: all 32 warps; narrow ones several of eight
int like_threads(int max_n) { return max_n >= 256 ? 1024 : 256; }

template <int K, int PW, bool NN>
cudaError_t launch_like_t(int dev, const Device::LikeDev &L, const float *x, float *y, const float *part, int nz, int64_t pstride,
                          cudaStream_t s)
{
    const int th = like_threads(L.max_n);
    const size_t smem = like_smem(L.max_n, PW, th);
    auto kern = hx_like_kernel<K, PW, NN>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    LikeArgs A{L.panels[K - 1], L.ptr, L.ent, part, nz, pstride};
    const int np = L.npanels[K - 1];
    if (np <= 0) return cudaSuccess;
    // several CTAs to a panel, each with some of its rows, until there are four for every
    // place on the chip (a panel is loaded in a fortieth of the time its rows take) or a
    // warp has only two rows left
    int nsm = 0, per = 0;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, th, smem)) != cudaSuccess) return e;
    const int want = (4 * nsm * std::max(per, 1) + np - 1) / np, most = std::max(1, L.max_n / (th / 32 * 2));
    kern<<<dim3((unsigned)np, (unsigned)std::max(1, std::min(want, most))), th, smem, s>>>(A, x, y);
    return cudaGetLastError();
}

template <int K>
cudaError_t launch_like_k(const Device &D, const float *x, float *y, const float *part, int nz, int64_t pstride, cudaStream_t s)
{
    cudaError_t e = D.like[1].pw == 64 ? launch_like_t<K, 64, true>(D.dev, D.like[1], x, y, nullptr, 0, 0, s)
                                       : launch_like_t<K, 32, true>(D.dev, D.like[1], x, y, nullptr, 0, 0, s);
    if (e != cudaSuccess) return e;
    return D.like[0].pw == 64 ? launch_like_t<K, 64, false>(D.dev, D.like[0], x, y, part, nz, pstride, s)
                              : launch_like_t<K, 32, false>(D.dev, D.like[0], x, y, part, nz, pstride, s);
}

}  // namespace

// Floats of a panel row for matrices of up to max_n rows; 0: none fits.
int like_panel_width(int max_n)
{
    for (int pw : {64, 32})
        if (like_smem(max_n, pw, like_threads(max_n)) <= kLikeSmem) return pw;
    return 0;
}

// y = nn + pp + the nz partial vectors; only where like_applies.
bool like_applies(const bs_ctx *c) { return c->dev.like[0].pw > 0 && c->dev.like[1].pw > 0; }

cudaError_t launch_hx_like(const bs_ctx *c, const float *x, float *y, int k, cudaStream_t s, const float *part, int nz)
{
    const int64_t ps = c->basis.dim * k;
    return k == 1 ? launch_like_k<1>(c->dev, x, y, part, nz, ps, s) : launch_like_k<2>(c->dev, x, y, part, nz, ps, s);
}

}  // namespace bs
