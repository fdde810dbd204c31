// Tables of the pair-core pn kernel (bs_hx_pair.cu).
//
// Between (Z-1)-proton and (N-1)-neutron determinants ("cores") the
// proton-neutron interaction is a plain matrix product: inserting the cores
// into both one-body operators of Eq. (xpndef),
//   sum W(ij,kl) (a+_i a_k)_p (a+_j a_l)_n
//     = sum_{cp,cn} sum_{ij,kl} a+_i a+_j |cp cn> W(ij,kl) <cp cn| a_l a_k,
// so for one proton core and all neutron cores of one (2M, parity) the
// gathered elements x[cp+k, cn+l] are a matrix [pairs kl] x [cores] that one
// constant matrix W [pairs ij] x [pairs kl] takes to the elements of y.
// Built here: the neutron cores grouped by (2M, parity) with the column of
// every cn + s, the W matrix of every pair key (2m, parity), and per proton
// core the list of its pairs and, as the work of one CTA, its tiles.  Bases
// whose proton cores have more output rows than the kernel's shared memory
// holds have no items.
#include <algorithm>
#include <map>
#include <new>
#include <tuple>

#include "bs_internal.h"

namespace bs {

namespace {

inline int below(uint64_t m, int s)
{
    return __builtin_popcountll(m & ((1ULL << s) - 1ULL)) & 1;   // 1: sign -1
}

struct CoreKey {
    int twoM, par;
    bool operator<(const CoreKey &o) const { return std::tie(twoM, par) < std::tie(o.twoM, o.par); }
};

// Determinants with one particle removed, unique, by (2M, parity), bitmask ascending inside.
void cores_of(const Basis &B, const Species &S, std::map<CoreKey, std::vector<uint64_t>> &out)
{
    const int ns = (int)B.st.size();
    std::vector<uint64_t> c;
    c.reserve(S.bits.size() * (size_t)std::max(1, S.nparticles));
    for (uint64_t b : S.bits)
        for (uint64_t m = b; m; m &= m - 1) c.push_back(b & ~(m & (~m + 1)));
    std::sort(c.begin(), c.end());
    c.erase(std::unique(c.begin(), c.end()), c.end());
    for (uint64_t b : c) {
        CoreKey k{0, 0};
        for (int s = 0; s < ns; ++s)
            if (b >> s & 1) {
                k.twoM += B.st[(size_t)s].twom;
                k.par ^= B.st[(size_t)s].par;
            }
        out[k].push_back(b);
    }
}

}  // namespace

// With max_cols >= 0, nothing is built where some proton core has more output columns.
void build_pair_tables(const Basis &B, const Interaction &I, PairTables &T, int64_t max_cols)
{
    T = PairTables();
    const int ns = (int)B.st.size();
    // the kernel's limits: one 32-bit sign mask per neutron core, 32-bit basis indices; a W-truncated basis splits the
    // groups into ones too small for it (pf 5p4n 4p-4h k = 4: 2.9 ms against 2.5 by the tiled kernel)
    if (B.trunc || ns > 32 || B.Z < 1 || B.N < 1 || B.dim >= (int64_t)1 << 31) return;
    const Species &P = B.sp[0], &Q = B.sp[1];
    // ---- neutron cores; every group starts at a multiple of 4 (its columns are read four cores at a time)
    std::map<CoreKey, std::vector<uint64_t>> ncore, pcore;
    cores_of(B, Q, ncore);
    cores_of(B, P, pcore);
    struct Group { CoreKey key; int start, count; std::vector<int> sec; };
    std::vector<Group> groups;
    size_t tot = 0;
    for (const auto &kv : ncore) {
        Group g{kv.first, (int)tot, (int)kv.second.size(), std::vector<int>((size_t)ns, -1)};
        tot += (kv.second.size() + 3) / 4 * 4;
        groups.push_back(std::move(g));
    }
    T.ncn = (int)tot;
    T.colpos.assign((size_t)ns * tot, 0xFFFF);
    T.nsign.assign(tot, 0u);
    {
        size_t gi = 0;
        for (const auto &kv : ncore) {
            Group &g = groups[gi++];
            for (size_t a = 0; a < kv.second.size(); ++a) {
                const uint64_t c = kv.second[a];
                uint32_t sg = 0;
                for (int s = 0; s < ns; ++s) {
                    if (below(c, s)) sg |= 1u << s;
                    if (c >> s & 1) continue;
                    auto it = Q.index.find(c | 1ULL << s);
                    if (it == Q.index.end()) continue;
                    const int sec = Q.sec_of_sd[(size_t)it->second];
                    g.sec[(size_t)s] = sec;
                    T.colpos[(size_t)s * tot + (size_t)g.start + a] = (uint16_t)(it->second - Q.sec[(size_t)sec].start);
                }
                T.nsign[(size_t)g.start + a] = sg;
            }
        }
    }
    // ---- pairs (proton state, neutron state) by (2m, parity), proton state outer, and their W matrices
    std::map<std::pair<int, int>, std::vector<std::pair<int, int>>> pairs;
    for (int i = 0; i < ns; ++i)
        for (int j = 0; j < ns; ++j)
            pairs[{B.st[(size_t)i].twom + B.st[(size_t)j].twom, B.st[(size_t)i].par ^ B.st[(size_t)j].par}].push_back({i, j});
    std::map<std::pair<int, int>, int64_t> woff;
    int64_t nw = 0;
    for (const auto &kv : pairs) {
        woff[kv.first] = nw;
        nw += (int64_t)kv.second.size() * (int64_t)kv.second.size();
    }
    if (nw >= (int64_t)1 << 31) return;
    T.w.assign((size_t)nw, 0.0);
    for (const auto &kv : pairs) {
        const auto &v = kv.second;
        const size_t np = v.size();
        double *w = T.w.data() + woff[kv.first];
        for (size_t a = 0; a < np; ++a)
            for (size_t b = 0; b < np; ++b) {   // row kl (a), column ij (b)
                const int op = v[b].first * ns + v[a].first, on = v[b].second * ns + v[a].second;
                const int g = I.ops.group_of_op[(size_t)op];
                if (g < 0) continue;
                const int h = I.conj_group[(size_t)g];
                if (h < 0 || I.ops.group_of_op[(size_t)on] != h) continue;
                w[a * np + b] = I.Wpn[(size_t)(I.wpn_off[(size_t)g] +
                                               (int64_t)I.ops.local_of_op[(size_t)op] * (int64_t)I.ops.ops[(size_t)h].size() +
                                               I.ops.local_of_op[(size_t)on])];
            }
    }
    // place of a state among those of equal (2m, parity): two neutron states of
    // different place never lead two cores of one group to the same column in the same round
    std::vector<int> place((size_t)ns, 0);
    for (int s = 0; s < ns; ++s)
        for (int t = 0; t < s; ++t)
            if (B.st[(size_t)t].twom == B.st[(size_t)s].twom && B.st[(size_t)t].par == B.st[(size_t)s].par)
                ++place[(size_t)s];
    // ---- blocks of every proton sector, in order, with their first column among the sector's
    std::vector<std::vector<int>> blk_of((size_t)P.sec.size());
    std::vector<int> colbase(B.blocks.size(), 0), width(P.sec.size(), 0);
    for (size_t b = 0; b < B.blocks.size(); ++b) {
        const int ps = B.blocks[b].ps;
        colbase[b] = width[(size_t)ps];
        width[(size_t)ps] += (int)B.blocks[b].nN;
        blk_of[(size_t)ps].push_back((int)b);
    }
    // ---- per proton core: its free states' rows, ...
    struct PC { CoreKey key; uint64_t bits; std::vector<int> psec, prow, ybase, order; int64_t y; };
    std::vector<PC> pcs;
    for (const auto &kv : pcore)
        for (uint64_t cp : kv.second) pcs.push_back(PC{kv.first, cp, std::vector<int>((size_t)ns, -1), std::vector<int>((size_t)ns, 0),
                                                       std::vector<int>((size_t)ns, -1), {}, 0});
    for (PC &c : pcs)
        for (int k = 0; k < ns; ++k) {
            if (c.bits >> k & 1) continue;
            auto it = P.index.find(c.bits | 1ULL << k);
            if (it == P.index.end()) continue;
            const int sec = P.sec_of_sd[(size_t)it->second];
            if (blk_of[(size_t)sec].empty()) continue;
            c.psec[(size_t)k] = sec;
            c.prow[(size_t)k] = (int)(it->second - P.sec[(size_t)sec].start);
            c.ybase[(size_t)k] = (int)c.y;
            c.y += width[(size_t)sec];
            c.order.push_back(k);
        }
    for (const PC &c : pcs)
        if ((max_cols >= 0 && c.y > max_cols) || c.y >= (int64_t)1 << 31) {
            T = PairTables();
            return;
        }
    // ... pair records by neutron group, and output rows
    struct Out { std::vector<PairRec> recs; std::vector<uint8_t> state; std::vector<PairGroup> grps; std::vector<PairRow> rows; };
    std::vector<Out> outs(pcs.size());
    auto records = [&](int64_t n) {
        const PC &c = pcs[(size_t)n];
        Out &o = outs[(size_t)n];
        if (c.order.empty()) return;
        for (const Group &g : groups) {
            const std::pair<int, int> key{B.twoM - c.key.twoM - g.key.twoM, B.par ^ c.key.par ^ g.key.par};
            auto pit = pairs.find(key);
            if (pit == pairs.end()) continue;
            PairGroup G;
            G.rec0 = (int)o.recs.size();
            const auto &v = pit->second;
            for (size_t a = 0; a < v.size(); ++a) {
                const int k = v[a].first, l = v[a].second;
                if (c.psec[(size_t)k] < 0 || g.sec[(size_t)l] < 0) continue;
                const int b = B.block_of(c.psec[(size_t)k], g.sec[(size_t)l]);
                if (b < 0) continue;
                const Block &K = B.blocks[(size_t)b];
                PairRec r;
                r.xoff = (uint32_t)(K.off + (int64_t)c.prow[(size_t)k] * K.nN);
                r.yoff = (uint32_t)(c.ybase[(size_t)k] + colbase[(size_t)b]);
                r.srec = (uint32_t)(31 - l) | (below(c.bits, k) ? 0x80000000u : 0u);
                r.wj = (uint32_t)a | (uint32_t)l << 16 | (uint32_t)place[(size_t)l] << 24;
                o.recs.push_back(r);
                o.state.push_back((uint8_t)k);
            }
            G.nrec = (int)o.recs.size() - G.rec0;
            if (!G.nrec) continue;
            G.core0 = g.start;
            G.ncore = g.count;
            G.woff = (int)woff.at(key);
            G.np = (int)v.size();
            o.grps.push_back(G);
        }
        for (int k : c.order)
            for (int b : blk_of[(size_t)c.psec[(size_t)k]]) {
                const Block &K = B.blocks[(size_t)b];
                PairRow R;
                R.elem = K.off + (int64_t)c.prow[(size_t)k] * K.nN;
                R.ycol = c.ybase[(size_t)k] + colbase[(size_t)b];
                R.n = (int)K.nN;
                R.part = __builtin_popcountll(c.bits & ((1ULL << k) - 1ULL));
                R.state = k;
                R.sign = below(c.bits, k);
                R.pad = 0;
                o.rows.push_back(R);
            }
    };
    bool failed = false;   // (no exception may leave the parallel region)
#pragma omp parallel for schedule(dynamic, 16)
    for (int64_t n = 0; n < (int64_t)pcs.size(); ++n) {
        try {
            records(n);
        } catch (const std::bad_alloc &) {
#pragma omp atomic write
            failed = true;
        }
    }
    if (failed) throw std::bad_alloc();
    for (size_t n = 0; n < pcs.size(); ++n) {
        Out &o = outs[n];
        if (o.rows.empty()) continue;
        PairCore pc;
        pc.rec0 = (int)T.recs.size();
        pc.nrec = (int)o.recs.size();
        pc.grp0 = (int)T.grps.size();
        pc.ngrp = (int)o.grps.size();
        pc.row0 = (int)T.rows.size();
        pc.nrow = (int)o.rows.size();
        T.recs.insert(T.recs.end(), o.recs.begin(), o.recs.end());
        T.rec_state.insert(T.rec_state.end(), o.state.begin(), o.state.end());
        T.grps.insert(T.grps.end(), o.grps.begin(), o.grps.end());
        T.rows.insert(T.rows.end(), o.rows.begin(), o.rows.end());
        T.max_rec = std::max(T.max_rec, pc.nrec);
        T.max_cols = std::max<int64_t>(T.max_cols, pcs[n].y);
        T.cores.push_back(pc);
        o = Out();
    }
    T.on = !T.cores.empty();
}

// Items, one for each proton core with all its free states, largest work first.  False where a core has more rows
// than a tile can name.
bool build_pair_items(const PairTables &T, PairItems &O)
{
    O = PairItems();
    struct U { double cost; PairItem it; std::vector<PairTile> tiles; std::vector<PairRec> rows; std::vector<PairRow> store; };
    std::vector<U> units;
    for (const PairCore &pc : T.cores) {
        U u;
        u.it = {};
        u.it.rec0 = pc.rec0;
        u.it.nrec = pc.nrec;
        u.store.assign(T.rows.begin() + pc.row0, T.rows.begin() + pc.row0 + pc.nrow);
        for (const PairRow &r : u.store) u.it.cols += r.n;
        // the states in four subsets, one per consumer group: each state, the one
        // with the most rows first, to the subset whose fullest neutron group grows least
        std::vector<int> states;
        for (const PairRow &r : u.store)
            if (states.empty() || states.back() != r.state) states.push_back(r.state);
        std::vector<std::vector<int>> cnt(states.size(), std::vector<int>((size_t)pc.ngrp, 0));
        std::vector<int> sub(64, -1);
        std::vector<size_t> by(states.size());
        std::vector<long> tot(states.size(), 0);
        for (size_t a = 0; a < states.size(); ++a) {
            by[a] = a;
            for (int g = 0; g < pc.ngrp; ++g) {
                const PairGroup &G = T.grps[(size_t)(pc.grp0 + g)];
                const uint8_t *st = T.rec_state.data() + pc.rec0 + G.rec0;
                for (int r = 0; r < G.nrec; ++r) cnt[a][(size_t)g] += st[r] == states[a];
                tot[a] += (long)cnt[a][(size_t)g] * G.nrec;
            }
        }
        std::stable_sort(by.begin(), by.end(), [&](size_t a, size_t b) { return tot[a] > tot[b]; });
        std::vector<std::vector<int>> load(4, std::vector<int>((size_t)pc.ngrp, 0));
        for (size_t a : by) {
            int best = 0;
            double bestc = 1e300;
            for (int q = 0; q < 4; ++q) {
                double c = 0;   // sum over groups of (load after)^2, heavier for long sums
                for (int g = 0; g < pc.ngrp; ++g) {
                    const double l = load[(size_t)q][(size_t)g], n = cnt[a][(size_t)g];
                    c += ((l + n) * (l + n) - l * l) * T.grps[(size_t)(pc.grp0 + g)].nrec;
                }
                if (c < bestc) { bestc = c; best = q; }
            }
            sub[(size_t)states[a]] = best;
            for (int g = 0; g < pc.ngrp; ++g) load[(size_t)best][(size_t)g] += cnt[a][(size_t)g];
        }
        u.cost = 2.0 * u.it.cols;
        for (int g = 0; g < pc.ngrp; ++g) {
            const PairGroup &G = T.grps[(size_t)(pc.grp0 + g)];
            std::vector<PairRec> list[4];
            for (int r = 0; r < G.nrec; ++r) {
                const int q = sub[T.rec_state[(size_t)(pc.rec0 + G.rec0 + r)]];
                list[q].push_back(T.recs[(size_t)(pc.rec0 + G.rec0 + r)]);
            }
            size_t most = 0;
            for (auto &v : list) {
                std::stable_sort(v.begin(), v.end(), [](const PairRec &a, const PairRec &b) { return a.wj >> 24 < b.wj >> 24; });
                most = std::max(most, v.size());
            }
            const int nch = (G.ncore + kPairCores - 1) / kPairCores;
            const int ch = ((G.ncore + nch - 1) / nch + 31) / 32 * 32;
            for (size_t p0 = 0; p0 < most; p0 += kPairRows) {
                PairTile t = {};
                t.rec0 = G.rec0;
                t.nrec = G.nrec;
                t.woff = G.woff;
                t.np = G.np;
                int rmax = 0;
                for (int q = 0; q < 4; ++q) {
                    t.row0[q] = (uint16_t)u.rows.size();
                    const size_t n = list[q].size() > p0 ? std::min<size_t>(kPairRows, list[q].size() - p0) : 0;
                    t.nrow[q] = (uint8_t)n;
                    rmax = std::max(rmax, (int)n);
                    t.first[q] = n > 0;
                    for (size_t r = 0; r < n; ++r) {
                        if (r && list[q][p0 + r].wj >> 24 != list[q][p0 + r - 1].wj >> 24) t.first[q] |= (uint16_t)(1u << r);
                        u.rows.push_back(list[q][p0 + r]);
                    }
                }
                for (int c0 = 0; c0 < G.ncore; c0 += ch) {
                    t.core0 = G.core0 + c0;
                    t.ncore = std::min(ch, G.ncore - c0);
                    u.tiles.push_back(t);
                    u.cost += (double)G.nrec * (rmax + 3) * (0.5 + t.ncore / 256.0) + 100.0;
                }
            }
        }
        if (u.rows.size() > 65535) return false;
        O.max_cols = std::max(O.max_cols, u.it.cols);
        O.max_tiles = std::max(O.max_tiles, (int)u.tiles.size());
        O.max_rows = std::max(O.max_rows, (int)u.rows.size());
        O.max_rec = std::max(O.max_rec, pc.nrec);
        units.push_back(std::move(u));
    }
    std::stable_sort(units.begin(), units.end(), [](const U &a, const U &b) { return a.cost > b.cost; });
    for (U &u : units) {
        u.it.tile0 = (int)O.tiles.size();
        u.it.ntile = (int)u.tiles.size();
        u.it.row0 = (int)O.rows.size();
        u.it.nrow = (int)u.rows.size();
        u.it.store0 = (int)O.store.size();
        u.it.nstore = (int)u.store.size();
        O.tiles.insert(O.tiles.end(), u.tiles.begin(), u.tiles.end());
        O.rows.insert(O.rows.end(), u.rows.begin(), u.rows.end());
        O.store.insert(O.store.end(), u.store.begin(), u.store.end());
        O.items.push_back(u.it);
    }
    return true;
}

}  // namespace bs
