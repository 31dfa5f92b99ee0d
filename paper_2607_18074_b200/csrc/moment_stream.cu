// Host side of the moment-form edge stream: sets, units and read-out tables of a direction, the choice between the two forms of the
// stream, and the launch.
#include <algorithm>
#include <cmath>

#include "moment_stream.h"

namespace sobek {

static bool build_moment_set(const sobek_plan* p, Direction& dir, int dual, int& nq_max);
static void stream_costs(const sobek_plan* p, Direction& dir, int dual);

// Both forms of each stream of a direction; a call takes one of them (moment_stream_pays).  The moment form only in the place of
// k_stream_tc: a profile that k_stream_tc does not fit keeps the FP32-pipe stream, whose rows and coupling values have 32 bits (error
// of gR, 2-norm against fp64, 192 x (0..3): 4.5e-6 there, 6.4e-6 in either form on the tensor cores).
void build_stream_sets(const sobek_plan* p, Direction& dir) {
    for (int dual = 0; dual < 2; ++dual) {
        build_tc_sets(p, dir, dual);
        if (!dir.tc[dual].ok || p->form == kFormCoupled) continue;
        for (int nq_max = 8; !build_moment_set(p, dir, dual, nq_max);) {}
        if (dir.ms[dual].ok) stream_costs(p, dir, dual);
    }
}

// Microseconds of either form, from the counts of the forms' tables: a launch, and on one SM a node and 16 of its edges, which the roles
// work at side by side: (a^p + b^p)^(1/p).  The constants are least-squares fits (of relative errors; 8 and 10 % left, dual 9 and 11 %)
// to the streams of 9,082 random layers, 8 to 128 multiplicities of orders up to 4, K = 1 .. 16, degrees 2 to 400, 64 to 8,000 nodes, in
// both directions.  On the half of the layers that a fit to the other half did not see the form taken is 0.2 % above the faster one on
// average (dual streams: 0.2 %), at worst 1.4 (1.3) times the coupled one; fixed forms: moment 4.8 % (2.5 %), coupled 44 % (64 %).
struct StreamFit {
    double launch, p;                                         // moment form
    double unit, pair, val, part, set;                        //   node: units, pairs of components per team and run, their radial indices, those of runs not whole
    double kcycle, w, row, pass, slot_unit;                   //   slot: products, rows of W, gathered slabs, passes, units
    double c_launch, c_p;                                     // coupled form (1: with one accumulator buffer, on top)
    double c_col, c_col1, c_node_set;                         //   node: accumulator columns, sets
    double c_slab, c_row, c_set, c_slab1;                     //   batch: built operand, gathered rows, hand-over
    double c2_slab, c2_row, c2_set, c2_set1;                  //   its second operand
    double geo[5], c_geo[5];                                  // phi and Y of a slot from edge vectors: constant, per radial index, per harmonic; p; launch
};
constexpr StreamFit kFit[2] = {
    {9.89, 1.26, 0.517, 0.398, 0.0255, 0.0437, 0.0989, 0.226, 0.00195, 0.0139, 0.259, 0.0568,
     14.6, 1.65, 0.0194, 0.00377, 0.182, 0.186, 0.0487, 0.789, 0.0515, 0, 0, 0, 0, {1.17, 0.0476, 0, 4.37, 7.59}, {1.02, 0.0633, 0.00452, 11.1, 7.54}},
    {10.9, 1.21, 0.553, 0.39, 0.0369, 0.0406, 0, 0.219, 0.00282, 0.0095, 0.352, 0,
     15.5, 1.36, 0.0176, 0.00402, 0.295, 0.274, 0.03, 1, 0.0395, 0.167, 0.061, 0.855, 0.093, {1.66, 0.182, 0.0134, 1.59, 5.18}, {1.09, 0.148, 0.0545, 3.94, 13.1}}};
static double side_by_side(double a, double b, double p) { return std::pow(std::pow(a, p) + std::pow(b, p), 1 / p); }

static void stream_costs(const sobek_plan* p, Direction& dir, int dual) {
    const StreamFit& F = kFit[dual];
    TcSets& T = dir.tc[dual];
    MomentSets& M = dir.ms[dual];
    double cols = 0, slabs = 0, rows = 0;
    const double sets = (double)T.sets.size(), one = T.nbuf == 1 ? 1 : 0;
    for (const TSet& S : T.sets) {
        slabs += S.nslab;
        for (int u = 0; u < S.nunit; ++u) cols += (T.blks[T.units[S.unit_begin + u].blk].ncols + 31) & ~31;
        for (int b = 0; b < S.nblk; ++b) rows += T.blks[S.blk_begin + b].d_src * ((T.blks[S.blk_begin + b].c_src + 63) / 64);
    }
    T.node_us = (F.c_col + one * F.c_col1) * cols + F.c_node_set * sets;
    T.slot_us = (F.c_slab + one * F.c_slab1) * slabs + F.c_row * rows + F.c_set * sets;
    T.slot2_us = F.c2_slab * slabs + F.c2_row * rows + (F.c2_set + one * F.c2_set1) * sets;
    double units = 0, pairs = 0, vals = 0, part = 0, kcycles = 0, w[2] = {0, 0}, gathered[2] = {0, 0}, passes[2] = {0, 0};      // [1]: slots that do not stay
    for (const MSet& S : M.sets) {
        gathered[0] += S.nslab; passes[0] += 1; passes[1] += S.npass;
        for (int g = 0; g < S.ngrp; ++g) {
            const MGrp& G = M.grps[S.grp_begin + g];
            w[0] += 2 * G.rows;
            for (int u = 0; u < G.nunit; ++u) {
                const MUnit& U = M.units[G.unit_begin + u];
                const double team = (double)U.n_pair / (U.c > 32 ? MS_NDT : U.c > 16 ? 2 * MS_NDT : 4 * MS_NDT);
                units += 1; pairs += U.nqs * team; vals += U.nqs * S.nq * team;
                for (int r = 1; r <= U.nqs; ++r)
                    if (U.q0 + 2 * S.nq * r > p->K) part += S.nq * team;
                kcycles += 6e-3 * U.d * std::max(41.0, U.N / 2.0);           // six products per component, at least 41 cycles each
                if (u & 1) continue;
                const MUnit& V = M.units[G.unit_begin + std::min(u + 1, G.nunit - 1)];               // two units' pass
                w[1] += 2 * (std::max(U.row0 + U.N, V.row0 + V.N) - std::min(U.row0, V.row0));
                gathered[1] += V.slab0 + V.d - U.slab0;
            }
        }
    }
    M.node_us = F.unit * units + F.pair * pairs + F.val * vals + F.part * part + F.set * M.sets.size();
    for (int k = 0; k < 2; ++k) {
        M.slot_us[k] = F.kcycle * kcycles + F.w * w[k] + F.row * gathered[k] + F.pass * passes[k] + F.slot_unit * units;
        M.passes[k] = passes[k];
    }
}

// The busiest SM counts: items are (set, node), dealt to 148 of them.  The slots of a node stay for all its units where they all fit the
// rings; the rows of the others are gathered, and their W built, for every two units.  Degrees spread around their mean: the share of the
// latter falls from all to none where the longest node that stays has 0.7 to 1.5 times the mean.  Below four nodes per SM the longest ones
// decide.  With the edge inputs computed from vectors (geo) one warp of either kernel makes the rows of every slot in every pass, a bound of
// its own.  (Of such layers that the fit did not see: 0.4 % above the faster form on average, dual streams 0.9 %, at worst 1.4 and 2.0 times
// the coupled one; moment throughout 7 % and 31 %.)
bool moment_stream_pays(const sobek_plan* p, const Direction& dir, int dual, int operands, bool geo, int64_t N, int64_t E) {
    const StreamFit& F = kFit[dual];
    const TcSets& T = dir.tc[dual];
    const MomentSets& M = dir.ms[dual];
    if (!M.ok || p->form != kFormAuto) return M.ok && p->form == kFormMoment;
    const double mean = (double)E / (double)std::max<int64_t>(N, 1), sets = (double)M.sets.size(), c_sets = (double)T.sets.size();
    const double per_sm = std::ceil((double)N * sets / 148) / sets, c_per_sm = std::ceil((double)N * c_sets / 148) / c_sets;
    const bool few = N < 4 * 148;
    const double batches = (few ? 1.15 : 1.0) * mean / MS_TB + 0.5, slots = batches * operands;
    const double longest = MS_TB * (double)(std::min(M.ns, M.nw) / operands), over = 1.5 * mean - longest;
    const double again = few ? (over > 0 ? 1 : 0) : std::min(1.0, std::max(0.0, over / (0.8 * mean)));
    auto mix = [&](const double* v) { return v[0] + again * (v[1] - v[0]); };
    double moment = F.launch + per_sm * side_by_side(M.node_us, slots * mix(M.slot_us), F.p),
           coupled = F.c_launch + c_per_sm * side_by_side(T.node_us, batches * (T.slot_us + (operands - 1) * T.slot2_us), F.c_p);
    if (geo) {
        auto rows = [&](const double* g, double passes) { return g[4] + slots * passes * (g[0] + g[1] * p->K + g[2] * p->dim_sh); };
        moment = side_by_side(moment, rows(F.geo, per_sm * mix(M.passes)), F.geo[3]);
        coupled = side_by_side(coupled, rows(F.c_geo, c_per_sm * c_sets), F.c_geo[3]);
    }
    return moment < coupled;
}

// Sets, units and tables with at most nq_max radial indices side by side.  False where parts of one block came into sets with
// different numbers of them (nq_max is then the smallest): the order of a path's state is one for all its multiplicities.
static bool build_moment_set(const sobek_plan* p, Direction& dir, int dual, int& nq_max) {
    constexpr int kSmem = 227 * 1024;
    constexpr int kSlotBytes = 37 * 1024;      // gathered rows of a slot, hi and lo, beyond which a block starts a set of its own
    constexpr int kWRows = 224;                // rows of W at a time (both lane halves) that several runs share; a single run may have more
    MomentSets& T = dir.ms[dual];
    T = MomentSets{};
    if (p->K > 16 || (dir.C_src & 7) || dir.paths.empty()) return true;
    bool ok = true;
    struct Pth { const DPath* P; int lb, group; };
    struct Blk { int so, c, d; std::vector<Pth> paths; };
    std::vector<Blk> blocks;
    for (size_t gi = 0; gi < dir.groups.size(); ++gi)
        for (int k = dir.groups[gi].path_begin; k < dir.groups[gi].path_end; ++k) {
            const DPath& P = dir.paths[k];
            if ((P.c_src & 7) || (P.src_off & 7)) ok = false;
            auto it = std::find_if(blocks.begin(), blocks.end(), [&](const Blk& b) { return b.so == P.src_off; });
            if (it == blocks.end()) { blocks.push_back(Blk{P.src_off, P.c_src, P.d_src, {}}); it = blocks.end() - 1; }
            it->paths.push_back(Pth{&P, (P.d_sh - 1) / 2, (int)gi});
        }
    if (!ok) return true;
    std::sort(blocks.begin(), blocks.end(), [](const Blk& x, const Blk& y) { return x.so < y.so; });
    const int raw = ((dual ? 2 : 1) * (p->K + p->dim_sh) * MS_PS * 4 + 1023) & ~1023;
    // blocks of more than 64 multiplicities are cut into equal parts
    struct Part { int blk, u0, c; };
    std::vector<Part> parts;
    for (size_t b = 0; b < blocks.size(); ++b) {
        const int n = (blocks[b].c + 63) / 64, per = ((blocks[b].c / 8 + n - 1) / n) * 8;
        for (int u = 0; u < blocks[b].c; u += per) parts.push_back(Part{(int)b, u, std::min(per, blocks[b].c - u)});
    }
    // Sets: consecutive parts whose rows of 16 edges leave room for four slots with their W (a node of 32 edges and the next
    // one's first rows); a wider part is a set of its own with the slots it leaves, at least two.
    int x_cap = 0;
    for (size_t i = 0; i < parts.size() && ok;) {
        MSet S{};
        S.blk_begin = (int)T.blks.size(); S.grp_begin = (int)T.grps.size();
        int slabs = 0, dmax = 0;
        size_t j = i;
        for (; j < parts.size(); ++j) {
            const Blk& B = blocks[parts[j].blk];
            if (j > i && 2 * (slabs + B.d) * MS_SLAB > kSlotBytes) break;
            T.blks.push_back(MBlk{B.so + parts[j].u0, parts[j].c, B.c, B.d, slabs, {0, 0, 0}});
            slabs += B.d;
            dmax = std::max(dmax, B.d);
        }
        S.nblk = (int)T.blks.size() - S.blk_begin;
        // a slab has room for 64 multiplicities: rows of up to 32 (16) go in twice (four times)
        S.slab_begin = (int)T.slabs.size(); S.nslab = slabs;
        for (int b = S.blk_begin; b < (int)T.blks.size(); ++b)
            for (int k = 0; k < T.blks[b].d_src; ++k) {
                const int chunks = (T.blks[b].c + 7) / 8;
                T.slabs.push_back(MSlab{T.blks[b].src_off + k * T.blks[b].c_row, chunks, chunks > 4 ? 7 : (chunks > 2 ? 3 : 1), 0});
            }
        x_cap = std::max(x_cap, slabs * MS_SLAB);
        // Rows of W: runs of nq radial indices (those of one lane half), per run the harmonics order by order, the radial
        // index fastest, so that one read-out instruction takes nq of them.  The orders are cut into segments of whole
        // groups of eight rows such that every block's components x a segment fit the columns of one TMEM half.
        const int KH = (p->K + 1) / 2;
        struct Seg { int l0, l1, row, rows; };
        std::vector<Seg> segs;
        // Eight at a time from 13 radial indices on.  At 16, where the run is whole, four at a time are 3 to 13 % slower (dual: 0 to 10 %);
        // at 13 to 15 within 2 % either way, one-order harmonics with long neighbourhoods 20 % slower.  At l_max 3 and 4 the run has 256 and
        // 400 rows of W, which take ring slots: four at a time are 12 to 30 % slower at 64 and 128 multiplicities and degrees to 30, and
        // 6 to 12 % faster in the dual streams of orders 0 and 1 at degree 120.
        int nq = std::min(nq_max, KH >= 7 ? 8 : KH >= 3 ? 4 : KH), rows_q = 0;
        for (; nq >= 1; nq >>= 1) {
            segs.clear(); rows_q = 0;
            bool fits = true;
            for (int l = 0; l <= p->l_max && fits;) {
                int e = l, rows = 0;
                for (; e <= p->l_max; ++e) {
                    const int r = (((e + 1) * (e + 1) - l * l) * nq + 7) & ~7;
                    if (dmax * r > MS_HALF) break;
                    rows = r;
                }
                if (e == l) { fits = false; break; }
                segs.push_back(Seg{l, e - 1, rows_q, rows});
                rows_q += rows;
                l = e;
            }
            if (fits) break;
        }
        if (!nq) { ok = false; break; }
        S.nq = nq;
        const int runs = (KH + nq - 1) / nq;                                  // runs of radial indices per lane half
        const int nqs = std::max(1, std::min(runs, kWRows / 2 / rows_q)), ngrp = (runs + nqs - 1) / nqs;
        const int nqs_g = (runs + ngrp - 1) / ngrp, rows_h = nqs_g * rows_q;
        S.ngrp = ngrp;
        T.w_bytes = std::max(T.w_bytes, 2 * rows_h * 64);
        const int row_begin = (int)T.rows.size();
        for (int h = 0; h < 2; ++h)
            for (int r = 0; r < nqs_g; ++r)
                for (const Seg& g : segs)
                    for (int n = 0; n < g.rows; ++n) {
                        const int nb = (g.l1 + 1) * (g.l1 + 1) - g.l0 * g.l0, m = std::min(n, nb * nq - 1);
                        T.rows.push_back((uint16_t)((2 * (r * nq + m % nq) + h) | ((g.l0 * g.l0 + m / nq) << 8)));
                    }
        // units of one group; `used` tells which segments a block has paths in
        std::vector<MUnit> us;
        for (size_t k = i; k < j; ++k) {
            const Blk& B = blocks[parts[k].blk];
            const MBlk& M = T.blks[S.blk_begin + (int)(k - i)];
            auto used = [&](size_t g) { return std::any_of(B.paths.begin(), B.paths.end(), [&](const Pth& t) { return t.lb >= segs[g].l0 && t.lb <= segs[g].l1; }); };
            auto emit = [&](int run, int n_runs, size_t ga, size_t gb) {          // segments [ga, gb)
                MUnit U{};
                U.slab0 = M.slab0; U.d = B.d; U.c = M.c; U.blk0 = (int)(k - i); U.nblk = 1;
                U.row0 = run * rows_q + segs[ga].row;
                U.N = n_runs > 1 ? n_runs * rows_q : segs[gb - 1].row + segs[gb - 1].rows - segs[ga].row;
                U.nqs = n_runs; U.rows_q = rows_q; U.q0 = 2 * run * nq;
                U.pad[0] = (int)ga; U.pad[1] = (int)gb;
                if (!us.empty()) {       // together with the block before it, where the columns hold both
                    MUnit& V = us.back();
                    if (V.row0 == U.row0 && V.N == U.N && V.c == U.c && V.blk0 + V.nblk == U.blk0 &&
                        V.slab0 + V.d == U.slab0 && (V.d + U.d) * U.N <= MS_HALF) {
                        V.d += U.d; ++V.nblk;
                        return;
                    }
                }
                us.push_back(U);
            };
            const size_t ns = segs.size();
            size_t ga = 0, gb = ns;
            while (ga < ns && !used(ga)) ++ga;
            while (gb > ga && !used(gb - 1)) --gb;
            if (ga == 0 && gb == ns && B.d * nqs_g * rows_q <= MS_HALF) { emit(0, nqs_g, 0, ns); continue; }
            for (int run = 0; run < nqs_g; ++run)
                for (size_t x = ga; x < gb;) {
                    if (!used(x)) { ++x; continue; }
                    size_t y = x + 1;
                    while (y < gb && B.d * (segs[y].row + segs[y].rows - segs[x].row) <= MS_HALF) ++y;
                    emit(run, 1, x, y);
                    x = y;
                }
        }
        // read-out tables (the same for every group)
        int pairs = 0;
        for (MUnit& U : us) {
            struct Comp { MOut e; std::vector<MTerm> t; };
            std::vector<Comp> comps;
            int s0 = 0;
            for (int k = 0; k < U.nblk; ++k) {
                const Part& Pt = parts[i + U.blk0 + k];
                const Blk& B = blocks[Pt.blk];
                for (int g = U.pad[0]; g < U.pad[1]; ++g)
                    for (const Pth& t : B.paths) {
                        if (t.lb < segs[g].l0 || t.lb > segs[g].l1) continue;
                        for (int o = 0; o < t.P->d_dst; ++o) {
                            const int ld = dir.nk_ld[t.group];
                            Comp C{MOut{(int64_t)o * ld + t.P->koff, t.P->d_dst * ld, B.c, Pt.u0, 0, 0, (int)dir.zb_off[t.group]}, {}};
                            const int col0 = segs[g].row - segs[U.pad[0]].row + (t.lb * t.lb - segs[g].l0 * segs[g].l0) * nq;
                            for (int sc = 0; sc < B.d; ++sc)
                                for (int z = p->tab_ptr[t.P->tabM + sc * t.P->d_dst + o]; z < p->tab_ptr[t.P->tabM + sc * t.P->d_dst + o + 1]; ++z)
                                    C.t.push_back(MTerm{(uint32_t)((s0 + sc) * U.N + col0 + p->tab_idx[z] * nq), p->tab_coef[z]});
                            if (C.t.empty()) C.t.push_back(MTerm{(uint32_t)col0, 0.f});
                            comps.push_back(C);
                        }
                    }
                s0 += B.d;
            }
            // pairs of about equally many terms; the shorter one reads its last column again, times zero
            std::stable_sort(comps.begin(), comps.end(), [](const Comp& x, const Comp& y) { return x.t.size() > y.t.size(); });
            U.out_begin = (int)T.outs.size();
            U.n_out = (int)comps.size();
            U.n_pair = (U.n_out + 1) / 2;
            U.pair0 = pairs;
            pairs += U.n_pair;
            for (size_t k = 0; k < comps.size(); k += 2) {
                const Comp& A = comps[k];
                Comp N = k + 1 < comps.size() ? comps[k + 1] : Comp{MOut{A.e.a, A.e.b, 0, 0, 0, 0, A.e.zoff}, {MTerm{A.t[0].col, 0.f}}};
                const int first = (int)T.terms.size(), n = (int)A.t.size();
                while (N.t.size() < A.t.size()) N.t.push_back(MTerm{N.t.back().col, 0.f});
                for (int z = 0; z < n; ++z) { T.terms.push_back(A.t[z]); T.terms.push_back(N.t[z]); }
                for (MOut e : {A.e, N.e}) { e.term = first; e.n = n; T.outs.push_back(e); }
            }
        }
        for (int g = 0; g < ngrp; ++g) {
            MGrp G{};
            G.q0 = 2 * g * nqs_g * nq; G.rows = rows_h; G.row_begin = row_begin; G.unit_begin = (int)T.units.size(); G.nunit = (int)us.size();
            for (MUnit U : us) { U.q0 += G.q0; U.pair0 += g * pairs; T.units.push_back(U); }
            T.grps.push_back(G);
        }
        S.nunit = ngrp * (int)us.size();
        S.gpass = ((int)us.size() + 1) / 2; S.npass = ngrp * S.gpass;
        T.sets.push_back(S);
        i = j;
    }
    if (!ok) { T = MomentSets{}; return true; }
    T.zq.assign(dir.paths.size(), 0);
    for (const MSet& S : T.sets)
        for (int b = 0; b < S.nblk; ++b) {
            const MBlk& B = T.blks[S.blk_begin + b];
            for (size_t k = 0; k < dir.paths.size(); ++k) {
                const DPath& P = dir.paths[k];
                if (B.src_off < P.src_off || B.src_off >= P.src_off + P.c_src) continue;
                if (T.zq[k] && T.zq[k] != S.nq) { nq_max = std::min(T.zq[k], S.nq); T = MomentSets{}; return false; }
                T.zq[k] = S.nq;
            }
        }
    const int tables = (int)(T.outs.size() * sizeof(MOut) + T.terms.size() * sizeof(MTerm) + T.sets.size() * sizeof(MSet) + T.grps.size() * sizeof(MGrp) +
                             T.slabs.size() * sizeof(MSlab) + T.units.size() * sizeof(MUnit) + T.rows.size() * 2 + 64);
    const int fixed = 1024 + MS_NBAR * 8 + 16 + tables;
    T.x_cap = x_cap;
    T.slot_bytes = 2 * x_cap + raw;
    // as many slots as fit with an entry of W each
    T.ns = T.nw = std::min(std::min(MS_MAXNS, MS_MAXNW), (kSmem - fixed) / (T.slot_bytes + T.w_bytes));
    if (fixed + T.ns * (T.slot_bytes + T.w_bytes) + T.w_bytes <= kSmem && T.nw < MS_MAXNW) ++T.nw;
    T.smem_bytes = fixed + T.ns * T.slot_bytes + T.nw * T.w_bytes;
    // Where the loaders are to copy phi and Y: at most twelve state components a set.  (2,000 random layers of 600 nodes and more, loaders
    // against edge warp: 1.5 to 15 % faster up to twelve; 21 to 30 components 0.2 to 0.5 % slower, above 30 0.5 to 1.4 %.)
    int n_out = 0;
    for (const MUnit& U : T.units) n_out += U.n_out;
    T.loaders_edge = n_out <= 12 * (int)T.sets.size();
    T.ok = T.ns >= 2;
    return true;
}

cudaError_t launch_moment_stream(const sobek_plan* p, const Direction& dir, const EdgeView& ev, int64_t node0, int64_t n_nodes,
                                 const SplitSrc& ss, const float* Y, const float* vY, const float* phi, const float* vphi, int dual,
                                 void* zh, void* zl, int* status, cudaStream_t s) {
    const MomentSets& T = dir.ms[dual ? 1 : 0];
    if (!T.ok || !ss.h || !ss.l) return cudaErrorInvalidValue;
    if (n_nodes <= 0) return cudaSuccess;
    MsArgs a{};
    a.sets = T.d_sets; a.grps = T.d_grps; a.slabs = T.d_slabs; a.units = T.d_units; a.outs = T.d_outs; a.terms = T.d_terms; a.rows = T.d_rows;
    a.nsets = (int)T.sets.size(); a.n_grps = (int)T.grps.size(); a.n_slabs = (int)T.slabs.size(); a.n_units = (int)T.units.size(); a.n_terms = (int)T.terms.size();
    a.n_outs = (int)T.outs.size(); a.n_rows = (int)T.rows.size();
    a.ev = ev; a.node0 = node0; a.n_nodes = n_nodes;
    a.oseg = ss.oseg ? ss.oseg + node0 : nullptr;
    a.sh = (const __nv_bfloat16*)ss.h; a.sl = (const __nv_bfloat16*)ss.l;
    a.vsh = (const __nv_bfloat16*)ss.vh; a.vsl = (const __nv_bfloat16*)ss.vl;
    a.Y = Y; a.vY = vY; a.phi = phi; a.vphi = vphi;
    a.rvec = ss.rvec; a.geo_rc = ss.geo_rc; a.geo_basis = ss.geo_basis; a.geo_p = ss.geo_p;
    a.vrvec = dual ? ss.vrvec : nullptr;
    a.zh = (__nv_bfloat16*)zh; a.zl = (__nv_bfloat16*)zl;
    a.K = p->K; a.dsh = p->dim_sh; a.C_src = dir.C_src;
    a.x_cap = T.x_cap; a.slot_bytes = T.slot_bytes; a.ns = T.ns; a.w_bytes = T.w_bytes; a.nw = T.nw;
    a.interleaved = p->uvu ? 0 : 1;      // (the channelwise node-side kernels read the state q-major)
    a.status = status;
    const int grid = (int)std::min<int64_t>(n_nodes * a.nsets, (int64_t)148);
    KernelTimer kt(K_STATE, s);
    const bool le = T.loaders_edge && !a.rvec && n_nodes >= 4 * 148;      // (a node or two per SM: two warps side by side, 26.7 against 27.8 us a call at 64 nodes)
    const cudaError_t e = dual ? moment_stream_dual(a, grid, T.smem_bytes, le, s) : moment_stream_plain(a, grid, T.smem_bytes, le, s);
    count_launch();
    return e;
}

}  // namespace sobek
