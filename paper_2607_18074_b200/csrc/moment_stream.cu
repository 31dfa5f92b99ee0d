// Host side of the moment-form edge stream: sets, units and read-out tables of a direction, and the launch.
#include <algorithm>

#include "moment_stream.h"

namespace sobek {

// Sets, units and read-out tables of one direction for the plain ([0]) and the dual ([1]) stream.
void build_moment_sets(const sobek_plan* p, Direction& dir) {
    constexpr int kSmem = 227 * 1024;
    for (int dual = 0; dual < 2; ++dual) {
        MomentSets& T = dir.ms[dual];
        T = MomentSets{};
        if (p->K > 16 || (dir.C_src & 7) || dir.paths.empty()) continue;
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
        if (!ok) continue;
        std::sort(blocks.begin(), blocks.end(), [](const Blk& x, const Blk& y) { return x.so < y.so; });
        const int raw = ((dual ? 2 : 1) * (p->K + p->dim_sh) * MS_PS * 4 + 1023) & ~1023;
        // blocks of more than 128 multiplicities are cut into equal parts
        struct Part { int blk, u0, c; };
        std::vector<Part> parts;
        for (size_t b = 0; b < blocks.size(); ++b) {
            const int n = (blocks[b].c + 127) / 128, per = ((blocks[b].c / 8 + n - 1) / n) * 8;
            for (int u = 0; u < blocks[b].c; u += per) parts.push_back(Part{(int)b, u, std::min(per, blocks[b].c - u)});
        }
        int max_rows = 16;
        std::vector<std::vector<MUnit>> units(parts.size());
        for (size_t pi = 0; pi < parts.size() && ok; ++pi) {
            const Blk& B = blocks[parts[pi].blk];
            const int halves = parts[pi].c > 64 ? 1 : 2, gran = halves == 2 ? 8 : 16;
            std::vector<int> lbs, lboff(1, 0);
            for (int lb = 0; lb <= p->l_max; ++lb)
                if (std::any_of(B.paths.begin(), B.paths.end(), [&](const Pth& t) { return t.lb == lb; })) { lbs.push_back(lb); lboff.push_back(lboff.back() + 2 * lb + 1); }
            // Harmonic orders that share a unit, and how many radial indices it takes: the partition with the fewest MMA cycles.
            // (see the rates at ms_issue: M = 64 takes about max(N/2, 16 + 0.24 N) cycles, M = 128 max(N/2, 27 + 0.23 N))
            const int nl = (int)lbs.size(), KH = (p->K + halves - 1) / halves;     // radial indices per lane half
            const int cap = std::min(MS_NMAX, MS_HALF / B.d & ~(gran - 1));
            auto cycles = [&](int n) { return halves == 2 ? 2.0 * std::max(0.5 * n, 16.0 + 0.24 * n) : std::max(0.5 * n, 27.0 + 0.23 * n); };
            // columns of nb harmonics x nq radial indices: the read-out takes four or eight indices at a time from three or five
            // on, and its last read may reach past them
            auto width = [&](int nb, int nq) { return (nb * nq + (nq > 4 ? (8 - nq % 8) % 8 : nq == 3 ? 1 : 0) + gran - 1) & ~(gran - 1); };
            double best = 1e30; int best_mask = 0; std::vector<int> best_nq;
            for (int mask = 0; mask < (1 << (nl - 1)); ++mask) {      // bit i: cut after order i
                double cost = 0; std::vector<int> nqs; bool good = true;
                for (int i = 0; i < nl && good;) {
                    int j = i;
                    while (j + 1 < nl && !((mask >> j) & 1)) ++j;
                    const int nb = lboff[j + 1] - lboff[i];
                    int nout = 0;
                    for (const Pth& t : B.paths) if (t.lb >= lbs[i] && t.lb <= lbs[j]) nout += t.P->d_dst;
                    // as many radial indices as fit, in equal units; then the cheapest count by products and read-out steps (some
                    // 8 + 4 R cycles per component)
                    double c_best = 1e30; int nq = 0;
                    for (int t = 1; t <= KH; ++t) {
                        if (width(nb, t) > cap) break;
                        const int nu = (KH + t - 1) / t;
                        const double c = nu * (B.d * 3.0 * cycles(width(nb, t)) + nout * (8.0 + 4.0 * (t > 4 ? 8 : (t > 2 ? 4 : t))));
                        if (c <= c_best) { c_best = c; nq = t; }
                    }
                    if (!nq) { good = false; break; }
                    cost += c_best;
                    nqs.push_back(nq);
                    i = j + 1;
                }
                if (good && cost < best) { best = cost; best_mask = mask; best_nq = nqs; }
            }
            if (best > 1e29) { ok = false; break; }
            for (int i = 0, gi = 0; i < nl; ++gi) {
                int j = i;
                while (j + 1 < nl && !((best_mask >> j) & 1)) ++j;
                const int nb = lboff[j + 1] - lboff[i], nq = best_nq[gi];
                MUnit U{};
                U.d_src = B.d; U.halves = halves; U.N = width(nb, nq); U.nq = nq; U.c = parts[pi].c; U.c_row = B.c;
                // columns: radial index fastest, so that one read-out instruction takes several of them
                U.row_begin = (int)T.rows.size();
                for (int h = 0; h < halves; ++h)
                    for (int n = 0; n < U.N; ++n) {
                        if (n >= nb * nq) { T.rows.push_back(0xffff); continue; }
                        int r = n / nq, b = 0;
                        for (int k = i; k <= j; ++k) { const int db = 2 * lbs[k] + 1; if (r < db) { b = lbs[k] * lbs[k] + r; break; } r -= db; }
                        T.rows.push_back((uint16_t)(((n % nq) * halves + h) | (b << 8)));
                    }
                U.out_begin = (int)T.outs.size();
                for (int k = i; k <= j; ++k)
                    for (const Pth& t : B.paths) {
                        if (t.lb != lbs[k]) continue;
                        for (int o = 0; o < t.P->d_dst; ++o) {
                            const int ld = dir.nk_ld[t.group];
                            MOut e{(int64_t)o * ld + t.P->koff + parts[pi].u0, dir.zb_off[t.group], t.P->d_dst * ld, (int)T.terms.size(), 0, 0};
                            for (int sc = 0; sc < B.d; ++sc)
                                for (int z = p->tab_ptr[t.P->tabM + sc * t.P->d_dst + o]; z < p->tab_ptr[t.P->tabM + sc * t.P->d_dst + o + 1]; ++z)
                                    T.terms.push_back(MTerm{(uint32_t)(sc * U.N + (lboff[k] - lboff[i] + p->tab_idx[z]) * nq), p->tab_coef[z]});
                            if ((int)T.terms.size() == e.term) T.terms.push_back(MTerm{0, 0.f});
                            if ((T.terms.size() - e.term) & 1) T.terms.push_back(MTerm{T.terms.back().col, 0.f});
                            e.n = (int)T.terms.size() - e.term;
                            T.outs.push_back(e);
                        }
                    }
                U.n_out = (int)T.outs.size() - U.out_begin;
                max_rows = std::max(max_rows, U.N * halves);
                for (int q0 = 0; q0 < p->K; q0 += nq * halves) { U.q0 = q0; units[pi].push_back(U); }
                i = j + 1;
            }
        }
        if (!ok) { T = MomentSets{}; continue; }
        size_t n_units = 0;
        for (const auto& u : units) n_units += u.size();
        T.w_bytes = max_rows * 64;
        const int tables = (int)(T.outs.size() * sizeof(MOut) + T.terms.size() * sizeof(MTerm) + parts.size() * (sizeof(MSet) + sizeof(MBlk)) + n_units * sizeof(MUnit) +
                                 T.rows.size() * 2 + 64);
        const int fixed = 1024 + MS_NW * T.w_bytes + MS_NBAR * 8 + 16 + tables;
        // Sets: consecutive parts whose rows of 16 edges leave room for four slots (a node of 32 edges and the next one's
        // first rows); a wider part is a set of its own with the slots it leaves, at least two.
        const int slot4 = ((kSmem - fixed) / 4) & ~1023;
        int x_cap = 0;
        for (size_t i = 0; i < parts.size();) {
            MSet S{};
            S.blk_begin = (int)T.blks.size(); S.unit_begin = (int)T.units.size();
            int slabs = 0;
            size_t j = i;
            for (; j < parts.size(); ++j) {
                const Blk& B = blocks[parts[j].blk];
                const int nch = (parts[j].c + 63) / 64;
                if (j > i && 2 * (slabs + B.d * nch) * MS_SLAB + raw > slot4) break;
                T.blks.push_back(MBlk{B.so + parts[j].u0, parts[j].c, B.c, B.d, slabs, nch, {0, 0}});
                for (MUnit U : units[j]) { U.slab0 = slabs; T.units.push_back(U); }
                slabs += B.d * nch;
            }
            S.nblk = (int)T.blks.size() - S.blk_begin; S.nunit = (int)T.units.size() - S.unit_begin;
            T.sets.push_back(S);
            x_cap = std::max(x_cap, slabs * MS_SLAB);
            i = j;
        }
        T.x_cap = x_cap;
        T.slot_bytes = 2 * x_cap + raw;
        T.ns = std::min(MS_MAXNS, (kSmem - fixed) / T.slot_bytes);
        T.smem_bytes = fixed + T.ns * T.slot_bytes;
        T.ok = T.ns >= 2;
    }
}

cudaError_t launch_moment_stream(const sobek_plan* p, const Direction& dir, const EdgeView& ev, int64_t node0, int64_t n_nodes,
                                 const SplitSrc& ss, const float* Y, const float* vY, const float* phi, const float* vphi, int dual,
                                 void* zh, void* zl, int* status, cudaStream_t s) {
    const MomentSets& T = dir.ms[dual ? 1 : 0];
    if (!T.ok || !ss.h || !ss.l) return cudaErrorInvalidValue;
    if (n_nodes <= 0) return cudaSuccess;
    MsArgs a{};
    a.sets = T.d_sets; a.blks = T.d_blks; a.units = T.d_units; a.outs = T.d_outs; a.terms = T.d_terms; a.rows = T.d_rows;
    a.nsets = (int)T.sets.size(); a.n_blks = (int)T.blks.size(); a.n_units = (int)T.units.size(); a.n_terms = (int)T.terms.size();
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
    a.x_cap = T.x_cap; a.slot_bytes = T.slot_bytes; a.ns = T.ns; a.w_bytes = T.w_bytes;
    a.status = status;
    const int grid = (int)std::min<int64_t>(n_nodes * a.nsets, (int64_t)148);
    KernelTimer kt(K_STATE, s);
    const cudaError_t e = dual ? moment_stream_dual(a, grid, T.smem_bytes, s) : moment_stream_plain(a, grid, T.smem_bytes, s);
    count_launch();
    return e;
}

}  // namespace sobek
