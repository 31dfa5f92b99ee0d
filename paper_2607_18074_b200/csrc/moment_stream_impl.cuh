// Edge stream in moment form (sm_100a, tcgen05 / TMEM), warp-specialised.
//
// The receiver state (Eqs. angular_path_contraction, receiver_state)
//     Z_i[path, o, q, u] = sum_e phi_e[q] sum_{s,b} c[s,b,o] Y_e[b] x_{src(e)}[s,u]
// is linear in the edge's outer product, so the Clebsch-Gordan coefficients come out of the sum over the edges:
//     P_i[q,b,s,u] = sum_e (phi_e[q] Y_e[b]) x_{src(e)}[s,u]          (moments of the neighbourhood, no coupling in them)
//     Z_i[path, o, q, u] = sum_{s,b} c[s,b,o] P_i[q,b,s,u]            (once per node)
// The first line is a dense contraction over the edges: per component s of a source block
//     D_s[u, (q,b)] = sum_e x_e[s,u] W_e[(q,b)],    W_e[(q,b)] = phi_e[q] Y_e[b],
// whose first operand is the gathered sender rows as they lie in memory and whose second is K x (harmonics) values per edge,
// whatever the multiplicity, the number of paths or their order.  The second line is a sparse sum (1.9 terms per moment at order 4)
// over the node's moments, independent of its degree.  Building the contraction's operand with the coupling folded in
// (phi_e[q] M_e[s,o]) takes K sum d_src d_dst values per edge instead: 1,840 against 144 at 64 x (0..2), K = 16, 20,832 against
// 400 at 64 x (0..4), and that build bound the kernel.  fp32 parity comes from the split-bf16 product
// a*b ~= a_hi*b_hi + a_hi*b_lo + a_lo*b_hi with fp32 accumulation in TMEM; the coupling sums run in fp32.
//
// Work items are (set, node): a set is a run of source blocks (64 multiplicities at most each, wider ones are cut) whose gathered
// rows of 16 edges fit one slot of the shared-memory ring.  W of a group of radial indices is built once per slot; an item's
// accumulators are then produced unit after unit: a unit is a run of components x a run of W's rows, at most 256 TMEM columns, so
// that the two TMEM halves alternate between products and read-out.  The products have M = 64, whose 64 rows take 16 lanes of
// each 32-lane quarter: the even radial indices go to the lower 16, the odd ones to the upper 16, and every lane has work in the
// read-out.  (M = 128 for wider blocks has half the products but needs slots twice as large: 128 x (0..2) ran 3 to 17 % slower.)
// When the slots of a node's edges all fit the rings they stay there for all units; longer segments are gathered again for every
// two units, whose accumulators then fill both TMEM halves side by side (the products of such a segment outlast the read-out).
//   loader warps   cp.async of the sender rows (MN-major, 128-byte swizzle) into the ring;
//   edge warp      phi and Y (transposed) into the ring, from memory or computed from the edge vectors (LE: the loader warps, from memory);
//   builder warps  W of one (group, slot): thread <-> (row (q,b), eight edges), bf16 hi / lo, K-major;
//   MMA warps      one per TMEM half, each with every second unit: one elected lane issues the three products per component and lane
//                  half.  (The steps around a slot's products take a warp about as long as the products themselves.)
//   drain warps    four teams of four warps (one per TMEM lane quarter) that share the state components of a unit: a lane holds one
//                  multiplicity, sums the coupling terms and writes bf16 hi / lo.  Rows of up to 32 multiplicities are gathered twice
//                  (up to 16: four times) side by side, so that no lane quarter is left without work.  All of them work on one accumulator while the
//                  other is filled: with a group of its own for each, the read-out took twice as long as the products and both
//                  waited a third of the time.
// All waits suspend their warp: polling ones took half of the issued instructions (64 x (0..2), K = 16, degree 32: 43.6 thousand
// a node), and without them the kernel is 5 to 9 % faster.
// With DUAL the kernel produces the directional state of the double backward (Eq. receiver_double_adjoint)
//     dP = sum_e (vphi Y + phi vY)[q,b] x[s,u] + (phi Y)[q,b] vx[s,u]
// as two slots per batch of edges.  The same kernel runs the sender-owned transposed traversal.  Every wait is bounded.
#pragma once
#include <cuda_bf16.h>

#include <algorithm>

#include "geometry.cuh"
#include "guard.cuh"
#include "moment_stream.h"
#include "ptx.cuh"

namespace sobek {
namespace {

using namespace ptx;

__device__ __forceinline__ int64_t owner_of(const int64_t* __restrict__ row_ptr, int64_t N, int64_t e) {
    int64_t lo = 0, hi = N;   // row_ptr[lo] <= e < row_ptr[hi]
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (__ldg(row_ptr + mid) <= e) lo = mid; else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4_zfill(uint32_t dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
// R consecutive columns of this thread's TMEM lane, not waited for
template <int R>
__device__ __forceinline__ void tm_ld(uint32_t t, float* p) {
    if constexpr (R == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(p[0]), "=f"(p[1]), "=f"(p[2]), "=f"(p[3]), "=f"(p[4]), "=f"(p[5]), "=f"(p[6]), "=f"(p[7]) : "r"(t) : "memory");
    else if constexpr (R == 4)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=f"(p[0]), "=f"(p[1]), "=f"(p[2]), "=f"(p[3]) : "r"(t) : "memory");
    else if constexpr (R == 2)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=f"(p[0]), "=f"(p[1]) : "r"(t) : "memory");
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=f"(p[0]) : "r"(t) : "memory");
}
// acc0 and acc1 += S steps of the coupling terms at tp, {column, coefficient} of either, summed straight out of TMEM
template <int R, int S>
__device__ __forceinline__ void add_terms(uint32_t t, const uint4* tp, float* acc0, float* acc1) {
    uint4 c[S];
    float p[2 * S][R];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        c[s] = tp[s];
        tm_ld<R>(t + c[s].x, p[2 * s]);
        tm_ld<R>(t + c[s].z, p[2 * s + 1]);
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int s = 0; s < 2 * S; ++s) {
        float* const acc = s & 1 ? acc1 : acc0;
        const float k = __uint_as_float(s & 1 ? c[s / 2].w : c[s / 2].y);
#pragma unroll
        for (int r = 0; r < R; ++r) asm volatile("" : "+f"(p[s][r]));      // (no use of a loaded value moves above the wait)
        if constexpr (R == 1) acc[0] = fmaf(k, p[s][0], acc[0]);
        else
#pragma unroll
            for (int r = 0; r < R; r += 2) unpack2(fma2(pack2(k, k), pack2(p[s][r], p[s][r + 1]), pack2(acc[r], acc[r + 1])), acc[r], acc[r + 1]);
    }
}
__device__ __forceinline__ void st_b32_if(uint32_t ok, void* p, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.global.b32 [%0], %1;\n\t}" ::"l"(p), "r"(v), "r"(ok) : "memory");
}
// One component, one run of radial indices from q0 on, into the state.  A whole run of 2 R radial indices leaves in the order that a
// lane holds it (state_pos with zq = R): 4 R bytes, one store each for the hi and the lo parts.
template <int R>
__device__ __forceinline__ void put_state(const MsArgs& a, const MOut& e, const float* acc, int nl, int q0, int u, int qh, bool ok) {
    const int64_t zr = e.a + (int64_t)nl * e.b + q0 * e.c;
    if (R > 1 && a.interleaved && q0 + 2 * R <= a.K) {
        constexpr int W = R > 1 ? R / 2 : 1;
        uint32_t hi[W], lo[W];
#pragma unroll
        for (int r = 0; r + 1 < R; r += 2) split2(pack2(acc[r], acc[r + 1]), hi[r / 2], lo[r / 2]);
        const int64_t z = zr + (qh * e.c + e.u0 + u) * R;
        if (ok) {
            if constexpr (R == 8) {
                *reinterpret_cast<uint4*>(a.zh + z) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                *reinterpret_cast<uint4*>(a.zl + z) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            } else if constexpr (R == 4) {
                *reinterpret_cast<uint2*>(a.zh + z) = make_uint2(hi[0], hi[1]);
                *reinterpret_cast<uint2*>(a.zl + z) = make_uint2(lo[0], lo[1]);
            } else {
                *reinterpret_cast<uint32_t*>(a.zh + z) = hi[0];
                *reinterpret_cast<uint32_t*>(a.zl + z) = lo[0];
            }
        }
    } else {
        // q-major.  Two neighbouring lanes swap halves: the even one writes the hi, the odd one the lo parts of both multiplicities.
        const uint32_t sel = u & 1 ? 0x1054u : 0x7632u;
        __nv_bfloat16* z = (u & 1 ? a.zl + u - 1 : a.zh + u) + zr + e.u0 + qh * e.c;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            uint32_t w, x;         // the value's bf16 in the high half, zero below: its fp32 pattern; then hi and lo together
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(acc[r]), "f"(0.f));
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(x) : "f"(acc[r]), "f"(acc[r] - __uint_as_float(w)));
            st_b32_if(ok && q0 + 2 * r + qh < a.K, z, __byte_perm(x, __shfl_xor_sync(0xffffffffu, x, 1), sel));
            z += 2 * e.c;
        }
    }
}

// Read-out of a unit by one warp: every n_team-th pair of components of the state, R radial indices (columns) at a time.  The coupling
// terms come from a table; TMEM serves the repeated reads at some ten cycles each.  A warp spends its time in the latency of one
// table entry, one TMEM read, one sum and one split after another (450 cycles a component with the terms and the stores left out), so
// two components go side by side.  (Unrolled over the terms with immediate coefficients, a function for every (source order, harmonic
// order), the kernel took 25.4 instead of 21.2 thousand cycles a node at 64 x (0..2), K = 16, degree 32.)
template <int R>
__device__ __forceinline__ void read_out(const MsArgs& a, const MUnit& U, const MOut* outs, const MTerm* terms, uint32_t t0, bool full, int nl,
                                         int first, int n_team, int u, int qh) {
    const int n_pair = U.n_pair, nqs = U.nqs, rows_q = U.rows_q;
    const bool lane_ok = u < U.c;
    outs += U.out_begin;
#pragma unroll 1
    for (int o = first; o < n_pair; o += n_team) {
        const MOut* const e = outs + 2 * o;
        uint32_t t = t0;
        int q0 = U.q0;
#pragma unroll 1
        for (int qc = 0; qc < nqs; ++qc, t += (uint32_t)rows_q, q0 += 2 * R) {
            float acc0[R], acc1[R];
#pragma unroll
            for (int r = 0; r < R; ++r) acc0[r] = acc1[r] = 0.f;
            const uint4* tp = reinterpret_cast<const uint4*>(terms + e->term);
            int n = full ? e->n : 0;
            constexpr int S = R == 8 ? 1 : 2;
#pragma unroll 1
            for (; n >= S; n -= S, tp += S) add_terms<R, S>(t, tp, acc0, acc1);
            if (S > 1 && n) add_terms<R, 1>(t, tp, acc0, acc1);
            put_state<R>(a, e[0], acc0, nl, q0, u, qh, lane_ok);
            put_state<R>(a, e[1], acc1, nl, q0, u, qh, lane_ok && e[1].c);
        }
    }
}

// Every role walks the same items; the next item's bounds are requested one item ahead.
struct MsItem { int set, nl, seg0, len, nslot; bool resident; };        // (node counts and edge counts are below 2^31)
struct MsWalk {
    const MsArgs& a;
    uint32_t v;
    int nl, s0, s1, set, nsub;
    int* st;
    __device__ MsWalk(const MsArgs& a_, int nsub_, int* st_) : a(a_), nl(0), s0(0), s1(0), nsub(nsub_), st(st_) {
        v = blockIdx.x % (uint32_t)a.n_nodes; set = (int)(blockIdx.x / (uint32_t)a.n_nodes);
        fetch();
    }
    __device__ void fetch() {
        if (set >= a.nsets) return;
        if (a.oseg) { const int4 q = __ldg(a.oseg + v); nl = q.x; s0 = q.y; s1 = q.z; return; }
        int64_t b, e;
        seg_bounds(a.ev.ptr, a.node0 + v, a.ev.E, st, b, e);
        nl = (int)v; s0 = (int)b; s1 = (int)e;
    }
    __device__ bool next(MsItem& it) {
        if (set >= a.nsets) return false;
        it.set = set; it.nl = nl; it.seg0 = s0; it.len = nsub ? s1 - s0 : 0;
        it.nslot = ((it.len + MS_TB - 1) / MS_TB) * nsub;
        it.resident = it.nslot <= min(a.ns, a.nw);
        v += gridDim.x;
        while (v >= (uint32_t)a.n_nodes && set < a.nsets) { v -= (uint32_t)a.n_nodes; ++set; }
        fetch();
        return true;
    }
};

// The slots in the order in which the roles meet them: for every item its passes over the edges, for every batch its operands.
struct MsSlots {
    MsWalk walk;
    MsItem it{};
    const MSet* sets;
    int nsub, rep = 0, nrep = 0, b0 = 0, sub = 0;
    __device__ MsSlots(const MsArgs& a, const MSet* s, int n, int* st) : walk(a, n, st), sets(s), nsub(n) {}
    __device__ bool first() {
        for (;;) {
            if (!walk.next(it)) return false;
            if (it.len == 0) continue;
            rep = 0; b0 = 0; sub = 0; nrep = it.resident ? 1 : sets[it.set].npass;
            return true;
        }
    }
    __device__ bool next() {
        if (++sub < nsub) return true;
        sub = 0; b0 += MS_TB;
        if (b0 < it.len) return true;
        b0 = 0;
        return ++rep < nrep || first();
    }
};

// The products of one slot: x_hi W_hi, x_hi W_lo, x_lo W_hi per component and lane half.  (x_hi stays in the collector for two
// products of one lane half; a product into the other half does not find it there.)
__device__ __forceinline__ void ms_issue(uint32_t d, uint32_t d0, uint64_t dX, uint32_t xlo16, uint64_t dW, uint32_t wlo16, uint32_t whalf16, uint32_t N,
                                         uint32_t idesc, uint32_t acc) {
#pragma unroll 2
    for (uint32_t s = 0; s < d; ++s, d0 += N, dX += MS_SLAB >> 4)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t w = dW + (h ? whalf16 : 0u);
            tc_mma_bf16_x3(d0 + (uint32_t)(h * 16 << 16), dX, dX + xlo16, w, w + wlo16, idesc, acc);
        }
}

// phi and Y (and their directions) of edge ee into a slot's transposed rows, every second radial index and harmonic from hf on
template <bool DUAL>
__device__ __forceinline__ void ms_edge_rows(const MsArgs& a, uint32_t raw, int64_t ee, uint32_t n, bool has_vphi, bool has_vY, int le, int hf) {
    uint32_t d = raw + (uint32_t)((hf * MS_PS + le) * 4);
    const uint32_t dv = (uint32_t)((a.K + a.dsh) * MS_PS * 4);
    const float* p = a.phi + ee * a.K;
    const float* pv = DUAL && has_vphi ? a.vphi + ee * a.K : p;
    for (int q = hf; q < a.K; q += 2, d += 2 * MS_PS * 4) {
        cp_async4_zfill(d, p + q, n);
        if (DUAL && has_vphi) cp_async4_zfill(d + dv, pv + q, n);
    }
    d = raw + (uint32_t)(((a.K + hf) * MS_PS + le) * 4);
    p = a.Y + ee * a.dsh;
    pv = DUAL && has_vY ? a.vY + ee * a.dsh : p;
    for (int b = hf; b < a.dsh; b += 2, d += 2 * MS_PS * 4) {
        cp_async4_zfill(d, p + b, n);
        if (DUAL && has_vY) cp_async4_zfill(d + dv, pv + b, n);
    }
}

// LE: the loader warps copy phi and Y as well (stored edge inputs only).  One warp for the edge rows of every slot bounds the nodes whose
// read-out is short, four share them among the loaders (64 x 0 -> 64 x 0, K = 8, 5,206 nodes of degree 11: 64 -> 52 us; 128 x 0 -> 128 x (0, 2),
// K = 16, degree 6, dual: 119 -> 97 us); behind a long read-out the loaders are the longer chain (64 x (0..2), K = 16: 171 -> 176 us).
template <bool DUAL, bool LE>
__global__ void __launch_bounds__(MS_TT, 1) k_moment_stream(const MsArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);       // (keeps the pointer in the shared address space)
    constexpr int TB = MS_TB, PS = MS_PS, SLAB = MS_SLAB, HALF = MS_HALF;
    constexpr int NLW = MS_NLW, NBW = MS_NBW, NDW = MS_NDW, W_LOAD = NDW, W_BUILD = W_LOAD + NLW, W_MMA = W_BUILD + NBW, W_EDGE = W_MMA + 2;
    const int NS = a.ns, NW = a.nw;
    uint8_t* sRing = smem;                                            // slots: x hi, x lo, raw phi / Y (+ directions)
    uint8_t* sW = sRing + (size_t)NS * a.slot_bytes;                  // W ring: hi rows, lo rows
    uint64_t* bars = reinterpret_cast<uint64_t*>(sW + (size_t)NW * a.w_bytes);
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + MS_NBAR);
    MTerm* sTerm = reinterpret_cast<MTerm*>(tmem_holder + 4);
    MOut* sOut = reinterpret_cast<MOut*>(sTerm + a.n_terms);
    MSet* sSet = reinterpret_cast<MSet*>(sOut + a.n_outs);
    MGrp* sGrp = reinterpret_cast<MGrp*>(sSet + a.nsets);
    MSlab* sSlab = reinterpret_cast<MSlab*>(sGrp + a.n_grps);
    MUnit* sUnit = reinterpret_cast<MUnit*>(sSlab + a.n_slabs);
    uint16_t* sRow = reinterpret_cast<uint16_t*>(sUnit + a.n_units);
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t bar_full = bar0, bar_sfree = bar0 + 8 * MS_MAXNS, bar_wfull = bar0 + 16 * MS_MAXNS, bar_wfree = bar_wfull + 8 * MS_MAXNW,
                   bar_accfull = bar_wfree + 8 * MS_MAXNW, bar_accfree = bar_accfull + 16;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool has_vx = DUAL && a.vsh != nullptr, has_vY = DUAL && (a.rvec ? a.vrvec != nullptr : a.vY != nullptr),
               has_vphi = DUAL && (a.rvec ? a.vrvec != nullptr : a.vphi != nullptr);
    const bool has_a1 = !DUAL || has_vY || has_vphi;   // operand 1: phi Y (plain) or vphi Y + phi vY (dual), times x
    const bool has_a2 = has_vx;                        // operand 2 (dual): phi Y, times vx
    const int nsub = (has_a1 ? 1 : 0) + (has_a2 ? 1 : 0);

    if (tid == 0) {
        for (int s = 0; s < MS_MAXNS; ++s) { mbar_init(bar_full + 8 * s, LE ? 32 : 64); mbar_init(bar_sfree + 8 * s, 2); }
        for (int s = 0; s < MS_MAXNW; ++s) { mbar_init(bar_wfull + 8 * s, NBW * 32); mbar_init(bar_wfree + 8 * s, 2); }
        for (int t = 0; t < 2; ++t) { mbar_init(bar_accfull + 8 * t, 1); mbar_init(bar_accfree + 8 * t, 4 * MS_NDT); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    {   // raw rows of absent directions stay zero for ever
        const int words = a.slot_bytes / 4, x_words = 2 * a.x_cap / 4;
        for (int s = 0; s < NS; ++s)
            for (int i = x_words + tid; i < words; i += MS_TT) reinterpret_cast<uint32_t*>(sRing + (size_t)s * a.slot_bytes)[i] = 0u;
    }
    auto table = [&](void* dst, const void* src, int bytes) {
        for (int i = tid; i < bytes / 2; i += MS_TT) reinterpret_cast<uint16_t*>(dst)[i] = reinterpret_cast<const uint16_t*>(src)[i];
    };
    table(sTerm, a.terms, a.n_terms * (int)sizeof(MTerm)); table(sSet, a.sets, a.nsets * (int)sizeof(MSet));
    table(sGrp, a.grps, a.n_grps * (int)sizeof(MGrp));
    table(sSlab, a.slabs, a.n_slabs * (int)sizeof(MSlab)); table(sUnit, a.units, a.n_units * (int)sizeof(MUnit)); table(sRow, a.rows, a.n_rows * 2);
    for (int i = tid; i < a.n_outs; i += MS_TT) {
        MOut e = a.outs[i];
        e.a += a.n_nodes * (int64_t)e.zoff;         // the groups of a chunk's state lie one after another
        sOut[i] = e;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;

    if (warp >= W_LOAD && warp < W_LOAD + NLW) {
        // =========================== loader warps ===========================
        // A slot is filled by one warp alone, the warps take turns: a warp spends most of its time on index arithmetic, a few cycles
        // an instruction whatever the others do.  (All four on one slot: 32 x (0..2) forward 312 instead of 294 us, 128/64/64
        // backward at degree 255, whose slots did not stay, 6.8 instead of 4.9 ms.  TMA gathers of four rows: 3 to 20 % slower.)
        const int me = warp - W_LOAD;
        MsSlots at(a, sSet, nsub, a.status);
        // Lane e < 16 holds edge e of the batch.  The ids of the next batch are requested one batch ahead and not looked at before
        // their turn (an id out of range turns the edge's copies into zero fills and is reported in the status word).
        struct Ids { int v, e; bool in; };
        auto request = [&]() -> Ids {
            Ids d{0, 0, at.b0 + lane < at.it.len && lane < TB};
            if (d.in) {
                const int pos = at.it.seg0 + at.b0 + lane;
                if (!a.ev.transposed) d.v = a.ev.col[pos];
                else d.v = a.ev.recv ? a.ev.recv[pos] : a.ev.perm[pos];
                if (LE) d.e = a.ev.perm ? a.ev.perm[pos] : pos;
            }
            return d;
        };
        int st = 0; uint32_t round = 0;      // of the slot at hand
        // its index mod the number of warps that take part: no more than slots, so that the free barrier of a slot is never waited
        // for two phases ahead
        const int nlw = min(NLW, NS);
        int turn = 0;
        auto to_mine = [&](bool first) -> bool {
            bool more = first ? at.first() : at.next();
            if (!first) { if (++st == NS) { st = 0; ++round; } if (++turn == nlw) turn = 0; }
            while (more && turn != me) {
                more = at.next();
                if (++st == NS) { st = 0; ++round; }
                if (++turn == nlw) turn = 0;
            }
            return more;
        };
        // 16 bytes = 8 multiplicities per copy: lane <-> piece j of eight rows' pieces; its four edges are lane / 8 + 0, 4, 8, 12
        const int j = lane & 7, e0 = lane >> 3;
        bool have = me < nlw && to_mine(true);
        Ids ids{0, 0, false};
        if (have) ids = request();
        while (have) {
            const int st_now = st; const uint32_t round_now = round;
            const MSet& S = sSet[at.it.set];
            int slab0 = 0, slab1 = S.nslab;
            if (!at.it.resident) {          // two units' turn: their slabs only (the same for every group)
                const MGrp& G = sGrp[S.grp_begin];
                const int u0 = 2 * (at.rep % S.gpass);
                const MUnit& U = sUnit[G.unit_begin + u0];
                const MUnit& V = sUnit[G.unit_begin + min(u0 + 1, G.nunit - 1)];
                slab0 = U.slab0; slab1 = V.slab0 + V.d;
            }
            const MSlab* const slabs = sSlab + S.slab_begin;
            const int op = has_a1 ? at.sub : 1;
            bool ok = ids.in;
            int sn = ids.v;
            if (ok && a.ev.transposed && !a.ev.recv) {
                ok = id_ok(sn, a.ev.E, a.status);
                if (ok) sn = (int)owner_of(a.ev.row_ptr, a.ev.N, sn);
            }
            ok = ok && id_ok(sn, a.ev.N, a.status);
            if (!ok) sn = 0;
            const uint32_t msk = __ballot_sync(0xffffffffu, ok);
            const int eid = LE && ids.in && id_ok(ids.e, a.ev.E, a.status) ? ids.e : -1;
            have = to_mine(false);
            if (have) ids = request();
            if (round_now > 0) mbar_wait(bar_sfree + 8 * st_now, (round_now & 1) ^ 1, a.status);
            if (LE) {
                const int ee = __shfl_sync(0xffffffffu, eid, lane & (TB - 1));
                ms_edge_rows<DUAL>(a, smem_u32(sRing + (size_t)st_now * a.slot_bytes + (size_t)2 * a.x_cap), ee < 0 ? 0 : ee, ee < 0 ? 0u : 4u, has_vphi, has_vY,
                                   lane & (TB - 1), lane >> 4);
            }
            const __nv_bfloat16* const baseh = op == 0 ? a.sh : a.vsh;
            const int64_t to_lo = (op == 0 ? a.sl : a.vsl) - baseh;
            const __nv_bfloat16* row[4];
            uint32_t n[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                row[i] = baseh + (int64_t)__shfl_sync(0xffffffffu, sn, e0 + 4 * i) * a.C_src;
                n[i] = ((msk >> (e0 + 4 * i)) & 1u) * 16u;
            }
            uint32_t dst = smem_u32(sRing + (size_t)st_now * a.slot_bytes) + (uint32_t)(slab0 * SLAB + e0 * 128 + ((j ^ e0) << 4));
#pragma unroll 1
            for (int k = slab0; k < slab1; ++k, dst += (uint32_t)SLAB) {
                const MSlab B = slabs[k];
                const int js = j & B.mask;
                if (js < B.chunks) {
                    const int off = B.off + 8 * js;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t d = (i & 1 ? dst ^ 64u : dst) + (uint32_t)(i * 512);
                        cp_async16_zfill(d, row[i] + off, n[i]);
                        cp_async16_zfill(d + (uint32_t)a.x_cap, row[i] + off + to_lo, n[i]);
                    }
                }
            }
            // this thread's arrival on the slot's barrier fires when all its copies above have landed
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar_full + 8 * st_now) : "memory");
        }
    } else if (!LE && warp == W_EDGE) {
        // =========================== edge warp ===========================
        // Walks the same slots as the loaders and fills their phi and Y rows, transposed: from memory, or computed from the edge vectors
        // (lane <-> edge lane & 15, half of the radial indices / harmonics each).
        if (a.rvec == nullptr) {
            MsSlots at(a, sSet, nsub, nullptr);
            const int le = lane & (TB - 1), hf = lane >> 4;
            int st = 0; uint32_t round = 0;
            auto request = [&](bool have, bool& in) -> int {       // one slot ahead
                in = have && at.b0 + le < at.it.len;
                const int pos = at.it.seg0 + at.b0 + le;
                return in && a.ev.perm ? a.ev.perm[pos] : pos;
            };
            bool have = at.first(), in;
            int e = request(have, in);
            while (have) {
                const bool ok = in && id_ok(e, a.ev.E, a.status);
                const int64_t ee = ok ? e : 0;
                const uint32_t n = ok ? 4u : 0u;
                have = at.next();
                e = request(have, in);
                if (round > 0) mbar_wait(bar_sfree + 8 * st, (round & 1) ^ 1, a.status);
                ms_edge_rows<DUAL>(a, smem_u32(sRing + (size_t)st * a.slot_bytes + (size_t)2 * a.x_cap), ee, n, has_vphi, has_vY, le, hf);
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar_full + 8 * st) : "memory");
                if (++st == NS) { st = 0; ++round; }
            }
        }
        if (a.rvec != nullptr) {
            MsWalk walk(a, nsub, nullptr);
            MsItem it{};
            const int le = lane & (TB - 1), hf = lane >> 4;
            int st = 0; uint32_t round = 0;
            while (walk.next(it)) {
                if (it.len == 0) continue;
                const int nrep = it.resident ? 1 : sSet[it.set].npass;
                for (int rep = 0; rep < nrep; ++rep)
                for (int b0 = 0; b0 < it.len; b0 += TB) {
                    bool okb = b0 + le < it.len;
                    int64_t ee = 0;
                    if (okb) { const int pos = it.seg0 + b0 + le; ee = a.ev.perm ? a.ev.perm[pos] : pos; okb = id_ok(ee, a.ev.E, a.status); }
                    float rx = 0.f, ry = 0.f, rz = 1.f;
                    if (okb) { const float* rp = a.rvec + ee * 3; rx = __ldg(rp); ry = __ldg(rp + 1); rz = __ldg(rp + 2); }
                    const float r = sqrtf(rx * rx + ry * ry + rz * rz), ir = 1.f / r;
                    const float ux = rx * ir, uy = ry * ir, uz = rz * ir;
                    // DUAL: the directions vphi = phi'(r) (u . v) and vY = grad F . (v - u (u . v)) / r of the edge-vector direction v
                    float uv = 0.f, tx = 0.f, ty = 0.f, tz = 0.f;
                    const bool dirs = DUAL && a.vrvec != nullptr;
                    if (dirs && okb) {
                        const float* vp = a.vrvec + ee * 3;
                        const float vx_ = __ldg(vp), vy_ = __ldg(vp + 1), vz_ = __ldg(vp + 2);
                        uv = ux * vx_ + uy * vy_ + uz * vz_;
                        tx = (vx_ - ux * uv) * ir; ty = (vy_ - uy * uv) * ir; tz = (vz_ - uz * uv) * ir;
                    }
                    for (int sub = 0; sub < nsub; ++sub) {       // the slots of the operand pairs need the same rows
                        if (round > 0) mbar_wait(bar_sfree + 8 * st, (round & 1) ^ 1, a.status);
                        float* F = reinterpret_cast<float*>(sRing + (size_t)st * a.slot_bytes + (size_t)2 * a.x_cap);
                        float* Yt = F + a.K * PS;
                        const int dv = (a.K + a.dsh) * PS, dsh = a.dsh;
                        geo_radial(r, a.K, a.geo_rc, a.geo_basis, a.geo_p, [&](int q, float f, float df) {
                            if ((q & 1) == hf) {
                                F[q * PS + le] = okb ? f : 0.f;
                                if (dirs) F[dv + q * PS + le] = okb ? df * uv : 0.f;
                            }
                        });
                        geo_sh(ux, uy, uz, [&](int b, float yb, float fx, float fy, float fz) {
                            if (b < dsh && (b & 1) == hf) {
                                Yt[b * PS + le] = okb ? yb : 0.f;
                                if (dirs) Yt[dv + b * PS + le] = okb ? fx * tx + fy * ty + fz * tz : 0.f;
                            }
                        });
                        mbar_arrive(bar_full + 8 * st);      // release: the stores above are visible to whoever sees the slot full
                        if (++st == NS) { st = 0; ++round; }
                    }
                }
            }
        }
    } else if (warp >= W_BUILD && warp < W_BUILD + NBW) {
        // =========================== builder warps ===========================
        const int bt = (warp - W_BUILD) * 32 + lane;
        MsWalk walk(a, nsub, nullptr);
        MsItem it{};
        int st0 = 0; uint32_t r0 = 0;          // slot and round of the item's first slot
        int ws = 0; uint32_t wr = 0;
        while (walk.next(it)) {
            if (it.len == 0) continue;
            const int g0 = sSet[it.set].grp_begin, g1 = g0 + sSet[it.set].ngrp;
            int st = st0; uint32_t rd = r0;
            for (int gi = g0; gi < g1; ++gi)
            for (int ps = 0; ps < (it.resident ? 1 : sSet[it.set].gpass); ++ps) {      // resident: one W for the units of the group
                if (it.resident) { st = st0; rd = r0; }
                const MGrp& G = sGrp[gi];
                const uint16_t* rt = sRow + G.row_begin;
                const int rows = 2 * G.rows, q_first = G.q0;
                int lo = 0, n_lo = rows, hi = 0, n_hi = 0;                             // rows [lo, lo + n_lo) and [hi, hi + n_hi)
                if (!it.resident) {
                    const MUnit& U = sUnit[G.unit_begin + 2 * ps];
                    const MUnit& V = sUnit[G.unit_begin + min(2 * ps + 1, G.nunit - 1)];
                    lo = min(U.row0, V.row0); hi = lo + G.rows;
                    n_lo = n_hi = max(U.row0 + U.N, V.row0 + V.N) - lo;
                }
                for (int j = 0; j < it.nslot; ++j) {
                    const int op = has_a1 ? (nsub == 2 ? (j & 1) : 0) : 1;
                    if (warp == W_BUILD) {
                        mbar_wait(bar_full + 8 * st, rd & 1, a.status);
                        if (wr > 0) mbar_wait(bar_wfree + 8 * ws, (wr & 1) ^ 1, a.status);
                    }
                    asm volatile("bar.sync 3, %0;" ::"n"(MS_NBW * 32) : "memory");
                    const float* F = reinterpret_cast<const float*>(sRing + (size_t)st * a.slot_bytes + (size_t)2 * a.x_cap);
                    const float* Yt = F + a.K * PS;
                    const int dv = (a.K + a.dsh) * PS;
                    uint8_t* w = sW + (size_t)ws * a.w_bytes;
                    auto build = [&](int i) {                  // (row, eight edges)
                        const int m = ((i >> 4) << 3) | (i & 7), h = (i >> 3) & 1, n = m < n_lo ? lo + m : hi + m - n_lo;
                        const uint32_t qb = rt[n];
                        const int q = min(q_first + (int)(qb & 255u), a.K - 1), b = (int)(qb >> 8);   // (indices past K: any value)
                        uint64_t f[4], y[4], v[4];                 // pairs of edges
                        auto row = [&](uint64_t* r, const float* p) {
                            const ulonglong2 p0 = *reinterpret_cast<const ulonglong2*>(p), p1 = *reinterpret_cast<const ulonglong2*>(p + 4);
                            r[0] = p0.x; r[1] = p0.y; r[2] = p1.x; r[3] = p1.y;
                        };
                        row(f, F + q * PS + 8 * h);
                        row(y, Yt + b * PS + 8 * h);
                        if (DUAL && op == 0) {
                            uint64_t vf[4], vy[4];
                            row(vf, F + dv + q * PS + 8 * h);
                            row(vy, Yt + dv + b * PS + 8 * h);
#pragma unroll
                            for (int e = 0; e < 4; ++e) v[e] = fma2(vf[e], y[e], mul2(f[e], vy[e]));
                        } else {
#pragma unroll
                            for (int e = 0; e < 4; ++e) v[e] = mul2(f[e], y[e]);
                        }
                        uint4 hi, lo;
                        split2(v[0], hi.x, lo.x); split2(v[1], hi.y, lo.y); split2(v[2], hi.z, lo.z); split2(v[3], hi.w, lo.w);
                        uint8_t* d = w + (n >> 3) * 256 + h * 128 + (n & 7) * 16;
                        *reinterpret_cast<uint4*>(d) = hi;
                        *reinterpret_cast<uint4*>(d + rows * 32) = lo;
                    };
                    int i = bt;
#pragma unroll 1
                    for (; !DUAL && i + NBW * 32 < 2 * (n_lo + n_hi); i += 2 * NBW * 32) { build(i); build(i + NBW * 32); }
#pragma unroll 1
                    for (; i < 2 * (n_lo + n_hi); i += NBW * 32) build(i);
                    fence_async_smem();
                    mbar_arrive(bar_wfull + 8 * ws);
                    if (++ws == NW) { ws = 0; ++wr; }
                    if (++st == NS) { st = 0; ++rd; }
                }
            }
            st0 = st; r0 = rd;
        }
    } else if (warp == W_MMA || warp == W_MMA + 1) {
        // =========================== MMA warps: one for each TMEM half, the units go to them in turn ===========================
        // Both follow every slot and every entry of W: each of these is free when both have passed it, and neither arrives there a
        // second time before it is full again.
        const uint32_t me = __shfl_sync(0xffffffffu, (uint32_t)(warp - W_MMA), 0);
        MsWalk walk(a, nsub, nullptr);
        MsItem it{};
        int st0 = 0; uint32_t r0 = 0;
        int ws = 0; uint32_t wr = 0, ai = 0;
        const uint32_t d0 = __shfl_sync(0xffffffffu, tmem_base, 0) + me * HALF;
        const uint64_t dX0 = make_desc(smem_u32(sRing), SLAB, 1024);          // 64 multiplicities per row
        const uint64_t dW0 = make_desc_plain(smem_u32(sW), 128, 256);
        const uint32_t slot16 = (uint32_t)a.slot_bytes >> 4, w16 = (uint32_t)a.w_bytes >> 4, xlo16 = (uint32_t)a.x_cap >> 4;
        while (walk.next(it)) {
            if (it.len == 0) continue;
            const int g0 = sSet[it.set].grp_begin, g1 = g0 + sSet[it.set].ngrp;
            int st = st0; uint32_t rd = r0;
            for (int gi = g0; gi < g1; ++gi) {
                const int nu = sGrp[gi].nunit, u_begin = sGrp[gi].unit_begin;
                const uint32_t grows = __shfl_sync(0xffffffffu, (uint32_t)sGrp[gi].rows, 0);
                // resident slots: my units of the group, one after another over the same slots and entries of W
                const int ws0 = ws; const uint32_t wr0 = wr;
                bool first = true;
                for (int ui = 0, n; ui < nu; ui += n, ai += n) {
                    n = it.resident ? 1 : min(2, nu - ui);             // slots that do not stay: one pass for two units, one of them mine
                    const uint32_t k = (ai ^ me) & 1, my = ai + k;
                    const bool mine = (int)k < n, last = it.resident ? ui + 2 >= nu : true;           // (of mine)
                    // a unit of the other warp: its slots pass by, unless the next one is mine and finds them
                    if (!mine && it.resident && (!first || ui + 1 < nu)) continue;
                    if (it.resident) { st = st0; rd = r0; ws = ws0; wr = wr0; }
                    const MUnit& U = sUnit[u_begin + ui + (mine ? (int)k : 0)];
                    const bool xlast = last && (gi + 1 == g1 || !it.resident);
                    const uint32_t uN = __shfl_sync(0xffffffffu, (uint32_t)U.N, 0), ud = __shfl_sync(0xffffffffu, (uint32_t)U.d, 0),
                                   x0 = __shfl_sync(0xffffffffu, (uint32_t)U.slab0 * (SLAB >> 4), 0), w0 = __shfl_sync(0xffffffffu, (uint32_t)U.row0 * 2u, 0);
                    // D = F32, A = B = BF16, A MN-major, B K-major, M = 64
                    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uN >> 3) << 17) | (4u << 24);
                    if (mine && my >= 2) mbar_wait(bar_accfree + 8 * me, ((my >> 1) & 1) ^ 1, a.status);
                    for (int j = 0; j < it.nslot; ++j) {
                        if (first || !it.resident) {         // (later units of a group find the slot's rows and W in place)
                            mbar_wait(bar_full + 8 * st, rd & 1, a.status);
                            mbar_wait(bar_wfull + 8 * ws, wr & 1, a.status);
                            fence_async_smem();      // the gathered rows were written through the generic proxy
                        }
                        tc_fence_after();
                        // (broadcasts: operands that the compiler knows to be uniform take no transfer per instruction)
                        const uint64_t dX = dX0 + (x0 + __shfl_sync(0xffffffffu, (uint32_t)st * slot16, 0)),
                                       dW = dW0 + (w0 + __shfl_sync(0xffffffffu, (uint32_t)ws * w16, 0));
                        if (elect_one()) {
                            if (mine) {
                                ms_issue(ud, d0, dX, xlo16, dW, grows * 4u, grows * 2u, uN, idesc, j > 0 ? 1u : 0u);
                                if (last) tc_commit(bar_wfree + 8 * ws);
                                if (xlast) tc_commit(bar_sfree + 8 * st);
                                if (j + 1 == it.nslot) tc_commit(bar_accfull + 8 * me);
                            } else {
                                mbar_arrive(bar_wfree + 8 * ws);
                                if (xlast) mbar_arrive(bar_sfree + 8 * st);
                            }
                        }
                        __syncwarp();
                        if (++ws == NW) { ws = 0; ++wr; }
                        if (++st == NS) { st = 0; ++rd; }
                    }
                    first = false;
                }
            }
            st0 = st; r0 = rd;
        }
    } else if (warp < NDW) {
        // =========================== drain warps ===========================
        const int quarter = warp & 3, team = warp >> 2;
        MsWalk walk(a, nsub, nullptr);
        MsItem it{};
        uint32_t ai = 0;
        while (walk.next(it)) {
            const int u_begin = sGrp[sSet[it.set].grp_begin].unit_begin, nunit = sSet[it.set].nunit, R = sSet[it.set].nq;
            const bool full = it.len > 0;
            for (int ui = 0; ui < nunit; ++ui) {
                const uint32_t buf = ai & 1, par = (ai >> 1) & 1;
                if (full) ++ai;
                const MUnit& U = sUnit[u_begin + ui];
                if (full) {
                    mbar_wait(bar_accfull + 8 * buf, par, a.status);
                    tc_fence_after();
                }
                // rows of at most 32 (16) multiplicities lie in the slots twice (four times), and so in the lanes: twice (four times) the teams
                const int lgq = U.c > 32 ? 2 : (U.c > 16 ? 1 : 0), lgt = 2 - lgq, qc = quarter & ((1 << lgq) - 1);
                if (qc * 16 < U.c) {
                    const uint32_t t0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * HALF;
                    const int u = qc * 16 + (lane & 15), qh = lane >> 4, n_team = MS_NDT << lgt;
                    const int first = ((team << lgt) + (quarter >> lgq) - U.pair0) & (n_team - 1);       // the set's pairs go to the teams in turn, across its units
#define SOBEK_READ(r) read_out<r>(a, U, sOut, sTerm, t0, full, it.nl, first, n_team, u, qh)
                    if (R == 8) SOBEK_READ(8);
                    else if (R == 4) SOBEK_READ(4);
                    else if (R == 2) SOBEK_READ(2);
                    else SOBEK_READ(1);
#undef SOBEK_READ
                }
                if (full) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_accfree + 8 * buf);
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

template <bool DUAL, bool LE>
cudaError_t moment_stream_launch(const MsArgs& a, int grid, int smem, cudaStream_t s) {
    cudaError_t e = allow_dynamic_smem(k_moment_stream<DUAL, LE>);
    if (e != cudaSuccess) return e;
    k_moment_stream<DUAL, LE><<<grid, MS_TT, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace
}  // namespace sobek
