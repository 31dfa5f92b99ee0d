// Receiver-owned edge pass in moment form (sm_100a, tcgen05 / TMEM), warp-specialised.
//
// The edge outputs of the backward program (Eqs. streamed_radial_adjoints, streamed_operand_adjoints) are adjoints of the moments
//     P_i[q,b,s,u] = sum_e phi_e[q] Y_e[b] x_{src(e)}[s,u],     Z_i[path,o,q,u] = sum_{s,b} c[s,b,o] P_i[q,b,s,u]
// so with the moments' adjoint, made once per node from the state's adjoint Zbar = gy R^T,
//     Pbar_i[(q,b),(s,u)] = sum_{path,o} c[s,b,o] Zbar_i[path,o,q,u]
// they are one dense contraction per node and two short sums per edge:
//     G_e[(q,b)] = sum_{s,u} x_{src(e)}[s,u] Pbar_i[(q,b),(s,u)]
//     gphi_e[q] = sum_b G_e[(q,b)] Y_e[b],     gY_e[b] = sum_q G_e[(q,b)] phi_e[q]
// G has K x (harmonics) values per edge; the contraction with the coupling left in (k_edge_tc) has K sum d_src d_dst of them, each
// of which its epilogue reads twice: 1,840 against 144 at 64 x (0..2), K = 16.  What binds here is building Pbar (per node, not
// per edge).  fp32 parity: coupling sums in fp32, split-bf16 product with fp32 accumulation in TMEM.
//
// The contraction is long (all multiplicities of all components of all blocks, 1,152 terms at 128 x (0..2); k_edge_tc adds its
// components in fp32 instead), and an accumulation in tensor memory rounds towards zero.  So the small products of the split have an
// accumulator of their own, in the lanes that a product of 64 rows leaves free, and the fourth of them, lo x lo, is taken along.
// Error of gY against fp64 (2-norm), 128 x (0..2), K = 16, channelwise: 6.0e-6 with the three products in one accumulator,
// 4.4e-6 in k_edge_tc, 3.4e-6 so; the pass takes 6 % longer up to degree 64 and 14 % above, where a TMEM half holds half as many edges.
//
// With DUAL the pass gives the second-order terms that share Zbar (Eq. streamed_operand_second_adjoints) from G (rows of x) and Gv
// (rows of vx):   hphi[q] = sum_b Gv Y + G vY,     hY[b] = sum_q Gv phi + G vphi.
//
// A CTA takes nodes round-robin.  A node's edges are taken in passes of as many tiles of 64 as the accumulators hold, the radial
// indices in runs of NQ; for every run the blocks' slabs (64 multiplicities of one component) go by:
//   state warps    cp.async of the Zbar rows of one (block, run), fp32, into shared memory;
//   builder warps  Pbar of one slab: a warp takes (harmonic b) x NQ rows, a lane two multiplicities; K-major, 128-byte swizzle;
//   row warps      cp.async of the sender rows of one (slab, tile), taking turns;
//   MMA warp       M = 64 edges, N = NQ x harmonics; hi x hi in the lower 16 lanes of each TMEM lane quarter, the small products in
//                  the upper 16;
//   output warps   the two sums, two threads per edge (one per accumulator); the two TMEM halves alternate between products and
//                  read-out.
// Every wait is bounded.  The MMA warp polls, on whose path every hand-over lies; all others suspend (all polling: 3 to 7 % slower at
// 64 multiplicities, none polling: 2 to 5 %).
#include <cuda_bf16.h>

#include <algorithm>

#include "guard.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace sobek {
namespace {

using namespace ptx;

constexpr int NOW = 4;                  // output warps (one per TMEM lane quarter)
constexpr int NBW = 12;                 // builder warps
constexpr int NXW = 4;                  // row warps
constexpr int NZW = 3;                  // state warps
constexpr int W_B = NOW, W_X = W_B + NBW, W_Z = W_X + NXW, W_M = W_Z + NZW;
constexpr int TT = (W_M + 1) * 32;
constexpr int TILE = 64;                // edges of a tile
constexpr int SLAB = TILE * 128;        // bytes of one copy of a (slab, tile): 64 edges x 64 bf16
constexpr int MAXNX = 8, MAXNP = 4, MAXNZ = 2;
constexpr int HALF = 256;
constexpr int ACC_KSTEPS = 80;          // EXACT: k-steps that one accumulator takes (its rounding stays below the rows' representation error)
constexpr int SET2 = HALF / 2;          // EXACT with more of them: first column of the accumulators of the second and the third run of k-steps
constexpr int NBAR = 2 * MAXNX + 2 * MAXNP + 2 * MAXNZ + 4;

struct MeArgs {
    const MEBlk* blks;
    const MEComp* comps;
    const int32_t* tptr;        // per (component of a block, harmonic): first term (MEBlk::t_begin)
    const MTerm* terms;         // {component of the block, coefficient}
    int32_t n_blks, n_comps, n_tptr, n_terms;
    const int64_t* row_ptr;
    const int32_t* col;
    int64_t node0, n_nodes, N, E;
    const int4* oseg;           // the chunk's nodes in processing order {local node, segment begin, end} or NULL
    const __nv_bfloat16 *sh, *sl, *vsh, *vsl;
    const float *Y, *vY, *phi, *vphi;
    const float* zbar;
    float *gphi, *gY;
    int32_t phi_mode, Y_mode;   // 0 skip, 1 overwrite, 2 accumulate
    int32_t K, dsh, C_src, N_cols, nx, np, nz, p_bytes, z_bytes;
    int32_t nacc, acc_ksteps;   // EXACT: accumulators of the hi x hi products, k-steps of each
    int* status;
};

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
// what a split leaves, in bf16 pairs
__device__ __forceinline__ uint32_t rest2(float a, float b, uint32_t hi, uint32_t lo) {
    const __nv_bfloat162 r = __floats2bfloat162_rn((a - __uint_as_float(hi << 16)) - __uint_as_float(lo << 16),
                                                   (b - __uint_as_float(hi & 0xffff0000u)) - __uint_as_float(lo & 0xffff0000u));
    return *reinterpret_cast<const uint32_t*>(&r);
}
// NQ columns of this thread's TMEM lane, waited for
template <int NQ>
__device__ __forceinline__ void tm_read(uint32_t t, float* v) {
    if constexpr (NQ == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\ttcgen05.wait::ld.sync.aligned;"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "r"(t) : "memory");
    else if constexpr (NQ == 4)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n\ttcgen05.wait::ld.sync.aligned;"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(t) : "memory");
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];\n\ttcgen05.wait::ld.sync.aligned;" : "=f"(v[0]), "=f"(v[1]) : "r"(t) : "memory");
}

// Nodes of a CTA; the next one's bounds are requested one node ahead.
struct Walk {
    const MeArgs& a;
    int64_t v, nl, s0, s1;
    int* st;
    __device__ Walk(const MeArgs& a_, int* st_) : a(a_), v(blockIdx.x), nl(0), s0(0), s1(0), st(st_) { fetch(); }
    __device__ void fetch() {
        if (v >= a.n_nodes) return;
        if (a.oseg) { const int4 q = __ldg(a.oseg + v); nl = q.x; s0 = q.y; s1 = q.z; return; }
        seg_bounds(a.row_ptr, a.node0 + v, a.E, st, s0, s1);
        nl = v;
    }
    __device__ bool next(int64_t& node, int64_t& seg0, int& len) {
        while (v < a.n_nodes) {
            node = nl; seg0 = s0; len = (int)(s1 - s0);
            v += gridDim.x;
            fetch();
            if (len > 0) return true;
        }
        return false;
    }
};

// The two sums of one run of radial indices for the edge of this thread and of lane ^ 16, which has the other accumulator.
template <int NQ, bool DUAL, bool EXACT>
__device__ __forceinline__ void edge_sums(const MeArgs& a, uint32_t t, uint32_t tv, int64_t e, bool ok, int part, int q0, bool first_run, bool has_vx) {
    float f[NQ], vf[NQ], gp[NQ];
    const bool has_vY = DUAL && a.vY, has_vphi = DUAL && a.vphi;
#pragma unroll
    for (int r = 0; r < NQ; ++r) {
        const bool in = ok && q0 + r < a.K;
        f[r] = in ? __ldg(a.phi + e * a.K + q0 + r) : 0.f;
        vf[r] = in && has_vphi ? __ldg(a.vphi + e * a.K + q0 + r) : 0.f;
        gp[r] = 0.f;
    }
#pragma unroll 2
    for (int b = 0; b < a.dsh; ++b) {
        const float y = ok ? __ldg(a.Y + e * a.dsh + b) : 0.f, vy = ok && has_vY ? __ldg(a.vY + e * a.dsh + b) : 0.f;
        float g[NQ], gv[NQ];
        auto read = [&](uint32_t at, float* v) {
            tm_read<NQ>(at, v);
            if (EXACT && a.nacc > 1) {         // the second accumulator beside the first, the third (if any) beside the small products
                float w[NQ];
                tm_read<NQ>(at + SET2, w);
#pragma unroll
                for (int r = 0; r < NQ; ++r) v[r] += part == 0 || a.nacc > 2 ? w[r] : 0.f;
            }
        };
        read(t + (uint32_t)(b * NQ), g);
        float gy = 0.f;
        if (DUAL) {
            if (has_vx) {
                read(tv + (uint32_t)(b * NQ), gv);
            } else {
#pragma unroll
                for (int r = 0; r < NQ; ++r) gv[r] = 0.f;
            }
#pragma unroll
            for (int r = 0; r < NQ; ++r) {
                gp[r] = fmaf(gv[r], y, fmaf(g[r], vy, gp[r]));
                if (q0 + r < a.K) gy = fmaf(gv[r], f[r], fmaf(g[r], vf[r], gy));       // (columns past K hold no sums)
            }
        } else {
#pragma unroll
            for (int r = 0; r < NQ; ++r) {
                gp[r] = fmaf(g[r], y, gp[r]);
                if (q0 + r < a.K) gy = fmaf(g[r], f[r], gy);
            }
        }
        gy += __shfl_xor_sync(0xffffffffu, gy, 16);
        if (ok && a.Y_mode && (b & 1) == part) {
            float* d = a.gY + e * a.dsh + b;
            *d = (first_run && a.Y_mode == 1) ? gy : *d + gy;
        }
    }
#pragma unroll
    for (int r = 0; r < NQ; ++r) gp[r] += __shfl_xor_sync(0xffffffffu, gp[r], 16);
    if (ok && a.phi_mode) {
#pragma unroll
        for (int r = 0; r < NQ; ++r)
            if (q0 + r < a.K && (r & 1) == part) {
                float* d = a.gphi + e * a.K + q0 + r;
                *d = a.phi_mode == 1 ? gp[r] : *d + gp[r];
            }
    }
}

// EXACT: Pbar in three parts instead of two, so that only the rows' representation error is left.
template <int NQ, bool DUAL, bool EXACT>
__global__ void __launch_bounds__(TT, 1) k_moment_edge(const MeArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);
    uint8_t* sX = smem;                                                // rows of (slab, tile): hi, lo
    uint8_t* sP = sX + (size_t)a.nx * 2 * SLAB;                        // Pbar of a slab: hi rows, lo rows (EXACT: the rest's rows)
    uint8_t* sZ = sP + (size_t)a.np * a.p_bytes;                       // Zbar of (block, run): [component][NQ][64]
    uint64_t* bars = reinterpret_cast<uint64_t*>(sZ + (size_t)a.nz * a.z_bytes);
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + NBAR);
    MEComp* sComp = reinterpret_cast<MEComp*>(tmem_holder + 4);
    MEBlk* sBlk = reinterpret_cast<MEBlk*>(sComp + a.n_comps);
    MTerm* sTerm = reinterpret_cast<MTerm*>(sBlk + a.n_blks);
    int32_t* sTp = reinterpret_cast<int32_t*>(sTerm + a.n_terms);
    const uint32_t bar0 = smem_u32(bars);
    const uint32_t bar_xfull = bar0, bar_xfree = bar0 + 8 * MAXNX, bar_pfull = bar_xfree + 8 * MAXNX, bar_pfree = bar_pfull + 8 * MAXNP,
                   bar_zfull = bar_pfree + 8 * MAXNP, bar_zfree = bar_zfull + 8 * MAXNZ, bar_accfull = bar_zfree + 8 * MAXNZ, bar_accfree = bar_accfull + 16;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool has_vx = DUAL && a.vsh != nullptr;
    const int nop = has_vx ? 2 : 1;                                    // operands: rows of x, of vx
    const int n_cols = a.N_cols, runs = (a.K + NQ - 1) / NQ;
    const int pass_tiles = (EXACT && a.nacc > 1 ? SET2 : HALF) / (n_cols * nop);      // tiles that one TMEM half holds
    if (tid == 0) {
        for (int s = 0; s < MAXNX; ++s) { mbar_init(bar_xfull + 8 * s, 32); mbar_init(bar_xfree + 8 * s, 1); }
        for (int s = 0; s < MAXNP; ++s) { mbar_init(bar_pfull + 8 * s, NBW * 32); mbar_init(bar_pfree + 8 * s, 1); }
        for (int s = 0; s < MAXNZ; ++s) { mbar_init(bar_zfull + 8 * s, NZW * 32); mbar_init(bar_zfree + 8 * s, NBW); }
        for (int t = 0; t < 2; ++t) { mbar_init(bar_accfull + 8 * t, 1); mbar_init(bar_accfree + 8 * t, NOW); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    auto table = [&](void* dst, const void* src, int bytes) {
        for (int i = tid; i < bytes / 4; i += TT) reinterpret_cast<uint32_t*>(dst)[i] = reinterpret_cast<const uint32_t*>(src)[i];
    };
    table(sComp, a.comps, a.n_comps * (int)sizeof(MEComp)); table(sBlk, a.blks, a.n_blks * (int)sizeof(MEBlk));
    table(sTerm, a.terms, a.n_terms * (int)sizeof(MTerm)); table(sTp, a.tptr, a.n_tptr * 4);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    int64_t node, seg0;
    int len;

    if (warp >= W_X && warp < W_X + NXW) {
        // =========================== row warps ===========================
        // An entry is one (run, block, slab, tile, operand), filled by one warp; the warps that take part (no more than entries,
        // so that a free barrier is never waited for two phases ahead) take turns.
        const int nw = min(NXW, a.nx), me = warp - W_X;
        Walk walk(a, a.status);
        int xs = 0; uint32_t xr = 0;
        int turn = 0;
        while (me < nw && walk.next(node, seg0, len)) {
            for (int p0 = 0; p0 < len; p0 += pass_tiles * TILE) {
                const int plen = min(len - p0, pass_tiles * TILE), tiles = (plen + TILE - 1) / TILE;
                int32_t id0 = 0, id1 = 0;
                uint32_t m0 = 0, m1 = 0;
                int have = -1;                                         // tile whose sender ids the lanes hold
                for (int run = 0; run < runs; ++run)
                for (int bi = 0; bi < a.n_blks; ++bi) {
                    const MEBlk B = sBlk[bi];
                    const int cpr = B.c >> 3, pieces = 2 * B.ksteps;   // 16-byte pieces with multiplicities / that the products read
                    for (int s = 0; s < B.d; ++s)
                    for (int t = 0; t < tiles; ++t)
                    for (int op = 0; op < nop; ++op) {
                        if (turn == me) {
                            if (have != t) {
                                const int64_t pos = seg0 + p0 + t * TILE + lane;
                                const int left = plen - t * TILE;
                                bool ok0 = lane < left, ok1 = lane + 32 < left;
                                const int64_t v0 = ok0 ? (int64_t)a.col[pos] : 0, v1 = ok1 ? (int64_t)a.col[pos + 32] : 0;
                                ok0 = ok0 && id_ok(v0, a.N, a.status); ok1 = ok1 && id_ok(v1, a.N, a.status);
                                id0 = ok0 ? (int32_t)v0 : 0; id1 = ok1 ? (int32_t)v1 : 0;
                                m0 = __ballot_sync(0xffffffffu, ok0); m1 = __ballot_sync(0xffffffffu, ok1);
                                have = t;
                            }
                            if (xr > 0) mbar_wait(bar_xfree + 8 * xs, (xr & 1) ^ 1, a.status);
                            const uint32_t dst0 = smem_u32(sX + (size_t)xs * 2 * SLAB);
                            const __nv_bfloat16* bh = (op == 0 ? a.sh : a.vsh) + B.src_off + s * B.c_row;
                            const __nv_bfloat16* bl = (op == 0 ? a.sl : a.vsl) + B.src_off + s * B.c_row;
                            const int j = lane & 7, rmax = min(TILE, plen - t * TILE);
                            const uint32_t d0 = dst0 + (uint32_t)((lane >> 3) * 128);
                            // eight threads per row, four rows at a time; nobody reads the rows past the edges
#pragma unroll 4
                            for (int r0 = 0; r0 < rmax; r0 += 4) {
                                const int r = (r0 & 31) + (lane >> 3);
                                const int32_t id = __shfl_sync(0xffffffffu, r0 < 32 ? id0 : id1, r);
                                const bool ok = (((r0 < 32 ? m0 : m1) >> r) & 1u) && j < cpr;
                                const int64_t g = (int64_t)id * a.C_src + 8 * j;
                                const uint32_t d = d0 + (uint32_t)(r0 * 128 + ((j ^ ((r0 + (lane >> 3)) & 7)) << 4));
                                if (j < pieces) {
                                    cp_async16_zfill(d, bh + (j < cpr ? g : 0), ok ? 16u : 0u);
                                    cp_async16_zfill(d + SLAB, bl + (j < cpr ? g : 0), ok ? 16u : 0u);
                                }
                            }
                            cp_async_arrive(bar_xfull + 8 * xs);
                        }
                        if (++turn == nw) turn = 0;
                        if (++xs == a.nx) { xs = 0; ++xr; }
                    }
                }
            }
        }
    } else if (warp >= W_Z && warp < W_Z + NZW) {
        // =========================== state warps ===========================
        // A component's NQ rows by one warp, sixteen threads per row of 64 multiplicities (index arithmetic once per component:
        // with it for every copy these warps held up all others: 42.5 instead of 26.5 thousand cycles a node at 64 x (0..2), K = 16).
        const int me = warp - W_Z, j = lane & 15, rr = lane >> 4;
        Walk walk(a, nullptr);
        int zs = 0; uint32_t zr = 0;
        while (walk.next(node, seg0, len)) {
            for (int p0 = 0; p0 < len; p0 += pass_tiles * TILE)
            for (int run = 0; run < runs; ++run)
            for (int bi = 0; bi < a.n_blks; ++bi) {
                const int c4 = sBlk[bi].c >> 2, ncomp = sBlk[bi].ncomp;
                const MEComp* cps = sComp + sBlk[bi].comp_begin;
                if (zr > 0) mbar_wait(bar_zfree + 8 * zs, (zr & 1) ^ 1, a.status);
                uint32_t dst = smem_u32(sZ + (size_t)zs * a.z_bytes) + (uint32_t)(((me * NQ + rr) * 64 + 4 * j) * 4);
                const int q0 = run * NQ + rr;
                for (int i = me; i < ncomp; i += NZW, dst += NZW * NQ * 256) {
                    const MEComp cp = cps[i];
                    const float* src = a.zbar + (a.n_nodes * cp.zoff + node * cp.b + cp.a + q0 * cp.c_row + 4 * j);
#pragma unroll
                    for (int r = 0; r < NQ; r += 2, src += 2 * cp.c_row) {
                        const bool ok = j < c4 && q0 + r < a.K;
                        cp_async16_zfill(dst + (uint32_t)(r * 256), ok ? src : a.zbar, ok ? 16u : 0u);
                    }
                }
                cp_async_arrive(bar_zfull + 8 * zs);
                if (++zs == a.nz) { zs = 0; ++zr; }
            }
        }
    } else if (warp >= W_B && warp < W_B + NBW) {
        // =========================== builder warps ===========================
        const int me = warp - W_B;
        Walk walk(a, nullptr);
        int zs = 0, ps = 0; uint32_t zr = 0, pr = 0;
        int turn = 0;                                                  // harmonics go round the warps
        while (walk.next(node, seg0, len)) {
            for (int p0 = 0; p0 < len; p0 += pass_tiles * TILE)
            for (int run = 0; run < runs; ++run)
            for (int bi = 0; bi < a.n_blks; ++bi) {
                const MEBlk B = sBlk[bi];
                mbar_wait(bar_zfull + 8 * zs, zr & 1, a.status);
                const float* z = reinterpret_cast<const float*>(sZ + (size_t)zs * a.z_bytes) + 2 * lane;
                const int32_t* tp = sTp + B.t_begin;
                for (int s = 0; s < B.d; ++s, tp += a.dsh) {
                    if (pr > 0) mbar_wait(bar_pfree + 8 * ps, (pr & 1) ^ 1, a.status);
                    uint8_t* P = sP + (size_t)ps * a.p_bytes;
                    int b = me - turn;
                    if (b < 0) b += NBW;
                    for (; b < a.dsh; b += NBW) {
                        uint64_t v[NQ];                                // two multiplicities each
#pragma unroll
                        for (int r = 0; r < NQ; ++r) v[r] = 0;
                        const int k1 = tp[b + 1];
#pragma unroll 1
                        for (int k = tp[b]; k < k1; ++k) {
                            const MTerm m = sTerm[k];
                            const float* zc = z + m.col;
                            const uint64_t c2 = pack2(m.coef, m.coef);
#pragma unroll
                            for (int r = 0; r < NQ; ++r) v[r] = fma2(c2, *reinterpret_cast<const uint64_t*>(zc + r * 64), v[r]);
                        }
                        uint8_t* d = P + (size_t)(b * NQ) * 128 + (lane & 3) * 4;
                        const int ch = lane >> 2;
#pragma unroll
                        for (int r = 0; r < NQ; ++r) {
                            uint32_t hi, lo, rest;
                            split2(v[r], hi, lo);
                            if (EXACT) {
                                float va, vb;
                                unpack2(v[r], va, vb);
                                rest = rest2(va, vb, hi, lo);
                            }
                            const uint32_t o = (uint32_t)(r * 128 + ((ch ^ ((b * NQ + r) & 7)) << 4));
                            *reinterpret_cast<uint32_t*>(d + o) = hi;
                            *reinterpret_cast<uint32_t*>(d + o + n_cols * 128) = lo;
                            if (EXACT) *reinterpret_cast<uint32_t*>(d + o + 2 * n_cols * 128) = rest;
                        }
                    }
                    turn = (turn + a.dsh) % NBW;
                    fence_async_smem();
                    mbar_arrive(bar_pfull + 8 * ps);
                    if (++ps == a.np) { ps = 0; ++pr; }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_zfree + 8 * zs);
                if (++zs == a.nz) { zs = 0; ++zr; }
            }
        }
    } else if (warp == W_M) {
        // =========================== MMA warp ===========================
        Walk walk(a, nullptr);
        int xs = 0, ps = 0; uint32_t xr = 0, pr = 0, ai = 0;
        // D = F32, A = B = BF16, both K-major, M = 64
        const uint32_t uN = __shfl_sync(0xffffffffu, (uint32_t)n_cols, 0), tm_u = __shfl_sync(0xffffffffu, tmem_base, 0);
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uN >> 3) << 17) | (4u << 24);
        const uint64_t dX0 = make_desc(smem_u32(sX), 16, 1024), dP0 = make_desc(smem_u32(sP), 16, 1024);
        while (walk.next(node, seg0, len)) {
            for (int p0 = 0; p0 < len; p0 += pass_tiles * TILE) {
                const int tiles = (min(len - p0, pass_tiles * TILE) + TILE - 1) / TILE;
                for (int run = 0; run < runs; ++run, ++ai) {
                    const uint32_t buf = __shfl_sync(0xffffffffu, ai & 1, 0);
                    if (ai >= 2) mbar_spin(bar_accfree + 8 * buf, ((ai >> 1) & 1) ^ 1, a.status);
                    tc_fence_after();
                    int k_acc = 0, i_acc = 0;          // EXACT: k-steps in the accumulator at hand, its number
                    for (int bi = 0; bi < a.n_blks; ++bi) {
                        const int d = sBlk[bi].d;
                        const uint32_t ks = __shfl_sync(0xffffffffu, (uint32_t)sBlk[bi].ksteps, 0);
                        for (int s = 0; s < d; ++s) {
                            mbar_spin(bar_pfull + 8 * ps, pr & 1, a.status);
                            const uint64_t dP = dP0 + __shfl_sync(0xffffffffu, (uint32_t)ps * ((uint32_t)a.p_bytes >> 4), 0);
                            const uint32_t acc = __shfl_sync(0xffffffffu, bi + s > 0 ? 1u : 0u, 0);
                            uint32_t acc_d = acc, main = 0;
                            if (EXACT) {
                                if (k_acc >= a.acc_ksteps && i_acc + 1 < a.nacc) { ++i_acc; k_acc = 0; }
                                acc_d = __shfl_sync(0xffffffffu, k_acc > 0 ? 1u : 0u, 0);
                                main = __shfl_sync(0xffffffffu, i_acc == 0 ? 0u : SET2 + (i_acc == 2 ? 16u << 16 : 0u), 0);
                                k_acc += (int)ks;
                            }
                            for (int t = 0; t < tiles; ++t)
                            for (int op = 0; op < nop; ++op) {
                                mbar_spin(bar_xfull + 8 * xs, xr & 1, a.status);
                                fence_async_smem();      // the gathered rows were written through the generic proxy
                                tc_fence_after();
                                const uint64_t dX = dX0 + __shfl_sync(0xffffffffu, (uint32_t)xs * (2u * SLAB >> 4), 0);
                                const uint32_t dt = tm_u + buf * HALF + __shfl_sync(0xffffffffu, (uint32_t)(t * nop + op) * uN, 0);
                                constexpr uint32_t small = 16u << 16;      // lanes of the small products
                                if (elect_one()) {
                                    auto kstep = [&](uint32_t k) {
                                        tc_mma_bf16_x4(dt + main, dt + small, dX + 2 * k, dX + 2 * k + (SLAB >> 4), dP + 2 * k, dP + 2 * k + uN * 8u, idesc,
                                                       k > 0 ? 1u : acc_d, k > 0 ? 1u : acc);
                                        if (EXACT) tc_mma_bf16(dt + small, dX + 2 * k, dP + 2 * k + uN * 16u, idesc, 1u);
                                    };
                                    if (ks == 4) {
#pragma unroll
                                        for (uint32_t k = 0; k < 4; ++k) kstep(k);
                                    } else {
#pragma unroll 1
                                        for (uint32_t k = 0; k < ks; ++k) kstep(k);
                                    }
                                    tc_commit(bar_xfree + 8 * xs);
                                    if (t + 1 == tiles && op + 1 == nop) {
                                        tc_commit(bar_pfree + 8 * ps);
                                        if (bi + 1 == a.n_blks && s + 1 == d) tc_commit(bar_accfull + 8 * buf);
                                    }
                                }
                                __syncwarp();
                                if (++xs == a.nx) { xs = 0; ++xr; }
                            }
                            if (++ps == a.np) { ps = 0; ++pr; }
                        }
                    }
                }
            }
        }
    } else if (warp < NOW) {
        // =========================== output warps ===========================
        Walk walk(a, nullptr);
        uint32_t ai = 0;
        while (walk.next(node, seg0, len)) {
            for (int p0 = 0; p0 < len; p0 += pass_tiles * TILE) {
                const int plen = min(len - p0, pass_tiles * TILE), tiles = (plen + TILE - 1) / TILE;
                for (int run = 0; run < runs; ++run, ++ai) {
                    const uint32_t buf = ai & 1;
                    if (warp == 0) mbar_wait(bar_accfull + 8 * buf, (ai >> 1) & 1, a.status);
                    asm volatile("bar.sync 1, %0;" ::"n"(NOW * 32) : "memory");
                    tc_fence_after();
                    for (int t = 0; t < tiles; ++t) {
                        const int le = t * TILE + warp * 16 + (lane & 15);
                        const bool ok = le < plen;
                        if (!__any_sync(0xffffffffu, ok)) continue;
                        const uint32_t td = tmem_base + ((uint32_t)(warp * 32) << 16) + buf * HALF + (uint32_t)(t * nop * n_cols);
                        edge_sums<NQ, DUAL, EXACT>(a, td, td + (uint32_t)n_cols, seg0 + p0 + (ok ? le : 0), ok, lane >> 4, run * NQ, run == 0, has_vx);
                    }
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

}  // namespace

// Tables of the receiver direction's edge pass in moment form.
void build_moment_edge(const sobek_plan* p, Direction& dir) {
    constexpr int kSmem = 227 * 1024;
    MomentEdge& T = dir.me;
    T = MomentEdge{};
    // In the place of k_edge_tc, or (EXACT) of the FP32-pipe pass, which holds rows and adjoint state in 32 bits.  There the error
    // against fp64 must not grow by the split: in the fully connected mode it does not, since Pbar then has three parts and the product
    // that makes its Zbar takes lo x lo along (2-norm of gY, 168 random profiles: 0.97 of the FP32 pipes' on average, 1.07 at most).  The
    // channelwise mode, whose Zbar has the error of one fp32 product, keeps the FP32 pipes (1e-7), and so does a contraction that is
    // too long for three accumulators (they round towards zero, a little with every k-step).
    const bool exact = !dir.etc[0].ok;
    if (exact && p->uvu) return;
    if (p->K > 16 || p->K < 2 || (dir.C_src & 7) || dir.paths.empty()) return;
    struct Blk { int so, c, d; std::vector<std::pair<const DPath*, int>> paths; };
    std::vector<Blk> blocks;
    for (size_t gi = 0; gi < dir.groups.size(); ++gi)
        for (int k = dir.groups[gi].path_begin; k < dir.groups[gi].path_end; ++k) {
            const DPath& P = dir.paths[k];
            if ((P.c_src & 7) || (P.src_off & 7)) return;
            auto it = std::find_if(blocks.begin(), blocks.end(), [&](const Blk& b) { return b.so == P.src_off; });
            if (it == blocks.end()) { blocks.push_back(Blk{P.src_off, P.c_src, P.d_src, {}}); it = blocks.end() - 1; }
            it->paths.push_back({&P, (int)gi});
        }
    std::sort(blocks.begin(), blocks.end(), [](const Blk& x, const Blk& y) { return x.so < y.so; });
    int max_comp = 0;
    for (const Blk& B : blocks) {
        int n = 0;
        for (const auto& t : B.paths) n += t.first->d_dst;
        max_comp = std::max(max_comp, n);
    }
    const int dsh = p->dim_sh;
    // the longest run of radial indices whose Pbar and Zbar leave room for four entries of gathered rows
    for (int nq : {8, 4, 2}) {
        if (nq > 2 && p->K <= nq / 2) continue;
        const int n_cols = (dsh * nq + 7) & ~7;
        if (n_cols > 128) continue;                                    // the dual pass holds two accumulators in a TMEM half
        T = MomentEdge{};
        T.nq = nq; T.n_cols = n_cols;
        for (const Blk& B : blocks) {
            const int parts = (B.c + 63) / 64, per = ((B.c / 8 + parts - 1) / parts) * 8;
            for (int u0 = 0; u0 < B.c; u0 += per) {
                MEBlk M{};
                M.src_off = B.so + u0; M.c = std::min(per, B.c - u0); M.c_row = B.c; M.d = B.d; M.ksteps = (M.c + 15) / 16;
                M.comp_begin = (int)T.comps.size();
                std::vector<int> first;
                for (const auto& t : B.paths) {
                    const DGroup& G = dir.groups[t.second];
                    first.push_back((int)T.comps.size() - M.comp_begin);
                    for (int o = 0; o < t.first->d_dst; ++o)
                        T.comps.push_back(MEComp{G.z_off, (int64_t)o * G.D + t.first->koff + u0, G.d_dst * G.D, B.c});
                }
                M.ncomp = (int)T.comps.size() - M.comp_begin;
                M.t_begin = (int)T.tptr.size();
                for (int s = 0; s < B.d; ++s)
                    for (int b = 0; b < dsh; ++b) {
                        T.tptr.push_back((int)T.terms.size());
                        for (size_t k = 0; k < B.paths.size(); ++k) {
                            const DPath& P = *B.paths[k].first;
                            if (b < P.sh_off || b >= P.sh_off + P.d_sh) continue;
                            for (int o = 0; o < P.d_dst; ++o)
                                for (int z = p->tab_ptr[P.tabM + s * P.d_dst + o]; z < p->tab_ptr[P.tabM + s * P.d_dst + o + 1]; ++z)
                                    if (P.sh_off + p->tab_idx[z] == b) T.terms.push_back(MTerm{(uint32_t)((first[k] + o) * nq * 64), p->tab_coef[z]});
                        }
                    }
                T.tptr.push_back((int)T.terms.size());
                T.blks.push_back(M);
                T.slabs += M.d; T.ksteps += M.d * M.ksteps;
                const int w = (M.c + 31) / 32;
                T.comps32 += w * M.ncomp; T.rows32 += w * M.d; T.terms32 += w * ((int)T.terms.size() - T.tptr[M.t_begin]);
            }
        }
        T.exact = exact;
        T.nacc = exact ? (T.ksteps + ACC_KSTEPS - 1) / ACC_KSTEPS : 1;
        if (T.nacc > 3) break;
        if (T.nacc > 1 && 2 * n_cols > SET2) continue;
        T.p_bytes = ((exact ? 3 : 2) * n_cols * 128 + 1023) & ~1023;
        T.z_bytes = (max_comp * nq * 256 + 1023) & ~1023;
        const int fixed = 1024 + NBAR * 8 + 16 + (int)(T.comps.size() * sizeof(MEComp) + T.blks.size() * sizeof(MEBlk) + T.terms.size() * sizeof(MTerm) + T.tptr.size() * 4 + 64);
        for (int np = 3, nz = 2;;) {
            const int left = kSmem - fixed - np * T.p_bytes - nz * T.z_bytes;
            if (left >= 4 * 2 * SLAB) {
                T.np = np; T.nz = nz; T.nx = std::min(MAXNX, left / (2 * SLAB));
                T.smem_bytes = fixed + np * T.p_bytes + nz * T.z_bytes + T.nx * 2 * SLAB;
                T.ok = true;
                break;
            }
            if (nz == 2 && T.z_bytes > T.p_bytes) nz = 1;
            else if (np == 3) np = 2;
            else if (nz == 2) nz = 1;
            else break;
        }
        if (T.ok) return;
    }
    T = MomentEdge{};
}

// Microseconds per node that one SM spends in either form of the pass, the adjoint state's product with it (fp32 for one, bf16 hi + lo
// for the other).  Least-squares fits (of relative errors, 11 % and 18 % left) to the passes of 531 random layers with
// multiplicities of 16 (and 250 channelwise ones), orders up to 4, K = 1 .. 16, degrees 2 to 400, 64 to 8,000 nodes.  The chosen form takes 1.6 % longer than the
// faster one on average (1.3 % in the dual pass), 37 % (50 %) at worst longer than the other.  (Lines at fixed degrees, drawn before
// the fp32 products wrote 16 bytes a lane and the small products had an accumulator of their own: 8.3 % and 11 %, up to 2.2 and 2.7
// times as long.)  Against the FP32-pipe pass (EXACT; its own fit from 219 layers, 31 % left, counts per 32 lanes): 1.6 % (1.2 %) above
// the faster one, 34 % (21 %) at worst longer than the FP32 pipes, where the moment form throughout is 20 % above and up to four times
// as long, with scalar outputs at low degrees, and the FP32 pipes 58 % (73 %).
// Since then its warps stopped polling and the pass became 3 to 7 % faster: the whole call of gphi and gY of 7,288 other layers takes 3.0 %
// longer than with the faster form on average (moment throughout 10 %, never 70 %; dual 2.9, 11 and 87 %).
bool moment_edge_pays(const sobek_plan* p, int dual, int operands, int64_t N, int64_t E, int64_t chunk) {
    const Direction& dir = p->fwd;
    const MomentEdge& M = dir.me;
    const TcSets& T = dir.etc[dual];
    if (!M.ok || p->form != kFormAuto) return M.ok && p->form == kFormMoment;
    if (!M.exact && !T.ok) return true;          // (the dual pass of a plan whose tensor-core pass fits in its plain form only)
    const double deg = (double)E / (double)std::max<int64_t>(N, 1), per_sm = std::max(1.0, (double)std::min(N, chunk) / 148.0);
    const double state = 1e-4 * (double)dir.state_floats;
    const double fp32 = (dual ? 0.88 : 1.12) + (p->uvu ? 1.9 : 0.0);     // (the channelwise mode writes fp32 rows at 0.6 of the rate of its bf16 ones)
    const double runs = (p->K + M.nq - 1) / M.nq, cap = TILE * ((M.nacc > 1 ? SET2 : HALF) / (M.n_cols * operands));      // edges of a pass
    const double builds = runs * (deg > 0.6 * cap ? std::max(1.0, deg / cap + 0.4) : 1.0);
    const double tiles = runs * (deg > 40 ? deg / TILE + 0.5 : 1.0) * operands;
    const double build = dual ? 0.88 + 0.364 * M.slabs + M.nq * (0.00135 * M.terms.size() + 0.00154 * M.slabs * p->dim_sh)
                              : 0.45 + 0.206 * M.slabs + M.nq * (0.00274 * M.terms.size() + 0.0006 * M.slabs * p->dim_sh);
    const double moment = 27.0 / per_sm + builds * build + tiles * (M.ksteps * (dual ? 0.055 + 0.00063 * M.n_cols : 0.053 + 0.00083 * M.n_cols) +
                          (dual ? 0.061 : 0.127) * p->dim_sh) + runs * operands * deg * 0.0035 * M.slabs + fp32 * state;
    if (M.exact)
        return 1.13 * moment < (dual ? 59.0 / per_sm + 1.1 + deg * (0.0092 * M.terms32 + 0.015 * M.rows32) + 21.0 * state
                                     : 52.0 / per_sm + deg * (0.004 * M.terms32 + 0.011 * M.rows32) + 11.5 * state + 0.0077 * p->K * M.comps32);
    double coupled = (dual ? 2.46 : 2.48) * state;
    for (const TcSets::ESetPar& e : T.epar) {
        const double batches = std::max(1.0, deg / e.tb + 0.45);
        coupled += 25.0 / per_sm + batches / e.ctas * (dual ? 5.97 + 0.0133 * e.acc_cols + 3.7e-5 * e.nnz * e.tb : 3.24 + 0.009 * e.acc_cols + 1.9e-5 * e.nnz * e.tb);
    }
    return moment < coupled;
}

cudaError_t launch_moment_edge(const sobek_plan* p, const Direction& dir, const EdgeView& ev, int64_t node0, int64_t n_nodes, const SplitSrc& ss,
                               const float* Y, const float* vY, const float* phi, const float* vphi, int dual, const float* zbar, float* gphi,
                               float* gY, int phi_mode, int Y_mode, int* status, cudaStream_t s) {
    const MomentEdge& T = dir.me;
    if (!T.ok || !ss.h || !ss.l || ss.rvec) return cudaErrorInvalidValue;
    if (n_nodes <= 0) return cudaSuccess;
    MeArgs a{};
    a.blks = T.d_blks; a.comps = T.d_comps; a.tptr = T.d_tptr; a.terms = T.d_terms;
    a.n_blks = (int)T.blks.size(); a.n_comps = (int)T.comps.size(); a.n_tptr = (int)T.tptr.size(); a.n_terms = (int)T.terms.size();
    a.row_ptr = ev.ptr; a.col = ev.col; a.node0 = node0; a.n_nodes = n_nodes; a.N = ev.N; a.E = ev.E;
    a.oseg = ss.oseg ? ss.oseg + node0 : nullptr;
    a.sh = (const __nv_bfloat16*)ss.h; a.sl = (const __nv_bfloat16*)ss.l;
    a.vsh = dual ? (const __nv_bfloat16*)ss.vh : nullptr; a.vsl = dual ? (const __nv_bfloat16*)ss.vl : nullptr;
    a.Y = Y; a.vY = vY; a.phi = phi; a.vphi = vphi; a.zbar = zbar; a.gphi = gphi; a.gY = gY;
    a.phi_mode = phi_mode; a.Y_mode = Y_mode;
    a.K = p->K; a.dsh = p->dim_sh; a.C_src = dir.C_src; a.N_cols = T.n_cols; a.nx = T.nx; a.np = T.np; a.nz = T.nz;
    a.nacc = T.nacc; a.acc_ksteps = (T.ksteps + T.nacc - 1) / T.nacc;
    a.p_bytes = T.p_bytes; a.z_bytes = T.z_bytes; a.status = status;
#define SOBEK_ME(x) (T.nq == 8 ? (dual ? k_moment_edge<8, true, x> : k_moment_edge<8, false, x>) \
                     : T.nq == 4 ? (dual ? k_moment_edge<4, true, x> : k_moment_edge<4, false, x>) \
                                 : (dual ? k_moment_edge<2, true, x> : k_moment_edge<2, false, x>))
    void (*kern)(const MeArgs) = T.exact ? SOBEK_ME(true) : SOBEK_ME(false);
#undef SOBEK_ME
    cudaError_t e = allow_dynamic_smem(kern);
    if (e != cudaSuccess) return e;
    KernelTimer kt(K_EDGE, s);
    kern<<<(int)std::min<int64_t>(n_nodes, 148), TT, T.smem_bytes, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sobek
