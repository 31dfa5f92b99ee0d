// Arguments and layout constants of the moment-form edge stream (moment_stream_impl.cuh), shared with its host side.
#pragma once
#include <cuda_bf16.h>

#include "internal.h"

namespace sobek {

constexpr int MS_TB = 16;               // edges per slot = k extent of one MMA
constexpr int MS_NDT = 4;               // drain teams (four warps each, one per TMEM lane quarter)
constexpr int MS_NDW = 4 * MS_NDT;
constexpr int MS_NLW = 4;               // loader warps
constexpr int MS_NBW = 4;               // builder warps
constexpr int MS_TT = (MS_NDW + MS_NLW + MS_NBW + 3) * 32;      // plus the two MMA warps and the edge warp
constexpr int MS_MAXNS = 8;             // ring slots at most
constexpr int MS_MAXNW = 8;             // entries of the W ring at most
constexpr int MS_HALF = 256;            // columns of one TMEM half
constexpr int MS_PS = 20;               // pitch (floats) of the transposed phi / Y rows: 16 values + 4 (bank spread)
constexpr int MS_SLAB = MS_TB * 128;    // bytes of 64 multiplicities of one component: 16 edges x 64 bf16
constexpr int MS_NBAR = 2 * MS_MAXNS + 2 * MS_MAXNW + 4;

struct MsArgs {
    const MSet* sets;
    const MGrp* grps;
    const MSlab* slabs;
    const MUnit* units;
    const MOut* outs;
    const MTerm* terms;
    const uint16_t* rows;
    int32_t nsets, n_grps, n_slabs, n_units, n_outs, n_terms, n_rows;
    EdgeView ev;
    int64_t node0, n_nodes;
    const int4* oseg;           // the chunk's nodes in processing order {local node, segment begin, end} or NULL
    const __nv_bfloat16* sh;    // bf16 hi / lo copies of the source features [N][C_src]
    const __nv_bfloat16* sl;
    const __nv_bfloat16* vsh;   // DUAL: the same for the source direction; NULL without it
    const __nv_bfloat16* vsl;
    const float* Y;
    const float* vY;
    const float* phi;
    const float* vphi;
    const float* rvec;          // edge vectors [E][3]: when set, Y and phi are recomputed from them (Y, phi are NULL then)
    const float* vrvec;         // DUAL, geometry mode: direction on the edge vectors; vY = J_Y vrvec, vphi = J_phi vrvec
    float geo_rc;
    int32_t geo_basis, geo_p;
    __nv_bfloat16* zh;
    __nv_bfloat16* zl;
    int32_t K, dsh, C_src;
    int32_t x_cap, slot_bytes, ns, w_bytes, nw;
    int32_t interleaved;        // the state's order has zq = MSet::nq (state_pos); 0: q-major
    int* status;
};

cudaError_t moment_stream_plain(const MsArgs& a, int grid, int smem, bool loaders_edge, cudaStream_t s);
cudaError_t moment_stream_dual(const MsArgs& a, int grid, int smem, bool loaders_edge, cudaStream_t s);

}  // namespace sobek
