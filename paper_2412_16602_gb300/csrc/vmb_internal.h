// vmb_internal.h - host-side plumbing between the C ABI (vmb_abi.cu) and the
// kernel launchers (cross_scan_merge.cu, full_scan.cu, mean_scan.cu).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "vmb.h"

namespace vmb {

// One scan problem as the ABI received it (shapes already validated).
struct ScanArgs {
    const void* u;
    const void* delta;
    const float* A;
    const void* Bs;
    const void* Cs;
    const float* Dskip;
    const float* bias;
    void* y;
    float* ybar;  // mean path only (may be null)
    int B, K, D, N, L;
    unsigned flags;
    vmb_dtype dtype;
    void* ws;
    size_t ws_bytes;
    bool no_bcast = false;  // mean path fused with the cross-merge: ybar only, no y
    int bc_group = 1;       // grouped basis: K and D above are K*G and D/G; B / C rows per G sequences
    int gather_h = 0;       // > 0: u is the map x [B, D, H, W] (H = gather_h, K = 4) and u_t its transpose
                            // [B, D, W, H]; directions 0 / 2 read x, 1 / 3 read u_t (no materialised
                            // cross-scan)
    const void* u_t = nullptr;
    float* saved = nullptr;  // mean path: the group means kept for the backward, [B*K][N + 1][L] fp32
    const float* Wup = nullptr;  // full path, low-rank Delta: delta is z [B*K][R][L] fp32 and
    int R = 0;                   // delta_raw = Wup z (Wup [K][D][R]); warp-specialised plans only
    bool no_tma = false;         // full path: plan as for tensors that tensor copies cannot read
};

// Execution plan of an L-chunked scan: how the (sequence, chunk) grid is cut
// and how much workspace its look-back needs.  Deterministic for a given
// problem, build and device, so that the workspace query and the launch agree.
struct ScanPlan {
    int np;            // padded state count (1, 2, 4, 8, 16)
    int split;         // tile-shape index (full path)
    int tile_rows;     // channels per CTA (full path) or 0 (mean path)
    int tiles_per_bk;  // channel tiles per (b, k)   (full path)
    int n_seq;         // independent sequences: channel tiles (full) or (b, k) pairs (mean)
    int n_chunks;      // chunks along L per sequence
    int chunk_len;     // steps per chunk (a multiple of the stage length)
    size_t state_floats;  // floats of one chunk's published state (per array)
    size_t ws_bytes;      // total workspace bytes
    bool early = true;    // may be launched before the previous kernel of the stream completes
};

// One instance of the warp-specialised full scan (full_ws.cuh): fn is null when
// it could not be set up.
struct WsKernel {
    const void* fn;
    int per_slot, fixed;  // shared memory: bytes per ring slot, and once
    int G, DT, threads, ts;
};
constexpr int kWsOneLane = 0, kWsTwoLanes = 1;  // variants of the 16-state kernel: lanes per channel
WsKernel ws_kernel_f32(int np, int variant, bool gather, int R);
WsKernel ws_kernel_bf16(int np, int variant, bool gather, int R);

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Workspace layout: [header 256 B][flags n_seq*n_chunks u32][agg_P][agg_H][inc_H]
struct WsLayout {
    size_t flags_off, aggP_off, aggH_off, incH_off, total;
};
inline WsLayout ws_layout(const ScanPlan& p) {
    WsLayout w;
    size_t slots = (size_t)p.n_seq * (size_t)p.n_chunks;
    w.flags_off = 256;
    w.aggP_off = align_up(w.flags_off + slots * 4, 256);
    size_t arr = align_up(slots * p.state_floats * 4, 256);
    w.aggH_off = w.aggP_off + arr;
    w.incH_off = w.aggH_off + arr;
    w.total = w.incH_off + arr;
    if (p.n_chunks <= 1) w.total = 256;  // single-chunk plans only use the header
    return w;
}

// The paper's scan-only setting (Sec. 4): discretisation into materialised
// fp32 operands, then the scan alone.
struct DiscArgs {
    const void* u;
    const void* delta;
    const float* A;
    const void* Bs;
    const float* bias;
    float* dA;   // [B][K][D][N][L], or [B][K][N][L] for the channel means
    float* dBu;  // same shape as dA
    int B, K, D, N, L;
    unsigned flags;
    vmb_dtype dtype;
};
struct OnlyArgs {
    const float* dA;   // [B][K][Dm][N][L]
    const float* dBu;  // [B][K][Dm][N][L]
    const void* Cs;    // [B][K][N][L], dtype
    float* y;          // [B][K][Dm][L]
    int B, K, Dm, N, L;
    vmb_dtype dtype;
};

// The selection functions of Eq. 6 (B, C and the raw Delta from the input).
struct SelArgs {
    const void* u;     // [B][K][D][L], dtype
    const float* WB;   // [K][N][D]
    const float* WC;   // [K][N][D]
    const float* Wz;   // [K][R][D]
    const float* Wup;  // [K][D][R]
    void* Bs;          // [B][K][N][L], dtype
    void* Cs;          // [B][K][N][L], dtype
    void* delta_raw;   // [B][K][D][L], dtype
    int B, K, D, N, R, L;
    vmb_dtype dtype;
    float* z = nullptr;  // not null: z [B][K][R][L] fp32 written instead of delta_raw (Wup unused)
};

// Gradients of the (grouped) channel-mean scan.
struct MeanBwdArgs {
    const void* u;
    const void* delta;  // raw Delta (before bias and softplus)
    const float* A;
    const void* Bs;
    const void* Cs;
    const float* Dskip;
    const float* bias;
    const void* gy;
    const float* saved;  // the forward's group means, or null (recomputed)
    void* gu;
    void* gdelta;
    float* gA;
    void* gBs;
    void* gCs;
    float* gDskip;
    float* gbias;
    int B, K, D, N, L, groups;
    unsigned flags;
    vmb_dtype dtype;
    void* ws;
    size_t ws_bytes;
};

int device_sm_count();

// CTAs of a kernel that fit on the current device at once (at least one per
// SM); 0 when the occupancy query fails.  The query costs about 2 us of host
// time and its answer is fixed for a kernel, block size and shared-memory size,
// so the answers are kept per device (a plan asks for up to eight, and a call
// makes up to three plans: 25 of a small call's 48 us were these queries).
long long resident_ctas(const void* fn, int threads, size_t smem);

// The argument checks of the scan entry points (shapes, flags, pointers,
// alignment); *empty is set for a problem with no elements.
vmb_status validate_scan(const ScanArgs& a, bool mean, bool* empty);

// Test-only plan overrides (vmb_testing.h); -1 / 0 when unset.
int forced_full_shape(int* chunks);
int forced_mean_chunk();
int forced_mean_steps();
bool refuse_tensor_maps();

vmb_status plan_full(const ScanArgs& a, ScanPlan* plan);
vmb_status plan_mean(const ScanArgs& a, ScanPlan* plan);
// (*refused: the driver's tensor-map encoder refused the tensors of a warp-specialised plan.  A
// scan of materialised sequences has then been launched with another plan; one that gathers or
// expands has not been, and its tensors have to be materialised, ScanArgs::no_tma.)
vmb_status launch_full(const ScanArgs& a, const ScanPlan& plan, cudaStream_t stream, bool* refused = nullptr);
int full_plan_launches(const ScanPlan& plan);  // kernels launch_full starts for this plan
// Whether launch_full can read the plan's u gathered from the map (ScanArgs::gather_h):
// the warp-specialised plans; or expand a low-rank Delta (ScanArgs::R): those of 16 states.
bool full_plan_gathers(const ScanPlan& plan);
bool full_plan_lowrank(const ScanPlan& plan);
// out [B,K,D,L] (dtype) = Wup z, the raw Deltas of the low-rank form.
vmb_status launch_lowrank_expand(const float* z, const float* Wup, void* out, int B, int K, int D, int R, int L,
                                 vmb_dtype dt, cudaStream_t stream);
// Short sequences held whole in shared memory (small_map.cu): lanes per channel
// of a plan that takes this kernel, 0 for the others; `map`: as the whole block.
int full_plan_small(const ScanPlan& plan);
constexpr size_t kSmallMaxSmem = 227 * 1024;
size_t small_scan_smem(int G, int L, bool map);
// out = null: the scan alone (a.u the sequences); else a.u is the map [B][D][H][W] and K = 4.
vmb_status launch_small(const ScanArgs& a, int G, void* out, int H, int W, cudaStream_t stream, bool early = true);
vmb_status launch_mean(const ScanArgs& a, const ScanPlan& plan, cudaStream_t stream);
bool mean_two_steps(long long n, int D, long long res1, long long res2, int sms, bool with_y);
// Kernels of the cross-scan and the cross-merge; `aligned`: both tensors 16-byte aligned.
enum class CsmKernel { kPlane, kBand, kGather };
CsmKernel csm_kernel(bool merge, vmb_dtype dt, long long planes, int H, int W, bool aligned, int sms);
vmb_status launch_cross_scan(const void* x, void* xs, int B, int D, int H, int W, vmb_dtype dt,
                             cudaStream_t stream);
vmb_status launch_cross_merge(const void* ys, void* out, int B, int D, int H, int W, vmb_dtype dt,
                              cudaStream_t stream);
// The transpose by whole planes (transpose_by_planes: they fit) runs as one CTA per SM of at
// most this shared memory (1 KB of the CTA's own included), beside which the scan starts;
// otherwise 32 x 32 tiles.
constexpr size_t kTransposeSmem = 33 * 1024;
bool transpose_by_planes(const void* x, const void* xt, int H, int W, vmb_dtype dt);
bool transpose_whole_vectors(const void* x, const void* xt, int H, int W, vmb_dtype dt);
vmb_status launch_map_transpose(const void* x, void* xt, int B, int D, int H, int W, vmb_dtype dt, bool planes,
                                cudaStream_t stream);
// Whether the channel-mean scan of this plan runs beside the transpose by planes.
bool mean_beside_transpose(const ScanArgs& a, const ScanPlan& plan, int H, int W);
vmb_status launch_discretise(const DiscArgs& a, bool mean, cudaStream_t stream);
bool selection_two_buffers(long long grid, int D, int sms);
vmb_status launch_selection(const SelArgs& a, cudaStream_t stream);
size_t mean_bwd_workspace_bytes(long long B, long long K, long long D, long long N, long long L, long long G);
vmb_status launch_mean_bwd(const MeanBwdArgs& a, cudaStream_t stream);
vmb_status launch_scan_only(const OnlyArgs& a, cudaStream_t stream);
vmb_status launch_mean_merge(const void* x, const float* ybar, const float* Dskip, void* out, int B, int D, int H,
                             int W, bool per_channel_skip, vmb_dtype dt, cudaStream_t stream);

}  // namespace vmb
