// vmb_testing.h - test-only controls of libvmb, not part of the public ABI
// (include/vmb.h does not declare them and production callers never call
// them).  The tests use them to run every tile shape and chunk length of the
// scans, which the planners would otherwise pick by problem size alone.
//
// The overrides are process-wide and take effect on the next plan; calls made
// while an override is set (by any thread) get the forced plan.  Restore the
// defaults (-1 / 0) when done.
#pragma once

#include <stddef.h>

#include "vmb.h"

#ifdef __cplusplus
extern "C" {
#endif

/* What the rules of the dispatch answer, without a launch (csm, mean steps and selection
 * also without a GPU).
 * vmb_testing_csm_kernel: kernel of a cross-scan (merge 0) or cross-merge (1) of
 *   `planes` maps: 0 whole planes, 1 bands, 2 the gather of single elements.
 * vmb_testing_mean_two_steps: 1 if `ctas` channel-mean CTAs take two steps per
 *   thread, given the CTAs that `sms` SMs hold at once with one and with two.
 * vmb_testing_selection_buffers: operand buffers of a selection grid.
 * vmb_testing_full_plan: out = {tile shape, L-chunks, launched early} of a full scan
 *   (map 1: as vmb_ss2d_full_fwd), with u or x (off & 1) or delta (off & 2) one element
 *   past 16-byte alignment.  Returns the status.
 * vmb_testing_mean_beside: 1 if the channel-mean scan of a block from the map runs beside
 *   the transpose by planes, with x one element past 16-byte alignment (off 1); -1: no plan. */
int vmb_testing_csm_kernel(int merge, vmb_dtype dtype, long long planes, int H, int W, int aligned, int sms);
int vmb_testing_mean_two_steps(long long ctas, int D, long long res_one, long long res_two, int sms, int with_y);
int vmb_testing_selection_buffers(long long grid, int D, int sms);
int vmb_testing_full_plan(int B, int K, int D, int N, int H, int W, unsigned flags, vmb_dtype dtype, int map, int off,
                          int* out);
int vmb_testing_mean_beside(int B, int D, int N, int H, int W, vmb_dtype dtype, int off);

/* Force the full scan's tile shape (0..23 for 16 states; taken modulo the
 * number of shapes of the padded state count) and, for the look-back and
 * warp-specialised shapes, the number of L-chunks (<= 1: one chunk).  shape < 0 restores the planner.
 * Ignored under VMB_FLAG_B_ZOH, which has one shape.  Returns 0. */
int vmb_testing_force_full_plan(int shape, int chunks);

/* Force the chunk length of the channel-mean scan (32, 64 or 128; 0 restores
 * the planner).  Returns 0, or 1 for another value (nothing changes). */
int vmb_testing_force_mean_chunk(int tc);

/* Force one or two steps per thread in the channel-mean scan (0 restores the
 * rule).  A call that cannot take two returns VMB_ERR_UNSUPPORTED while two are
 * forced.  Returns 0, or 1 for another value (nothing changes). */
int vmb_testing_force_mean_steps(int steps);

/* Let every tensor-map encoding fail (1), as a driver that refuses the tensors
 * would (0 restores it).  Returns 0. */
int vmb_testing_refuse_tensor_maps(int on);

/* Workspace bytes of the plan one scan call with these exact flags would run
 * (vmb_scan_workspace_bytes returns the larger over the two Bbar forms).
 * 0 for invalid arguments. */
size_t vmb_testing_plan_workspace_bytes(int path, unsigned flags, int B, int K, int D, int N, int H, int W,
                                        vmb_dtype dtype);

#ifdef __cplusplus
}
#endif
