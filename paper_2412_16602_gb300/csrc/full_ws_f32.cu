// full_ws_f32.cu - the warp-specialised full scan, fp32 storage (full_ws.cuh).
#include "full_ws.cuh"

namespace vmb {
WsKernel ws_kernel_f32(int np, int variant, bool gather, int R) { return ws_pick<float>(np, variant, gather, R); }
}  // namespace vmb
