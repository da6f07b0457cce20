// full_ws_bf16.cu - the warp-specialised full scan, bf16 storage (full_ws.cuh).
#include "full_ws.cuh"

namespace vmb {
WsKernel ws_kernel_bf16(int np, int variant, bool gather, int R) { return ws_pick<__nv_bfloat16>(np, variant, gather, R); }
}  // namespace vmb
