// full_common.cuh - what the kernels of the full-channel scan share: the launch
// parameters, row loads and row stores (full_scan.cu, full_ws.cu).
#pragma once

#include <cuda.h>

#include "vmb_common.cuh"

namespace vmb {

struct FullParams {
    const void* u;
    const void* dl;
    const float* A;
    const void* Bs;
    const void* Cs;
    const float* Dskip;
    const float* bias;
    void* y;
    int K, D, N, L;
    int softplus_on;
    int tiles_per_bk, n_tiles, n_chunks, chunk_len;
    int vec;       // rows are 16-byte aligned: cp.async 16-byte path and vector stores
    int suppress;  // test hook: chunk 0 does not publish
    const float* Wup;  // low-rank Delta (warp-specialised variant only): dl is z [B*K][R][L] fp32 and
    int R;             // delta_raw[b,k,d,l] = sum_r Wup[k,d,r] z[b,k,r,l]
    int nstg;          // warp-specialised variant: ring slots
    int phase;         // warp-specialised variant: 0 one pass, 1 / 2 the two launches of its chunked form
    WsHeader* hdr;
    unsigned* flags;
    float* aggP;   // per chunk: sum of delta per channel (DT floats, rest unused)
    float* aggH;
    float* incH;
};

// The warp-specialised variant's tensor maps.
struct TensorMaps {
    CUtensorMap u, dl, B, C;  // [B*K][D][L] (u, delta) and [B*K][N][L] (B, C)
    CUtensorMap u2;           // gathering from the map: u is x [B][D][L] and u2 its transpose xt
};

__host__ __device__ constexpr size_t a16(size_t v) { return (v + 15) / 16 * 16; }

// Four consecutive elements of one row as fp32 (16-byte / 8-byte aligned reads).
__device__ __forceinline__ void load4(const float* p, float (&v)[4]) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
}
__device__ __forceinline__ void load4(const __nv_bfloat16* p, float (&v)[4]) {
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    v[0] = __uint_as_float(q.x << 16);
    v[1] = __uint_as_float(q.x & 0xffff0000u);
    v[2] = __uint_as_float(q.y << 16);
    v[3] = __uint_as_float(q.y & 0xffff0000u);
}

// Store n consecutive outputs of one row (n = 4, 2 or 1), vectorised when aligned.
template <typename T, int NV>
__device__ __forceinline__ void store_row(T* dst, const float (&v)[NV], int nvalid_here, bool vec) {
    if (vec && nvalid_here >= NV) {
        if constexpr (sizeof(T) == 4 && NV == 4) {
            *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
            return;
        } else if constexpr (sizeof(T) == 4 && NV == 2) {
            *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
            return;
        } else if constexpr (sizeof(T) == 2 && NV == 4) {
            const unsigned lo = __bfloat16_as_ushort(io<T>::to(v[0])) | ((unsigned)__bfloat16_as_ushort(io<T>::to(v[1])) << 16);
            const unsigned hi = __bfloat16_as_ushort(io<T>::to(v[2])) | ((unsigned)__bfloat16_as_ushort(io<T>::to(v[3])) << 16);
            *reinterpret_cast<uint2*>(dst) = make_uint2(lo, hi);
            return;
        } else if constexpr (sizeof(T) == 2 && NV == 2) {
            *reinterpret_cast<unsigned*>(dst) =
                __bfloat16_as_ushort(io<T>::to(v[0])) | ((unsigned)__bfloat16_as_ushort(io<T>::to(v[1])) << 16);
            return;
        }
    }
#pragma unroll
    for (int j = 0; j < NV; ++j)
        if (j < nvalid_here) dst[j] = io<T>::to(v[j]);
}

}  // namespace vmb
