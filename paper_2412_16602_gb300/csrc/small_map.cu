// small_map.cu - the full-channel selective scan (App. A, Eqs. 3, 4, 6) of
// short sequences, alone or as the whole scan side of an SS2D block
// (cross-scan, scan of the four directions and cross-merge in one launch).
//
// A warp owns 32 / G channels of one (batch, direction), G lanes a channel and
// 16 / G states a lane, and holds their whole sequences in shared memory: it
// copies its u, raw Delta, B and C rows in (4-byte asynchronous copies, so rows
// of any length and alignment take the same path), turns Delta into
// softplus(raw + bias) in place, runs the recurrence reading B and C as
// broadcast rows [t][B0..15, C0..15], leaves y in place of Delta and writes it
// out as one contiguous run.  Nothing but the warp itself is waited for.
// As the block (MAP), the four warps of a CTA are the four directions of the
// same channels: they share one tile of the map, which direction k reads at
// its own pixel order (no cross-scanned sequences), and after one barrier the
// CTA adds the four directions' y of every pixel from shared memory.
//
// Why: at these lengths the streaming kernels spend their time on stage
// prologues and element-wise loads (rows of 49 steps are not 16-byte
// multiples), and a block of three launches spends it on the launches.
// Bound by instruction dispatch (the update loop, and about as many again for
// staging short rows): block of 32 maps of 7x7x1536 213 -> 69 us, of one 14x14x192 map 38.5
// -> 11 us on the device.  Which lengths and row counts take it, with both
// sides measured: small_rule in full_scan.cu.
#include <mutex>

#include "vmb_common.cuh"
#include "vmb_internal.h"

namespace vmb {
namespace {

constexpr int kSmThreads = 128;  // four warps
constexpr int kNP = 16;          // states, zero padded
constexpr int kBC = 2 * kNP;     // floats of one step's B and C

struct SmallParams {
    const void* u;  // [B][K][D][L], or (MAP) the map x [B][D][L]
    const void* dl;
    const float* A;
    const void* Bs;
    const void* Cs;
    const float* Dskip;
    const float* bias;
    void* y;
    void* out;  // MAP: [B][D][L]
    int K, D, N, L, H, W;
    int softplus_on;
    int tiles;        // channel tiles per (b, k)
    long long units;  // warps with work: B * K * tiles (MAP: CTAs, B * tiles)
    int RX;           // row stride (floats) of the u, Delta / y and map tiles: odd, so that the lanes' rows
                      // start in distinct banks
    FastDiv fL, fW;
};

__device__ __forceinline__ void load_elem(float* dst, const float* src) { cp_async4(dst, src, 4); }
__device__ __forceinline__ void load_elem(float* dst, const __nv_bfloat16* src) { *dst = __bfloat162float(*src); }

// `rows` consecutive rows of L elements into rows of stride RX, by `step`
// threads of which this is number `i0`.
template <typename T>
__device__ __forceinline__ void load_rows(float* dst, const T* src, int rows, const SmallParams& p, int i0, int step) {
    const int n = rows * p.L;
#pragma unroll 4
    for (int i = i0; i < n; i += step) {
        const int c = (int)fdiv((unsigned)i, p.fL), t = i - c * p.L;
        load_elem(dst + c * p.RX + t, src + i);
    }
}

// Word of column q (B: q = 0..15, C: 16 + the same) at step t: the columns of a
// step are rotated by four per step, so that the stores of one column at
// consecutive steps spread over eight banks; a quad of columns stays contiguous.
__device__ __forceinline__ int bc_word(int t, int q) { return t * kBC + ((q + 4 * t) & (kBC - 1)); }

// Sum of v[0..G) over the G lanes of a channel, transposed: lane g ends with
// the sum for index g in v[0].
template <int G>
__device__ __forceinline__ void reduce_lanes(float (&v)[G], int g) {
#pragma unroll
    for (int m = G / 2; m >= 1; m /= 2) {
        const bool up = g & m;
#pragma unroll
        for (int i = 0; i < m; ++i) {
            const float keep = up ? v[i + m] : v[i];
            const float send = up ? v[i] : v[i + m];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
    }
}

template <typename T, int G, bool MAP>
__global__ void __launch_bounds__(kSmThreads) small_scan_kernel(const SmallParams p) {
    constexpr int CT = 32 / G, NG = kNP / G, BS = G > 4 ? G : 4;  // channels a warp, states a lane, steps a block
    extern __shared__ __align__(16) float sm[];
    pdl_wait();
    pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int L = p.L, RX = p.RX;
    const long long unit = MAP ? (long long)blockIdx.x : blockIdx.x * 4LL + warp;
    if (!MAP && unit >= p.units) return;  // the whole warp: no CTA barrier follows
    const long long seq = unit / p.tiles;  // (b, k), or b
    const int d0 = (int)(unit % p.tiles) * CT;
    const int rows = min(CT, p.D - d0);
    const long long bk = MAP ? seq * 4 + warp : seq;
    const int k = MAP ? warp : (int)(bk % p.K);
    // shared memory: the map tile (MAP) or each warp's u rows, then each warp's
    // Delta / y rows, then each warp's B and C rows
    float* ut = sm + (MAP ? 0 : warp * CT * RX);
    float* yt0 = sm + (MAP ? 1 : 4) * CT * RX;
    float* yt = yt0 + warp * CT * RX;
    float* bc = sm + ((MAP ? 5 : 8) * CT * RX + 3) / 4 * 4 + warp * L * kBC;
    const T* Bs = static_cast<const T*>(p.Bs) + (size_t)bk * p.N * L;
    const T* Cs = static_cast<const T*>(p.Cs) + (size_t)bk * p.N * L;
    const size_t row0 = (size_t)bk * p.D + d0;
    if (MAP)
        load_rows<T>(ut, static_cast<const T*>(p.u) + ((size_t)seq * p.D + d0) * L, rows, p, threadIdx.x, kSmThreads);
    else
        load_rows<T>(ut, static_cast<const T*>(p.u) + row0 * L, rows, p, lane, 32);
    load_rows<T>(yt, static_cast<const T*>(p.dl) + row0 * L, rows, p, lane, 32);
    if (p.N < kNP)
        for (int i = lane; i < L * kBC; i += 32) bc[i] = 0.0f;
    __syncwarp();
    // lane g owns the states g, g + G, ...: their columns lie together
#pragma unroll 4
    for (int i = lane; i < p.N * L; i += 32) {
        const int n = (int)fdiv((unsigned)i, p.fL), t = i - n * L;
        const int q = G == 4 ? (n & 3) * 4 + (n >> 2) : n;
        load_elem(bc + bc_word(t, q), Bs + i);
        load_elem(bc + bc_word(t, kNP + q), Cs + i);
    }
    cp_async_commit();
    const int c = lane / G, g = lane % G;
    const int d = d0 + c;
    const bool cval = d < p.D;
    const float bias = cval ? __ldg(p.bias + (size_t)k * p.D + d) : 0.0f;
    const float dsk = cval ? __ldg(p.Dskip + (size_t)k * p.D + d) : 0.0f;
    float A2[NG], h[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) {
        const int n = g + i * G;
        A2[i] = (cval && n < p.N) ? __ldg(p.A + ((size_t)k * p.D + d) * p.N + n) * kLog2e : 0.0f;
        h[i] = 0.0f;
    }
    cp_async_wait<0>();
    if (MAP)
        __syncthreads();  // the map tile is every warp's
    else
        __syncwarp();
    float* yr = yt + c * RX;
    const float* ur = ut + c * RX;
    // delta = softplus(raw + bias) (Eq. 6), once per element, two steps at a time
    if (cval) {
        for (int t = 2 * g; t < L; t += 2 * G) {
            const bool two = t + 1 < L;
            float2 v = make_float2(yr[t] + bias, (two ? yr[t + 1] : 0.0f) + bias);
            if (p.softplus_on) v = softplus2(v);
            yr[t] = v.x;
            if (two) yr[t + 1] = v.y;
        }
    }
    __syncwarp();
    // the pixel (MAP) or step that step t of this direction reads: row by row,
    // column by column, or their reverses
    int pos = (MAP && k >= 2) ? L - 1 : 0;
    const int inc = !MAP ? 1 : (k & 1 ? p.W : 1) * (k >= 2 ? -1 : 1);
    auto block = [&](int t0, auto tail_tag) {
        constexpr bool TAIL = decltype(tail_tag)::value;
        float us[BS], yp[BS];
#pragma unroll
        for (int j = 0; j < BS; ++j) {
            const bool in = !TAIL || t0 + j < L;  // past the end: delta = u = 0, an identity step
            const int t = in ? t0 + j : 0;
            const float dv = in ? yr[t] : 0.0f;
            us[j] = in ? ur[pos] : 0.0f;
            pos += inc;
            if (MAP) {
                if (pos >= L) pos -= L - 1;
                if (pos < 0) pos += L - 1;
            }
            const float du = dv * us[j];
            if constexpr (NG == 1) {
                const float b = bc[bc_word(t, g)], cc = bc[bc_word(t, kNP + g)];
                h[0] = fmaf(ex2(dv * A2[0]), h[0], du * b);
                yp[j] = cc * h[0];
            } else {
                // sum over the states: one chain, as in the other kernels with one lane
                // a channel, or (G = 4) the first two levels of the tree over the 16
                // states that the lane-per-state kernels add across lanes (scalar additions,
                // with which the products are not fused)
                const float2 dd = make_float2(dv, dv), uu = make_float2(du, du);
                float2 ya = make_float2(0.0f, 0.0f), half = ya;
#pragma unroll
                for (int q = 0; q < NG / 4; ++q) {
                    const float4 b = *reinterpret_cast<const float4*>(bc + bc_word(t, g * NG + 4 * q));
                    const float4 cc = *reinterpret_cast<const float4*>(bc + bc_word(t, kNP + g * NG + 4 * q));
                    const float2 b2[2] = {make_float2(b.x, b.y), make_float2(b.z, b.w)};
                    const float2 c2[2] = {make_float2(cc.x, cc.y), make_float2(cc.z, cc.w)};
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int n = 4 * q + 2 * e;
                        const float2 x = __fmul2_rn(dd, make_float2(A2[n], A2[n + 1]));
                        const float2 hn = __ffma2_rn(make_float2(ex2(x.x), ex2(x.y)), make_float2(h[n], h[n + 1]),
                                                     __fmul2_rn(uu, b2[e]));
                        h[n] = hn.x;
                        h[n + 1] = hn.y;
                        if constexpr (G == 1) ya = __ffma2_rn(c2[e], hn, ya);
                        else if (e == 0) half = __fmul2_rn(c2[0], hn);
                        else {
                            const float2 p1 = __fmul2_rn(c2[1], hn);
                            ya = make_float2(__fadd_rn(half.x, p1.x), __fadd_rn(half.y, p1.y));
                        }
                    }
                }
                yp[j] = ya.x + ya.y;
            }
        }
        // y = sum over the channel's lanes + D u, rounded to the storage type,
        // in place of Delta (every lane has read the block's Deltas)
        if constexpr (G == 1) {
#pragma unroll
            for (int j = 0; j < BS; ++j)
                if (cval && (!TAIL || t0 + j < L)) yr[t0 + j] = io<T>::cvt(io<T>::to(fmaf(dsk, us[j], yp[j])));
        } else {
            // lane g keeps step g (BS = G)
            float uo = us[0];
#pragma unroll
            for (int j = 1; j < BS; ++j) uo = g == j ? us[j] : uo;
            reduce_lanes<G>(yp, g);
            __syncwarp();
            if (cval && (!TAIL || t0 + g < L)) yr[t0 + g] = io<T>::cvt(io<T>::to(fmaf(dsk, uo, yp[0])));
        }
    };
    int t0 = 0;
#pragma unroll 1
    for (; t0 + BS <= L; t0 += BS) block(t0, std::false_type{});
    if (t0 < L) block(t0, std::true_type{});
    __syncwarp();
    // y of the warp's channels: one contiguous run
    T* yo = static_cast<T*>(p.y) + row0 * L;
    const int n = rows * L;
#pragma unroll 4
    for (int i = lane; i < n; i += 32) {
        const int cc = (int)fdiv((unsigned)i, p.fL);
        yo[i] = io<T>::to(yt[cc * RX + i - cc * L]);
    }
    if (!MAP) return;
    // cross-merge: out = (y0 + y2) + (y1 + y3) at every pixel, in this order
    __syncthreads();
    T* oo = static_cast<T*>(p.out) + ((size_t)seq * p.D + d0) * L;
    const int ys = CT * RX;
    for (int i = threadIdx.x; i < n; i += kSmThreads) {
        const int cc = (int)fdiv((unsigned)i, p.fL), pos0 = i - cc * L;
        const int hh = (int)fdiv((unsigned)pos0, p.fW), ww = pos0 - hh * p.W;
        const int pos1 = ww * p.H + hh;
        const float* r = yt0 + cc * RX;
        const float a = r[pos0] + r[2 * ys + L - 1 - pos0];
        const float b = r[ys + pos1] + r[3 * ys + L - 1 - pos1];
        oo[i] = io<T>::to(a + b);
    }
}

template <typename T, int G, bool MAP>
const void* small_fn() {
    const void* fn = reinterpret_cast<const void*>(&small_scan_kernel<T, G, MAP>);
    static std::once_flag once;
    static cudaError_t err = cudaSuccess;
    std::call_once(once, [&] {
        err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallMaxSmem);
    });
    return err == cudaSuccess ? fn : nullptr;
}

template <typename T, bool MAP>
const void* small_pick(int G) {
    return G == 1 ? small_fn<T, 1, MAP>() : G == 4 ? small_fn<T, 4, MAP>() : small_fn<T, 16, MAP>();
}

}  // namespace

size_t small_scan_smem(int G, int L, bool map) {
    const size_t ct = 32 / G, rx = (size_t)L | 1;
    return (((map ? 5 : 8) * ct * rx + 3) / 4 * 4 + (size_t)4 * L * kBC) * 4;
}

vmb_status launch_small(const ScanArgs& a, int G, void* out, int H, int W, cudaStream_t stream, bool early) {
    const bool map = out != nullptr;
    const void* fn = a.dtype == VMB_BF16 ? (map ? small_pick<__nv_bfloat16, true>(G) : small_pick<__nv_bfloat16, false>(G))
                                         : (map ? small_pick<float, true>(G) : small_pick<float, false>(G));
    if (!fn) return VMB_ERR_CUDA;
    SmallParams p{};
    p.u = a.u;
    p.dl = a.delta;
    p.A = a.A;
    p.Bs = a.Bs;
    p.Cs = a.Cs;
    p.Dskip = a.Dskip;
    p.bias = a.bias;
    p.y = a.y;
    p.out = out;
    p.K = a.K;
    p.D = a.D;
    p.N = a.N;
    p.L = a.L;
    p.H = H;
    p.W = W;
    p.softplus_on = (a.flags & VMB_FLAG_SOFTPLUS) ? 1 : 0;
    p.tiles = (a.D + 32 / G - 1) / (32 / G);
    p.units = (map ? (long long)a.B : (long long)a.B * a.K) * p.tiles;
    p.RX = a.L | 1;
    p.fL = make_fastdiv((unsigned)a.L);
    p.fW = make_fastdiv((unsigned)(W > 0 ? W : 1));
    const long long grid = map ? p.units : (p.units + 3) / 4;
    void* args[] = {&p};
    return launch_kernel(fn, dim3((unsigned)grid), dim3(kSmThreads), small_scan_smem(G, a.L, map), args, stream, early) ==
                   cudaSuccess
               ? VMB_OK
               : VMB_ERR_CUDA;
}

}  // namespace vmb
