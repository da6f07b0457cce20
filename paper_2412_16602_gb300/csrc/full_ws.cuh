// full_ws.cuh - the warp-specialised full scan (tensor copies, mbarrier stage
// hand-over); full_ws_f32.cu and full_ws_bf16.cu instantiate it.
//
// A CTA is CW consumer warps and one producer warp over 32 CW / G channels of
// one (b, k): G adjacent lanes share a channel, each owning NP / G of its
// states in registers.  The producer issues, per stage of TS steps, four tiled
// tensor copies (u and delta: DT rows x TS steps, B and C: NP rows x TS steps)
// into a ring (nstg stages) and, once a stage has landed, converts its B and C rows
// into fp32 [t][B0..NP-1, C0..NP-1] rows for broadcast reads.  Stages are handed
// over with mbarriers (landed / ready / released), so no barrier spans the CTA
// and the copies of the next stages overlap the consumers' arithmetic.  Each
// consumer lane computes delta = softplus(raw + bias) of its channel (the G
// lanes split the stage's steps), runs the update and stores y from registers.
// The state update is packed (f32x2): per pair of states and step one product
// delta (A log2 e), two ex2, one product (delta u) B and two FMAs; with 16
// states and G = 1 the operations and their order are those of
// full_packed_kernel (y is bit-identical).
//
// The u and delta rows are 16 to 64 bytes apart in shared memory; the tensor
// copies swizzle their 16-byte pieces so that a quarter warp's 128-bit reads of
// one piece of consecutive rows hit distinct banks.
//
// What bounds it: at 16 states the dispatch of the packed update (about 6.4
// cycles of a scheduler per update: a packed FMA with three register operands takes
// 3.3, a product 2.1, an ex2 1) and the softplus; at one state HBM (90% of it).  GB300,
// fp32, us: 128 maps of 56x56x256, 16 states, one lane 1448, two 1535; 24576 rows of
// 56x56 471 with one lane, 350 with two (a warp per scheduler leaves the step's
// latency open, 106 ns a step with one lane and 51 with two); one state 1355 with
// barrier-staged tiles, 795 here.  Eight steps are unrolled together with one lane, 16 with
// two (4: 10% slower; 16 with one lane spill); starting the next stage's softplus
// before this stage's updates was 20% slower.
//
// Requires rows of 16-byte multiples and 16-byte aligned tensors (the host
// picks this variant only then); every wait is bounded.
// Gathering from the map (GATHER, App. A cross-scan without the cross-scanned
// sequences): direction k's u rows are the (b, d) planes of x (k = 0, 2) or of
// its transpose xt (k = 1, 3), and the reversed directions (k = 2, 3) load the
// mirrored box, steps [L - (s+1) TS, L - s TS), and read it from the end, so
// each step sees the value the cross-scan would have put there (the same
// operations: y is bit-identical to the scan of xs).
// Low-rank Delta (RP > 0, Eq. 6's s_Delta = Linear_D(Linear_R(u)) with the
// rank-R expansion fused into the scan): the second box of a stage is z
// (16 rows x TS steps, fp32, rows past R zero) instead of the raw Deltas, and
// each consumer lane forms its channel's raw Delta per step as
// sum_r Wup[k,d,r] z_r (r in order, as the selection kernel's epilogue does,
// so fp32 results are bit-identical to selection -> raw Deltas -> scan), with
// its Wup row (RP >= R values, zero-padded) in shared memory.
// Chunked form (phase 1 and 2; few channel rows): L is cut into P + 1 chunks.
// Launch 1 runs chunk 0 in full, leaving its end state, and next to it chunks
// 1 .. P - 1 from h = 0 for their aggregates (the sum of delta, so that the
// product of Abar_n is 2^(A_n log2 e S), and the end state); launch 2 runs chunks
// 1 .. P in full from the carry that each folds from chunk 0's end state and
// the aggregates before it, in chunk order.  2 P chunk passes for P + 1 chunks,
// P of them at a time: two launches without waits between CTAs.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <mutex>
#include <type_traits>

#include "full_common.cuh"
#include "vmb_internal.h"

namespace vmb {

template <int NP_, int G_, int CW_, int TS_, int ST_, int MINB_, int RP_ = 0, bool GATHER_ = false>
struct WsShape {
    static constexpr int NP = NP_, G = G_, CW = CW_, TS = TS_, ST = ST_, MINB = MINB_, RP = RP_;
    static constexpr bool GATHER = GATHER_;  // u gathered from the map (see above)
};

__host__ __device__ constexpr int a128(int v) { return (v + 127) / 128 * 128; }

template <typename T, class WS>
struct WsTileLayout {
    static constexpr int G = WS::G, CW = WS::CW, DT = 32 * CW / G, NP = WS::NP, TS = WS::TS;
    static constexpr int THREADS = 32 * CW + 32;
    static constexpr int ROW = TS * (int)sizeof(T);  // bytes of one u (or delta) row of a stage
    static constexpr int U_BYTES = DT * ROW;         // one u (or delta) box
    static constexpr int DL_BYTES = WS::RP ? 16 * TS * 4 : U_BYTES;  // the delta box, or the z box (fp32)
    static constexpr int BC_BYTES = NP * ROW;                        // one B (or C) box
    static constexpr int B_OFF = U_BYTES + DL_BYTES;
    static constexpr int C_OFF = B_OFF + a128(BC_BYTES);
    static constexpr int TX = U_BYTES + DL_BYTES + 2 * BC_BYTES;  // bytes that land per stage
    static constexpr int RAW_STAGE = (C_OFF + BC_BYTES + 511) / 512 * 512;
    static constexpr int BCT_STAGE = TS * 2 * NP * 4;  // fp32 [TS][B0..NP-1, C0..NP-1]
    // the ring's slots are followed by the converted B / C rows of each slot, the
    // low rank's Wup rows (fp32 [DT][RP + 1]) and three mbarriers per slot; its
    // depth is the launch's (the host fills the shared memory that the CTAs per SM leave)
    static constexpr int WUP_BYTES = WS::RP ? (DT * (WS::RP + 1) * 4 + 15) / 16 * 16 : 0;
    static constexpr int PER_SLOT = RAW_STAGE + BCT_STAGE + 24;
    static constexpr size_t bytes(int nstg) { return (size_t)nstg * PER_SLOT + WUP_BYTES; }
    static_assert(U_BYTES % 512 == 0 && DL_BYTES % 128 == 0 && ROW % 16 == 0 && ROW <= 64 && TS % 8 == 0,
                  "tensor-copy boxes: rows of 16, 32 or 64 bytes, swizzle-aligned boxes");
    static_assert(NP % G == 0 && (G == 1 || G == 2) && (G == 1 || NP / G >= 2), "states per lane");
    // Byte offset of 16-byte piece `j` of row `r` of a u or delta box: the copies' swizzle
    // (32-byte rows: bit 4 ^= bit 7; 64-byte rows: bits 4-5 ^= bits 7-8 of the offset)
    static __device__ __forceinline__ int piece(int r, int j) {
        if constexpr (ROW == 64) return r * 64 + 16 * (j ^ ((r >> 1) & 3));
        else if constexpr (ROW == 32) return r * 32 + 16 * (j ^ ((r >> 2) & 1));
        else return r * 16;
    }
};

// One value per step of a stage.
template <int TS>
struct Steps {
    float v[TS];
    __device__ __forceinline__ float& operator[](int j) { return v[j]; }
    __device__ __forceinline__ float operator[](int j) const { return v[j]; }
};

constexpr uint64_t kStageWaitNs = 1000000000ull;  // 1 s per stage hand-over

// Eight outputs of one row as one 32-byte store (the row's address is 32-byte aligned).
__device__ __forceinline__ void store8(float* p, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

template <typename T, class WS>
__global__ void __launch_bounds__(WsTileLayout<T, WS>::THREADS, WS::MINB)
    full_ws_kernel(const FullParams p, const __grid_constant__ TensorMaps tm) {
    // Launch 2 of the chunked form starts its copies before launch 1 is done: its
    // inputs were complete before launch 1 passed its own wait.  Its consumers wait
    // for launch 1 before they read the carries or write.
    const bool late = p.phase == 2;
    // Gathering, the kernel before this one writes xt, which only the column-major
    // directions read: the CTAs of directions 0 and 2 (the first half of the grid)
    // do not wait for it.  What they touch was complete before that kernel passed its
    // own wait, and this grid's dependents are released by its waiting CTAs.
    const int tiles = p.n_tiles;
    int tile = blockIdx.x % tiles;
    bool own = true;
    if constexpr (WS::GATHER) {
        // tiles of directions 0, 2 of every b, then of 1, 3
        const int t2 = 2 * p.tiles_per_bk, half = tiles / 2, odd = tile >= half;
        const int r = tile - odd * half, b = r / t2, w = r % t2;
        tile = (b * 4 + 2 * (w / p.tiles_per_bk) + odd) * p.tiles_per_bk + w % p.tiles_per_bk;
        own = odd;
    }
    if (!late) {
        if (own) pdl_wait();
        pdl_launch_dependents();
    }
    using LY = WsTileLayout<T, WS>;
    constexpr int DT = LY::DT, NP = LY::NP, G = LY::G, TS = LY::TS, ST = WS::ST, NG = NP / G, CPW = 32 / G;
    extern __shared__ __align__(1024) unsigned char smem_ws[];
    unsigned char* smem = smem_ws;
    const uint32_t sbase = smem_u32(smem);
    const int nstg = p.nstg;  // ring slots
    const uint32_t bct_off = (uint32_t)(nstg * LY::RAW_STAGE), wup_off = bct_off + (uint32_t)(nstg * LY::BCT_STAGE);
    const uint32_t bar0 = sbase + wup_off + (uint32_t)LY::WUP_BYTES;
    // landed[i]: the four copies of the stage in slot i arrived; ready[i]: its
    // B/C rows are converted; released[i]: every consumer warp is done with it
    auto landed = [&](int i) { return bar0 + 24u * i; };
    auto ready = [&](int i) { return bar0 + 24u * i + 8u; };
    auto released = [&](int i) { return bar0 + 24u * i + 16u; };
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int chunk = (int)(blockIdx.x / tiles) + (p.phase == 2 ? 1 : 0);
    const bool agg = p.phase == 1 && chunk > 0;  // aggregate only: no y
    const int bk = tile / p.tiles_per_bk;
    const int d0 = (tile % p.tiles_per_bk) * DT;
    const int k = bk % p.K;
    const int L = p.L;
    const int l_begin = p.phase ? chunk * p.chunk_len : 0;  // chunk_len: a multiple of TS
    const int l_end = p.phase ? min(L, l_begin + p.chunk_len) : L;
    const int nst = (l_end - l_begin + TS - 1) / TS;
    const int cwarps = min(LY::CW, (p.D - d0 + CPW - 1) / CPW);  // consumer warps with at least one channel
    if (tid == 0) {
        for (int i = 0; i < nstg; ++i) {
            mbarrier_init(landed(i), 1);
            mbarrier_init(ready(i), 32);
            mbarrier_init(released(i), cwarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    if (warp == LY::CW) {
        // ------------------------------------------------------ producer warp
        // u: the rows of (b, k), or gathered from x / xt (see above)
        constexpr bool gather = WS::GATHER;
        const CUtensorMap* um = (gather && (k & 1)) ? &tm.u2 : &tm.u;
        const int uz = gather ? bk / p.K : bk;
        const bool urev = gather && k >= 2;
        int issued = 0;  // stages whose copies have been issued (0 .. issued-1)
        auto issue = [&](int s, int slot) {
            issued = s + 1;
            const int l0 = l_begin + s * TS;
            const uint32_t dst = sbase + (uint32_t)(slot * LY::RAW_STAGE);
            mbarrier_expect_tx(landed(slot), (unsigned)LY::TX);
            tma_load_3d(dst, um, urev ? L - l0 - TS : l0, d0, uz, landed(slot));
            tma_load_3d(dst + LY::U_BYTES, &tm.dl, l0, WS::RP ? 0 : d0, bk, landed(slot));
            tma_load_3d(dst + LY::B_OFF, &tm.B, l0, 0, bk, landed(slot));
            tma_load_3d(dst + LY::C_OFF, &tm.C, l0, 0, bk, landed(slot));
        };
        if (lane == 0)
            for (int s = 0; s < nstg && s < nst; ++s) issue(s, s);
        issued = __shfl_sync(0xffffffffu, issued, 0);
        int seen = 0;  // stages whose copies this warp has seen land
        bool ok = true;
        // (every wait's outcome is made warp-uniform, so that no lane leaves a
        // loop whose warp-wide operations the others still execute)
        int slot = 0, prev = 0;            // slots of stages s and s - 1
        unsigned par = 0, prev_par = 0;    // and the parities of their phases
        for (int s = 0; s < nst; ++s) {
            if (!(ok = __all_sync(0xffffffffu, mbarrier_wait(landed(slot), par, kStageWaitNs)))) break;
            seen = s + 1;
            // lane (row, part) converts four-step pieces of row `row` of
            // [B rows 0..NP-1, C rows 0..NP-1] into column `row`
            constexpr int PARTS = 32 / (2 * NP);
            const int row = lane % (2 * NP), part = lane / (2 * NP);
            const T* rb = reinterpret_cast<const T*>(smem + slot * LY::RAW_STAGE + (row < NP ? LY::B_OFF : LY::C_OFF)) +
                          (row % NP) * TS;
            float* bo = reinterpret_cast<float*>(smem + bct_off + slot * LY::BCT_STAGE) + row;
#pragma unroll
            for (int t = 4 * part; t < TS; t += 4 * PARTS) {
                float q[4];
                load4(rb + t, q);
#pragma unroll
                for (int e = 0; e < 4; ++e) bo[(t + e) * 2 * NP] = q[e];
            }
            __syncwarp();
            // (test hook: the first stage is never handed over, so every wait on it runs out)
            if (!(p.suppress && s == 0)) mbarrier_arrive(ready(slot));
            // refill the slot of stage s - 1 once the consumers released it
            if (s >= 1 && s - 1 + nstg < nst) {
                if (!(ok = __all_sync(0xffffffffu, mbarrier_wait(released(prev), prev_par, kStageWaitNs)))) break;
                if (lane == 0) issue(s - 1 + nstg, prev);
                issued = __shfl_sync(0xffffffffu, issued, 0);
            }
            prev = slot, prev_par = par;
            if (++slot == nstg) slot = 0, par ^= 1u;
        }
        if (!ok) {
            if (lane == 0) atomicOr(&p.hdr->err, kErrTimeout);
            // every copy issued must land before the CTA exits
            for (int s = seen; s < issued; ++s) mbarrier_wait(landed(s % nstg), (s / nstg) & 1, kStageWaitNs);
        }
        return;
    }
    if (late) {
        pdl_wait();
        pdl_launch_dependents();
    }
    if (warp >= cwarps) return;  // a tile's channels past D: no work, not counted by `released`
    // -------------------------------------------------------- consumer warps
    const bool urev = WS::GATHER && k >= 2;  // u arrives mirrored (see above)
    const int c = tid / G, g = tid % G;
    const int d = d0 + c;
    const bool cval = d < p.D;
    const size_t row0 = (size_t)bk * p.D + d0;
    const float bias = cval ? p.bias[(size_t)k * p.D + d] : 0.0f;
    const float dsk = cval ? p.Dskip[(size_t)k * p.D + d] : 0.0f;
    const float* Ad = p.A + ((size_t)k * p.D + d) * p.N;
    float A2[NG], h[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) {
        const int n = g * NG + i;
        A2[i] = (cval && n < p.N) ? Ad[n] * kLog2e : 0.0f;
        h[i] = 0.0f;
    }
    const size_t sfl = (size_t)DT * NP;  // floats of one chunk's published state
    const size_t my_off = (size_t)c * NP + (size_t)g * NG;
    if (p.phase == 2) {
        // the carry into this chunk, folded in chunk order
        const size_t s0 = (size_t)tile * p.n_chunks;
#pragma unroll
        for (int i = 0; i < NG; ++i) h[i] = ld_cg(&p.incH[s0 * sfl + my_off + i]);
        constexpr int FB = 4;  // aggregates whose loads are in flight together
        for (int m0 = 1; m0 < chunk; m0 += FB) {
            float S[FB], H[FB][NG];
#pragma unroll
            for (int q = 0; q < FB; ++q) {
                const size_t sm = s0 + min(m0 + q, chunk - 1);
                S[q] = ld_cg(&p.aggP[sm * sfl + c]);
#pragma unroll
                for (int i = 0; i < NG; ++i) H[q][i] = ld_cg(&p.aggH[sm * sfl + my_off + i]);
            }
#pragma unroll
            for (int q = 0; q < FB; ++q) {
                if (m0 + q >= chunk) break;
#pragma unroll
                for (int i = 0; i < NG; ++i) h[i] = fmaf(ex2(A2[i] * S[q]), h[i], H[q][i]);
            }
        }
    }
    float ssum = 0.0f;  // this lane's share of the chunk's sum of delta (aggregate only)
    T* yrow = static_cast<T*>(p.y) + (row0 + c) * (size_t)L;
    const bool wide = sizeof(T) == 4 && (L & 7) == 0 && (reinterpret_cast<uintptr_t>(p.y) & 31) == 0;
    constexpr int RP = WS::RP > 0 ? WS::RP : 1;
    // low rank: this channel's Wup row, in shared memory (a padded stride:
    // conflict-free) to leave the registers to the states
    float* wr = reinterpret_cast<float*>(smem + wup_off) + c * (RP + 1);
    if constexpr (WS::RP > 0) {
        if (g == 0) {
#pragma unroll
            for (int r = 0; r < RP; ++r) wr[r] = (cval && r < p.R) ? p.Wup[((size_t)k * p.D + d) * p.R + r] : 0.0f;
        }
        __syncwarp();
    }
    // u and delta = softplus(raw + bias) of this channel over steps t0 .. t0 + ST - 1 of
    // the stage in `slot`
    auto block_in = [&](int slot, int t0, Steps<WS::ST>& uv, Steps<WS::ST>& dv) {
        const unsigned char* ru = smem + slot * LY::RAW_STAGE;
        const unsigned char* rd = ru + LY::U_BYTES;
        constexpr int E = 16 / (int)sizeof(T);  // elements of a 16-byte piece
        auto at = [&](const unsigned char* b, int t) {  // address of step t (a multiple of 4) of this channel's row
            return reinterpret_cast<const T*>(b + LY::piece(c, t / E)) + t % E;
        };
#pragma unroll
        for (int j = 0; j < ST; j += 4) {
            float q[4];
            if (urev) {
                // the mirrored box, read from its end
                load4(at(ru, TS - 4 - t0 - j), q);
#pragma unroll
                for (int e = 0; e < 4; ++e) uv[j + e] = q[3 - e];
            } else {
                load4(at(ru, t0 + j), q);
#pragma unroll
                for (int e = 0; e < 4; ++e) uv[j + e] = q[e];
            }
        }
        // this lane's steps: t0 + g ST / G .. t0 + (g + 1) ST / G - 1
        constexpr int SPL = ST / G;
        static_assert(SPL % 4 == 0, "steps per lane: whole reads of four");
        float own[SPL];
        if constexpr (WS::RP == 0) {
#pragma unroll
            for (int j = 0; j < SPL; j += 4) {
                float w[4];
                load4(at(rd, t0 + g * SPL + j), w);
#pragma unroll
                for (int e = 0; e < 4; ++e) own[j + e] = w[e] + bias;
            }
        } else {
            // raw Delta = sum_r Wup[r] z_r, r in order (the z rows are broadcast reads)
            // (packed: each lane of a pair is the same fused multiply-add as fmaf)
            const float* zr = reinterpret_cast<const float*>(rd) + t0 + g * SPL;
            float2 raw[SPL / 2];
#pragma unroll
            for (int j = 0; j < SPL / 2; ++j) raw[j] = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int r = 0; r < RP; ++r) {
                if (r < p.R) {
                    const float2 w2 = make_float2(wr[r], wr[r]);
#pragma unroll
                    for (int j = 0; j < SPL; j += 2)
                        raw[j / 2] = __ffma2_rn(w2, *reinterpret_cast<const float2*>(zr + r * TS + j), raw[j / 2]);
                }
            }
#pragma unroll
            for (int j = 0; j < SPL; j += 2) {
                own[j] = raw[j / 2].x + bias;
                own[j + 1] = raw[j / 2].y + bias;
            }
        }
        if (p.softplus_on) {
#pragma unroll
            for (int j = 0; j < SPL; j += 2) {
                const float2 v = softplus2(make_float2(own[j], own[j + 1]));
                own[j] = v.x;
                own[j + 1] = v.y;
            }
        }
        if constexpr (G == 1) {
#pragma unroll
            for (int j = 0; j < ST; ++j) dv[j] = own[j];
        } else {
#pragma unroll
            for (int j = 0; j < SPL; ++j) {
                const float o = __shfl_xor_sync(0xffffffffu, own[j], 1);
                dv[j] = g ? o : own[j];
                dv[SPL + j] = g ? own[j] : o;
            }
        }
    };
    // those steps of the recurrence; yv: the sums over this lane's states
    auto update = [&](int slot, int t0, const Steps<WS::ST>& uv, const Steps<WS::ST>& dv, auto y_tag, Steps<WS::ST>& yv) {
        constexpr bool WITH_Y = decltype(y_tag)::value;
        const float* bct = reinterpret_cast<const float*>(smem + bct_off + slot * LY::BCT_STAGE) + t0 * 2 * NP + g * NG;
#pragma unroll
        for (int j = 0; j < ST; ++j) {
            const float du = dv[j] * uv[j];
            const float* bt = bct + j * 2 * NP;
            if constexpr (NG == 1) {
                const float2 bc = *reinterpret_cast<const float2*>(bt);
                h[0] = fmaf(ex2(dv[j] * A2[0]), h[0], du * bc.x);
                if constexpr (WITH_Y) yv[j] = bc.y * h[0];
            } else {
                const float2 dd = make_float2(dv[j], dv[j]), uu = make_float2(du, du);
                float2 ya = make_float2(0.0f, 0.0f);
                auto pair = [&](int n, float2 b, float2 cc) {
                    const float2 x = __fmul2_rn(dd, make_float2(A2[n], A2[n + 1]));
                    const float2 hn = __ffma2_rn(make_float2(ex2(x.x), ex2(x.y)), make_float2(h[n], h[n + 1]),
                                                 __fmul2_rn(uu, b));
                    h[n] = hn.x;
                    h[n + 1] = hn.y;
                    if constexpr (WITH_Y) ya = __ffma2_rn(cc, hn, ya);
                };
                if constexpr (NG % 4 == 0) {
#pragma unroll
                    for (int q = 0; q < NG / 4; ++q) {
                        const float4 b = *reinterpret_cast<const float4*>(bt + 4 * q);
                        const float4 cc = WITH_Y ? *reinterpret_cast<const float4*>(bt + NP + 4 * q)
                                                 : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        pair(4 * q, make_float2(b.x, b.y), make_float2(cc.x, cc.y));
                        pair(4 * q + 2, make_float2(b.z, b.w), make_float2(cc.z, cc.w));
                    }
                } else {
                    pair(0, *reinterpret_cast<const float2*>(bt), *reinterpret_cast<const float2*>(bt + NP));
                }
                if constexpr (WITH_Y) yv[j] = ya.x + ya.y;
            }
        }
    };
    // y = sum over the channel's lanes + D u, stored from registers
    auto store = [&](int l0, const Steps<WS::ST>& uv, const Steps<WS::ST>& yv) {
        const int nvalid = l_end - l0;
        if constexpr (G == 1) {
            float o[ST];
#pragma unroll
            for (int j = 0; j < ST; ++j) o[j] = fmaf(dsk, uv[j], yv[j]);
            if (!cval) return;
            bool done = false;
            if constexpr (sizeof(T) == 4 && ST == 8) {
                if (wide && nvalid >= 8) {
                    store8(reinterpret_cast<float*>(yrow) + l0, o);
                    done = true;
                }
            }
            if (!done) {
#pragma unroll
                for (int j = 0; j < ST; j += 4) {
                    const float q[4] = {o[j], o[j + 1], o[j + 2], o[j + 3]};
                    store_row<T, 4>(yrow + l0 + j, q, nvalid - j, true);
                }
            }
        } else {
            // lane g keeps its half of the steps
            constexpr int SPL = ST / 2;
            float o[SPL];
#pragma unroll
            for (int j = 0; j < SPL; ++j) {
                const float keep = g ? yv[SPL + j] : yv[j], send = g ? yv[j] : yv[SPL + j];
                const float sum = keep + __shfl_xor_sync(0xffffffffu, send, 1);
                o[j] = fmaf(dsk, g ? uv[SPL + j] : uv[j], sum);
            }
            if (!cval) return;
#pragma unroll
            for (int j = 0; j < SPL; j += 4) {
                const float q[4] = {o[j], o[j + 1], o[j + 2], o[j + 3]};
                store_row<T, 4>(yrow + l0 + g * SPL + j, q, nvalid - g * SPL - j, true);
            }
        }
    };
    auto run = [&](auto y_tag) -> bool {
        constexpr bool WITH_Y = decltype(y_tag)::value;
        int slot = 0;
        unsigned par = 0;
#pragma unroll 1
        for (int s = 0; s < nst; ++s) {
            if (!__all_sync(0xffffffffu, mbarrier_wait(ready(slot), par, kStageWaitNs))) return false;
#pragma unroll 1
            for (int t0 = 0; t0 < TS; t0 += ST) {
                Steps<WS::ST> uv, dv, yv;
                block_in(slot, t0, uv, dv);
                update(slot, t0, uv, dv, y_tag, yv);
                if constexpr (WITH_Y) {
                    store(l_begin + s * TS + t0, uv, yv);
                } else {
#pragma unroll
                    for (int j = 0; j < ST; ++j) ssum += dv[j];  // every step of an aggregated chunk is in range
                }
            }
            __syncwarp();
            if (lane == 0) mbarrier_arrive(released(slot));
            if (++slot == nstg) slot = 0, par ^= 1u;
        }
        return true;
    };
    const bool done = agg ? run(std::false_type{}) : run(std::true_type{});
    if (!done) {
        if (lane == 0) atomicOr(&p.hdr->err, kErrTimeout);
        return;
    }
    if (p.phase == 1) {
        const size_t slot = (size_t)tile * p.n_chunks + chunk;
        float* dst = (agg ? p.aggH : p.incH) + slot * sfl + my_off;
#pragma unroll
        for (int i = 0; i < NG; ++i) dst[i] = h[i];
        if (agg && g == 0) p.aggP[slot * sfl + c] = ssum;
    }
}

template <typename T, class WS>
WsKernel ws_info() {
    using LY = WsTileLayout<T, WS>;
    const void* fn = reinterpret_cast<const void*>(&full_ws_kernel<T, WS>);
    static std::once_flag once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(once, [&] {
        attr_err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallMaxSmem);
    });
    return {attr_err == cudaSuccess ? fn : nullptr, LY::PER_SLOT, LY::WUP_BYTES, LY::G, LY::DT, LY::THREADS, LY::TS};
}

// The instances of one storage type by padded state count and variant (16
// states), gathering from the map, or of the low-rank form of rank <= 8 or
// <= 16 (16 states only).
template <typename T, int NP, int G, int TS, int ST, int MINB>
WsKernel ws_pick_form(bool gather, int R) {
    if (gather) return ws_info<T, WsShape<NP, G, 4, TS, ST, MINB, 0, true>>();
    if constexpr (NP == 16) {
        if (R > 8) return ws_info<T, WsShape<NP, G, 4, TS, ST, MINB, 16>>();
        if (R > 0) return ws_info<T, WsShape<NP, G, 4, TS, ST, MINB, 8>>();
    }
    return ws_info<T, WsShape<NP, G, 4, TS, ST, MINB>>();
}

template <typename T>
WsKernel ws_pick(int np, int variant, bool gather, int R) {
    switch (np) {
    case 1: return ws_pick_form<T, 1, 1, 16, 8, 3>(gather, 0);
    case 2: return ws_pick_form<T, 2, 1, 16, 8, 3>(gather, 0);
    case 4: return ws_pick_form<T, 4, 1, 16, 8, 3>(gather, 0);
    case 8:
        if (variant == kWsTwoLanes) return ws_pick_form<T, 8, 2, 16, 16, 3>(gather, 0);
        return ws_pick_form<T, 8, 1, 8, 8, 4>(gather, 0);
    default:
        if (variant == kWsTwoLanes) return ws_pick_form<T, 16, 2, 16, 16, 3>(gather, R);
        return ws_pick_form<T, 16, 1, 8, 8, 4>(gather, R);
    }
}

}  // namespace vmb
