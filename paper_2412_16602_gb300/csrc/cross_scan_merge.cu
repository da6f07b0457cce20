// cross_scan_merge.cu - SS2D cross-scan and cross-merge (App. A, "VMamba") for sm_103a.
//
// cross-scan: x[B,D,H,W] -> xs[B,4,D,L], direction 0 row-major, 1 column-major,
// 2 and 3 the reverses of 0 and 1.  cross-merge: ys[B,4,D,L] -> out[B,D,H,W],
// out = (ys0[p0] + ys2[p2]) + (ys1[p1] + ys3[p3]) in fp32 in that order.
// Maps below 1024 pixels: a CTA stages ppc whole maps (planes) in shared memory
// with a padded row stride, which keeps the column-major accesses free of bank
// conflicts; global loads and stores are 16-byte vectors when rows are 16-byte
// aligned.  Larger maps use band kernels: one CTA per band of rows of one map
// (eight for the scan, up to 32 for the merge; see below), which keeps batch-1
// problems parallel.  Which kernel takes rows too long for that: csm_kernel.
#include <algorithm>
#include <type_traits>

#include "vmb_common.cuh"
#include "vmb_internal.h"

namespace vmb {
namespace {

constexpr int kThreads = 256;
constexpr size_t kMaxSmem = 200 * 1024;

struct CsmParams {
    const void* in;
    void* out;
    int D, H, W, L;
    long long planes;  // B * D
    int ppc;           // planes per CTA
    int tabn;          // entries of one index table, padded (8-byte multiple)
    int vec;
    FastDiv fL, fW, fH, fD;
};

template <typename T>
union Vec {
    uint4 v;
    T e[16 / sizeof(T)];
};

// Tile indices of a plane's positions, computed once per CTA (the planes of a CTA
// share them; a division per element and plane was half of these kernels'
// instructions): row[r] of pixel r in row-major order, col[m] of the m-th pixel in
// column-major order.
__device__ __forceinline__ void plane_tables(unsigned short* row, unsigned short* col, const CsmParams& p, bool by_col) {
    for (int i = threadIdx.x; i < p.L; i += kThreads) {
        const int h = (int)fdiv((unsigned)i, p.fW), w = i - h * p.W;
        row[i] = (unsigned short)(by_col ? w * (p.H + 1) + h : h * (p.W + 1) + w);
        const int w1 = (int)fdiv((unsigned)i, p.fH), h1 = i - w1 * p.H;
        col[i] = (unsigned short)(by_col ? w1 * (p.H + 1) + h1 : h1 * (p.W + 1) + w1);
    }
}

// Without tables (TAB false: planes of kBandMinL pixels or more, whose tables would
// take shared memory from the plane and are used for one plane only) the indices
// are computed where they are used.
struct PlaneIndex {
    const unsigned short* tab;
    FastDiv f;   // positions along one row of this order
    int sm, sq;  // tile strides of the quotient and of the remainder
    template <bool TAB>
    __device__ __forceinline__ unsigned at(unsigned i) const {
        if constexpr (TAB) return tab[i];
        const unsigned q = fdiv(i, f);
        return q * sm + (i - q * f.d) * sq;
    }
};
// Index of the tile [H][W+1] (by_col false) or [W][H+1] in row-major and column-major order.
__device__ __forceinline__ PlaneIndex row_index(const unsigned short* tab, const CsmParams& p, bool by_col) {
    return {tab, p.fW, by_col ? 1 : p.W + 1, by_col ? p.H + 1 : 1};
}
__device__ __forceinline__ PlaneIndex col_index(const unsigned short* tab, const CsmParams& p, bool by_col) {
    return {tab, p.fH, by_col ? p.H + 1 : 1, by_col ? 1 : p.W + 1};
}

// Directions 0 and 2 are written straight from the loaded values, 1 and 3 (the same
// values in opposite orders) from the staged planes.
template <typename T, bool TAB>
__global__ void __launch_bounds__(kThreads) cross_scan_kernel(const CsmParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = p.L, PS = p.H * (p.W + 1);
    unsigned short* rtab = reinterpret_cast<unsigned short*>(smem_raw);  // [L] (TAB)
    unsigned short* ctab = rtab + p.tabn;                                // [L]
    T* sp = reinterpret_cast<T*>(ctab + p.tabn);                         // [ppc][H][W+1]
    constexpr int VE = 16 / sizeof(T);
    if constexpr (TAB) plane_tables(rtab, ctab, p, false);
    const PlaneIndex row = row_index(rtab, p, false), col = col_index(ctab, p, false);
    pdl_wait();
    pdl_launch_dependents();
    __syncthreads();
    const T* x = static_cast<const T*>(p.in);
    T* xs = static_cast<T*>(p.out);
    const long long p0 = (long long)blockIdx.x * p.ppc;
    const int np = (int)min((long long)p.ppc, p.planes - p0);
    const unsigned n = (unsigned)(np * L);
    const T* src = x + p0 * L;
    const size_t DL = (size_t)p.D * L;
    // direction 0's row of a plane; direction k's is k DL further
    auto base = [&](unsigned j) {
        const unsigned pi = (unsigned)(p0 + j), b = fdiv(pi, p.fD);
        return xs + ((size_t)pi + (size_t)3 * p.D * b) * L;
    };
    if (p.vec) {
#pragma unroll 2
        for (unsigned i = threadIdx.x * VE; i < n; i += kThreads * VE) {
            Vec<T> v, r;
            v.v = *reinterpret_cast<const uint4*>(src + i);
            const unsigned j = fdiv(i, p.fL), l = i - j * L;
#pragma unroll
            for (int q = 0; q < VE; ++q) {
                sp[j * PS + row.template at<TAB>(l + q)] = v.e[q];
                r.e[q] = v.e[VE - 1 - q];
            }
            T* o = base(j);
            *reinterpret_cast<uint4*>(o + l) = v.v;
            *reinterpret_cast<uint4*>(o + 2 * DL + (L - VE - l)) = r.v;
        }
    } else {
#pragma unroll 2
        for (unsigned i = threadIdx.x; i < n; i += kThreads) {
            const T v = src[i];
            const unsigned j = fdiv(i, p.fL), l = i - j * L;
            sp[j * PS + row.template at<TAB>(l)] = v;
            T* o = base(j);
            o[l] = v;
            o[2 * DL + (L - 1 - l)] = v;
        }
    }
    __syncthreads();
    if (p.vec) {
#pragma unroll 2
        for (unsigned i = threadIdx.x * VE; i < n; i += kThreads * VE) {
            const unsigned j = fdiv(i, p.fL), l = i - j * L;
            Vec<T> v, r;
#pragma unroll
            for (int q = 0; q < VE; ++q) {
                v.e[q] = sp[j * PS + col.template at<TAB>(l + q)];
                r.e[VE - 1 - q] = v.e[q];
            }
            T* o = base(j);
            *reinterpret_cast<uint4*>(o + DL + l) = v.v;
            *reinterpret_cast<uint4*>(o + 3 * DL + (L - VE - l)) = r.v;
        }
    } else {
#pragma unroll 2
        for (unsigned i = threadIdx.x; i < n; i += kThreads) {
            const unsigned j = fdiv(i, p.fL), l = i - j * L;
            const T v = sp[j * PS + col.template at<TAB>(l)];
            T* o = base(j);
            o[DL + l] = v;
            o[3 * DL + (L - 1 - l)] = v;
        }
    }
}

// ys1 + ys3 of every pixel is formed in column-major order and staged in fp32,
// then added to ys0 + ys2 in row order (the sums and their order as stated above).
template <typename T, bool TAB>
__global__ void __launch_bounds__(kThreads) cross_merge_kernel(const CsmParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = p.L, PS = p.W * (p.H + 1);
    unsigned short* rtab = reinterpret_cast<unsigned short*>(smem_raw);  // [L] (TAB)
    unsigned short* ctab = rtab + p.tabn;                                // [L]
    float* sp = reinterpret_cast<float*>(ctab + p.tabn);                 // [ppc][W][H+1]
    constexpr int VE = 16 / sizeof(T);
    if constexpr (TAB) plane_tables(rtab, ctab, p, true);
    const PlaneIndex row = row_index(rtab, p, true), col = col_index(ctab, p, true);
    pdl_wait();
    pdl_launch_dependents();
    __syncthreads();
    const long long p0 = (long long)blockIdx.x * p.ppc;
    const int np = (int)min((long long)p.ppc, p.planes - p0);
    const T* ys = static_cast<const T*>(p.in);
    T* out = static_cast<T*>(p.out) + p0 * L;
    const unsigned n = (unsigned)(np * L);
    const size_t DL = (size_t)p.D * L;
    auto base = [&](unsigned j) {
        const unsigned pi = (unsigned)(p0 + j), b = fdiv(pi, p.fD);
        return ys + ((size_t)pi + (size_t)3 * p.D * b) * L;
    };
    if (p.vec) {
#pragma unroll 2
        for (unsigned i = threadIdx.x * VE; i < n; i += kThreads * VE) {
            const unsigned j = fdiv(i, p.fL), l = i - j * L;
            const T* o = base(j);
            Vec<T> v1, v3;
            v1.v = *reinterpret_cast<const uint4*>(o + DL + l);
            v3.v = *reinterpret_cast<const uint4*>(o + 3 * DL + (L - VE - l));  // reversed block
#pragma unroll
            for (int q = 0; q < VE; ++q) sp[j * PS + col.template at<TAB>(l + q)] = io<T>::cvt(v1.e[q]) + io<T>::cvt(v3.e[VE - 1 - q]);
        }
    } else {
#pragma unroll 2
        for (unsigned i = threadIdx.x; i < n; i += kThreads) {
            const unsigned j = fdiv(i, p.fL), l = i - j * L;
            const T* o = base(j);
            sp[j * PS + col.template at<TAB>(l)] = io<T>::cvt(o[DL + l]) + io<T>::cvt(o[3 * DL + (L - 1 - l)]);
        }
    }
    __syncthreads();
    if (p.vec) {
#pragma unroll 2
        for (unsigned i = threadIdx.x * VE; i < n; i += kThreads * VE) {
            const unsigned j = fdiv(i, p.fL), l = i - j * L;
            const T* y = base(j);
            Vec<T> v0, v2, o;
            v0.v = *reinterpret_cast<const uint4*>(y + l);
            v2.v = *reinterpret_cast<const uint4*>(y + 2 * DL + (L - VE - l));  // reversed block
#pragma unroll
            for (int q = 0; q < VE; ++q) {
                const float a = io<T>::cvt(v0.e[q]) + io<T>::cvt(v2.e[VE - 1 - q]);
                o.e[q] = io<T>::to(a + sp[j * PS + row.template at<TAB>(l + q)]);
            }
            *reinterpret_cast<uint4*>(out + i) = o.v;
        }
    } else {
#pragma unroll 2
        for (unsigned i = threadIdx.x; i < n; i += kThreads) {
            const unsigned j = fdiv(i, p.fL), l = i - j * L;
            const T* y = base(j);
            const float a = io<T>::cvt(y[l]) + io<T>::cvt(y[2 * DL + (L - 1 - l)]);
            out[i] = io<T>::to(a + sp[j * PS + row.template at<TAB>(l)]);
        }
    }
}

// ---------------------------------------------------------------- band kernels
// Maps of at least kBandMinL pixels: one CTA per band of rows of one map, so
// that even a batch-1 problem has enough CTAs.  Directions 0 and 2 of a band are
// one contiguous run of the sequence; directions 1 and 3 are W runs of one step
// per row of the band, written from (scan) or read into (merge) a [rows][W+1]
// shared tile.  The scan takes bands of kRB rows; the merge takes taller bands
// (mrb rows, chosen on the host), whose runs of directions 1 and 3 are longer
// reads (measured on GB300: 32-row fp32 bands 305 us against 337 us for 8 rows
// on the batch-128 56x56 map; 16 rows best for bf16).
constexpr int kRB = 8;
constexpr int kBandMinL = 1024;
constexpr int kBandThreads = 128;

// Rows of a merge band: 32 (fp32) or 16 (bf16), fewer while the tiles would not fit.
inline int merge_band_rows(int W, int es) {
    int mrb = es == 4 ? 32 : 16;
    while (mrb > kRB && (size_t)2 * mrb * (W + 1) * es > kMaxSmem) mrb /= 2;
    return mrb;
}

struct BandParams {
    const void* in;
    void* out;
    int D, H, W, L;
    int nbands;  // bands per map
    int vec;     // W and H multiples of the vector width, 16-byte aligned bases
    int mrb;     // merge: rows per band (a multiple of 8)
};

template <typename T>
__global__ void __launch_bounds__(kBandThreads) cross_scan_band_kernel(const BandParams p) {
    pdl_wait();
    pdl_launch_dependents();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* tile = reinterpret_cast<T*>(smem_raw);  // [kRB][W+1]
    constexpr int VE = 16 / sizeof(T);
    const int W = p.W, H = p.H, L = p.L, WP = p.W + 1;
    const long long plane = blockIdx.x / p.nbands;
    const int band = blockIdx.x % p.nbands;
    const int h0 = band * kRB;
    const int rb = min(kRB, H - h0);
    const int n = rb * W;
    const long long b = plane / p.D, d = plane % p.D;
    const T* src = static_cast<const T*>(p.in) + plane * L + (long long)h0 * W;
    T* xs = static_cast<T*>(p.out);
    T* row0 = xs + ((b * 4 + 0) * p.D + d) * L;
    T* row1 = xs + ((b * 4 + 1) * p.D + d) * L;
    T* row2 = xs + ((b * 4 + 2) * p.D + d) * L;
    T* row3 = xs + ((b * 4 + 3) * p.D + d) * L;
    if (p.vec) {
        for (int e = threadIdx.x * VE; e < n; e += kBandThreads * VE) {
            Vec<T> v, r;
            v.v = *reinterpret_cast<const uint4*>(src + e);
            const int j = e / W, w = e - j * W;  // a vector never crosses a row (W % VE == 0)
#pragma unroll
            for (int q = 0; q < VE; ++q) {
                tile[j * WP + w + q] = v.e[q];
                r.e[q] = v.e[VE - 1 - q];
            }
            *reinterpret_cast<uint4*>(row0 + (long long)h0 * W + e) = v.v;           // direction 0
            *reinterpret_cast<uint4*>(row2 + L - (long long)h0 * W - e - VE) = r.v;  // direction 2
        }
    } else {
        for (int e = threadIdx.x; e < n; e += kBandThreads) {
            const T v = src[e];
            const int j = e / W, w = e - j * W;
            tile[j * WP + w] = v;
            row0[(long long)h0 * W + e] = v;
            row2[L - 1 - (long long)h0 * W - e] = v;
        }
    }
    __syncthreads();
    // directions 1 and 3: for each column w, the steps w*H + h0 .. w*H + h0 + rb - 1
    if (p.vec && rb == kRB) {
        constexpr int RV = kRB / VE;  // vectors per run
        for (int i = threadIdx.x; i < W * RV; i += kBandThreads) {
            const int w = i / RV, jv = (i - w * RV) * VE;
            Vec<T> v, r;
#pragma unroll
            for (int q = 0; q < VE; ++q) {
                v.e[q] = tile[(jv + q) * WP + w];
                r.e[q] = tile[(jv + VE - 1 - q) * WP + w];
            }
            const long long pos = (long long)w * H + h0 + jv;
            *reinterpret_cast<uint4*>(row1 + pos) = v.v;
            *reinterpret_cast<uint4*>(row3 + L - pos - VE) = r.v;
        }
    } else {
        for (int e = threadIdx.x; e < n; e += kBandThreads) {
            const int w = e / rb, j = e - w * rb;
            const T v = tile[j * WP + w];
            const long long pos = (long long)w * H + h0 + j;
            row1[pos] = v;
            row3[L - 1 - pos] = v;
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(kBandThreads) cross_merge_band_kernel(const BandParams p) {
    pdl_wait();
    pdl_launch_dependents();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int W = p.W, H = p.H, L = p.L, WP = p.W + 1;
    T* s1 = reinterpret_cast<T*>(smem_raw);  // [mrb][W+1]: ys1 at pixel (h0 + j, w)
    T* s3 = s1 + p.mrb * WP;                   // [mrb][W+1]: ys3 at pixel (h0 + j, w)
    constexpr int VE = 16 / sizeof(T);
    const long long plane = blockIdx.x / p.nbands;
    const int band = blockIdx.x % p.nbands;
    const int h0 = band * p.mrb;
    const int rb = min(p.mrb, H - h0);
    const int n = rb * W;
    const long long b = plane / p.D, d = plane % p.D;
    const T* ys = static_cast<const T*>(p.in);
    const T* row0 = ys + ((b * 4 + 0) * p.D + d) * L;
    const T* row1 = ys + ((b * 4 + 1) * p.D + d) * L;
    const T* row2 = ys + ((b * 4 + 2) * p.D + d) * L;
    const T* row3 = ys + ((b * 4 + 3) * p.D + d) * L;
    T* out = static_cast<T*>(p.out) + plane * L + (long long)h0 * W;
    // stage directions 1 and 3 of the band's pixels
    if (p.vec && rb % VE == 0) {
        const int RV = rb / VE;  // vectors per run
        for (int i = threadIdx.x; i < W * RV; i += kBandThreads) {
            const int w = i / RV, jv = (i - w * RV) * VE;
            const long long pos = (long long)w * H + h0 + jv;
            Vec<T> v1, v3;
            v1.v = *reinterpret_cast<const uint4*>(row1 + pos);
            v3.v = *reinterpret_cast<const uint4*>(row3 + L - pos - VE);
#pragma unroll
            for (int q = 0; q < VE; ++q) {
                s1[(jv + q) * WP + w] = v1.e[q];
                s3[(jv + q) * WP + w] = v3.e[VE - 1 - q];
            }
        }
    } else {
        for (int e = threadIdx.x; e < n; e += kBandThreads) {
            const int w = e / rb, j = e - w * rb;
            const long long pos = (long long)w * H + h0 + j;
            s1[j * WP + w] = row1[pos];
            s3[j * WP + w] = row3[L - 1 - pos];
        }
    }
    __syncthreads();
    // out = (ys0 + ys2) + (ys1 + ys3), in this order
    if (p.vec) {
        for (int e = threadIdx.x * VE; e < n; e += kBandThreads * VE) {
            const int j = e / W, w = e - j * W;
            const long long pos = (long long)h0 * W + e;
            Vec<T> v0, v2, o;
            v0.v = *reinterpret_cast<const uint4*>(row0 + pos);
            v2.v = *reinterpret_cast<const uint4*>(row2 + L - pos - VE);
#pragma unroll
            for (int q = 0; q < VE; ++q) {
                const float a = io<T>::cvt(v0.e[q]) + io<T>::cvt(v2.e[VE - 1 - q]);
                const float c = io<T>::cvt(s1[j * WP + w + q]) + io<T>::cvt(s3[j * WP + w + q]);
                o.e[q] = io<T>::to(a + c);
            }
            *reinterpret_cast<uint4*>(out + e) = o.v;
        }
    } else {
        for (int e = threadIdx.x; e < n; e += kBandThreads) {
            const int j = e / W, w = e - j * W;
            const long long pos = (long long)h0 * W + e;
            const float a = io<T>::cvt(row0[pos]) + io<T>::cvt(row2[L - 1 - pos]);
            const float c = io<T>::cvt(s1[j * WP + w]) + io<T>::cvt(s3[j * WP + w]);
            out[e] = io<T>::to(a + c);
        }
    }
}

// Rows too long for a band in shared memory: one thread per element, plain gathers.
template <typename T>
__global__ void cross_scan_direct(const T* x, T* xs, int D, int H, int W, long long total) {
    pdl_wait();
    pdl_launch_dependents();
    const long long L = (long long)H * W;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const long long l = e % L, row = e / L;  // row = (b*4 + kd)*D + d
        const long long d = row % D, bk = row / D, kd = bk % 4, b = bk / 4;
        const long long m = kd >= 2 ? L - 1 - l : l;
        const long long h = (kd & 1) ? m % H : m / W;
        const long long w = (kd & 1) ? m / H : m % W;
        xs[e] = x[((b * D + d) * H + h) * W + w];
    }
}

template <typename T>
__global__ void cross_merge_direct(const T* ys, T* out, int D, int H, int W, long long total) {
    pdl_wait();
    pdl_launch_dependents();
    const long long L = (long long)H * W;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const long long pos = e % L, pl = e / L, d = pl % D, b = pl / D;
        const long long h = pos / W, w = pos % W, p1 = w * H + h;
        const T* r = ys + (b * 4 * D + d) * L;
        const long long st = (long long)D * L;
        const float a = io<T>::cvt(r[pos]) + io<T>::cvt(r[2 * st + L - 1 - pos]);
        const float c = io<T>::cvt(r[st + p1]) + io<T>::cvt(r[3 * st + L - 1 - p1]);
        out[e] = io<T>::to(a + c);
    }
}

}  // namespace

// Kernel of a cross-scan or cross-merge.  Below 1024 pixels whole planes are staged
// with index tables.  From there on bands of rows, or, where a row is too long for a band,
// whole planes with their indices computed (merges: if there is a plane for every SM and whole
// vectors can be copied; scans: for an eighth as many, or half as many element by element, as
// the gather reads every element four times); and where neither fits, or a plane takes more
// than kMaxSmem of staging (counted as two storage-type planes for the merge), bands only
// where enough of them share an SM, else the gather of single elements.  GB300, us,
// planes x H x W: scan, staged and gather, 40x1x9000 fp32 5.3 and 10.6, 16x1x9000 5.3 and 5.5,
// 40x12x3760 18.6 and 35, 192x8x6000 72 and 170; out of line 80x3x7001 bf16 22 and 33, 80x9x5001 fp32 45 and 66,
// 152x7x7743 bf16 54 and 145, 152x9x5001 99 and 125;
// merge 192x2x8000 12 and 18, 16x2x8000 8.7 and 3.9, 192x4x6000 (117 KB staged) 41 and 29.  Merge in bands and
// gather: 192x256x256 fp32 (64 KB a band) 92 and 104, bf16 30 and 102; 192x64x800 fp32
// (100 KB) 99 and 80; 16x512x512 fp32 (128 KB) 60 and 36; rows out of line 192x201x201 fp32
// (50 KB) 127 and 61, 16x401x399 bf16 (25 KB) 17 and 22, 192x7001x12 bf16 166 and 91.
// Scan in bands and gather 192x15x2999 fp32 out of line (94 KB) 188 and 160, 192x61x997 (31 KB) 123 and 219.
CsmKernel csm_kernel(bool merge, vmb_dtype dt, long long planes, int H, int W, bool aligned, int sms) {
    const long long L = (long long)H * W, es = dt == VMB_BF16 ? 2 : 4;
    if (planes >= (1ll << 31) || L * 4 >= (1ll << 31)) return CsmKernel::kGather;
    if (L < kBandMinL) return CsmKernel::kPlane;
    const bool band_fits = 2ll * kRB * (W + 1) * es <= (long long)kMaxSmem &&
                           planes * ((H + kRB - 1) / kRB) < (1ll << 31);
    const long long staged = merge ? 2ll * W * (H + 1) * es : (long long)H * (W + 1) * es;
    if (!band_fits) {
        const bool vec = aligned && L * es % 16 == 0;
        const bool whole = staged <= (long long)kMaxSmem &&
                           (merge ? vec && planes >= sms : vec ? 8 * planes >= sms : 2 * planes >= sms);
        return whole ? CsmKernel::kPlane : CsmKernel::kGather;
    }
    if (staged <= (long long)kMaxSmem) return CsmKernel::kBand;
    const int VE = (int)(16 / es);
    const bool vec = aligned && W % VE == 0 && H % VE == 0;
    const long long smem = merge ? 2ll * merge_band_rows(W, (int)es) * (W + 1) * es : (long long)kRB * (W + 1) * es;
    const bool fast = merge ? (vec ? smem <= 65 * 1024 : smem <= 32 * 1024 && (W >= 64 || planes < sms)) : vec || smem <= 64 * 1024;
    return fast ? CsmKernel::kBand : CsmKernel::kGather;
}

namespace {

template <typename T>
vmb_status launch_csm(bool merge, const void* in, void* outp, int B, int D, int H, int W, cudaStream_t stream) {
    const int L = H * W;
    const long long planes = (long long)B * D;
    const size_t es = sizeof(T);
    const auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    const bool aligned = al16(in) && al16(outp);
    const CsmKernel kernel = csm_kernel(merge, sizeof(T) == 2 ? VMB_BF16 : VMB_F32, planes, H, W, aligned, device_sm_count());
    if (kernel == CsmKernel::kGather) {
        const long long total = merge ? planes * L : planes * 4 * L;
        const int grid = (int)std::min<long long>((total + kThreads - 1) / kThreads, 152ll * 32);
        const void* fn = merge ? reinterpret_cast<const void*>(&cross_merge_direct<T>)
                               : reinterpret_cast<const void*>(&cross_scan_direct<T>);
        const T* src = static_cast<const T*>(in);
        T* dst = static_cast<T*>(outp);
        void* args[] = {&src, &dst, &D, &H, &W, const_cast<long long*>(&total)};
        return launch_kernel(fn, dim3(grid), dim3(kThreads), 0, args, stream) == cudaSuccess ? VMB_OK : VMB_ERR_CUDA;
    }
    if (kernel == CsmKernel::kBand) {
        BandParams bp{};
        bp.in = in;
        bp.out = outp;
        bp.D = D;
        bp.H = H;
        bp.W = W;
        bp.L = L;
        const int mrb = merge_band_rows(W, (int)es);
        bp.mrb = mrb;
        bp.nbands = merge ? (H + mrb - 1) / mrb : (H + kRB - 1) / kRB;
        const int VE = (int)(16 / es);
        bp.vec = (W % VE == 0) && (H % VE == 0) && aligned;
        const size_t smem = merge ? 2 * (size_t)mrb * (W + 1) * es : (size_t)kRB * (W + 1) * es;
        const void* fn = merge ? reinterpret_cast<const void*>(&cross_merge_band_kernel<T>)
                               : reinterpret_cast<const void*>(&cross_scan_band_kernel<T>);
        if (smem > 48 * 1024 &&
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) != cudaSuccess)
            return VMB_ERR_CUDA;
        void* args[] = {&bp};
        const unsigned nblk = (unsigned)(planes * bp.nbands);
        return launch_kernel(fn, dim3(nblk), dim3(kBandThreads), smem, args, stream) == cudaSuccess ? VMB_OK
                                                                                                     : VMB_ERR_CUDA;
    }
    // about 8K elements per CTA, bounded by shared memory, fewer while the grid would
    // leave SMs idle
    const bool tab = L < kBandMinL;  // index tables
    const int tabn = tab ? (L + 7) / 8 * 8 : 0;
    const size_t tables = (size_t)2 * tabn * 2, plane = merge ? (size_t)W * (H + 1) * 4 : (size_t)H * (W + 1) * es;
    long long want = std::max<long long>(1, std::min<long long>(8192 / L, planes / (4LL * device_sm_count())));
    while (want > 1 && tables + (size_t)want * plane > kMaxSmem) --want;
    const int ppc = (int)want;
    CsmParams p{};
    p.in = in;
    p.out = outp;
    p.D = D;
    p.H = H;
    p.W = W;
    p.L = L;
    p.planes = planes;
    p.ppc = ppc;
    p.tabn = tabn;
    p.vec = ((size_t)L * es % 16 == 0) && aligned;
    p.fL = make_fastdiv((unsigned)L);
    p.fW = make_fastdiv((unsigned)W);
    p.fH = make_fastdiv((unsigned)H);
    p.fD = make_fastdiv((unsigned)D);
    const size_t smem = tables + (size_t)ppc * plane;
    const void* fn = merge ? (tab ? reinterpret_cast<const void*>(&cross_merge_kernel<T, true>)
                                  : reinterpret_cast<const void*>(&cross_merge_kernel<T, false>))
                           : (tab ? reinterpret_cast<const void*>(&cross_scan_kernel<T, true>)
                                  : reinterpret_cast<const void*>(&cross_scan_kernel<T, false>));
    if (smem > 48 * 1024 && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) != cudaSuccess)
        return VMB_ERR_CUDA;
    const unsigned grid = (unsigned)((planes + ppc - 1) / ppc);
    void* args[] = {&p};
    return launch_kernel(fn, dim3(grid), dim3(kThreads), smem, args, stream) == cudaSuccess ? VMB_OK : VMB_ERR_CUDA;
}

}  // namespace

vmb_status launch_cross_scan(const void* x, void* xs, int B, int D, int H, int W, vmb_dtype dt, cudaStream_t stream) {
    return dt == VMB_BF16 ? launch_csm<__nv_bfloat16>(false, x, xs, B, D, H, W, stream)
                          : launch_csm<float>(false, x, xs, B, D, H, W, stream);
}

vmb_status launch_cross_merge(const void* ys, void* out, int B, int D, int H, int W, vmb_dtype dt, cudaStream_t stream) {
    return dt == VMB_BF16 ? launch_csm<__nv_bfloat16>(true, ys, out, B, D, H, W, stream)
                          : launch_csm<float>(true, ys, out, B, D, H, W, stream);
}

// ------------------------------------------- channel-mean path: broadcast + merge
// The channel-mean scan's output is y_k[b,d,l] = ybar_k[b,l] + Dskip[kD+d] u_k[b,d,l]
// (Eq. 9 broadcast), and every direction's u at the position it merges into is
// the map itself: u_k[b,d,p_k(h,w)] = x[b,d,h,w].  So the merged map is
//   out[b,d,h,w] = (y0 + y2) + (y1 + y3),  y_k = ybar_k[b, p_k] + Dskip[kD+d] x[b,d,h,w]
// (y_k = ybar_k[b, p_k] when the skip term is already folded into ybar), read
// from x and the four ybar rows of (b, .) without y ever being written.  The
// fp32 operations and their order are those of the broadcast and of the
// cross-merge, so fp32 results are bit-identical to the unfused path; bf16
// rounds once, at the end.  A thread owns MP consecutive positions and keeps
// their four ybar values in registers across the CTA's channels; MP is the most that 16-byte
// accesses and the row length allow (GB300, with four channels in flight, block from the map: 8 maps of
// 128x128x192 bf16 349 us with two positions, 328 with eight; 32 maps of 28x28x384 fp32 161 and 148).
namespace {
constexpr int kMMThreads = 128;
constexpr int kMMAhead = 4;  // channels whose loads a thread has in flight
constexpr int kMMMaxDC = 64;

struct MeanMergeParams {
    const void* x;
    void* out;
    const float* ybar;   // [B, 4, L]
    const float* Dskip;  // [4 D]
    int B, D, H, W;
    int per_channel;  // 0: skip already in ybar
    int vec;          // MP positions of a row vector-accessible (aligned rows, L % MP == 0)
    int dc;           // channels per CTA
};

// MP consecutive elements as fp32, and back (MP sizeof(T) bytes at once).
template <typename T, int MP>
struct MmVec {
    static constexpr int W = MP * (int)sizeof(T) / 4;  // 32-bit words
    static __device__ __forceinline__ void load(const T* q, unsigned (&r)[W]) {
        if constexpr (W == 4) {
            const uint4 v = *reinterpret_cast<const uint4*>(q);
            r[0] = v.x, r[1] = v.y, r[2] = v.z, r[3] = v.w;
        } else if constexpr (W == 2) {
            const uint2 v = *reinterpret_cast<const uint2*>(q);
            r[0] = v.x, r[1] = v.y;
        } else {
            r[0] = *reinterpret_cast<const unsigned*>(q);
        }
    }
    static __device__ __forceinline__ float get(const unsigned (&r)[W], int j) {
        if constexpr (sizeof(T) == 4) return __uint_as_float(r[j]);
        else return __uint_as_float((j & 1) ? (r[j / 2] & 0xffff0000u) : (r[j / 2] << 16));
    }
    static __device__ __forceinline__ void store(T* q, const float (&o)[MP], uint64_t pol) {
        unsigned r[W];
#pragma unroll
        for (int i = 0; i < W; ++i) {
            if constexpr (sizeof(T) == 4) r[i] = __float_as_uint(o[i]);
            else r[i] = __bfloat16_as_ushort(io<T>::to(o[2 * i])) |
                        ((unsigned)__bfloat16_as_ushort(io<T>::to(o[2 * i + 1])) << 16);
        }
        if constexpr (W == 4)
            asm volatile("st.global.L2::cache_hint.v4.b32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(q), "r"(r[0]), "r"(r[1]),
                         "r"(r[2]), "r"(r[3]), "l"(pol)
                         : "memory");
        else if constexpr (W == 2)
            asm volatile("st.global.L2::cache_hint.v2.b32 [%0], {%1, %2}, %3;" ::"l"(q), "r"(r[0]), "r"(r[1]), "l"(pol)
                         : "memory");
        else
            asm volatile("st.global.L2::cache_hint.b32 [%0], %1, %2;" ::"l"(q), "r"(r[0]), "l"(pol) : "memory");
    }
};

template <typename T, int MP>
__global__ void __launch_bounds__(kMMThreads) mean_merge_kernel(const MeanMergeParams p) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ float sd[4][kMMMaxDC];
    const int H = p.H, W = p.W, L = H * W;
    const int b = blockIdx.y;
    const int dbeg = blockIdx.z * p.dc, dn = min(p.dc, p.D - dbeg);
    for (int i = threadIdx.x; i < 4 * kMMMaxDC; i += kMMThreads) {
        const int kd = i / kMMMaxDC, j = i % kMMMaxDC;
        sd[kd][j] = (p.per_channel && j < dn) ? __ldg(p.Dskip + (size_t)kd * p.D + dbeg + j) : 0.0f;
    }
    const int pos0 = (blockIdx.x * kMMThreads + threadIdx.x) * MP;
    const float* yb = p.ybar + (size_t)b * 4 * L;
    float y0[MP], y1[MP], y2[MP], y3[MP];
#pragma unroll
    for (int j = 0; j < MP; ++j) {
        const int pos = pos0 + j;
        if (pos < L) {
            const int h = pos / W, w = pos - h * W, p1 = w * H + h;
            y0[j] = __ldg(yb + pos);
            y2[j] = __ldg(yb + 2 * (size_t)L + (L - 1 - pos));
            y1[j] = __ldg(yb + (size_t)L + p1);
            y3[j] = __ldg(yb + 3 * (size_t)L + (L - 1 - p1));
        } else {
            y0[j] = y1[j] = y2[j] = y3[j] = 0.0f;
        }
    }
    __syncthreads();
    if (pos0 >= L) return;
    const T* x = static_cast<const T*>(p.x) + ((size_t)b * p.D + dbeg) * L + pos0;
    T* out = static_cast<T*>(p.out) + ((size_t)b * p.D + dbeg) * L + pos0;
    const uint64_t ev = l2_evict_first();
    auto merged = [&](int dd, int j, float xv) {
        const float a = fmaf(sd[0][dd], xv, y0[j]) + fmaf(sd[2][dd], xv, y2[j]);
        const float c = fmaf(sd[1][dd], xv, y1[j]) + fmaf(sd[3][dd], xv, y3[j]);
        return a + c;
    };
    if (p.vec) {  // L is a multiple of MP: all of a thread's positions are in range
        using V = MmVec<T, MP>;
        for (int d0 = 0; d0 < dn; d0 += kMMAhead) {
            unsigned r[kMMAhead][V::W];
#pragma unroll
            for (int q = 0; q < kMMAhead; ++q)
                if (d0 + q < dn) V::load(x + (size_t)(d0 + q) * L, r[q]);
#pragma unroll
            for (int q = 0; q < kMMAhead; ++q) {
                if (d0 + q >= dn) break;
                float o[MP];
#pragma unroll
                for (int j = 0; j < MP; ++j) o[j] = merged(d0 + q, j, V::get(r[q], j));
                V::store(out + (size_t)(d0 + q) * L, o, ev);
            }
        }
        return;
    }
    for (int dd = 0; dd < dn; ++dd, x += L, out += L) {
#pragma unroll
        for (int j = 0; j < MP; ++j)
            if (pos0 + j < L) out[j] = io<T>::to(merged(dd, j, io<T>::cvt(x[j])));
    }
}

template <typename T, int MP>
vmb_status launch_mean_merge_mp(const void* x, const float* ybar, const float* Dskip, void* out, int B, int D, int H,
                                int W, bool per_channel, cudaStream_t stream) {
    const long long L = (long long)H * W;
    const unsigned nblk = (unsigned)((L + kMMThreads * MP - 1) / (kMMThreads * MP));
    // channels per CTA: enough CTAs for a few waves, each amortising its ybar
    // reads over as many channels as that leaves
    const long long per_ch = (long long)nblk * B;
    long long dc = per_ch * D / (8LL * device_sm_count());
    dc = dc < 8 ? 8 : dc > kMMMaxDC ? kMMMaxDC : dc;
    if (dc > D) dc = D;
    const auto al = [](const void* q, size_t a) { return (reinterpret_cast<uintptr_t>(q) % a) == 0; };
    MeanMergeParams p{};
    p.x = x;
    p.out = out;
    p.ybar = ybar;
    p.Dskip = Dskip;
    p.B = B;
    p.D = D;
    p.H = H;
    p.W = W;
    p.per_channel = per_channel ? 1 : 0;
    p.vec = (L % MP == 0) && al(x, MP * sizeof(T)) && al(out, MP * sizeof(T));
    p.dc = (int)dc;
    const dim3 grid(nblk, (unsigned)B, (unsigned)((D + dc - 1) / dc));
    if (grid.y > 65535u || grid.z > 65535u) return VMB_ERR_UNSUPPORTED;
    void* args[] = {&p};
    return launch_kernel(reinterpret_cast<const void*>(&mean_merge_kernel<T, MP>), grid, dim3(kMMThreads), 0, args,
                         stream) == cudaSuccess
               ? VMB_OK
               : VMB_ERR_CUDA;
}

template <typename T>
vmb_status launch_mean_merge_t(const void* x, const float* ybar, const float* Dskip, void* out, int B, int D, int H,
                               int W, bool per_channel, cudaStream_t stream) {
    const long long L = (long long)H * W;
    const auto fits = [&](int mp) {
        return L % mp == 0 && reinterpret_cast<uintptr_t>(x) % (mp * sizeof(T)) == 0 &&
               reinterpret_cast<uintptr_t>(out) % (mp * sizeof(T)) == 0;
    };
    if (sizeof(T) == 2 && fits(8))
        return launch_mean_merge_mp<T, sizeof(T) == 2 ? 8 : 4>(x, ybar, Dskip, out, B, D, H, W, per_channel, stream);
    if (fits(4)) return launch_mean_merge_mp<T, 4>(x, ybar, Dskip, out, B, D, H, W, per_channel, stream);
    return launch_mean_merge_mp<T, 2>(x, ybar, Dskip, out, B, D, H, W, per_channel, stream);
}
// ------------------------------------------------------------ map transpose
// xt[b, d, w, h] = x[b, d, h, w]: the column-major order of every (b, d) plane,
// which the column-major directions of the cross-scan (1 and 3) read as
// contiguous rows.  The scan that follows reads xt in half of its CTAs only (see
// pdl_wait in the gathering scans), so this kernel is built to run beside the
// other half: one CTA per SM, which starts, and lets the scan be launched, at
// once, and walks over the planes with the next item's loads in flight while the
// current one is written.  Both sides are contiguous runs of whole planes.  VEC
// (W and H multiples of a 16-byte vector): the pieces of a transposed row are
// permuted by the column's vector index, so that the element stores of a
// vector's columns and the vector reads of a row both spread over the banks.
constexpr int kTrThreads = 512;
constexpr int kTrVals = 4;    // vectors (VEC) or 4-element groups a thread holds
constexpr size_t kTrSmem = kTransposeSmem - 1024;

struct TransposeParams {
    const void* x;
    void* xt;
    int H, W, HP;      // HP: row stride of the transposed tile (elements)
    int ppi;           // planes per item
    long long planes, items;
    FastDiv fP, fA, fB;  // units per plane, per row of x, per row of xt
};

inline bool transpose_vec(const void* x, const void* xt, int H, int W, int es) {
    return W % (16 / es) == 0 && H % (16 / es) == 0 && ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(xt)) & 15u) == 0;
}
inline int transpose_stride(int H, int VE, bool vec) { return vec ? (H + 8 * VE - 1) / (8 * VE) * (8 * VE) : H | 1; }

template <typename T, bool VEC>
__global__ void __launch_bounds__(kTrThreads) map_transpose_kernel(const TransposeParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sp = reinterpret_cast<T*>(smem_raw);  // [ppi][W][HP]
    constexpr int VE = VEC ? 16 / (int)sizeof(T) : 1;  // elements per unit
    constexpr int NV = VEC ? kTrVals : 4 * kTrVals;    // units per thread and item
    using U = typename std::conditional<VEC, uint4, T>::type;
    pdl_wait();
    pdl_launch_dependents();
    const unsigned per_plane = p.fP.d;  // units per plane
    const U* x = static_cast<const U*>(p.x);
    U* xt = static_cast<U*>(p.xt);
    U v[NV];
    auto load = [&](long long item) {
        const long long p0 = item * p.ppi;
        const unsigned n = (unsigned)min((long long)p.ppi, p.planes - p0) * per_plane;
        const U* src = x + p0 * per_plane;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const unsigned i = threadIdx.x + q * kTrThreads;
            if (i < n) v[q] = src[i];
        }
    };
    long long item = blockIdx.x;
    if (item < p.items) load(item);
    for (; item < p.items; item += gridDim.x) {
        const long long p0 = item * p.ppi;
        const unsigned n = (unsigned)min((long long)p.ppi, p.planes - p0) * per_plane;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const unsigned i = threadIdx.x + q * kTrThreads;
            if (i >= n) break;
            const unsigned j = fdiv(i, p.fP), r = i - j * per_plane;
            const unsigned h = fdiv(r, p.fA), c = r - h * p.fA.d;  // row, unit within it
            if constexpr (VEC) {
                Vec<T> w;
                w.v = v[q];
                T* dst = sp + (size_t)(j * p.W + c * VE) * p.HP + (h ^ ((c & 7) * VE));
#pragma unroll
                for (int e = 0; e < VE; ++e) dst[e * p.HP] = w.e[e];
            } else {
                sp[(size_t)(j * p.W + c) * p.HP + h] = v[q];
            }
        }
        __syncthreads();
        if (item + gridDim.x < p.items) load(item + gridDim.x);
        U* dst = xt + p0 * per_plane;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const unsigned i = threadIdx.x + q * kTrThreads;
            if (i >= n) break;
            const unsigned j = fdiv(i, p.fP), r = i - j * per_plane;
            const unsigned w = fdiv(r, p.fB), u = r - w * p.fB.d;  // column, unit within it
            const T* src = sp + (size_t)(j * p.W + w) * p.HP + (VEC ? (u ^ ((w / VE) & 7)) * VE : u);
            dst[i] = *reinterpret_cast<const U*>(src);
        }
        __syncthreads();  // the tile is rewritten by the next item
    }
}

// Maps that do not fit an item, or as the caller asks: 32 x 32 tiles through shared memory (one padded
// column so the transposed reads hit distinct banks), coalesced on both sides.
constexpr int kTT = 32, kTR = 8;  // tile edge, rows per thread pass

template <typename T>
__global__ void __launch_bounds__(kTT * kTR) tile_transpose_kernel(const T* x, T* xt, int H, int W, int tiles_w,
                                                                  int tiles_per_plane) {
    __shared__ T tile[kTT][kTT + 1];
    pdl_wait();
    pdl_launch_dependents();
    const long long plane = blockIdx.x / tiles_per_plane;
    const int t = blockIdx.x % tiles_per_plane;
    const int h0 = (t / tiles_w) * kTT, w0 = (t % tiles_w) * kTT;
    const T* src = x + plane * (long long)H * W;
    T* dst = xt + plane * (long long)H * W;
    const int tx = threadIdx.x % kTT, ty = threadIdx.x / kTT;
#pragma unroll
    for (int r = ty; r < kTT; r += kTR) {
        const int h = h0 + r, w = w0 + tx;
        if (h < H && w < W) tile[r][tx] = src[(long long)h * W + w];
    }
    __syncthreads();
#pragma unroll
    for (int r = ty; r < kTT; r += kTR) {
        const int w = w0 + r, h = h0 + tx;
        if (h < H && w < W) dst[(long long)w * H + h] = tile[tx][r];
    }
}


template <typename T>
vmb_status launch_plane_transpose(const void* x, void* xt, long long planes, int H, int W, cudaStream_t stream) {
    const int VE = 16 / (int)sizeof(T);
    const bool vec = transpose_vec(x, xt, H, W, (int)sizeof(T));
    const int ve = vec ? VE : 1, nv = vec ? kTrVals : 4 * kTrVals;
    TransposeParams p{};
    p.x = x;
    p.xt = xt;
    p.H = H;
    p.W = W;
    p.HP = transpose_stride(H, VE, vec);
    const long long L = (long long)H * W;
    const size_t plane_bytes = (size_t)W * p.HP * sizeof(T);
    const long long fit = std::min<long long>((long long)nv * kTrThreads * ve / L, (long long)(kTrSmem / plane_bytes));
    const int sms = device_sm_count();
    p.ppi = (int)std::max<long long>(1, std::min(fit, (planes + sms - 1) / sms));
    p.planes = planes;
    p.items = (planes + p.ppi - 1) / p.ppi;
    p.fP = make_fastdiv((unsigned)(L / ve));
    p.fA = make_fastdiv((unsigned)(W / ve));
    p.fB = make_fastdiv((unsigned)(H / ve));
    void* args[] = {&p};
    const void* fn = vec ? reinterpret_cast<const void*>(&map_transpose_kernel<T, true>)
                         : reinterpret_cast<const void*>(&map_transpose_kernel<T, false>);
    return launch_kernel(fn, dim3((unsigned)std::min<long long>(p.items, sms)), dim3(kTrThreads), p.ppi * plane_bytes,
                         args, stream) == cudaSuccess
               ? VMB_OK
               : VMB_ERR_CUDA;
}

}  // namespace

bool transpose_by_planes(const void* x, const void* xt, int H, int W, vmb_dtype dt) {
    const int es = dt == VMB_BF16 ? 2 : 4, VE = 16 / es;
    const bool vec = transpose_vec(x, xt, H, W, es);
    return (long long)H * W <= (long long)(vec ? kTrVals * VE : 4 * kTrVals) * kTrThreads &&
           (size_t)W * transpose_stride(H, VE, vec) * es <= kTrSmem;
}

bool transpose_whole_vectors(const void* x, const void* xt, int H, int W, vmb_dtype dt) {
    return transpose_vec(x, xt, H, W, dt == VMB_BF16 ? 2 : 4);
}

vmb_status launch_map_transpose(const void* x, void* xt, int B, int D, int H, int W, vmb_dtype dt, bool planes,
                                cudaStream_t stream) {
    if (planes)
        return dt == VMB_BF16 ? launch_plane_transpose<__nv_bfloat16>(x, xt, (long long)B * D, H, W, stream)
                              : launch_plane_transpose<float>(x, xt, (long long)B * D, H, W, stream);
    const int tiles_h = (H + kTT - 1) / kTT, tiles_w = (W + kTT - 1) / kTT;
    const long long grid = (long long)B * D * tiles_h * tiles_w;
    if (grid > INT32_MAX) return VMB_ERR_UNSUPPORTED;
    int tpp = tiles_h * tiles_w, tw = tiles_w;
    const void* xp = x;
    void* args[] = {&xp, &xt, &H, &W, &tw, &tpp};
    const void* fn = dt == VMB_BF16 ? reinterpret_cast<const void*>(&tile_transpose_kernel<__nv_bfloat16>)
                                    : reinterpret_cast<const void*>(&tile_transpose_kernel<float>);
    return launch_kernel(fn, dim3((unsigned)grid), dim3(kTT * kTR), 0, args, stream) == cudaSuccess ? VMB_OK
                                                                                                  : VMB_ERR_CUDA;
}

vmb_status launch_mean_merge(const void* x, const float* ybar, const float* Dskip, void* out, int B, int D, int H,
                             int W, bool per_channel_skip, vmb_dtype dt, cudaStream_t stream) {
    return dt == VMB_BF16
               ? launch_mean_merge_t<__nv_bfloat16>(x, ybar, Dskip, out, B, D, H, W, per_channel_skip, stream)
               : launch_mean_merge_t<float>(x, ybar, Dskip, out, B, D, H, W, per_channel_skip, stream);
}

}  // namespace vmb
