// Layout conversion, the unfused one-thread-per-cell Yee step, and the FP64
// energy/divergence reductions.
//
// The unfused step is two launches per step (Listing 1: curl H components,
// then curl E components), each updating one copy of the fields in place; it
// is the debugging baseline of the fused kernels and the path for coefficient
// sets too varied for a one-byte material id (COEF_FULL) with a single step, a
// current or a probe, or when it is asked for.
#include <algorithm>

#include "df.cuh"
#include "launch.h"

namespace fdtd {

namespace {

constexpr int BXs = 32, BYs = 8;

// Up to six canonical arrays of one launch (read by pack and maxabs, written by unpack).
struct Canon6 {
    float *f[6];
};

// Layout conversion.  A warp takes one canonical row (component, k, j), its lanes step along x: the row's
// kind (cells, or one of the far faces) is the same for the whole warp, the active-layout side is 128-byte
// aligned, and kLayU loads per lane are issued before their stores.  16-bit rows move two cells per lane, so
// that a warp still writes (reads) 128 bytes of the active layout at a time.  One launch takes ncomp
// components: six launches per load cost a small cavity more than the copying did.  Bound by HBM; with
// one thread per (i, j) and four planes per thread (no row knowledge, single 16-bit stores) the six
// components took 600 us to load and 834 us to read back at 384^3 FP16, now 358 us (5.7 TB/s) and
// 476 us; at 256^3 FP32 192 and 166 us, now 144 and 148 us.  Threads over the flat (j, i) index measured
// 817 and 948 us (stores straddle rows).
constexpr int kLayThreads = 256, kLayU = 4;

struct LayoutRow {
    int q, comp, j, k;     // slot in Canon6, component, row
    bool ok;
};
__device__ __forceinline__ LayoutRow layout_row(const CavityDesc &d, int comp0, int ncomp) {
    LayoutRow r;
    const unsigned w = blockIdx.x * (kLayThreads / 32) + (threadIdx.x >> 5);
    const unsigned NY1 = d.ny + 1, NZ1 = d.nz + 1;
    const unsigned kq = w / NY1;
    r.j = (int)(w - kq * NY1);
    r.q = (int)(kq / NZ1);
    r.k = (int)(kq - (unsigned)r.q * NZ1);
    r.comp = comp0 + r.q;
    r.ok = r.q < ncomp;
    return r;
}

template <typename T> struct LayPack;   // cells per lane and the store / load of them
template <> struct LayPack<float> {
    static constexpr int V = 1;
    __device__ __forceinline__ static void st(float *p, const float *v) { *p = v[0]; }
    __device__ __forceinline__ static void ld(const float *p, float *v) { v[0] = *p; }
};
template <> struct LayPack<__half> {
    static constexpr int V = 2;
    __device__ __forceinline__ static void st(__half *p, const float *v) {
        *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(v[0], v[1]);
    }
    __device__ __forceinline__ static void ld(const __half *p, float *v) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(p));
        v[0] = f.x;
        v[1] = f.y;
    }
};
template <> struct LayPack<__nv_bfloat16> {
    static constexpr int V = 2;
    __device__ __forceinline__ static void st(__nv_bfloat16 *p, const float *v) {
        *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(v[0], v[1]);
    }
    __device__ __forceinline__ static void ld(const __nv_bfloat16 *p, float *v) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
        v[0] = f.x;
        v[1] = f.y;
    }
};

// Value of a far-face H entry after the storage rounding.
template <typename T> __device__ __forceinline__ float face_round(const CavityDesc &d, int comp, float v) {
    return Storage<T>::scaled ? Storage<T>::load(Storage<T>::store(v * d.scale[comp])) * d.inv_scale[comp] : v;
}

// Canonical components -> active layout (scaled, rounded; tangential E zeroed) and far faces.  Rows are
// padded to a pitch of 32 elements, so a pair that starts inside a row never leaves it; the cell past an odd
// nx is written 0, as the context's first clear left it.
template <typename T>
__global__ void __launch_bounds__(kLayThreads) pack_kernel(const CavityDesc d, int copy, int comp0, int ncomp,
                                                           const Canon6 canon) {
    constexpr int V = LayPack<T>::V;
    const LayoutRow r = layout_row(d, comp0, ncomp);
    if (!r.ok) return;
    const int nx = d.nx, ny = d.ny, nz = d.nz, lane = threadIdx.x & 31;
    const float *__restrict__ src = canon.f[r.q] + ((long long)r.k * (ny + 1) + r.j) * (nx + 1);
    float *face = r.comp >= 3 ? const_cast<float *>(d.face[r.comp - 3]) : nullptr;
    if (r.j < ny && r.k < nz) {
        T *dst = static_cast<T *>(d.buf[copy][r.comp]) + (long long)r.k * d.plane + (long long)r.j * d.pitch;
        // Ex is tangential on j = 0 and k = 0, Ey on i = 0 and k = 0, Ez on i = 0 and j = 0
        const bool zero_row = r.comp < 3 && ((r.k == 0 && r.comp != 2) || (r.j == 0 && r.comp != 1));
        const bool zero_i0 = r.comp == 1 || r.comp == 2;
        const float sc = d.scale[r.comp];
        for (int i0 = lane * V; i0 < nx; i0 += 32 * V * kLayU) {
            float v[kLayU][V];
#pragma unroll
            for (int u = 0; u < kLayU; ++u)
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    const int i = i0 + 32 * V * u + e;
                    v[u][e] = i < nx && !zero_row && !(zero_i0 && i == 0) ? src[i] : 0.f;
                }
#pragma unroll
            for (int u = 0; u < kLayU; ++u) {
                const int i = i0 + 32 * V * u;
                if (Storage<T>::scaled)
#pragma unroll
                    for (int e = 0; e < V; ++e) v[u][e] *= sc;
                if (i < nx) LayPack<T>::st(dst + i, v[u]);
            }
        }
        if (r.comp == 3 && lane == 0) face[(long long)r.k * ny + r.j] = face_round<T>(d, 3, src[nx]);
        return;
    }
    // far-face normal H (FP32, after the same storage rounding)
    if (r.comp == 4 && r.j == ny && r.k < nz)
        for (int i = lane; i < nx; i += 32) face[(long long)r.k * nx + i] = face_round<T>(d, 4, src[i]);
    if (r.comp == 5 && r.k == nz && r.j < ny)
        for (int i = lane; i < nx; i += 32) face[(long long)r.j * nx + i] = face_round<T>(d, 5, src[i]);
}

// Active layout (and far faces) -> canonical components, zero outside the extents.
template <typename T>
__global__ void __launch_bounds__(kLayThreads) unpack_kernel(const CavityDesc d, int copy, int comp0, int ncomp,
                                                             const Canon6 canon) {
    constexpr int V = LayPack<T>::V;
    const LayoutRow r = layout_row(d, comp0, ncomp);
    if (!r.ok) return;
    const int nx = d.nx, ny = d.ny, nz = d.nz, lane = threadIdx.x & 31;
    float *__restrict__ dst = canon.f[r.q] + ((long long)r.k * (ny + 1) + r.j) * (nx + 1);
    if (r.j < ny && r.k < nz) {
        const T *__restrict__ src =
            static_cast<const T *>(d.buf[copy][r.comp]) + (long long)r.k * d.plane + (long long)r.j * d.pitch;
        const float is = d.inv_scale[r.comp];
        for (int i0 = lane * V; i0 < nx; i0 += 32 * V * kLayU) {
            float v[kLayU][V];
#pragma unroll
            for (int u = 0; u < kLayU; ++u) {
                const int i = i0 + 32 * V * u;
                if (i < nx) LayPack<T>::ld(src + i, v[u]);
            }
#pragma unroll
            for (int u = 0; u < kLayU; ++u)
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    const int i = i0 + 32 * V * u + e;
                    if (i < nx) dst[i] = Storage<T>::scaled ? v[u][e] * is : v[u][e];
                }
        }
        if (lane == 0) dst[nx] = r.comp == 3 ? d.face[0][(long long)r.k * ny + r.j] : 0.f;
        return;
    }
    const float *__restrict__ face = nullptr;
    if (r.comp == 4 && r.j == ny && r.k < nz) face = d.face[1] + (long long)r.k * nx;
    if (r.comp == 5 && r.k == nz && r.j < ny) face = d.face[2] + (long long)r.j * nx;
    for (int i = lane; i <= nx; i += 32) dst[i] = face && i < nx ? face[i] : 0.f;
}

__device__ __forceinline__ bool in_extent(int comp, int i, int j, int k, int nx, int ny, int nz) {
    switch (comp) {
        case 0: return i < nx;
        case 1: return j < ny;
        case 2: return k < nz;
        case 3: return j < ny && k < nz;
        case 4: return i < nx && k < nz;
        default: return i < nx && j < ny;
    }
}

// max |canon| over the component's extent into out[component].  A warp takes whole extent rows (so no
// element needs its own index arithmetic), kMaxRows of them at a time, a lane two loads of each; a block
// reduces in shared memory and issues one atomic.  Bound by HBM reads: 281 us for the six 384^3 components
// (4.9 TB/s), 27 us for 200 x 131 x 120; one row and four loads at a time 331 and 40 us.  One atomic per warp,
// all on one address per component, took 7.6 ms.
constexpr int kMaxThreads = 256, kMaxRows = 4;
__global__ void __launch_bounds__(kMaxThreads) maxabs_kernel(const Canon6 canon, int comp0, int nx, int ny, int nz,
                                                             unsigned *out) {
    __shared__ float sh[kMaxThreads / 32];
    const int comp = comp0 + blockIdx.y;
    const float *__restrict__ src = canon.f[blockIdx.y];
    const int ex = nx + (in_extent(comp, nx, 0, 0, nx, ny, nz) ? 1 : 0);
    const int ey = ny + (in_extent(comp, 0, ny, 0, nx, ny, nz) ? 1 : 0);
    const int ez = nz + (in_extent(comp, 0, 0, nz, nx, ny, nz) ? 1 : 0);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned rows = (unsigned)ey * (unsigned)ez, stride = gridDim.x * (kMaxThreads / 32);   // at most 32769^2
    // kMaxRows rows at a time: their loads are in flight together (one row at a time leaves a short row's latency
    // to every step)
    float m[kMaxRows];
#pragma unroll
    for (int u = 0; u < kMaxRows; ++u) m[u] = 0.f;
    for (unsigned r0 = blockIdx.x * (kMaxThreads / 32) + w; r0 < rows; r0 += kMaxRows * stride) {
        const float *row[kMaxRows];
#pragma unroll
        for (int u = 0; u < kMaxRows; ++u) {
            const unsigned r = r0 + u * stride < rows ? r0 + u * stride : r0, k = r / (unsigned)ey;
            row[u] = src + ((long long)k * (ny + 1) + (r - k * (unsigned)ey)) * (nx + 1);
        }
        int i = lane;
        for (; i + 32 < ex; i += 64)
#pragma unroll
            for (int u = 0; u < kMaxRows; ++u) m[u] = fmaxf(m[u], fmaxf(fabsf(row[u][i]), fabsf(row[u][i + 32])));
        if (i < ex)
#pragma unroll
            for (int u = 0; u < kMaxRows; ++u) m[u] = fmaxf(m[u], fabsf(row[u][i]));
    }
    float v = 0.f;
#pragma unroll
    for (int u = 0; u < kMaxRows; ++u) v = fmaxf(v, m[u]);
    // (fmaxf passes over NaN, as the extent scan always did)
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) sh[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < kMaxThreads / 32; ++q) v = fmaxf(v, sh[q]);
        if (v > 0.f) atomicMax(out + comp, __float_as_uint(v));
    }
}

// H^{n+1/2} = H^{n-1/2} - ch curl E^n, one thread per cell (E beyond the active range is 0).
template <typename T>
__global__ void simple_h_kernel(const CavityDesc d, int copy) {
    const int i = blockIdx.x * BXs + threadIdx.x, j = blockIdx.y * BYs + threadIdx.y, k = blockIdx.z;
    const int nx = d.nx, ny = d.ny, nz = d.nz;
    if (i >= nx || j >= ny) return;
    const long long P = d.pitch, Z = d.plane;
    const long long o = (long long)k * Z + (long long)j * P + i;
    const float ex = ld_field<T>(d, copy, 0, o), ey = ld_field<T>(d, copy, 1, o), ez = ld_field<T>(d, copy, 2, o);
    const float ex_j1 = j + 1 < ny ? ld_field<T>(d, copy, 0, o + P) : 0.f;
    const float ex_k1 = k + 1 < nz ? ld_field<T>(d, copy, 0, o + Z) : 0.f;
    const float ey_i1 = i + 1 < nx ? ld_field<T>(d, copy, 1, o + 1) : 0.f;
    const float ey_k1 = k + 1 < nz ? ld_field<T>(d, copy, 1, o + Z) : 0.f;
    const float ez_i1 = i + 1 < nx ? ld_field<T>(d, copy, 2, o + 1) : 0.f;
    const float ez_j1 = j + 1 < ny ? ld_field<T>(d, copy, 2, o + P) : 0.f;
    const float hx = ld_field<T>(d, copy, 3, o) - ld_coef(d, 3, o) * ((ez_j1 - ez) - (ey_k1 - ey));
    const float hy = ld_field<T>(d, copy, 4, o) - ld_coef(d, 4, o) * ((ex_k1 - ex) - (ez_i1 - ez));
    const float hz = ld_field<T>(d, copy, 5, o) - ld_coef(d, 5, o) * ((ey_i1 - ey) - (ex_j1 - ex));
    st_field<T>(d, copy, 3, o, hx);
    st_field<T>(d, copy, 4, o, hy);
    st_field<T>(d, copy, 5, o, hz);
}

// E^{n+1} = E^n + ce curl H^{n+1/2} on entries not tangential to a face.
template <typename T>
__global__ void simple_e_kernel(const CavityDesc d, int copy) {
    const int i = blockIdx.x * BXs + threadIdx.x, j = blockIdx.y * BYs + threadIdx.y, k = blockIdx.z;
    const int nx = d.nx, ny = d.ny;
    if (i >= nx || j >= ny) return;
    const long long P = d.pitch, Z = d.plane;
    const long long o = (long long)k * Z + (long long)j * P + i;
    const float hx = ld_field<T>(d, copy, 3, o), hy = ld_field<T>(d, copy, 4, o), hz = ld_field<T>(d, copy, 5, o);
    if (j >= 1 && k >= 1) {
        const float c = (hz - ld_field<T>(d, copy, 5, o - P)) - (hy - ld_field<T>(d, copy, 4, o - Z));
        st_field<T>(d, copy, 0, o, ld_field<T>(d, copy, 0, o) + ld_coef(d, 0, o) * c);
    }
    if (i >= 1 && k >= 1) {
        const float c = (hx - ld_field<T>(d, copy, 3, o - Z)) - (hz - ld_field<T>(d, copy, 5, o - 1));
        st_field<T>(d, copy, 1, o, ld_field<T>(d, copy, 1, o) + ld_coef(d, 1, o) * c);
    }
    if (i >= 1 && j >= 1) {
        const float c = (hy - ld_field<T>(d, copy, 4, o - 1)) - (hx - ld_field<T>(d, copy, 3, o - P));
        st_field<T>(d, copy, 2, o, ld_field<T>(d, copy, 2, o) + ld_coef(d, 2, o) * c);
    }
}

constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 1216;     // partials allocated: 8 x 152 SMs, the fourth-order reductions' grid
constexpr int kRedPerSM = 3;                 // blocks per SM of the second-order reductions (their registers allow no more):
constexpr int kRed2Blocks = 152 * kRedPerSM;   // one wave; grids are fixed so that the summation order is reproducible

__device__ __forceinline__ double block_sum(double v, double *sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < kRedThreads / 32; ++i) r += sh[i];
    return r;
}

// 1/ch at far-face entry fi of face array c, as a pair and in FP64.
__device__ __forceinline__ df::F2 face_inv_ch_df(const CavityDesc &d, int c, long long fi) {
    return df::recip(d.coef_mode == COEF_SCALAR ? d.ch[c] : d.face_ch[c][fi]);
}
__device__ __forceinline__ double face_inv_ch64(const CavityDesc &d, int c, long long fi) {
    return d.coef_mode == COEF_SCALAR ? 1.0 / (double)d.ch[c] : 1.0 / (double)d.face_ch[c][fi];
}

// Two adjacent values of field f from an even x index (rows are 128-byte aligned; past an odd nx lies padding).
template <typename T> __device__ __forceinline__ float2 ld_pair(const CavityDesc &d, int copy, int f, long long off) {
    const T *p = static_cast<const T *>(d.buf[copy][f]) + off;
    float2 v;
    if constexpr (Storage<T>::kind == 0) v = *reinterpret_cast<const float2 *>(p);
    else if constexpr (Storage<T>::kind == 1) v = __half22float2(*reinterpret_cast<const __half2 *>(p));
    else v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
    if (Storage<T>::scaled) {
        v.x *= d.inv_scale[f];
        v.y *= d.inv_scale[f];
    }
    return v;
}

// Per block, in a fixed order (a warp per (j, k) row, a lane two adjacent cells; far-face H appended):
//   WHAT == 0: energy sum  E^2/ce + H^2/ch - H curl E   (W without the 1/2 dt/dx factor)
//   WHAT == 1: sum of divE^2 over interior nodes and of divH^2 over cells.
// Every term is formed from the stored values with error-free FP32 transformations (the curl differences
// as exact pairs, the reciprocal coefficients as pairs; df.cuh) and a lane accumulates its cells of a row
// with Dot2, about 2^-48 relative; the row sums are added in FP64, then per block and over blocks in a fixed
// order, so the result is deterministic.  (GB300's FP64 rate made the same sums in FP64 eight times slower
// at 512^3.)  CHC: one ch everywhere, far faces included: H^2 takes no lookups, and divH is an exact sum of six
// values, scaled once.
// Bound by the compensated FP32 arithmetic and the latency of the loads that 24 warps per SM (80 registers) leave:
// packed pairs and separate accumulator chains against one cell and one chain per lane took the energy of 320^3
// FP32 cells from 369 to 300 us and the divergences from 645 to 389 us (a DRAM pass over the state is 121 us).
// Two blocks per SM (99-120 registers) 306 and 500 us; an L2 prefetch of the warp's next row: no gain.
template <typename T, int WHAT, bool CHC>
__global__ void __launch_bounds__(kRedThreads, kRedPerSM) reduce_kernel(const CavityDesc d, int copy, double *partial) {
    __shared__ double sh[kRedThreads / 32];
    __shared__ float thi[6 * kMaxTable], tlo[6 * kMaxTable];   // 1/ce xyz, 1/ch xyz by material id, as pairs
    const int nx = d.nx, ny = d.ny, nz = d.nz;
    const long long P = d.pitch, Z = d.plane;
    double s0 = 0.0, s1 = 0.0;
    const bool ids = d.coef_mode == COEF_ID8, scalar = d.coef_mode == COEF_SCALAR;
    // a uniform cavity is one entry of the table (read at index 0 by every lane)
    const int ntab = ids ? d.ntab : scalar ? 1 : 0;
    for (int e = threadIdx.x; e < 6 * ntab; e += blockDim.x) {
        const int c = e / ntab, m = e - c * ntab;
        const df::F2 r = df::recip(scalar ? (c < 3 ? d.ce[c] : d.ch[c - 3]) : d.table[8 * m + (c < 3 ? c : c + 1)]);
        thi[c * kMaxTable + m] = r.hi;
        tlo[c * kMaxTable + m] = r.lo;
    }
    const df::F2 ich = df::recip(d.ch[0]);   // CHC
    const df::F22 ich2{make_float2(ich.hi, ich.hi), make_float2(ich.lo, ich.lo)};
    const float pch = exp2f((float)ilogbf(ich.hi));   // the power of two at or below 1/ch
    const float2 pch2 = make_float2(pch, pch);
    __syncthreads();
    const float2 zero = make_float2(0.f, 0.f);
    // material ids of the two cells at off (packed), and 1/ce or 1/ch (c) of them
    auto IDS = [&](long long off) -> unsigned { return ids ? *reinterpret_cast<const uint16_t *>(d.id + off) : 0u; };
    bool two = true;   // the pair's second cell lies in the cavity (past an odd nx coefficient arrays hold 0)
    auto IC = [&](int c, unsigned m, long long off) -> df::F22 {
        if (d.coef_mode == COEF_FULL) {
            const df::F2 a = df::recip(d.coef[c][off]), b = two ? df::recip(d.coef[c][off + 1]) : a;
            return df::F22{make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)};
        }
        const float *h = thi + c * kMaxTable, *l = tlo + c * kMaxTable;
        return df::F22{make_float2(h[m & 0xff], h[m >> 8]), make_float2(l[m & 0xff], l[m >> 8])};
    };
    const int lane = threadIdx.x & 31;
    // rows of the planes [kr_lo, kr_hi) (the owned cells of a z-slab; every plane otherwise)
    // (at most 32768^2 of them: 32 bits; a 64-bit division per row showed)
    const unsigned nrows = (unsigned)ny * (unsigned)(d.kr_hi - d.kr_lo);
    const unsigned nwarps = (gridDim.x * kRedThreads) >> 5;
    for (unsigned r = (blockIdx.x * kRedThreads + threadIdx.x) >> 5; r < nrows; r += nwarps) {
        const unsigned kr = r / (unsigned)ny;
        const int j = (int)(r - kr * (unsigned)ny), k = d.kr_lo + (int)kr;
        df::Acc2 a0, a1, a2;
        for (int i = 2 * lane; i < nx; i += 64) {
            const long long o = (long long)k * Z + (long long)j * P + i;
            two = i + 1 < nx;
            auto F = [&](int f, long long off) -> float2 {
                float2 v = ld_pair<T>(d, copy, f, off);
                if (!two) v.y = 0.f;
                return v;
            };
            // the pair one cell up in x: (v.y, the cell after)
            auto up = [&](int f, float2 v) -> float2 {
                return make_float2(v.y, i + 2 < nx ? ld_field<T>(d, copy, f, o + 2) : 0.f);
            };
            const float2 ex = F(0, o), ey = F(1, o), ez = F(2, o), hx = F(3, o), hy = F(4, o), hz = F(5, o);
            const unsigned m = IDS(o);
            if (WHAT == 0) {
                const float2 ex_j1 = j + 1 < ny ? F(0, o + P) : zero, ez_j1 = j + 1 < ny ? F(2, o + P) : zero;
                const float2 ex_k1 = k + 1 < nz ? F(0, o + Z) : zero, ey_k1 = k + 1 < nz ? F(1, o + Z) : zero;
                const float2 ey_i1 = up(1, ey), ez_i1 = up(2, ez);
                a0.sq_times(ex, IC(0, m, o));
                a0.sq_times(ey, IC(1, m, o));
                a0.sq_times(ez, IC(2, m, o));
                // (H^2 summed first and scaled once is cheaper and 1.5 times less exact: the unscaled squares of
                // short-mantissa values round with a bias)
                a1.sq_times(hx, CHC ? ich2 : IC(3, m, o));
                a1.sq_times(hy, CHC ? ich2 : IC(4, m, o));
                a1.sq_times(hz, CHC ? ich2 : IC(5, m, o));
                // past an odd nx the second cell's H is 0, so its curl does not count
                a2.prod(hx, df::diff22(ez_j1, ez, ey_k1, ey));
                a2.prod(hy, df::diff22(ex_k1, ex, ez_i1, ez));
                a2.prod(hz, df::diff22(ey_i1, ey, ex_j1, ex));
            } else {
                if (j >= 1 && k >= 1) {
                    df::Acc2 de;   // sum over c of D_c(node) - D_c(node - e_c), D = E / ce
                    df::F22 cx = IC(0, m, o), cl;
                    float2 exl;    // the pair one cell down in x
                    exl.y = ex.x;
                    cl.hi.y = cx.hi.x;
                    cl.lo.y = cx.lo.x;
                    if (i > 0) {
                        exl.x = ld_field<T>(d, copy, 0, o - 1);
                        if (d.coef_mode == COEF_FULL) {
                            const df::F2 q = df::recip(d.coef[0][o - 1]);
                            cl.hi.x = q.hi;
                            cl.lo.x = q.lo;
                        } else {
                            const int q = ids ? d.id[o - 1] : 0;
                            cl.hi.x = thi[q];
                            cl.lo.x = tlo[q];
                        }
                    } else {
                        exl.x = cl.hi.x = cl.lo.x = 0.f;
                    }
                    de.prod(ex, cx);
                    de.prod(df::neg2(exl), cl);
                    de.prod(ey, IC(1, m, o));
                    de.prod(df::neg2(F(1, o - P)), IC(1, IDS(o - P), o - P));
                    de.prod(ez, IC(2, m, o));
                    de.prod(df::neg2(F(2, o - Z)), IC(2, IDS(o - Z), o - Z));
                    df::F22 v = de.pair();
                    if (i == 0) v.hi.x = v.lo.x = 0.f;       // not a node inside
                    if (!two) v.hi.y = v.lo.y = 0.f;
                    a0.square(v);
                }
                // sum over c of B_c(cell + e_c) - B_c(cell), B = H / ch
                const long long fx = (long long)k * ny + j, fy = (long long)k * nx + i, fz = (long long)j * nx + i;
                float2 hx1 = up(3, hx), hy1, hz1;
                if (i + 1 >= nx) hx1.x = d.face[0][fx];
                else if (i + 2 >= nx) hx1.y = d.face[0][fx];
                auto face2 = [&](const float *f, long long at) { return make_float2(f[at], two ? f[at + 1] : 0.f); };
                hy1 = j + 1 < ny ? F(4, o + P) : face2(d.face[1], fy);
                hz1 = k + 1 < nz ? F(5, o + Z) : face2(d.face[2], fz);
                if (CHC) {   // the difference as an exact sum; 1/ch^2 scales the total
                    // The leading part u cancels where the field is free of divergence, and what the sum's roundings
                    // left can exceed it: the pair is normalised before it is squared.  Then times the power of two
                    // next to 1/ch, so that weak fields square within the same range as H / ch does.
                    float2 x, exx, y, eyy, z, ezz, t, et, u, eu;
                    df::two_diff2(hx1, hx, x, exx);
                    df::two_diff2(hy1, hy, y, eyy);
                    df::two_diff2(hz1, hz, z, ezz);
                    df::two_sum2(x, y, t, et);
                    df::two_sum2(t, z, u, eu);
                    df::F22 v;
                    df::two_sum2(u, df::add2(df::add2(df::add2(exx, eyy), df::add2(ezz, et)), eu), v.hi, v.lo);
                    v.hi = df::mul2(v.hi, pch2);
                    v.lo = df::mul2(v.lo, pch2);
                    if (!two) v.hi.y = v.lo.y = 0.f;
                    a1.square(v);
                } else {
                    df::F22 c;
                    auto set = [](df::F22 &f, int e, df::F2 v) {
                        if (e == 0) { f.hi.x = v.hi; f.lo.x = v.lo; }
                        else { f.hi.y = v.hi; f.lo.y = v.lo; }
                    };
                    auto one = [&](int q, long long off) -> df::F2 {   // 1/ch component q at one cell
                        if (d.coef_mode == COEF_FULL) return df::recip(d.coef[3 + q][off]);
                        const int n = ids ? d.id[off] : 0;
                        return df::F2{thi[(3 + q) * kMaxTable + n], tlo[(3 + q) * kMaxTable + n]};
                    };
                    df::Acc2 dh;
                    set(c, 0, i + 1 < nx ? one(0, o + 1) : face_inv_ch_df(d, 0, fx));
                    set(c, 1, i + 2 < nx ? one(0, o + 2) : face_inv_ch_df(d, 0, fx));
                    dh.prod(hx1, c);
                    if (j + 1 < ny) c = IC(4, IDS(o + P), o + P);
                    else for (int e = 0; e < 2; ++e) set(c, e, face_inv_ch_df(d, 1, two ? fy + e : fy));
                    dh.prod(hy1, c);
                    if (k + 1 < nz) c = IC(5, IDS(o + Z), o + Z);
                    else for (int e = 0; e < 2; ++e) set(c, e, face_inv_ch_df(d, 2, two ? fz + e : fz));
                    dh.prod(hz1, c);
                    dh.prod(df::neg2(hx), IC(3, m, o));
                    dh.prod(df::neg2(hy), IC(4, m, o));
                    dh.prod(df::neg2(hz), IC(5, m, o));
                    df::F22 v = dh.pair();
                    if (!two) v.hi.y = v.lo.y = 0.f;
                    a1.square(v);
                }
            }
        }
        // the row's sum in FP64 (one pair per row: FP64 additions are the scarce operation)
        if (WHAT == 0) {
            const df::F2 c = a2.take(), t = df::add(df::add(a0.take(), a1.take()), df::F2{-c.hi, -c.lo});
            s0 += (double)t.hi + (double)t.lo;
        } else {
            const df::F2 e = a0.take(), h = a1.take();
            s0 += (double)e.hi + (double)e.lo;
            s1 += (double)h.hi + (double)h.lo;
        }
    }
    if (WHAT == 0) {
        // constant far-face normal H: curl E vanishes there, so its energy term is H^2/ch (the x and y
        // faces over the summed planes, the z face when the range reaches it); few terms: FP64
        const int nk = d.kr_hi - d.kr_lo;
        const long long nfx = (long long)ny * nk, nfy = (long long)nx * nk, nfz = d.face_top ? (long long)nx * ny : 0;
        for (long long n = blockIdx.x * (long long)kRedThreads + threadIdx.x; n < nfx + nfy + nfz;
             n += (long long)gridDim.x * kRedThreads) {
            int c;
            long long fi;
            if (n < nfx) { c = 0; fi = n + (long long)d.kr_lo * ny; }
            else if (n < nfx + nfy) { c = 1; fi = n - nfx + (long long)d.kr_lo * nx; }
            else { c = 2; fi = n - nfx - nfy; }
            const double h = d.face[c][fi];
            s0 += h * h * (CHC ? 1.0 / (double)d.ch[0] : face_inv_ch64(d, c, fi));
        }
    } else if (CHC) {
        const double q = 1.0 / ((double)d.ch[0] * (double)pch);
        s1 *= q * q;
    }
    const double a = block_sum(s0, sh);
    const double b = block_sum(s1, sh);
    if (threadIdx.x == 0) {
        partial[3 * blockIdx.x + 0] = WHAT == 0 ? a : 0.0;
        partial[3 * blockIdx.x + 1] = WHAT == 1 ? a : 0.0;
        partial[3 * blockIdx.x + 2] = b;
    }
}

// Sums of the block partials (in a fixed order) and the status word: one read-back for both.
__global__ void __launch_bounds__(kRedThreads) reduce_final_kernel(const double *partial, int nblocks, const int *status,
                                                                   double *out) {
    __shared__ double sh[3][kRedThreads / 32];
    double v[3] = {0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += kRedThreads)
#pragma unroll
        for (int q = 0; q < 3; ++q) v[q] += partial[3 * b + q];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
        if ((threadIdx.x & 31) == 0) sh[q][threadIdx.x >> 5] = v[q];
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double r = 0.0;
        for (int i = 0; i < kRedThreads / 32; ++i) r += sh[threadIdx.x][i];
        out[threadIdx.x] = r;
    }
    if (threadIdx.x == 3) out[3] = (double)*status;
}

template <typename T>
cudaError_t simple_step_typed(const CavityDesc &d, int copy, cudaStream_t s) {
    dim3 blk(BXs, BYs), grd((d.nx + BXs - 1) / BXs, (d.ny + BYs - 1) / BYs, d.nz);
    simple_h_kernel<T><<<grd, blk, 0, s>>>(d, copy);
    simple_e_kernel<T><<<grd, blk, 0, s>>>(d, copy);
    return cudaGetLastError();
}

#define FDTD_STORAGE_DISPATCH(storage, ...)                 \
    do {                                                     \
        if (storage == 0) { using T = float; __VA_ARGS__; }         \
        else if (storage == 1) { using T = __half; __VA_ARGS__; }   \
        else { using T = __nv_bfloat16; __VA_ARGS__; }              \
    } while (0)

}  // namespace

// Device memory bounds ny nz at about 3.6e8 (rows are padded to 32 elements, 12 arrays of them must fit), so row
// numbers fit 32 bits.
static unsigned layout_blocks(const CavityDesc &d, int ncomp) {
    const unsigned long long rows = (unsigned long long)ncomp * (d.ny + 1) * (d.nz + 1);
    return (unsigned)((rows + kLayThreads / 32 - 1) / (kLayThreads / 32));
}

cudaError_t launch_pack(int storage, const CavityDesc &d, int copy, int comp0, int ncomp, const float *const *canon,
                        cudaStream_t s) {
    Canon6 c{};
    for (int q = 0; q < ncomp; ++q) c.f[q] = const_cast<float *>(canon[q]);
    const unsigned grd = layout_blocks(d, ncomp);
    FDTD_STORAGE_DISPATCH(storage, pack_kernel<T><<<grd, kLayThreads, 0, s>>>(d, copy, comp0, ncomp, c));
    return cudaGetLastError();
}

cudaError_t launch_unpack(int storage, const CavityDesc &d, int copy, int comp0, int ncomp, float *const *canon,
                          cudaStream_t s) {
    Canon6 c{};
    for (int q = 0; q < ncomp; ++q) c.f[q] = canon[q];
    const unsigned grd = layout_blocks(d, ncomp);
    FDTD_STORAGE_DISPATCH(storage, unpack_kernel<T><<<grd, kLayThreads, 0, s>>>(d, copy, comp0, ncomp, c));
    return cudaGetLastError();
}

cudaError_t launch_maxabs(const float *const *canon, int comp0, int ncomp, int nx, int ny, int nz, unsigned *out,
                          cudaStream_t s) {
    Canon6 c{};
    for (int q = 0; q < ncomp; ++q) c.f[q] = const_cast<float *>(canon[q]);
    // enough warps for every row once, at most about eight blocks per SM over the launch's components
    const long long rows = (long long)(ny + 1) * (nz + 1), per = kMaxThreads / 32;
    const int blocks = (int)std::min<long long>((rows + per - 1) / per, 1216 / ncomp + 1);
    maxabs_kernel<<<dim3(blocks, ncomp), kMaxThreads, 0, s>>>(c, comp0, nx, ny, nz, out);
    return cudaGetLastError();
}

cudaError_t launch_simple_step(int storage, const CavityDesc &d, int copy, cudaStream_t s) {
    cudaError_t e;
    FDTD_STORAGE_DISPATCH(storage, e = simple_step_typed<T>(d, copy, s));
    return e;
}

int reduction_blocks() { return kRedBlocks; }

cudaError_t launch_reductions(int storage, const CavityDesc &d, int copy, int what, double *partial, int nblocks,
                              const int *status, double *out, cudaStream_t s, int order) {
    if (order == 4) {
        cudaError_t e = launch_reductions4(storage, d, copy, what, partial, nblocks, s);
        if (e != cudaSuccess) return e;
    } else {
        nblocks = kRed2Blocks;
        if (what == 0 && d.ch_const)
            FDTD_STORAGE_DISPATCH(storage, (reduce_kernel<T, 0, true><<<nblocks, kRedThreads, 0, s>>>(d, copy, partial)));
        else if (what == 0)
            FDTD_STORAGE_DISPATCH(storage, (reduce_kernel<T, 0, false><<<nblocks, kRedThreads, 0, s>>>(d, copy, partial)));
        else if (d.ch_const)
            FDTD_STORAGE_DISPATCH(storage, (reduce_kernel<T, 1, true><<<nblocks, kRedThreads, 0, s>>>(d, copy, partial)));
        else
            FDTD_STORAGE_DISPATCH(storage, (reduce_kernel<T, 1, false><<<nblocks, kRedThreads, 0, s>>>(d, copy, partial)));
    }
    reduce_final_kernel<<<1, kRedThreads, 0, s>>>(partial, nblocks, status, out);
    return cudaGetLastError();
}

}  // namespace fdtd
