// Many leapfrog steps of a small cavity in one launch, the state held on chip (sm_103a).
//
// A cavity of up to about a million cells fits the chip's registers and shared memory, so a step need not
// move its state at all: the cavity is cut into boxes of at most 32 x 16 x 14 cells, one persistent CTA
// each, and per step a CTA exchanges only the E values of its box's surface with its neighbours through
// L2.  The update is that of k_fused.cu (Eq. 2 of the paper in the order of Listing 1), value by value the
// same operations, so FP32 results are those of every other kernel bit for bit.  16-bit storage is read
// at the first step of a launch and written after its last one, with FP32 in between: fewer roundings.
//
// Per CTA: warp j owns row j of the box, lane i column i, and a thread keeps the six field values of its
// column's BZ cells in registers.  Shared memory holds the values that neighbouring threads read:
//   E on [-1, bx] x [-1, by] x [-1, bz] (the own cells and a one-cell shell from the neighbours),
//   H on [-1, bx) x [-1, by) x [0, bz).
// The E update of the box's first row and column needs H one cell below it.  Those H values are computed
// here too, from the shell, so that one exchange per step suffices.
// Cells outside the cavity hold E = 0.  PEC faces are materials: a cell's id (1 + material + ntab faces;
// for a uniform cavity 1 + faces, made here) selects a table entry whose tangential E coefficients are 0.
// The plane loops run all BZ planes of the instance without a test per plane (a box one plane shorter
// computes values that nothing reads): with a branch per plane no load could be issued ahead of the
// previous plane's arithmetic, and a step took three times as long.
//
// Exchange: the E values of a surface cell travel as one 16-byte word of three values and a step tag,
// written with a single store into the owner's packed surface buffer (two, used in turn) and polled by its
// reader until the tag is the step's: one store and one load between two steps, no fence, no flag.  (A
// flag per CTA behind a fence, then a poll, then the loads: four dependent L2 round trips.)  A buffer is used
// again two steps later: a CTA that has received all its words of step s + 1 knows that those neighbours had
// taken theirs of step s, because they send after a barrier behind their loads, and neighbours read each
// other in pairs.  Tags go on from launch to launch (a device counter that the last CTA to read it advances),
// so buffers are never cleared.
// All CTAs run at once (cooperative launch).  Waits are bounded in poll rounds (kPolls); the first to run out
// latches STATUS_TIMEOUT, which every wait looks at, so that all CTAs leave without a result.
#include <algorithm>

#include "fused_common.cuh"
#include "launch.h"

namespace fdtd {

namespace {

constexpr int NT = 512, NW = 16, BXR = 32;       // threads, rows and columns of a box
using u64 = unsigned long long;

template <int BZ> struct Lay {
    static constexpr int EX = BXR + 2, EY = NW + 2, EZ = BZ + 2;   // E: index - 1 is the shell
    static constexpr int HX = BXR + 1, HY = NW + 1, HZ = BZ;       // H: x and y index - 1 are halo
    static constexpr int EF = EX * EY * EZ, HF = HX * HY * HZ;
    __device__ __forceinline__ static int e(int i, int j, int k) { return ((k + 1) * EY + (j + 1)) * EX + (i + 1); }
    __device__ __forceinline__ static int h(int i, int j, int k) { return (k * HY + (j + 1)) * HX + (i + 1); }
    // packed surface of a box, in words: last / first column (x), row (y) and plane (z)
    static constexpr int XP = 0, XM = XP + BZ * NW, YP = XM + BZ * NW, YM = YP + BZ * BXR, ZP = YM + BZ * BXR,
                         ZM = ZP + NW * BXR, W = ZM + NW * BXR;
};

struct OwnSource {
    short tid, k;       // owning thread and plane
    short comp, q;      // component, index of the source
    float cd;           // ce dx (unscaled)
};
struct OwnProbe {
    unsigned short at, q;   // offset in the shared fields, index of the probe
    short comp, pad;
};

template <int BZ> __host__ __device__ constexpr int fields_bytes() {
    return ((3 * Lay<BZ>::EF + 3 * Lay<BZ>::HF) * 4 + 15) / 16 * 16;
}
template <int BZ> constexpr int smem_bytes(int ntab, int nsrc, int nprobe) {
    return fields_bytes<BZ>() + 32 * ntab + (int)sizeof(OwnSource) * nsrc + (int)sizeof(OwnProbe) * nprobe;
}

// Three values and the step tag as one 16-byte access (a .b128 access is one memory operation, never torn).
struct Word {
    u64 lo, hi;
    __device__ __forceinline__ float a() const { return __uint_as_float((unsigned)lo); }
    __device__ __forceinline__ float b() const { return __uint_as_float((unsigned)(lo >> 32)); }
    __device__ __forceinline__ float c() const { return __uint_as_float((unsigned)hi); }
    __device__ __forceinline__ unsigned tag() const { return (unsigned)(hi >> 32); }
};
struct alignas(16) WordMem {
    u64 w[2];
};
__device__ __forceinline__ Word ld_word(const WordMem *p) {
    Word v;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(v.lo), "=l"(v.hi)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ void st_word(WordMem *p, float a, float b, float c, unsigned tag) {
    const u64 lo = ((u64)__float_as_uint(b) << 32) | __float_as_uint(a), hi = ((u64)tag << 32) | __float_as_uint(c);
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
}
// Polls the wanted words (bit c of want) until every tag is the step's: all missing words of a round are
// loaded together.  Gives up after `polls` rounds, or when another CTA has, and looks at either every 256.  A round is
// an L2 round trip, about a microsecond, so kPolls are some seconds; a timer read per round would cost as much.
constexpr int kPolls = 1 << 22;
template <int N>
__device__ __forceinline__ void wait_words(const WordMem *const *p, Word *v, unsigned want, unsigned tag, int polls,
                                           int *status, int *abort) {
    for (int n = 1;; ++n) {
        bool miss = false;
#pragma unroll
        for (int c = 0; c < N; ++c)
            if (((want >> c) & 1u) && v[c].tag() != tag) {
                miss = true;
                v[c] = ld_word(p[c]);
            }
        if (!miss) return;
        if ((n & 255) == 0) {
            if (n >= polls) atomicOr(status, STATUS_TIMEOUT);
            if (*(volatile int *)status != 0) {   // a wait ran out, here or in another CTA
                *(volatile int *)abort = 1;
                return;
            }
        }
    }
}
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }

// A field array of either storage; the storage is a template parameter of the code that loads or stores many
// values (a test per value would serialise the loads).
template <typename T> __device__ __forceinline__ float ld_state(const void *p, long long o) {
    if constexpr (sizeof(T) == 4) return __ldcg(static_cast<const float *>(p) + o);
    const unsigned short v = __ldcg(static_cast<const unsigned short *>(p) + o);
    if constexpr (Storage<T>::kind == 1) return __half2float(__ushort_as_half(v));
    return __bfloat162float(__ushort_as_bfloat16(v));
}
template <typename F> __device__ __forceinline__ void by_storage(int storage, F f) {
    if (storage == 0) f(float{});
    else if (storage == 1) f(__half{});
    else f(__nv_bfloat16{});
}

// HID: ch differs between materials (else three ch for the whole cavity).
template <int BZ, bool HID>
__global__ void __launch_bounds__(NT, 1) resident_kernel(const ResidentParams P) {
    using L = Lay<BZ>;
    extern __shared__ __align__(16) unsigned char smem[];
    float *se = reinterpret_cast<float *>(smem), *sh = se + 3 * L::EF;
    float4 *stab = reinterpret_cast<float4 *>(smem + fields_bytes<BZ>());
    OwnSource *srcs = reinterpret_cast<OwnSource *>(stab + 2 * P.ntab);
    OwnProbe *probes = reinterpret_cast<OwnProbe *>(srcs + P.X.nsrc);
    __shared__ int s_abort, s_nsrc, s_nprobe;
    __shared__ unsigned s_tag;
    __shared__ long long s_n0;

    const int t = threadIdx.x, j = t >> 5, i = t & 31;
    const int b = blockIdx.x;
    const int qx = b % P.px, qy = (b / P.px) % P.py, qz = b / (P.px * P.py);
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x0 = (int)((long long)qx * nx / P.px), bx = (int)((long long)(qx + 1) * nx / P.px) - x0;
    const int y0 = (int)((long long)qy * ny / P.py), by = (int)((long long)(qy + 1) * ny / P.py) - y0;
    const int z0 = (int)((long long)qz * nz / P.pz), bz = (int)((long long)(qz + 1) * nz / P.pz) - z0;
    const int pitch = P.pitch, plane = P.plane;      // a resident cavity's offsets fit 32 bits
    const bool act = i < bx && j < by;
    const int o0 = z0 * plane + (y0 + j) * pitch + x0 + i;          // own column's first cell
    const bool z_lo = qz > 0, z_hi = qz + 1 < P.pz, y_lo = qy > 0, y_hi = qy + 1 < P.py, x_lo = qx > 0, x_hi = qx + 1 < P.px;
    const ExtrasParams &X = P.X;

    // ---------------- set-up: zero shared fields (the shell outside the cavity stays 0), table, lists
    for (int q = t; q < 3 * L::EF + 3 * L::HF; q += NT) se[q] = 0.f;
    if (P.id) {
        for (int q = t; q < 2 * P.ntab; q += NT) stab[q] = P.table[q];
    } else if (t < 9) {   // uniform cavity: entry 0 outside, 1 + faces inside
        const int f = t - 1;
        const bool in = t > 0, i0 = f & 1, j0 = f & 2, k0 = f & 4;
        stab[2 * t] = make_float4(in && !j0 && !k0 ? P.ce[0] : 0.f, in && !i0 && !k0 ? P.ce[1] : 0.f,
                                  in && !i0 && !j0 ? P.ce[2] : 0.f, 0.f);
        stab[2 * t + 1] = make_float4(P.ch[0], P.ch[1], P.ch[2], 0.f);
    }
    if (t == 0) {
        s_abort = s_nsrc = s_nprobe = 0;
        // the launch's first tag and step index; the last CTA to have read them moves them past the launch
        const unsigned tag = *(volatile unsigned *)P.epoch;
        const long long n0 = X.clock ? *(volatile long long *)X.clock : 0;
        s_tag = tag;
        s_n0 = n0;
        __threadfence();
        if (atomicAdd(P.epoch + 1, 1u) == gridDim.x - 1) {
            *(volatile unsigned *)(P.epoch + 1) = 0u;
            *(volatile unsigned *)P.epoch = tag + (unsigned)P.steps;
            if (X.clock) *(volatile long long *)X.clock = n0 + P.steps;
        }
    }
    __syncthreads();
    const unsigned tag0 = s_tag;
    if (P.lose_polls > 0 && b == 0) {   // diagnostic: CTA 0 waits for a tag that nobody sends, its neighbours then for it
        if (t == 0) {
            const WordMem *const p[1] = {static_cast<const WordMem *>(P.words)};
            Word v[1] = {{0, 0}};
            wait_words<1>(p, v, 1u, tag0 ^ (1u << 31), P.lose_polls, P.status, &s_abort);
        }
        __syncthreads();
        if (s_abort) return;
    }
    unsigned src_mask = 0;   // planes of this thread's column that hold a current
    if (X.nsrc | X.nprobe) {
        // position of an active-array offset relative to the box
        auto locate = [&](long long off, int &li, int &lj, int &lk) {
            const int o = (int)off, k = o / plane, r = o - k * plane;
            lk = k - z0;
            lj = r / pitch - y0;
            li = r % pitch - x0;
            return li >= 0 && li < bx && lj >= 0 && lj < by && lk >= 0 && lk < bz;
        };
        int li, lj, lk;
        if (t == 0)   // in the callers' order: currents at one position add up serially
            for (int q = 0; q < X.nsrc; ++q)
                if (locate(X.src_off[q], li, lj, lk)) {
                    const int c = X.src_comp[q];
                    const float ce = P.id_mat ? P.table_mat[8 * P.id_mat[X.src_off[q]] + c] : P.ce_mat[c];
                    srcs[s_nsrc++] = OwnSource{(short)(lj * 32 + li), (short)lk, (short)c, (short)q, ce * X.dx};
                }
        for (int q = t; q < X.nprobe; q += NT)
            if (locate(X.probe_off[q], li, lj, lk)) {
                const int c = X.probe_comp[q];
                const int at = c < 3 ? c * L::EF + L::e(li, lj, lk) : 3 * L::EF + (c - 3) * L::HF + L::h(li, lj, lk);
                probes[atomicAdd(&s_nprobe, 1)] = OwnProbe{(unsigned short)at, (unsigned short)q, (short)c, 0};
            }
        __syncthreads();
        for (int q = 0; q < s_nsrc; ++q)
            if (srcs[q].tid == t) src_mask |= 1u << srcs[q].k;
    }

    // ---------------- initial state
    // A deep box keeps Ex and Ey in shared memory alone (30 registers less; with all six in registers the 14-plane
    // instance spilled and took 6.3 instead of 4.7 us a step on 128 x 96 x 80).
    constexpr bool DEEP = BZ > 8;
    constexpr int NE = DEEP ? 1 : BZ + 1;
    float ex[NE], ey[NE], ez[BZ], hx[BZ], hy[BZ], hz[BZ];   // ex, ey: index bz is the neighbour's plane
    uint32_t ids[(BZ + 3) / 4];
    const long long fs = P.fstride;
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
        uint32_t m = 0;
        if (act && k < bz)
            m = P.id ? P.id[o0 + k * plane]
                     : 1u + (x0 + i == 0 ? 1u : 0u) + (y0 + j == 0 ? 2u : 0u) + (z0 + k == 0 ? 4u : 0u);
        if (k % 4 == 0) ids[k / 4] = 0;
        ids[k / 4] |= m << (8 * (k % 4));
    }
    // H one cell below the box: z (own column), y (plane k = j of row -1), x (row hj, plane hk of column -1)
    const int hj = t & 15, hk = t >> 4;
    const bool ytask = i < bx && j < bz, xtask = hj < by && hk < bz;
    const int oy = (z0 + j) * plane + (y0 - 1) * pitch + x0 + i, ox = (z0 + hk) * plane + (y0 + hj) * pitch + x0 - 1;
    float hzx = 0.f, hzy = 0.f;
    by_storage(P.storage, [&](auto type) __attribute__((always_inline)) {
        using T = decltype(type);
        auto ld = [&](int f, int o) { return ld_state<T>(P.src, f * fs + o); };
#pragma unroll
        for (int k = 0; k < BZ + 1; ++k) {
            const bool in = act && k < bz, top = act && k == bz && z_hi;
            const int o = o0 + k * plane;
            const float x = in || top ? ld(0, o) : 0.f, y = in || top ? ld(1, o) : 0.f;
            if constexpr (DEEP) {
                if (in || top) {
                    se[L::e(i, j, k)] = x;
                    se[L::EF + L::e(i, j, k)] = y;
                }
            } else {
                ex[k] = x;
                ey[k] = y;
            }
            if (k < BZ) {
                ez[k] = in ? ld(2, o) : 0.f;
                hx[k] = in ? ld(3, o) : 0.f;
                hy[k] = in ? ld(4, o) : 0.f;
                hz[k] = in ? ld(5, o) : 0.f;
            }
        }
        if (act && z_lo) {
            hzx = ld(3, o0 - plane);
            hzy = ld(4, o0 - plane);
        }
        if (ytask && y_lo) {
            sh[L::h(i, -1, j)] = ld(3, oy);
            sh[2 * L::HF + L::h(i, -1, j)] = ld(5, oy);
        }
        if (xtask && x_lo) {
            sh[L::HF + L::h(-1, hj, hk)] = ld(4, ox);
            sh[2 * L::HF + L::h(-1, hj, hk)] = ld(5, ox);
        }
        // the shell: a warp takes the rows (lj, lk) around the box in turn, whole rows outside it and the two ends
        // of the rows beside it, where they lie in the cavity
        for (int r = j; r < (by + 2) * (bz + 2); r += NW) {
            const int lk = r / (by + 2) - 1, lj = r - (lk + 1) * (by + 2) - 1, gj = y0 + lj, gk = z0 + lk;
            if (gj < 0 || gj >= ny || gk < 0 || gk >= nz) continue;
            const bool beside = lj >= 0 && lj < by && lk >= 0 && lk < bz;
            for (int li = i - 1; li <= bx; li += 32) {
                const int gi = x0 + li;
                if (gi < 0 || gi >= nx || (beside && li >= 0 && li < bx)) continue;
                const int o = gk * plane + gj * pitch + gi, q = L::e(li, lj, lk);
                const float a = ld(0, o), b2 = ld(1, o), c = ld(2, o);
                se[q] = a;
                se[L::EF + q] = b2;
                se[2 * L::EF + q] = c;
            }
        }
    });
    if (act)
#pragma unroll
        for (int k = 0; k < BZ; ++k)
            if (k < bz) {
                if constexpr (!DEEP) {
                    se[L::e(i, j, k)] = ex[k];
                    se[L::EF + L::e(i, j, k)] = ey[k];
                }
                se[2 * L::EF + L::e(i, j, k)] = ez[k];
            }
    uint32_t hid = 0;   // HID: material codes of the three halo cells
    if (HID) {
        if (act && z_lo) hid |= P.id[o0 - plane];
        if (ytask && y_lo) hid |= (uint32_t)P.id[oy] << 8;
        if (xtask && x_lo) hid |= (uint32_t)P.id[ox] << 16;
    }
    // surface buffers: this CTA's and its neighbours' (word offsets; the step's parity is added)
    const int dx = L::W, dy = P.px * L::W, dz = P.px * P.py * L::W;
    WordMem *const words = static_cast<WordMem *>(P.words), *const own = words + (size_t)b * L::W;
    // box edges, one value each: warps 0 .. 5 take one edge line, a lane one word
    int e_src = b * L::W, e_dst = -1;   // e_dst < 0: none
    {
        const int w = j, l = i;
        if (w == 0 && l < by && x_lo && z_hi) { e_src += -dx + dz + L::XP + l; e_dst = L::e(-1, l, bz); }
        if (w == 1 && l < bz && x_lo && y_hi) { e_src += -dx + dy + L::XP + l * NW; e_dst = L::e(-1, by, l); }
        if (w == 2 && l < bx && y_lo && z_hi) { e_src += -dy + dz + L::YP + l; e_dst = L::EF + L::e(l, -1, bz); }
        if (w == 3 && l < bz && x_hi && y_lo) { e_src += dx - dy + L::YP + l * BXR; e_dst = L::EF + L::e(bx, -1, l); }
        if (w == 4 && l < bx && y_hi && z_lo) { e_src += dy - dz + L::ZP + l; e_dst = 2 * L::EF + L::e(l, by, -1); }
        if (w == 5 && l < by && x_hi && z_lo) { e_src += dx - dz + L::ZP + l * BXR; e_dst = 2 * L::EF + L::e(bx, l, -1); }
    }
    const bool edge = e_dst >= 0;
    const float4 chu = make_float4(P.ch[0], P.ch[1], P.ch[2], 0.f);
    const size_t par_words = (size_t)gridDim.x * L::W;
    __syncthreads();

    const int T_ = P.steps;
    for (int s = 0; s < T_; ++s) {
        // ---------------- H^{n+1/2} on the own cells ...
        {
            const float *q = se + L::e(i, j, 0);
            float x = DEEP ? q[0] : ex[0], y = DEEP ? q[L::EF] : ey[0];
#pragma unroll
            for (int k = 0; k < BZ; ++k) {
                const int o = k * L::EX * L::EY;
                const float x1 = DEEP ? q[o + L::EX * L::EY] : ex[DEEP ? 0 : k + 1],
                            y1 = DEEP ? q[L::EF + o + L::EX * L::EY] : ey[DEEP ? 0 : k + 1];
                const float ex_j1 = q[o + L::EX], ez_j1 = q[2 * L::EF + o + L::EX];
                const float ey_i1 = q[L::EF + o + 1], ez_i1 = q[2 * L::EF + o + 1];
                const float4 ch = HID ? stab[2 * ((ids[k / 4] >> (8 * (k % 4))) & 0xff) + 1] : chu;
                hx[k] = __fmaf_rn(ch.x, sub(sub(y1, y), sub(ez_j1, ez[k])), hx[k]);
                hy[k] = __fmaf_rn(ch.y, sub(sub(ez_i1, ez[k]), sub(x1, x)), hy[k]);
                hz[k] = __fmaf_rn(ch.z, sub(sub(ex_j1, x), sub(ey_i1, y)), hz[k]);
                x = x1;
                y = y1;
            }
        }
        // ---------------- ... and one cell below the box
        if (act && z_lo) {
            const float4 ch = HID ? stab[2 * (hid & 0xff) + 1] : chu;
            const float *q = se + L::e(i, j, -1);
            const float z = q[2 * L::EF];
            hzx = __fmaf_rn(ch.x, sub(sub(DEEP ? q[L::EF + L::EX * L::EY] : ey[0], q[L::EF]), sub(q[2 * L::EF + L::EX], z)), hzx);
            hzy = __fmaf_rn(ch.y, sub(sub(q[2 * L::EF + 1], z), sub(DEEP ? q[L::EX * L::EY] : ex[0], q[0])), hzy);
        }
        if (ytask && y_lo) {
            const float4 ch = HID ? stab[2 * ((hid >> 8) & 0xff) + 1] : chu;
            const float *q = se + L::e(i, -1, j);
            float *h = sh + L::h(i, -1, j);
            const float y = q[L::EF];
            h[0] = __fmaf_rn(ch.x, sub(sub(q[L::EF + L::EX * L::EY], y), sub(q[2 * L::EF + L::EX], q[2 * L::EF])), h[0]);
            h[2 * L::HF] = __fmaf_rn(ch.z, sub(sub(q[L::EX], q[0]), sub(q[L::EF + 1], y)), h[2 * L::HF]);
        }
        if (xtask && x_lo) {
            const float4 ch = HID ? stab[2 * ((hid >> 16) & 0xff) + 1] : chu;
            const float *q = se + L::e(-1, hj, hk);
            float *h = sh + L::h(-1, hj, hk);
            const float x = q[0];
            h[L::HF] = __fmaf_rn(ch.y, sub(sub(q[2 * L::EF + 1], q[2 * L::EF]), sub(q[L::EX * L::EY], x)), h[L::HF]);
            h[2 * L::HF] = __fmaf_rn(ch.z, sub(sub(q[L::EX], x), sub(q[L::EF + 1], q[L::EF])), h[2 * L::HF]);
        }
        if (act) {
            float *q = sh + L::h(i, j, 0);
#pragma unroll
            for (int k = 0; k < BZ; ++k) {   // planes past bz: rows that nothing reads
                q[k * L::HX * L::HY] = hx[k];
                q[L::HF + k * L::HX * L::HY] = hy[k];
                q[2 * L::HF + k * L::HX * L::HY] = hz[k];
            }
        }
        __syncthreads();
        // ---------------- E^{n+1} on the own cells (planes past bz: id 0, ce = 0)
        {
            const float *q = sh + L::h(i, j, 0);
            float *const e = se + L::e(i, j, 0);
#pragma unroll
            for (int k = 0; k < BZ; ++k) {
                const int o = k * L::HX * L::HY;
                const float hx_jm = q[o - L::HX], hz_jm = q[2 * L::HF + o - L::HX];
                const float hy_im = q[L::HF + o - 1], hz_im = q[2 * L::HF + o - 1];
                const float hx_km = k ? hx[k ? k - 1 : 0] : hzx, hy_km = k ? hy[k ? k - 1 : 0] : hzy;
                const float4 ce = stab[2 * ((ids[k / 4] >> (8 * (k % 4))) & 0xff)];
                const float cx = sub(sub(hz[k], hz_jm), sub(hy[k], hy_km)), cy = sub(sub(hx[k], hx_km), sub(hz[k], hz_im));
                if constexpr (DEEP) {   // neighbours read these after the barrier only; planes past bz: E + 0
                    float *const g = e + k * L::EX * L::EY;
                    const float x = __fmaf_rn(ce.x, cx, g[0]), y = __fmaf_rn(ce.y, cy, g[L::EF]);
                    if (act) {
                        g[0] = x;
                        g[L::EF] = y;
                    }
                } else {
                    ex[k] = __fmaf_rn(ce.x, cx, ex[k]);
                    ey[k] = __fmaf_rn(ce.y, cy, ey[k]);
                }
                ez[k] = __fmaf_rn(ce.z, sub(sub(hy[k], hy_im), sub(hx[k], hx_jm)), ez[k]);
            }
        }
        if (src_mask) {   // point currents: E -= ce dx J of this step, in the callers' order
#pragma unroll
            for (int k = 0; k < BZ; ++k)
                if ((src_mask >> k) & 1u)
                    for (int q = 0; q < s_nsrc; ++q)
                        if (srcs[q].tid == t && srcs[q].k == k) {
                            const long long n = s_n0 + s;
                            const float J = n < X.wave_len ? X.wave[(size_t)srcs[q].q * X.wave_len + n] * P.scale_e : 0.f;
                            if (J == 0.f) continue;
                            const float cd = srcs[q].cd;
                            if (DEEP && srcs[q].comp < 2) {
                                float &g = se[srcs[q].comp * L::EF + L::e(i, j, k)];
                                g = __fmaf_rn(-cd, J, g);
                            } else if (srcs[q].comp == 0) ex[DEEP ? 0 : k] = __fmaf_rn(-cd, J, ex[DEEP ? 0 : k]);
                            else if (srcs[q].comp == 1) ey[DEEP ? 0 : k] = __fmaf_rn(-cd, J, ey[DEEP ? 0 : k]);
                            else ez[k] = __fmaf_rn(-cd, J, ez[k]);
                        }
        }
        if (act) {
            float *q = se + L::e(i, j, 0);
#pragma unroll
            for (int k = 0; k < BZ; ++k)
                if (k < bz) {
                    if constexpr (!DEEP) {
                        q[k * L::EX * L::EY] = ex[k];
                        q[L::EF + k * L::EX * L::EY] = ey[k];
                    }
                    q[2 * L::EF + k * L::EX * L::EY] = ez[k];
                }
        }
        __syncthreads();
        const bool last = s == T_ - 1;
        if (!last) {
            // ---------------- send the surface, take the shell of the next step
            const unsigned tag = tag0 + (unsigned)s + 1u;
            const size_t par = (s & 1) ? par_words : 0;
            WordMem *const o = own + par;
            const bool zl = act && z_lo, zh = act && z_hi, yl = ytask && y_lo, yh = ytask && y_hi, xl = xtask && x_lo,
                       xh = xtask && x_hi;
            const int wz = t, wy = t, wx = hk * NW + hj;   // (j, i), (plane j, i), (hk, hj) in their faces
            if (zh) {
                const float *q = se + L::e(i, j, bz - 1);
                st_word(o + L::ZP + wz, q[0], q[L::EF], q[2 * L::EF], tag);
            }
            if (zl) {
                const float *q = se + L::e(i, j, 0);
                st_word(o + L::ZM + wz, q[0], q[L::EF], 0.f, tag);
            }
            if (yh) {
                const float *q = se + L::e(i, by - 1, j);
                st_word(o + L::YP + wy, q[0], q[L::EF], q[2 * L::EF], tag);
            }
            if (yl) {
                const float *q = se + L::e(i, 0, j);
                st_word(o + L::YM + wy, q[0], 0.f, q[2 * L::EF], tag);
            }
            if (xh) {
                const float *q = se + L::e(bx - 1, hj, hk);
                st_word(o + L::XP + wx, q[0], q[L::EF], q[2 * L::EF], tag);
            }
            if (xl) {
                const float *q = se + L::e(0, hj, hk);
                st_word(o + L::XM + wx, 0.f, q[L::EF], q[2 * L::EF], tag);
            }
            const WordMem *const p[7] = {o - dz + L::ZP + wz, o + dz + L::ZM + wz, words + par + e_src, o - dy + L::YP + wy,
                                         o + dy + L::YM + wy, o - dx + L::XP + wx, o + dx + L::XM + wx};
            const unsigned want = (zl ? 1u : 0u) | (zh ? 2u : 0u) | (edge ? 4u : 0u) | (yl ? 8u : 0u) | (yh ? 16u : 0u) |
                                  (xl ? 32u : 0u) | (xh ? 64u : 0u);
            Word v[7];
#pragma unroll
            for (int c = 0; c < 7; ++c)
                if ((want >> c) & 1u) v[c] = ld_word(p[c]);
            wait_words<7>(p, v, want, tag, kPolls, P.status, &s_abort);
            if (zl) {
                float *q = se + L::e(i, j, -1);
                q[0] = v[0].a();
                q[L::EF] = v[0].b();
                q[2 * L::EF] = v[0].c();
            }
            if (zh) {
                if constexpr (DEEP) {
                    se[L::e(i, j, bz)] = v[1].a();
                    se[L::EF + L::e(i, j, bz)] = v[1].b();
                } else {
#pragma unroll
                    for (int k = 1; k < NE; ++k) {
                        ex[k] = k == bz ? v[1].a() : ex[k];
                        ey[k] = k == bz ? v[1].b() : ey[k];
                    }
                }
            }
            if (edge) se[e_dst] = j < 2 ? v[2].a() : j < 4 ? v[2].b() : v[2].c();
            if (yl) {
                float *q = se + L::e(i, -1, j);
                q[0] = v[3].a();
                q[L::EF] = v[3].b();
                q[2 * L::EF] = v[3].c();
            }
            if (yh) {
                float *q = se + L::e(i, by, j);
                q[0] = v[4].a();
                q[2 * L::EF] = v[4].c();
            }
            if (xl) {
                float *q = se + L::e(-1, hj, hk);
                q[0] = v[5].a();
                q[L::EF] = v[5].b();
                q[2 * L::EF] = v[5].c();
            }
            if (xh) {
                float *q = se + L::e(bx, hj, hk);
                q[L::EF] = v[6].b();
                q[2 * L::EF] = v[6].c();
            }
        }
        const long long slot = s_n0 + s - X.probe_start;
        if (slot >= 0 && slot < X.capacity)
            for (int q = t; q < s_nprobe; q += NT) {
                const OwnProbe pr = probes[q];
                X.probe_buf[(size_t)pr.q * X.capacity + slot] = se[pr.at] * (pr.comp < 3 ? P.inv_scale_e : P.inv_scale_h);
            }
        if (last) break;
        __syncthreads();
        if (s_abort) return;   // a wait ran out here or elsewhere: the status is latched
    }

    // ---------------- final state
    if (act)
        by_storage(P.storage, [&](auto type) __attribute__((always_inline)) {
            using T = decltype(type);
            T *const d = static_cast<T *>(P.dst);
#pragma unroll
            for (int k = 0; k < BZ; ++k)
                if (k < bz && fused::store_ok(P.status, o0 + k * plane, 1, fs)) {
                    T *const g = d + o0 + k * plane;
                    g[0] = Storage<T>::store(DEEP ? se[L::e(i, j, k)] : ex[DEEP ? 0 : k]);
                    g[fs] = Storage<T>::store(DEEP ? se[L::EF + L::e(i, j, k)] : ey[DEEP ? 0 : k]);
                    g[2 * fs] = Storage<T>::store(ez[k]);
                    g[3 * fs] = Storage<T>::store(hx[k]);
                    g[4 * fs] = Storage<T>::store(hy[k]);
                    g[5 * fs] = Storage<T>::store(hz[k]);
                }
        });
}

template <int BZ, bool HID> cudaError_t launch_typed(const ResidentParams &P, int ctas, cudaStream_t s) {
    ResidentParams p = P;
    if (!p.id) p.ntab = 9;
    const int smem = smem_bytes<BZ>(p.ntab, p.X.nsrc, p.X.nprobe);
    auto kern = resident_kernel<BZ, HID>;
    cudaError_t e = allow_all_smem(kern, 64);   // static: 32 bytes
    if (e != cudaSuccess) return e;
    void *args[] = {&p};
    return cudaLaunchCooperativeKernel((const void *)kern, dim3(ctas), dim3(NT), args, smem, s);
}

template <int BZ> cudaError_t launch_bz(const ResidentParams &P, int ctas, cudaStream_t s) {
    return P.id && !P.ch_uniform ? launch_typed<BZ, true>(P, ctas, s) : launch_typed<BZ, false>(P, ctas, s);
}

// Planes of the instance that runs boxes of bz planes.
int instance_bz(int bz) { return bz <= 2 ? 2 : bz <= 4 ? 4 : bz <= 6 ? 6 : bz <= 8 ? 8 : bz <= 11 ? 11 : 14; }

}  // namespace

// The split into boxes: the fewest rows and columns of boxes, then the least depth that max_ctas boxes allow, then the
// fewest boxes of the instance for that depth.  A warp works through its planes one after the other and all warps run
// the plane loops, so a step takes as long as the instance is deep (us a step with 2, 4, 6, 8, 11, 14 planes: 1.9, 2.4,
// 2.8, 3.4, 4.2, 4.7) and hardly depends on the rows or columns of a box.  Boxes beyond that only keep other streams'
// launches from the SMs: 24 x 20 x 17 cells take 1.75 us a step in 90 boxes and 1.89 in 18; eight such contexts on
// eight streams 1.74 and 0.25 us per step and context, since several of the launches then fit at once (32^3: 128
// boxes 1.73 and 1.71, 32 boxes 1.88 and 0.47; 18 x 11 x 22: 121 boxes 1.79 and 1.73, 11 boxes 1.54 and 0.24).
// Parts are equal to one cell, so the fullest CTA has ceil(n / parts) per axis.
bool resident_split(int nx, int ny, int nz, int max_ctas, int parts[3]) {
    const int px = (nx + BXR - 1) / BXR, py = (ny + NW - 1) / NW;
    if ((long long)px * py > max_ctas) return false;
    const int most = std::min(nz, max_ctas / (px * py)), bz = (nz + most - 1) / most;
    if (bz > kResidentMaxBZ) return false;
    parts[0] = px;
    parts[1] = py;
    parts[2] = (nz + instance_bz(bz) - 1) / instance_bz(bz);
    return true;
}

size_t resident_word_bytes(int nz, const int parts[3]) {
    const int bz = instance_bz((nz + parts[2] - 1) / parts[2]);
    const int w = bz == 2 ? Lay<2>::W : bz == 4 ? Lay<4>::W : bz == 6 ? Lay<6>::W : bz == 8 ? Lay<8>::W
                  : bz == 11 ? Lay<11>::W : Lay<14>::W;
    return sizeof(WordMem) * 2 * (size_t)w * parts[0] * parts[1] * parts[2];
}

cudaError_t launch_resident(const ResidentParams &P, cudaStream_t s) {
    const int ctas = P.px * P.py * P.pz;
    switch (instance_bz((P.nz + P.pz - 1) / P.pz)) {
        case 2: return launch_bz<2>(P, ctas, s);
        case 4: return launch_bz<4>(P, ctas, s);
        case 6: return launch_bz<6>(P, ctas, s);
        case 8: return launch_bz<8>(P, ctas, s);
        case 11: return launch_bz<11>(P, ctas, s);
        default: return launch_bz<14>(P, ctas, s);
    }
}

}  // namespace fdtd
