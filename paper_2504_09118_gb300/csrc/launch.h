// Host-side launchers of libfdtd's kernels (C++ linkage, internal to the library).
#pragma once

#include "fdtd_internal.cuh"

namespace fdtd {

// Canonical FP32 components comp0 .. comp0 + ncomp - 1 (canon[0 .. ncomp)) -> active arrays (scaled, rounded
// to storage), tangential E zeroed, far-face normal H -> the face arrays (FP32, after the same rounding).
cudaError_t launch_pack(int storage, const CavityDesc &d, int copy, int comp0, int ncomp, const float *const *canon,
                        cudaStream_t s);
// Active arrays (+ faces) -> canonical FP32 components, zero outside the extents.
cudaError_t launch_unpack(int storage, const CavityDesc &d, int copy, int comp0, int ncomp, float *const *canon,
                          cudaStream_t s);
// max |canon[q]| over each component's extent, as float bits atomically max-ed into out[comp0 + q] (0 at start).
cudaError_t launch_maxabs(const float *const *canon, int comp0, int ncomp, int nx, int ny, int nz, unsigned *out,
                          cudaStream_t s);
// One unfused step in place on copy `copy`: H kernel then E kernel.
cudaError_t launch_simple_step(int storage, const CavityDesc &d, int copy, cudaStream_t s);
// Reductions accumulated in FP64: what == 0 gives out[0] = sum E^2/ce + H.(H - ch curl E)/ch;
// what == 1 gives out[1] = sum divE^2, out[2] = sum divH^2.  partial holds nblocks*3 doubles.
// order 4 takes the curl and divergences of the fourth-order scheme.
// out[3] = the device status word.
cudaError_t launch_reductions(int storage, const CavityDesc &d, int copy, int what, double *partial, int nblocks,
                              const int *status, double *out, cudaStream_t s, int order = 2);
// Fourth-order scheme (k_order4.cu): one unfused step in place on copy `copy`, and the per-block
// partials of its reductions (same layout as launch_reductions' partial).
cudaError_t launch_simple4_step(int storage, const CavityDesc &d, int copy, cudaStream_t s);
cudaError_t launch_reductions4(int storage, const CavityDesc &d, int copy, int what, double *partial, int nblocks,
                               cudaStream_t s);
int reduction_blocks();

struct FusedLaunch {
    const TileRec *recs;       // device array, one record per tile
    // device step clock compared with TileRec::stop (NULL: no tile skipped), then a CTA count: the two-step kernel
    // (one row per warp) moves the clock itself, after the others launch_step_counter does
    long long *step;
    int ntiles;
    int parity;
    int *status;
    int tile_y;
    int stages;
    int grid;
    int inject_timeout_us;     // >0: do not issue the CTA 0's first unit; wait limit in us
    const int *first;          // device, grid + 1 entries: CTA b takes tiles [first[b], first[b+1]) in order
                               // (NULL: CTA b takes tiles b, b + grid, b + 2 grid, ...)
    int launch_steps;          // two-step kernel: 2, or 1 (every tile stores its level-1 result only)
    int rows_per_warp;         // two-step kernel: 1 (k_fused2.cu) or 2 (k_fused2r.cu); 0 means 1
    bool overlap;              // start as SMs fall free of the launch before (launch_overlapped)
    int coef_class;            // CoefClass shared by every tile (COEF_CLASS_ANY*: read from each record)
};
// Lets launches of a kernel instance use all the dynamic shared memory a block can have (227 KB less the instance's own
// static part).  The limit belongs to the function, not to a launch: the same value every time, so that host threads
// launching one instance with different needs (ring depths, material tables, probes) never lower it for each other.
constexpr int kMaxSmem = 227 * 1024;
template <typename Kernel> inline cudaError_t allow_all_smem(Kernel kern, int static_bytes = 0) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem - static_bytes);
}

// Launch a kernel whose CTAs may start while the previous kernel of the stream ends (it calls grid_wait_previous
// before it touches the fields).  Back to back, a tiled launch otherwise pays its launch latency, barrier set-up and
// first ring fill after the slowest CTA of the launch before it: per launch 2-4 us of 30-40 (200 x 131 x 120 BF16: a
// 64-step pass 1.44 -> 1.34 ms; 160 x 150 x 140 per-position 1.49 -> 1.39 ms).  CTAs started that way land on the SMs
// in the order these fall free, which moves neighbouring tiles apart and costs large FP32 cavities halo reads.  Two-step
// kernel, us a step without and with overlap, FP32: 211 x 198 x 368 (1.5e7 cells) 79.3 / 77.8, 256^3 81.2 / 79.7,
// 234 x 379 x 230 (2.0e7) 96.2 / 100.0, 115 x 354 x 521 (2.1e7) 108.0 / 109.6, 247 x 328 x 271 (2.2e7) 110.5 / 109.1,
// 288^3 (2.4e7) 103.5 / 102.0, 320^3 145.7 / 145.0, 384^3 248.2 / 248.9, 512^3 596 / 600; BF16: 256^3 69.9 / 68.4, 288^3
// 85.0 / 83.1, 384^3 204.7 / 202.8, 512^3 459 / 460.  So FP32 launches overlap below 2e7 cells, where all gain, and 16-bit
// ones below 3e7 (a batch: its running members' cells).
constexpr long long kOverlapCells32 = 20000000, kOverlapCells16 = 30000000, kOverlapCellsBatch = 30000000;
template <typename Kernel, typename Params>
inline cudaError_t launch_overlapped(Kernel kern, int grid, int threads, int smem, cudaStream_t s, const Params &p,
                                     bool overlap) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, p);
}
// Coefficient layout shared by all tiles of a launch, so that a kernel can be compiled for it.
enum CoefClass : int {
    COEF_CLASS_ANY = 0,        // tiles may differ (batches of mixed members): the record's mode decides
    COEF_CLASS_SCALAR = 1,     // COEF_SCALAR: three ce and three ch for the whole cavity
    COEF_CLASS_ID_UNIFORM_H = 2,  // COEF_ID8 with the same ch in every cell
    COEF_CLASS_ID = 3,         // COEF_ID8 with ce and ch per material id
    // COEF_ID8 whose ids and table code the PEC faces (fdtd_ctx::id_pec): no per-cell masks in the kernel
    COEF_CLASS_PEC_ID_UNIFORM_H = 4,
    COEF_CLASS_PEC_ID = 5,
    // COEF_FULL: per-position FP32 ce arrays (and ch arrays) streamed with the fields
    COEF_CLASS_FULL_UNIFORM_H = 6,
    COEF_CLASS_FULL = 7,
    COEF_CLASS_ANY_STEADY = 8,    // a batch's tiles may differ, and most are deep enough for a steady-state body per layout
};
inline int coef_class_of(int coef_mode, int ch_uniform, bool pec_ids) {
    if (coef_mode == COEF_SCALAR) return COEF_CLASS_SCALAR;
    if (coef_mode == COEF_ID8) {
        if (pec_ids) return ch_uniform ? COEF_CLASS_PEC_ID_UNIFORM_H : COEF_CLASS_PEC_ID;
        return ch_uniform ? COEF_CLASS_ID_UNIFORM_H : COEF_CLASS_ID;
    }
    if (coef_mode == COEF_FULL) return ch_uniform ? COEF_CLASS_FULL_UNIFORM_H : COEF_CLASS_FULL;
    return COEF_CLASS_ANY;
}
// Shared memory bytes and max co-resident CTAs per SM for a fused configuration.
int fused_smem_bytes(int storage, int tile_y, int stages);
cudaError_t fused_occupancy(int storage, int tile_y, int stages, int *ctas_per_sm);
cudaError_t launch_fused_step(int storage, const FusedLaunch &L, cudaStream_t s);
// Point currents and probes applied after a step (k_extras.cu).
struct ExtrasParams {
    long long *clock;          // device: steps taken since fdtd_set_fields; advanced by the launch
    int nsrc, wave_len;
    const int *src_comp;       // 0..2 (Ex, Ey, Ez)
    const long long *src_off;  // active-array offsets
    const float *wave;         // nsrc x wave_len: J^{n+1/2} of step n
    float dx;
    int nprobe, capacity;
    long long probe_start;     // step index of the probe buffer's first sample
    const int *probe_comp;     // 0..5
    const long long *probe_off;
    float *probe_buf;          // nprobe x capacity, physical units
};
cudaError_t launch_extras(int storage, const CavityDesc &d, int copy, const ExtrasParams &X, cudaStream_t s);

// Many steps of a small cavity in one cooperative launch, the state on chip (k_resident.cu).
constexpr int kResidentMaxBZ = 14;       // cells per box along z (at most 32 along x, 16 along y)
constexpr int kResidentMaxSources = 32, kResidentMaxProbes = 256;
struct ResidentParams {
    const void *src;           // first of the six source arrays, fstride elements apart
    void *dst;                 // first of the six result arrays
    int storage;
    int fstride;
    int nx, ny, nz, pitch, plane;
    int px, py, pz;            // boxes along each axis
    int steps;
    float ce[3], ch[3];        // in storage units (TileRec); ch also when ch_uniform
    const uint8_t *id;         // PEC-coded ids (NULL: uniform cavity) and their table, ntab entries
    const float4 *table;
    int ntab, ch_uniform;
    float scale_e, inv_scale_e, inv_scale_h;
    float ce_mat[3];           // unscaled coefficients for currents: scalars, or table by plain id
    const uint8_t *id_mat;
    const float *table_mat;
    void *words;               // surface buffers of every box, two copies (resident_word_bytes, zero at first)
    unsigned *epoch;           // step tag the next launch starts from, and a count of CTAs (both 0 at first)
    int *status;
    int lose_polls;            // diagnostic, > 0: a wait of CTA 0 runs out after this many poll rounds
    ExtrasParams X;            // currents and probes (nsrc = nprobe = 0: none); advances X.clock
};
bool resident_split(int nx, int ny, int nz, int max_ctas, int parts[3]);
size_t resident_word_bytes(int nz, const int parts[3]);
cudaError_t launch_resident(const ResidentParams &P, cudaStream_t s);

// Adds inc to the device step clock of a batch (one thread; ordered after the launch it follows; not for the two-step
// kernel with one row per warp).
cudaError_t launch_step_counter(long long *counter, int inc, cudaStream_t s);
// Two-step (temporal blocking) kernel: output tile width along x, shared memory, occupancy, launch.
int fused2_tile_w(int storage);
int fused2_smem_bytes(int storage, int tile_y, int stages);
// The same for per-position coefficients (tile height 12 only; the class is one of COEF_CLASS_FULL*).
constexpr int kFullTileY = 12;
int fused2_full_smem_bytes(int storage, int coef_class, int stages);
cudaError_t fused2_occupancy(int storage, int tile_y, int stages, int *ctas_per_sm);
cudaError_t launch_fused2_step(int storage, const FusedLaunch &L, cudaStream_t s);
// The two-step kernel with two rows per consumer warp (k_fused2r.cu; tile heights 12 and 16): the same
// tiles, boxes and results, a different split of the rows over the warps.
int fused2r_smem_bytes(int storage, int tile_y, int stages);
cudaError_t fused2r_occupancy(int storage, int tile_y, int stages, int *ctas_per_sm);
cudaError_t launch_fused2r_step(int storage, const FusedLaunch &L, cudaStream_t s);
// Three-step (T = 3) kernel (k_fused3.cu; single cavities, tile heights 8, 10 and 12): output tile width along x,
// shared memory, occupancy, launch.
int fused3_tile_w();
int fused3_smem_bytes(int storage, int tile_y, int stages);
cudaError_t fused3_occupancy(int storage, int tile_y, int stages, int *ctas_per_sm);
cudaError_t launch_fused3_step(int storage, const FusedLaunch &L, cudaStream_t s);
// Fused fourth-order kernel (k_fused4.cu): shared memory, occupancy, launch (stages 4..8).
int fused4_smem_bytes(int storage, int tile_y, int stages);
cudaError_t fused4_occupancy(int storage, int tile_y, int stages, int *ctas_per_sm);
cudaError_t launch_fused4_step(int storage, const FusedLaunch &L, cudaStream_t s);
// Box sizes used to encode the tensor maps of the fused kernel.
void fused_box(int storage, int tile_y, int *box_x, int *box_y, int *halo_x);

}  // namespace fdtd
