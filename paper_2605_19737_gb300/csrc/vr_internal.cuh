// vr_internal.cuh -- declarations shared by the library's translation units.
//
// Volume storage. Interpolation cell i0 spans voxels i0 and i0+1 along each axis;
// a sample whose clamped coordinate u_c has floor cell i0 = min(floor(u_c), N-2)
// lies in that cell. Two brick grids cut the cells:
//  * storage bricks of 8^3 cells hold the intensities (and the second channel)
//    for the per-sample stencils: a dense 12^3 float32 block of voxels
//    [8b-1, 8b+11) per axis with clamp-to-edge values outside the volume, so the
//    4-tap stencils of a cell (voxels i0-1 .. i0+2) fall inside it; 6912 bytes
//    (a multiple of 16), one bulk copy moves it;
//  * skip bricks of B^3 cells (B = 2^bs, 4, 8 or 16; 8 by default) carry the
//    quantised min/max grid, the empty flags and the
//    derived bricks of the voxel-wise derivatives, (B+1)^3 corners each.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "vr.h"
#include "vr_async.cuh"
#include "vr_df.cuh"

namespace vr {

constexpr int kCells = 8;                          // interpolation cells per brick edge
constexpr int kEdge = 12;                          // stored brick edge (1 low + 8 + 3 high apron)
constexpr int kBrickVox = kEdge * kEdge * kEdge;   // 1728 floats
constexpr int kBrickBytes = kBrickVox * 4;         // 6912 bytes
constexpr int kMaxCamsPerLaunch = 64;

// Derived bricks: per skip brick the (B+1)^3 corner voxels [Bb, Bb+B] (clamped) of
// its cells, the voxel-wise derivatives of Sec. 2.3 in mm units: (I, gx, gy, gz), (Hxx, Hyy,
// Hzz, Hxy) and (Hxz, Hyz) of every corner, read by a 16-, a 16- and an 8-byte load. A
// brick's place in the store is 12 floats per corner (B = 8: 9^3 corners, 34,992 B).
constexpr int kDerFloats = 12;
constexpr int kMinBrickShift = 2, kMaxBrickShift = 4;  // skip bricks of 4^3 .. 16^3 cells

__host__ __device__ __forceinline__ constexpr int der_edge(int bs) { return (1 << bs) + 1; }
__host__ __device__ __forceinline__ constexpr long long der_brick_floats(int bs) {
    const long long e = der_edge(bs);
    return e * e * e * kDerFloats;
}

// Where a corner's three pieces lie in its brick. The raymarch kernels are bound by the L1
// data stage (68-70 % of its passes in the 540p frame and its backward): the 16-byte loads
// of a quarter warp go through in one pass only if they meet different 16-byte columns of
// the 128-byte lines. In records of 48 bytes in rows of B + 1, a corner's neighbours along
// x, y and z all lie 3 columns on; a load took 5.1 passes (4 without conflicts). For B = 8
// and 16 the pieces are therefore three planes, and what they leave of the brick's place
// pads their rows and slices so that neighbours lie x 1, y 2, z 4 columns on: the corners
// of a cell, or one corner of eight neighbouring cells, on eight columns. Without a
// curvature term only the first plane is read, 16 of 16 bytes instead of 16 of 48.
// Measured, records -> planes: 1080p frame of the 181x217x181 head 1.88 -> 1.82 ms, its
// 540p at B = 16 0.84 -> 0.77, 32 views without curvature 8.88 -> 8.27, fit step of 8 views
// 6.90 -> 6.07. What a sparse ray with curvature reads lies on twice the lines that records did
// (12-13 a sample instead of 6-7; 64x64 of the head at one lane per ray and 64 registers 1195 ->
// 1645 us): launches of few rays give a ray several lanes or a warp more registers, after which
// they are faster than with records. B = 4 has no room for the padding (planes:
// 700x600 0.78 -> 0.81 ms) and keeps the records. Kernels take the layout of a fixed B: as
// run-time values it cost the launches of several lanes per ray 3 %.
struct DerLayout {
    int row, slice;  // records to a corner's neighbours along y and z
    int rec, m;      // float4 per record, and from its first to its second piece
    int t, trec;     // float2 from the brick's start to record 0's third piece, and per record
};
__host__ __device__ __forceinline__ constexpr DerLayout der_planes(int row, int slice, int B) {
    const int n = B * (slice + row + 1) + 1;  // records of a padded plane
    return DerLayout{row, slice, 1, n, 4 * n, 1};
}
__host__ __device__ __forceinline__ constexpr DerLayout der_layout(int bs) {
    return bs == 2 ? DerLayout{5, 25, 3, 1, 4, 6} : bs == 3 ? der_planes(10, 92, 8) : der_planes(18, 308, 16);
}
static_assert(10 * der_layout(3).m <= der_brick_floats(3) && 10 * der_layout(4).m <= der_brick_floats(4),
              "the planes fit a brick's place");

// Skip field: per interpolation cell one byte, the Chebyshev distance in cells to the
// nearest cell that may hold opacity under the current transfer function, capped (0: the
// cell itself may, so its samples are evaluated). Cells are stored in 4x4 columns of
// (y, z), 16 bytes each, so that a 32-byte sector covers 2x4x4 cells and a line
// 8x4x4: neighbouring rays and consecutive samples stay in a few sectors.
struct SkipDims {
    int cx, cy, cz;     // cells per axis, n - 1
    int wx;             // 32-cell words per row of the cell bit grid
    int bx, by, bz;     // 4^3-cell blocks per axis
    int bwx;            // 32-block words per row of the block bit grid
};
__host__ __device__ __forceinline__ SkipDims skip_dims(const int n[3]) {
    SkipDims d;
    d.cx = n[0] - 1, d.cy = n[1] - 1, d.cz = n[2] - 1;
    d.wx = (d.cx + 31) >> 5;
    d.bx = (d.cx + 3) >> 2, d.by = (d.cy + 3) >> 2, d.bz = (d.cz + 3) >> 2;
    d.bwx = (d.bx + 31) >> 5;
    return d;
}
__host__ __device__ __forceinline__ size_t skip_index(int x, int y, int z, int cx, int by) {
    return (size_t)(unsigned)(((z >> 2) * by + (y >> 2)) * cx + x) * 16 + (((y & 3) << 2) | (z & 3));
}
// One allocation holds the field and the scratch of its construction.
struct SkipStore {
    uint8_t* field;       // skip_index order
    uint32_t* cell_bits;  // [cz][cy][wx], bit set = cell empty
    uint32_t* block_bits; // [bz][by][bwx], bit set = 4^3 block empty
    uint4* block_dist;    // [bz][by][bwx] distance in blocks to the nearest non-empty block, capped,
                          // as four bit planes of 32 blocks
    int* limits;          // [kMaxTableWidth] the table's column limits
};
constexpr int kMaxTableWidth = 4096;
inline size_t skip_store_bytes(const int n[3]) {
    const SkipDims d = skip_dims(n);
    const size_t f = (size_t)d.bz * d.by * d.cx * 16;
    const size_t c = ((size_t)d.cz * d.cy * d.wx * 4 + 15) & ~(size_t)15;
    const size_t b = ((size_t)d.bz * d.by * d.bwx * 4 + 15) & ~(size_t)15;
    return f + c + b + (size_t)d.bz * d.by * d.bwx * 16 + sizeof(int) * kMaxTableWidth;
}
inline SkipStore skip_store(uint8_t* p, const int n[3]) {
    const SkipDims d = skip_dims(n);
    SkipStore s;
    s.field = p;
    p += (size_t)d.bz * d.by * d.cx * 16;
    s.cell_bits = reinterpret_cast<uint32_t*>(p);
    p += ((size_t)d.cz * d.cy * d.wx * 4 + 15) & ~(size_t)15;
    s.block_bits = reinterpret_cast<uint32_t*>(p);
    p += ((size_t)d.bz * d.by * d.bwx * 4 + 15) & ~(size_t)15;
    s.block_dist = reinterpret_cast<uint4*>(p);
    p += (size_t)d.bz * d.by * d.bwx * 16;
    s.limits = reinterpret_cast<int*>(p);
    return s;
}
constexpr int kSMs = 152;
// Planes that a CTA of a kernel marching along z walks, `columns` CTAs covering a plane:
// as many as keep `resident` CTAs for every SM, from 1 to `most`. Long walks read the two
// border planes once for more planes of output; but a walk is a serial chain of plane
// loads, so a launch that does not fill the chip takes the time of one walk.
inline int march_planes(long long columns, int nz, int resident, int most) {
    const long long p = columns * nz / ((long long)kSMs * resident);
    return p < 1 ? 1 : p > most ? most : (int)p;
}
// Cells of the min/max grid per row, padded to whole warps.
__host__ __device__ __forceinline__ int cellq_pitch(int nx) { return (nx - 1 + 31) & ~31; }
inline size_t cellq_cells(const int n[3]) { return (size_t)cellq_pitch(n[0]) * (n[1] - 1) * (n[2] - 1); }
constexpr size_t kDerivedBudgetBytes = (size_t)16 << 30;  // default: built only up to this size

struct CamDev {
    float eye[3], fwd[3], right[3], up[3];
};

struct TissueDev {
    int tf_mode, tf_w, tf_h, grad_mod, shading;
    float gamma, kappa_ref, w_max, ka, kd, ks, opacity_scale, et_threshold, step_vox;
    float alpha_exp;  // dt / opacity_ref_step for the step-size opacity correction; 0 = off
    // Samples per cell of leap: from a cell at distance d of the skip field, the d - 1
    // layers of cells around it are empty and a sample moves no axis by more than step_vox
    // cells, so the next floor((d - 1) leap_per_cell) samples are empty too and the one
    // after is looked at. leap_per_cell = (1 - 1e-6) / step_vox: the margin exceeds the
    // rounding of the step (2^-32 voxel per sample), so a leap never lands outside them.
    float leap_per_cell;
    float gk, inv_kref;  // gamma / kappa_ref and 1 / kappa_ref (rounded from double on the host)
    unsigned* status;    // the context's device status word (debug builds report failed index checks there)
};

// Index checks of the debug library (VR_DEBUG): VR_CHECK(status, cond) is cond,
// and when cond is false it also sets kStatusBounds in status[0] and records the
// source line of the first failed check in status[1]; the caller skips the access.
// Without VR_DEBUG it is the constant true and the check compiles away.
#ifdef VR_DEBUG
__device__ __forceinline__ bool debug_check(bool ok, unsigned* status, int line) {
    if (!ok && status) {
        atomicOr(status, kStatusBounds);
        atomicCAS(status + 1, 0u, (unsigned)line);
    }
    return ok;
}
#define VR_CHECK(status, cond) ::vr::debug_check((cond), (status), __LINE__)
#else
#define VR_CHECK(status, cond) true
#endif

// Per-volume constants that kernels read from device memory (so that host code
// never waits for the reductions that produce them).
struct VolConst {
    float imin, imax, range, gmax;
};

struct VolumeDev {
    int n[3];       // voxels per axis
    int nb[3];      // skip bricks per axis = ceil((n-1)/B)
    int nsb[3];     // storage bricks per axis = ceil((n-1)/8)
    int bs;         // log2 B, cells per skip-brick edge
    int der_stride; // floats per derived brick, der_brick_floats(bs)
    DerLayout der;  // der_layout(bs)
    float s[3];     // spacing (mm)
    const float* bricks;     // storage bricks x kBrickVox
    const float* vbricks;    // vesselness storage bricks (same layout) or nullptr
    const float* dbricks;    // derived skip bricks or nullptr (then the per-sample stencils are used)
    const uint8_t* empty;    // skip-brick flags, 1 = skip
    const uint8_t* skipf;    // skip field (nullptr before the precompute)
    int skip_cx, skip_by;    // its cells per row and 4-cell blocks along y
    const VolConst* vc;
};

// Per-launch constants of the ray setup, computed once on the host in FP64 and
// passed as double-floats (hi + lo).
struct RayConsts {
    dfloat_h two_over_w, two_over_h;  // 2/W, 2/H
    dfloat_h inv_s[3];                // 1/spacing
    dfloat_h dt;                      // sample spacing step_vox * min(s)
    float inv_dt;                     // 1/dt (only for the sample-count estimate)
};

inline RayConsts make_ray_consts(int W, int H, const float s[3], float step_vox) {
    RayConsts c;
    c.two_over_w = df_split(2.0 / (double)W);
    c.two_over_h = df_split(2.0 / (double)H);
    for (int q = 0; q < 3; ++q) c.inv_s[q] = df_split(1.0 / (double)s[q]);
    const float smin = s[0] < s[1] ? (s[0] < s[2] ? s[0] : s[2]) : (s[1] < s[2] ? s[1] : s[2]);
    const double dt = (double)step_vox * (double)smin;
    c.dt = df_split(dt);
    c.inv_dt = (float)(1.0 / dt);
    return c;
}

struct RenderLaunch {
    VolumeDev vol;
    TissueDev tp;
    RayConsts rc;
    const float* tf;           // [tf_h][tf_w][4]
    float* out;                // [n_cams][H][W][4]
    vr_counters* counters;     // nullable
    unsigned* ray_samples;     // nullable, [n_cams][H][W][2]
    float2* ray_state;         // nullable, [n_cams][H][W]: (last sample index as int bits, transmittance before it)
    int W, H, n_cams, cam_offset;
    int skip;
    int packet_w, packet_h;    // ray packet of a warp (packet_w * packet_h == 32); per-lane kernels: 4, 8 or 16 wide
    int tile_w, tile_h;        // per-lane kernels: CTA tile in pixels (tile_packets_x packets across)
    int tile_sx;               // log2 of the packets across the tile
    int lanes;                 // k_render_lanes: lanes per ray
    unsigned* work_counter;    // staged kernel work queue (zeroed before launch)
    unsigned* status;          // device status word (kStatusTimeout on an expired wait)
    int n_packets_x, n_packets_y, n_work;
    CamDev cams[kMaxCamsPerLaunch];
};

// CTA tile of a per-lane kernel: `warps` warp packets of packet_w x (32 / packet_w)
// rays (packet_w in {4, 8, 16}), min(warps, 16 / packet_w) packets across and the
// rest down: 4 warps give 16 x 8 pixels for every packet shape, 2 warps 8 x 8 or
// 16 x 4, 8 warps 16 x 16.
__host__ __device__ __forceinline__ int tile_packets_x(int packet_w, int warps) {
    return warps < 16 / packet_w ? warps : 16 / packet_w;
}

// Pixel offset (di, dj) of lane l of warp w within that tile (2^sx packets across).
__device__ __forceinline__ void tile_pixel(int packet_w, int sx, int w, int l, int& di, int& dj) {
    const int pl = __ffs(packet_w) - 1;  // log2 packet_w
    const int wx = w & ((1 << sx) - 1), wy = w >> sx;
    di = (wx << pl) + (l & (packet_w - 1));
    dj = wy * (32 >> pl) + (l >> pl);
}

// floats per lookup cell in a private copy of the transfer-function gradient
constexpr int kTfCellFloats = 16;

struct BackwardLaunch {
    RenderLaunch r;
    const float* dl_drgba;  // [n_cams][H][W][4] upstream gradient
    float* dtf;             // [tf_h][tf_w][4], zeroed by the caller
    double* dparams;        // sums for gamma, ka, kd, ks, opacity_scale, zeroed by the caller, or nullptr
    float* dvol;            // nvox or nullptr, zeroed by the caller
    float* dtf_copies;      // n_copies zeroed private copies of the transfer-function gradient, one
                            // 16-float record per lookup cell (TfGradSink); CTA c adds into copy c % n_copies
    int n_copies;
    float* dgrad;           // derived-brick path with dvol: zeroed channel gradients (10 floats per voxel
                            // in three planes, chan_index), else nullptr
};

// One view of a batched render (device-resident table).
struct ViewDev {
    VolumeDev vol;
    TissueDev tp;
    RayConsts rc;
    const float* tf;
    CamDev cam;
    float* out;     // [H][W][4]
    int W, H;
};

struct BatchLaunch {
    const ViewDev* views;
    const int* packet_prefix;  // n_views entries: first packet of each view
    int n_views, n_work;
    int packet_w, packet_h;
    unsigned* work_counter;    // zeroed before every launch
    vr_counters* counters;     // nullable
    int skip;
};

// Record `msg` as the context's last error and return `status`.
vr_status set_error(vr_ctx* ctx, vr_status status, const char* msg);

// Process-unique id of the calling thread's current CUDA context, 0 when there is none or
// the driver cannot tell.
unsigned long long current_cuda_context();

// ---------------------------------------------------------------- launchers
// All return cudaSuccess or the launch error; all enqueue on `st`.
cudaError_t launch_minmax_partials(const void* data, vr_dtype dt, long long n, float* partials, int nblocks,
                                   cudaStream_t st);
cudaError_t launch_minmax_final(const float* partials, int nblocks, float* out2, cudaStream_t st);
int minmax_blocks(long long n);

cudaError_t launch_normalize(const void* raw, vr_dtype dt, long long n, const float* minmax2, VolConst* vc,
                             float* norm, cudaStream_t st);
// Storage bricks (8^3 cells) of `nb` storage bricks per axis.
cudaError_t launch_make_bricks(const float* norm, const int n[3], const int nb[3], float* bricks, cudaStream_t st);
// Skip bricks of 2^bs cells per edge, `nb` per axis.
cudaError_t launch_brick_minmax(const float* norm, const int n[3], const int nb[3], int bs, uint16_t* grid,
                                cudaStream_t st);
cudaError_t launch_make_derived(const float* norm, const int n[3], const int nb[3], int bs, const float s[3],
                                float* dbricks, cudaStream_t st);
cudaError_t launch_gmax(const float* norm, const int n[3], const float s[3], VolConst* vc, cudaStream_t st);
cudaError_t launch_classify(const uint16_t* grid, long long nbricks, const float* tf, int tf_w, int tf_h,
                            uint8_t* empty, int* prefix_scratch /* tf_w + 1 ints */, cudaStream_t st);
// Per interpolation cell the quantised (min, max) of its 8 corner voxels, low and high
// 16 bits: [nz - 1][ny - 1][cellq_pitch(nx)].
cudaError_t launch_cell_minmax(const float* norm, const int n[3], uint32_t* cellq, cudaStream_t st);
// The skip field, and the brick flags of launch_classify, under a transfer function
// (prefix_scratch: tf_w + 1 ints).
cudaError_t launch_skip_field(const uint32_t* cellq, const int n[3], const uint16_t* grid, long long nbricks,
                              const float* tf, int tf_w, int tf_h, int* prefix_scratch, uint8_t* empty,
                              const SkipStore& s, cudaStream_t st);

// Multi-scale vesselness of `norm` into V (both nvox floats); tmp_a and tmp_b are
// nvox floats of scratch each, smax receives each scale's max Hessian norm.
cudaError_t launch_frangi(const float* norm, const int n[3], const float* sigmas, int n_sigmas, float* tmp_a,
                          float* tmp_b, float* smax, float* V, cudaStream_t st);

// 256-bin histogram of the normalised volume (zeroes hist first) and its three tissue peaks
// (peaks4 = three ascending bins, -1 padded, then the count).
cudaError_t launch_histogram(const float* norm, long long n, unsigned long long* hist, cudaStream_t st);
cudaError_t launch_tissue_peaks(const unsigned long long* hist, int lo, int hi, int* peaks4, cudaStream_t st);

// Pre-filters: 3x3x3 median; separable Gaussian (out = G * in, tmp is scratch; in != out).
cudaError_t launch_median3(const float* in, float* out, const int n[3], cudaStream_t st);
cudaError_t launch_gauss3d(const float* in, float* out, float* tmp, const int n[3], float sigma, cudaStream_t st);

// warps: warps per CTA (2, 4 or 8), tiled by tile_pixel.
cudaError_t launch_render_gather(const RenderLaunch& L, int warps, cudaStream_t st);
cudaError_t launch_render_backward(const BackwardLaunch& B, bool staged, cudaStream_t st);
// dtf += the entries' shares of the cell records of every copy; out_params (nullable) =
// the uniform gradients' sums rounded to float
cudaError_t launch_sum_copies(const float* copies, int n_copies, int tf_w, int tf_h, float* dtf,
                              const double* dparams, float* out_params, cudaStream_t st);
cudaError_t launch_fma_peak(float* out, int blocks, int iters, cudaStream_t st);
cudaError_t launch_wait_probe(unsigned* status, long long budget_cycles, cudaStream_t st);
// One thread fails one index check (debug builds record it; release builds do nothing).
cudaError_t launch_check_probe(unsigned* status, cudaStream_t st);
cudaError_t launch_channels_to_voxels(const float* dgrad, const int n[3], const float s[3], float* dvol,
                                      cudaStream_t st);
// The kernels of a batch: some volume without derived bricks; few packets (curved: some view has
// a curvature term); any other.
enum class BatchKind { kMixed, kFew, kMany };
BatchKind batch_kind(int packets, bool all_derived, bool curved);
// CTAs of a kind's kernels that an SM holds.
cudaError_t batch_ctas_per_sm(int warps_per_block, BatchKind kind, int* per_sm);
// bs: the skip-brick size (log2 cells) every view shares, or 0 when they differ.
cudaError_t launch_render_batch(const BatchLaunch& B, int warps_per_block, int ctas, BatchKind kind, int bs,
                                cudaStream_t st);
cudaError_t launch_render_staged(const RenderLaunch& L, int warps_per_block, int ctas, cudaStream_t st);
// The staged design on the derived bricks (skip bricks of 4^3 or 8^3 cells, bs 2 or 3).
cudaError_t launch_render_staged_derived(const RenderLaunch& L, int warps_per_block, int ctas, cudaStream_t st);
int staged_derived_smem_bytes(int warps_per_block, int bs);
cudaError_t staged_derived_config(int warps_per_block, int bs, int* ctas_per_sm);
int staged_smem_bytes(int warps_per_block, bool vessel);
// Set the kernel's dynamic shared-memory limit and report resident CTAs per SM.
cudaError_t staged_config(int warps_per_block, bool vessel, int* ctas_per_sm);

}  // namespace vr
