// vr_volume.cu -- per-volume stages: the parallel reductions of Eq. 1 and
// Eq. 4 (Sec. 2.2, Sec. 4), min-max normalisation (Eq. 1), bricking with a
// clamp-to-edge apron, the quantised per-brick min/max grid and the
// transfer-function-driven empty-brick classification (the calvarium culling
// by transfer-function clipping of Sec. 2.2, used for empty-space skipping).
//
// All of these are HBM-bound streaming kernels: coalesced x-fastest access,
// 16-byte vector loads where the layout allows, grids sized in multiples of
// the SM count.
#include <math.h>

#include "vr_internal.cuh"

namespace vr {

namespace {

constexpr int kReduceThreads = 256;

__device__ __forceinline__ void warp_minmax(float& lo, float& hi) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
}

// Block-wide min/max; result valid in thread 0.
__device__ __forceinline__ void block_minmax(float& lo, float& hi) {
    __shared__ float slo[32], shi[32];
    warp_minmax(lo, hi);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        slo[w] = lo;
        shi[w] = hi;
    }
    __syncthreads();
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        lo = l < nw ? slo[l] : INFINITY;
        hi = l < nw ? shi[l] : -INFINITY;
        warp_minmax(lo, hi);
    }
}

__device__ __forceinline__ void acc(float v, float& lo, float& hi) {
    lo = fminf(lo, v);
    hi = fmaxf(hi, v);
}

// Per-block partial min/max over a grid-stride range; float32 input read as float4.
__global__ void __launch_bounds__(kReduceThreads) k_minmax_partials_f32(const float* __restrict__ x, long long n,
                                                                        float* __restrict__ partials) {
    float lo = INFINITY, hi = -INFINITY;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const bool aligned = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
    long long done = 0;
    if (aligned) {
        const long long n4 = n >> 2;
        const float4* x4 = reinterpret_cast<const float4*>(x);
        for (long long i = tid; i < n4; i += stride) {
            float4 v = __ldg(x4 + i);
            acc(v.x, lo, hi);
            acc(v.y, lo, hi);
            acc(v.z, lo, hi);
            acc(v.w, lo, hi);
        }
        done = n4 << 2;
    }
    for (long long i = done + tid; i < n; i += stride) acc(__ldg(x + i), lo, hi);
    block_minmax(lo, hi);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = lo;
        partials[2 * blockIdx.x + 1] = hi;
    }
}

// uint16 input read as 8 values per 16-byte load.
__global__ void __launch_bounds__(kReduceThreads) k_minmax_partials_u16(const uint16_t* __restrict__ x, long long n,
                                                                        float* __restrict__ partials) {
    float lo = INFINITY, hi = -INFINITY;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const bool aligned = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
    long long done = 0;
    if (aligned) {
        const long long n8 = n >> 3;
        const uint4* x8 = reinterpret_cast<const uint4*>(x);
        for (long long i = tid; i < n8; i += stride) {
            uint4 v = __ldg(x8 + i);
            const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                acc((float)(w[q] & 0xffffu), lo, hi);
                acc((float)(w[q] >> 16), lo, hi);
            }
        }
        done = n8 << 3;
    }
    for (long long i = done + tid; i < n; i += stride) acc((float)__ldg(x + i), lo, hi);
    block_minmax(lo, hi);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = lo;
        partials[2 * blockIdx.x + 1] = hi;
    }
}

__global__ void __launch_bounds__(1024) k_minmax_final(const float* __restrict__ partials, int nblocks,
                                                       float* __restrict__ out2) {
    float lo = INFINITY, hi = -INFINITY;
    for (int i = threadIdx.x; i < nblocks; i += blockDim.x) {
        lo = fminf(lo, partials[2 * i]);
        hi = fmaxf(hi, partials[2 * i + 1]);
    }
    block_minmax(lo, hi);
    if (threadIdx.x == 0) {
        out2[0] = lo;
        out2[1] = hi;
    }
}

// Eq. 1 in float32, one IEEE round-to-nearest operation at a time:
// d = x - I_min; I_norm = d / (I_max - I_min). Also publishes the constants.
template <typename T>
__global__ void k_normalize(const T* __restrict__ raw, long long n, const float* __restrict__ mm,
                            VolConst* __restrict__ vc, float* __restrict__ out) {
    const float imin = __ldg(mm), imax = __ldg(mm + 1);
    const float range = __fsub_rn(imax, imin);
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid == 0) {
        vc->imin = imin;
        vc->imax = imax;
        vc->range = range;
    }
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = tid; i < n; i += stride) out[i] = __fdiv_rn(__fsub_rn((float)__ldg(raw + i), imin), range);
}

// Voxels [8b-1, 8b+11) per axis (clamped) of each brick into its 12^3 block: a thread per
// 16-byte piece of the output (432 per brick), so that stores are whole vectors and the
// index arithmetic is paid once per four voxels (181x217x181: 44 us with one voxel per
// thread -> 36 us, 99 MB written).
constexpr int kBrickPieces = kBrickVox / 4;
__global__ void __launch_bounds__(256) k_make_bricks(const float* __restrict__ norm, int nx, int ny, int nz, int nbx,
                                                     int nby, long long npieces, float4* __restrict__ bricks) {
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    if (i >= npieces) return;
    const int b = (int)(i / kBrickPieces), e = (int)(i - (long long)b * kBrickPieces);
    const int bx = b % nbx, by = (b / nbx) % nby, bz = b / (nbx * nby);
    const int px = e % 3, ly = (e / 3) % kEdge, lz = e / (3 * kEdge);
    const int x = kCells * bx - 1 + 4 * px;
    const int y = min(max(kCells * by - 1 + ly, 0), ny - 1);
    const int z = min(max(kCells * bz - 1 + lz, 0), nz - 1);
    const float* row = norm + ((long long)z * ny + y) * nx;
    float4 v;
    v.x = __ldg(row + min(max(x, 0), nx - 1));
    v.y = __ldg(row + min(x + 1, nx - 1));
    v.z = __ldg(row + min(x + 2, nx - 1));
    v.w = __ldg(row + min(x + 3, nx - 1));
    bricks[i] = v;
}

// One CTA per skip brick: the voxel-wise intensity, central-difference gradient
// (Eq. 2) and second/mixed differences (Sec. 2.3) of the brick's (B+1)^3 corner
// voxels, with clamp-to-edge neighbours, divided by the spacing -- the per-voxel
// morphology the paper's compute shader produces, laid out as der_layout says. Stores are
// whole lines: in the planes a warp writes 32 consecutive pieces, the padding (zeros)
// among them (without it the rows' last sectors are half written: 181x217x181 at B = 8,
// whole precompute 213 us, with it 145; as records 159); the 48-byte records of B = 4 go through shared
// memory (stored straight from the threads that computed them, a warp's store wrote 16 of
// every 48 bytes: 322 us, staged 267). kBS (log2 B) at compile time keeps the divisions by
// the edges out.
template <int kBS>
__global__ void __launch_bounds__(256) k_make_derived(const float* __restrict__ norm, int nx, int ny, int nz, int nbx,
                                                      int nby, float hx, float hy, float hz, float* __restrict__ out) {
    // the brick's corner voxels and their neighbours, [Bb - 1, Bb + B + 2) per axis,
    // clamped to the volume (so neighbour i +- 1 of a corner is tile entry t +- 1)
    constexpr int B = 1 << kBS, E = B + 1, T = B + 3;
    __shared__ float tile[T * T * T];
    constexpr bool kRecords = kBS == 2;
    __shared__ float4 stage[kRecords ? 8 : 1][96];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int b = blockIdx.x;
    const int bx = b % nbx, by = (b / nbx) % nby, bz = b / (nbx * nby);
    const int x0 = B * bx - 1, y0 = B * by - 1, z0 = B * bz - 1;
    for (int e = threadIdx.x; e < T * T * T; e += 256) {
        const int tx = e % T, ty = (e / T) % T, tz = e / (T * T);
        const int x = min(max(x0 + tx, 0), nx - 1), y = min(max(y0 + ty, 0), ny - 1), z = min(max(z0 + tz, 0), nz - 1);
        tile[e] = __ldg(norm + ((long long)z * ny + y) * nx + x);
    }
    __syncthreads();
    constexpr DerLayout d = der_layout(kBS);
    float4* dst = reinterpret_cast<float4*>(out + (size_t)(unsigned)b * (unsigned)der_brick_floats(kBS));
    constexpr int R = kRecords ? E : d.row, S = kRecords ? E * E : d.slice, N = kRecords ? E * E * E : d.m;
    for (int e0 = wid * 32; e0 < N; e0 += 256) {
        const int e = min(e0 + lane, N - 1);
        const int lz = e / S, ly = min(e % S / R, E - 1), lx = min(e % S % R, E - 1);
        const bool pad = lx + R * ly + S * lz != e;
        // the corner voxel (clamped as in the per-voxel definition) in tile coordinates
        const int tx = min(B * bx + lx, nx - 1) - x0, ty = min(B * by + ly, ny - 1) - y0,
                  tz = min(B * bz + lz, nz - 1) - z0;
        const float* t0 = tile + (tz * T + ty) * T + tx;
        auto at = [&](int dx, int dy, int dz) { return t0[(dz * T + dy) * T + dx]; };
        const float c = at(0, 0, 0), c2 = 2.0f * c;
        float4 a, m;
        float2 t;
        a.x = c;
        a.y = (at(1, 0, 0) - at(-1, 0, 0)) * (0.5f * hx);
        a.z = (at(0, 1, 0) - at(0, -1, 0)) * (0.5f * hy);
        a.w = (at(0, 0, 1) - at(0, 0, -1)) * (0.5f * hz);
        m.x = (at(1, 0, 0) - c2 + at(-1, 0, 0)) * (hx * hx);
        m.y = (at(0, 1, 0) - c2 + at(0, -1, 0)) * (hy * hy);
        m.z = (at(0, 0, 1) - c2 + at(0, 0, -1)) * (hz * hz);
        m.w = ((at(1, 1, 0) - at(1, -1, 0)) - (at(-1, 1, 0) - at(-1, -1, 0))) * (0.25f * hx * hy);
        t.x = ((at(1, 0, 1) - at(1, 0, -1)) - (at(-1, 0, 1) - at(-1, 0, -1))) * (0.25f * hx * hz);
        t.y = ((at(0, 1, 1) - at(0, 1, -1)) - (at(0, -1, 1) - at(0, -1, -1))) * (0.25f * hy * hz);
        if (kRecords) {
            float4* sp = stage[kRecords ? wid : 0];
            sp[3 * lane] = a;
            sp[3 * lane + 1] = m;
            sp[3 * lane + 2] = make_float4(t.x, t.y, 0.0f, 0.0f);
            __syncwarp();
            const int left = 3 * (N - e0);  // pieces from e0 on
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (lane + 32 * q < left) dst[3 * e0 + lane + 32 * q] = sp[lane + 32 * q];
            __syncwarp();
        } else if (e0 + lane < N) {
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            dst[e] = pad ? zero : a;
            dst[d.m + e] = pad ? zero : m;
            reinterpret_cast<float2*>(dst)[d.t + e] = pad ? make_float2(0.f, 0.f) : t;
        }
    }
}

// Min/max of I_norm over each skip brick's corner voxels [Bb, min(Bb+B, N-1)] per axis,
// quantised to qlo = floor(min*65535), qhi = ceil(max*65535) (float32 round-to-nearest
// products). A CTA owns 32/B bricks along x at one (y, z): its eight warps share the
// (B+1)^2 voxel rows, each read as 32 consecutive values plus one, reduced over the B
// lanes of a brick, whose last corner is the next brick's first lane (181x217x181, one
// warp per brick with divisions per voxel: 28 -> 16 us).
template <int kBS>
__global__ void __launch_bounds__(256) k_brick_minmax(const float* __restrict__ norm, int nx, int ny, int nz, int nbx,
                                                      uint16_t* __restrict__ grid) {
    constexpr int B = 1 << kBS, E = B + 1;
    __shared__ float slo[8][32], shi[8][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * B, z0 = blockIdx.z * B;
    const int xa = min(x0 + lane, nx - 1), xb = min(x0 + 32, nx - 1);
    float lo = INFINITY, hi = -INFINITY, elo = INFINITY, ehi = -INFINITY;  // own column; lane 31: the 33rd
#pragma unroll 4
    for (int r = wid; r < E * E; r += 8) {
        const int y = min(y0 + r % E, ny - 1), z = min(z0 + r / E, nz - 1);
        const float* row = norm + ((long long)z * ny + y) * nx;
        acc(__ldg(row + xa), lo, hi);
        if (lane == 31) acc(__ldg(row + xb), elo, ehi);
    }
    // the brick's columns are its B lanes and the lane after them
    float nlo = __shfl_down_sync(0xffffffffu, lo, 1), nhi = __shfl_down_sync(0xffffffffu, hi, 1);
    if (lane == 31) nlo = elo, nhi = ehi;
    lo = fminf(lo, nlo);
    hi = fmaxf(hi, nhi);
#pragma unroll
    for (int o = B / 2; o; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    slo[wid][lane] = lo;
    shi[wid][lane] = hi;
    __syncthreads();
    const int bx = blockIdx.x * (32 / B) + lane / B;
    if (wid == 0 && (lane & (B - 1)) == 0 && bx < nbx) {
#pragma unroll
        for (int w = 1; w < 8; ++w) {
            lo = fminf(lo, slo[w][lane]);
            hi = fmaxf(hi, shi[w][lane]);
        }
        const long long b = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * nbx + bx;
        // codes clamp to [0, 65535]: intensities set outside [0, 1] (vr_set_normalized)
        // look up the transfer function's end entries, which the clamped range covers
        grid[2 * b] = (uint16_t)fminf(fmaxf(floorf(__fmul_rn(lo, 65535.0f)), 0.0f), 65535.0f);
        grid[2 * b + 1] = (uint16_t)fminf(fmaxf(ceilf(__fmul_rn(hi, 65535.0f)), 0.0f), 65535.0f);
    }
}

// |grad I|_max: largest voxel-wise central-difference gradient magnitude
// (Eq. 2 with clamp-to-edge neighbours), reduced per block then combined with
// an integer atomicMax on the (non-negative) float's bit pattern.
// A thread walks kGmaxPlanes planes along z with the centre values of the planes below and
// above in registers: four in-plane neighbour loads and one new centre per voxel instead of
// seven loads (256x256x176: 53 -> 30 us).
constexpr int kGmaxPlanes = 8;
__global__ void __launch_bounds__(256) k_gmax(const float* __restrict__ I, int nx, int ny, int nz, float hx, float hy,
                                              float hz, VolConst* __restrict__ vc) {
    const int i = blockIdx.x * 32 + (threadIdx.x & 31);
    const int j = blockIdx.y * 8 + (threadIdx.x >> 5);
    const int k0 = blockIdx.z * kGmaxPlanes;
    float m = 0.0f;
    if (i < nx && j < ny) {
        const long long row = (long long)ny * nx;
        const float* c = I + (long long)k0 * row + (long long)j * nx + i;
        const int xp = i + 1 < nx ? 1 : 0, xm = i > 0 ? -1 : 0, yp = j + 1 < ny ? nx : 0, ym = j > 0 ? -nx : 0;
        float zm = __ldg(c - (k0 > 0 ? row : 0)), z0 = __ldg(c);
#pragma unroll
        for (int q = 0; q < kGmaxPlanes; ++q) {
            const int k = k0 + q;
            if (k >= nz) break;
            const float zp = k + 1 < nz ? __ldg(c + row) : z0;
            const float gx = (__ldg(c + xp) - __ldg(c + xm)) * hx;
            const float gy = (__ldg(c + yp) - __ldg(c + ym)) * hy;
            const float gz = (zp - zm) * hz;
            m = fmaxf(m, sqrtf(gx * gx + gy * gy + gz * gz));
            zm = z0;
            z0 = zp;
            c += row;
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    __shared__ float sm[8];
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) m = fmaxf(m, sm[w]);
        atomicMax(reinterpret_cast<int*>(&vc->gmax), __float_as_int(m));
    }
}

// Largest upper code of a range that stays below the first opaque column f (w: none).
__device__ __forceinline__ int column_limit(int f, int w) {
    return f >= w ? 65535 : (f < 2 ? -1 : (f - 2) * 65535 / (w - 1));
}

// For every intensity column j of the transfer function: 1 if any row has a
// non-zero opacity; then an exclusive prefix count, so that a brick's column
// range can be tested in O(1), and (when `limit` is wanted) per lower column j the
// largest upper code qhi that still leaves the range empty: with f the first column >= j
// with opacity, ceil(qhi (w - 1) / 65535) + 1 < f means qhi <= (f - 2) 65535 / (w - 1)
// (none: -1; no f: every code).
// One block of 1024 threads, each reading a column of rows with its loads issued back to
// back; each thread then owns four consecutive columns of the scans (w <= 4096).
__global__ void __launch_bounds__(1024) k_tf_alpha_prefix(const float* __restrict__ tf, int w, int h,
                                                          int* __restrict__ prefix, int* __restrict__ limit) {
    __shared__ int col[4096];
    __shared__ int warp_sum[32], warp_first[32];
    for (int j = threadIdx.x; j < w; j += blockDim.x) col[j] = 0;
    __syncthreads();
    const int groups = max(1, (int)blockDim.x / w);  // row groups that work on one column
    for (int j0 = threadIdx.x; j0 < w * groups; j0 += blockDim.x) {
        const int j = j0 % w, g = j0 / w;
        bool any = false;
        for (int k = g; k < h; k += 8 * groups) {
            float a[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int kk = k + q * groups;
                a[q] = kk < h ? __ldg(tf + 4 * ((size_t)kk * w + j) + 3) : 0.0f;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) any |= a[q] != 0.0f;
        }
        if (any) col[j] = 1;  // racing writes all store 1
    }
    __syncthreads();
    const int j0 = 4 * threadIdx.x;
    int c[4], s = 0, first = w;
#pragma unroll
    for (int q = 3; q >= 0; --q) {
        c[q] = j0 + q < w ? col[j0 + q] : 0;
        s += c[q];
        if (c[q]) first = j0 + q;
    }
    // exclusive scan of the per-thread sums, and a suffix minimum of the first opaque
    // columns: within each warp, then over the warps
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = s, suf = first;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o), m = __shfl_down_sync(0xffffffffu, suf, o);
        if (lane >= o) incl += v;
        if (lane + o < 32) suf = min(suf, m);
    }
    if (lane == 31) warp_sum[wid] = incl;
    if (lane == 0) warp_first[wid] = suf;
    __syncthreads();
    if (wid == 0) {
        int t = warp_sum[lane], f = warp_first[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, t, o), m = __shfl_down_sync(0xffffffffu, f, o);
            if (lane >= o) t += v;
            if (lane + o < 32) f = min(f, m);
        }
        warp_sum[lane] = t - warp_sum[lane];  // exclusive over warps
        const int after = __shfl_down_sync(0xffffffffu, f, 1);
        warp_first[lane] = lane < 31 ? after : w;  // first opaque column of the later warps
    }
    __syncthreads();
    int run = warp_sum[wid] + incl - s;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (j0 + q < w) prefix[j0 + q] = run;
        run += c[q];
    }
    if (j0 < w && j0 + 4 >= w) prefix[w] = run;  // the thread holding the last column
    if (limit) {
        const int later = __shfl_down_sync(0xffffffffu, suf, 1);
        int nx = min(lane < 31 ? later : w, warp_first[wid]);  // first opaque column after this thread's four
#pragma unroll
        for (int q = 3; q >= 0; --q) {
            if (c[q]) nx = j0 + q;
            if (j0 + q < w) limit[j0 + q] = column_limit(nx, w);
        }
    }
}

// A brick is empty when no transfer-function column in
// [floor(qlo*(w-1)/65535) - 1, ceil(qhi*(w-1)/65535) + 1] has any opacity.
__global__ void k_classify(const uint16_t* __restrict__ grid, long long nbricks, const int* __restrict__ prefix,
                           int w, uint8_t* __restrict__ empty) {
    const long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbricks) return;
    const long long ql = grid[2 * b], qh = grid[2 * b + 1];
    long long jl = (ql * (w - 1)) / 65535 - 1;
    long long jh = (qh * (w - 1) + 65534) / 65535 + 1;
    if (jl < 0) jl = 0;
    if (jh > w - 1) jh = w - 1;
    empty[b] = (uint8_t)(prefix[jh + 1] - prefix[jl] == 0);
}

// Per interpolation cell the quantised min/max of I_norm over its 8 corner voxels, with
// the brick grid's rounding; cells of the row padding get the empty range (65535, 0).
// A warp owns 32 cells of a row and walks kRun rows along y: each voxel row is loaded
// once per z plane, x neighbours come from a shuffle and the previous row's result is
// kept, so a cell costs two 4-byte loads instead of eight (181x217x181: 50 -> 22 us).
constexpr int kCellRun = 8;
__global__ void __launch_bounds__(256) k_cell_minmax(const float* __restrict__ norm, int nx, int ny, int nz, int pitch,
                                                     uint32_t* __restrict__ cellq) {
    const int lane = threadIdx.x & 31;
    const int x = blockIdx.x * 32 + lane;
    const int y0 = (blockIdx.y * 8 + (threadIdx.x >> 5)) * kCellRun;
    const int z = blockIdx.z;
    if (y0 >= ny - 1) return;
    const int xc = min(x, nx - 1), xe = min(blockIdx.x * 32 + 32, nx - 1);
    const float* p = norm + ((long long)z * ny + y0) * nx;
    const long long plane = (long long)ny * nx;
    const int rows = min(kCellRun, ny - 1 - y0);
    float a[kCellRun + 1], b[kCellRun + 1], ea[kCellRun + 1], eb[kCellRun + 1];
#pragma unroll
    for (int r = 0; r <= kCellRun; ++r) {
        const float* q = p + (long long)min(r, rows) * nx;
        a[r] = __ldg(q + xc);
        b[r] = __ldg(q + plane + xc);
        ea[r] = lane == 31 ? __ldg(q + xe) : 0.0f;
        eb[r] = lane == 31 ? __ldg(q + plane + xe) : 0.0f;
    }
    float plo = 0.0f, phi = 0.0f;
#pragma unroll
    for (int r = 0; r <= kCellRun; ++r) {
        float lo = fminf(a[r], b[r]), hi = fmaxf(a[r], b[r]);
        float nlo = __shfl_down_sync(0xffffffffu, lo, 1), nhi = __shfl_down_sync(0xffffffffu, hi, 1);
        if (lane == 31) {
            nlo = fminf(ea[r], eb[r]);
            nhi = fmaxf(ea[r], eb[r]);
        }
        lo = fminf(lo, nlo);
        hi = fmaxf(hi, nhi);
        if (r > 0 && r <= rows) {
            const float l = fminf(lo, plo), h = fmaxf(hi, phi);
            unsigned ql = (unsigned)fminf(fmaxf(floorf(__fmul_rn(l, 65535.0f)), 0.0f), 65535.0f);
            unsigned qh = (unsigned)fminf(fmaxf(ceilf(__fmul_rn(h, 65535.0f)), 0.0f), 65535.0f);
            if (x >= nx - 1) ql = 65535u, qh = 0u;
            cellq[((long long)z * (ny - 1) + (y0 + r - 1)) * pitch + x] = ql | (qh << 16);
        }
        plo = lo;
        phi = hi;
    }
}

// Cell bits of the skip field. A cell is empty under the brick rule applied to its own
// range: no transfer-function column in [floor(qlo*(w-1)/65535) - 1,
// ceil(qhi*(w-1)/65535) + 1] has any opacity (every sample in the cell interpolates its
// 8 corners, so its intensity lies in the range). A CTA classifies 32 x 4 x 16 cells
// (each of its warps eight rows, loads issued back to back), one ballot per row, and
// then the 8 x 1 x 4 blocks of 4^3 cells they make. Cells past the volume are empty.
// The rule is one division and one comparison with the lower column's limit from shared
// memory (qlo (w - 1) < 2^29: 32-bit arithmetic); two lookups of a prefix table in global
// memory bound this kernel by L1 wavefronts (181x217x181: 20.6 -> 15.9 us, the 30 MB of codes read from HBM).
// The same launch classifies the skip bricks (grid layers past the cells').
// A 1D table's limits are computed by every CTA for itself (one scan of w columns), which
// saves the launch that reduces a 2D table's rows first.
__device__ __forceinline__ int lower_column(unsigned ql, int w) {
    return max((int)(ql * (unsigned)(w - 1) / 65535u) - 1, 0);
}

// lim[j], j < w: from `limit`, or from the columns of the 1D table `tf1` (w <= 1024).
__device__ __forceinline__ void load_limits(const int* __restrict__ limit, const float* __restrict__ tf1, int w,
                                            int* lim) {
    if (!tf1) {
        for (int j = threadIdx.x; j < w; j += 256) lim[j] = __ldg(limit + j);
        __syncthreads();
        return;
    }
    __shared__ int first[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, j0 = 4 * threadIdx.x;
    bool c[4];
    int f = w;
#pragma unroll
    for (int q = 3; q >= 0; --q) {
        c[q] = j0 + q < w && __ldg(tf1 + 4 * (j0 + q) + 3) != 0.0f;
        if (c[q]) f = j0 + q;
    }
    int suf = f;  // suffix minimum of the first opaque columns
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int m = __shfl_down_sync(0xffffffffu, suf, o);
        if (lane + o < 32) suf = min(suf, m);
    }
    if (lane == 0) first[wid] = suf;
    __syncthreads();
    int nx = __shfl_down_sync(0xffffffffu, suf, 1);
    if (lane == 31) nx = w;
    for (int q = wid + 1; q < 8; ++q) nx = min(nx, first[q]);
#pragma unroll
    for (int q = 3; q >= 0; --q) {
        if (c[q]) nx = j0 + q;
        if (j0 + q < w) lim[j0 + q] = column_limit(nx, w);
    }
    __syncthreads();
}

__global__ void __launch_bounds__(256) k_cell_bits(const uint32_t* __restrict__ cellq, SkipDims d, int pitch,
                                                   const int* __restrict__ limit, const float* __restrict__ tf1, int w,
                                                   uint32_t* __restrict__ cell_bits, uint8_t* __restrict__ block_bits,
                                                   int cell_layers, const uint16_t* __restrict__ grid,
                                                   long long nbricks, uint8_t* __restrict__ empty) {
    __shared__ uint32_t rows[64];  // [z 0..15][y 0..3]
    __shared__ int lim[4096];
    if ((int)blockIdx.z >= cell_layers) {
        load_limits(limit, tf1, w, lim);
        const long long stride = (long long)(gridDim.z - cell_layers) * gridDim.y * gridDim.x * 256;
        for (long long b = (((long long)(blockIdx.z - cell_layers) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) *
                               256 + threadIdx.x;
             b < nbricks; b += stride) {
            const unsigned q = __ldg(reinterpret_cast<const unsigned*>(grid) + b);
            empty[b] = (uint8_t)((int)(q >> 16) <= lim[lower_column(q & 0xffffu, w)]);
        }
        return;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int x = blockIdx.x * 32 + lane, y0 = blockIdx.y * 4, z0 = blockIdx.z * 16 + wid * 2;
    const long long r0 = (long long)z0 * d.cy + y0;  // the warp's rows: (z0, z0 + 1) x (y0 .. y0 + 3)
    const int ny = min(4, d.cy - y0), nz = d.cz - z0;
    unsigned q[8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
        q[r] = (r & 3) < ny && (r >> 2) < nz ? __ldg(cellq + (r0 + (r >> 2) * d.cy + (r & 3)) * pitch + x) : 65535u;
    load_limits(limit, tf1, w, lim);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int jl = lower_column(q[r] & 0xffffu, w);
        // cells past the volume hold the code pair (65535, 0), the only one with qlo > qhi
        const unsigned bits = __ballot_sync(0xffffffffu, (int)(q[r] >> 16) <= lim[jl] || q[r] == 65535u);
        if (lane == 0) {
            rows[wid * 8 + r] = bits;
            if ((r & 3) < ny && (r >> 2) < nz) cell_bits[(r0 + (r >> 2) * d.cy + (r & 3)) * d.wx + blockIdx.x] = bits;
        }
    }
    __syncthreads();
    if (threadIdx.x < 4) {  // one z block each: the AND over its 16 rows, four cells per bit
        unsigned a = 0xffffffffu;
#pragma unroll
        for (int r = 0; r < 16; ++r) a &= rows[threadIdx.x * 16 + r];
        a &= a >> 1;
        a &= a >> 2;
        unsigned b = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) b |= ((a >> (4 * i)) & 1u) << i;
        const int bz = blockIdx.z * 4 + threadIdx.x;
        if (bz < d.bz) {
            uint8_t* o = block_bits + ((long long)bz * d.by + blockIdx.y) * d.bwx * 4;
            o[blockIdx.x] = (uint8_t)b;
            if ((int)blockIdx.x == d.wx - 1)
                for (int q = d.wx; q < 4 * d.bwx; ++q) o[q] = 0xff;  // the row's padding is empty
        }
    }
}

// Chebyshev distance of every empty cell (or 4^3 block) to the nearest non-empty one,
// capped at kE + 1, on bit grids: kE erosions by the 3x3x3 cube, counted per bit.
//   E_0 = the empty bits, E_{l+1} = erode(E_l), distance = number of l with the bit set
// (0: not empty). A CTA owns 32 x T x T bits, T = 32 - 2 kE, with a halo of kE rows in y
// and z and 16 bits in x: lane = row along y, a warp holds four rows along z, so the
// erosion is bit shifts in x, shuffles in y and registers (two rows through shared
// memory per warp) in z. Everything outside the grid counts as empty: no sample lies
// there. Distances are right up to the cap because each erosion consumes one row of the
// halo. Counts are kept as four bit planes.
// Cells take kE = 4 (T = 24), blocks kE = 8: the farther layers are the blocks' part
// (8 erosions of the cells, T = 16: 20.9 us for 181x217x181 against 11.9, the frames equal;
// 4 erosions of the blocks: the 256x256x176 vessel frame 6 % slower).
struct EdgeRows {
    uint64_t edge[8][2][32];
};
// Per-bit counts of the warp's four rows, as bit planes.
struct CountPlanes {
    uint32_t c0[4], c1[4], c2[4], c3[4];
};

__device__ __forceinline__ uint64_t shfl_up64(uint64_t v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ uint64_t shfl_dn64(uint64_t v) { return __shfl_down_sync(0xffffffffu, v, 1); }

template <int kE>
__device__ __forceinline__ void erode_tile(const uint32_t* __restrict__ bits, int wx, int ny, int nz, int xw, int y0,
                                           int z0, EdgeRows& sm, CountPlanes& c) {
    static_assert(kE % 4 == 0 && kE <= 8, "whole warps of the tile, counts of four bits");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int y = y0 - kE + lane;
    uint64_t e[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int z = z0 - kE + wid * 4 + r;
        uint64_t v = ~0ull;
        if (y >= 0 && y < ny && z >= 0 && z < nz) {
            const uint32_t* row = bits + ((long long)z * ny + y) * wx;
            const uint32_t l = xw > 0 ? __ldg(row + xw - 1) : 0xffffffffu, m = __ldg(row + xw),
                           h = xw + 1 < wx ? __ldg(row + xw + 1) : 0xffffffffu;
            v = (uint64_t)(l >> 16) | ((uint64_t)m << 16) | ((uint64_t)h << 48);
        }
        e[r] = v;
        c.c0[r] = (uint32_t)(v >> 16);
        c.c1[r] = c.c2[r] = c.c3[r] = 0u;
    }
#pragma unroll 1
    for (int l = 0; l < kE; ++l) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            uint64_t a = e[r] & ((e[r] << 1) | 1ull) & ((e[r] >> 1) | (1ull << 63));
            const uint64_t up = shfl_up64(a), dn = shfl_dn64(a);
            if (lane > 0) a &= up;
            if (lane < 31) a &= dn;
            e[r] = a;
        }
        sm.edge[wid][0][lane] = e[0];
        sm.edge[wid][1][lane] = e[3];
        __syncthreads();
        const uint64_t below = wid > 0 ? sm.edge[wid - 1][1][lane] : ~0ull,
                       above = wid < 7 ? sm.edge[wid + 1][0][lane] : ~0ull;
        const uint64_t e0 = e[0], e1 = e[1], e2 = e[2], e3 = e[3];
        e[0] = below & e0 & e1;
        e[1] = e0 & e1 & e2;
        e[2] = e1 & e2 & e3;
        e[3] = e2 & e3 & above;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 4; ++r) {  // count += bit, a ripple over the planes
            uint32_t carry = (uint32_t)(e[r] >> 16), n;
            n = c.c0[r] & carry, c.c0[r] ^= carry, carry = n;
            n = c.c1[r] & carry, c.c1[r] ^= carry, carry = n;
            n = c.c2[r] & carry, c.c2[r] ^= carry;
            c.c3[r] |= n;
        }
    }
}

// The rows of the tile itself, without the halo.
template <int kE>
__device__ __forceinline__ bool tile_row() {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    return wid >= kE / 4 && wid < 8 - kE / 4 && lane >= kE && lane < 32 - kE;
}

constexpr int kCellErosions = 4, kBlockErosions = 8;

// Block distances, left as four bit planes per 32 blocks: [bz][by][bwx] uint4.
__global__ void __launch_bounds__(256) k_block_dist(const uint32_t* __restrict__ bits, SkipDims d,
                                                    uint4* __restrict__ dist) {
    constexpr int kE = kBlockErosions, T = 32 - 2 * kE;
    __shared__ EdgeRows sm;
    CountPlanes c;
    erode_tile<kE>(bits, d.bwx, d.by, d.bz, blockIdx.x, blockIdx.y * T, blockIdx.z * T, sm, c);
    const int y = blockIdx.y * T - kE + (threadIdx.x & 31);
    if (!tile_row<kE>() || y >= d.by) return;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int z = blockIdx.z * T - kE + (threadIdx.x >> 5) * 4 + r;
        if (z < d.bz)
            dist[((long long)z * d.by + y) * d.bwx + blockIdx.x] = make_uint4(c.c0[r], c.c1[r], c.c2[r], c.c3[r]);
    }
}

__device__ __forceinline__ unsigned plane_count(const uint4& p, int x) {
    return ((p.x >> x) & 1u) | (((p.y >> x) & 1u) << 1) | (((p.z >> x) & 1u) << 2) | (((p.w >> x) & 1u) << 3);
}

// The field: distance in cells to the nearest non-empty cell, the larger of the cell's
// own (up to 5) and what its block's promises: with the block at distance c, the
// 4 (c - 1) layers of cells around the block are empty, so the cell is at 4 c - 3 at
// least (up to 33).
// kFused: the CTA erodes the blocks around its tile itself instead of reading
// k_block_dist's result: three times the erosions, so only where the launch is too small
// to fill the chip and the saved launch is worth more (64^3: 5 + 6.2 -> 9.4 us).
template <bool kFused>
__global__ void __launch_bounds__(256) k_skip_field(const uint32_t* __restrict__ bits, SkipDims d,
                                                    const uint32_t* __restrict__ block_bits,
                                                    const uint4* __restrict__ block_dist,
                                                    uint8_t* __restrict__ field) {
    constexpr int kE = kCellErosions, T = 32 - 2 * kE, TB = T / 4;
    __shared__ EdgeRows sm;
    __shared__ uint4 plane[T][T];       // [z][y] of the tile
    __shared__ uint4 bplane[TB][TB];    // kFused: of its blocks
    const int xl = threadIdx.x & 31, x = blockIdx.x * 32 + xl;
    CountPlanes p;
    if (kFused) {
        constexpr int kB = kBlockErosions;
        erode_tile<kB>(block_bits, d.bwx, d.by, d.bz, blockIdx.x >> 2, blockIdx.y * TB, blockIdx.z * TB, sm, p);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int z = (threadIdx.x >> 5) * 4 + r - kB, y = xl - kB;
            if (z >= 0 && z < TB && y >= 0 && y < TB) bplane[z][y] = make_uint4(p.c0[r], p.c1[r], p.c2[r], p.c3[r]);
        }
        __syncthreads();  // the edge rows are used again
    }
    erode_tile<kE>(bits, d.wx, d.cy, d.cz, blockIdx.x, blockIdx.y * T, blockIdx.z * T, sm, p);
    if (tile_row<kE>()) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
            plane[(threadIdx.x >> 5) * 4 + r - kE][xl - kE] = make_uint4(p.c0[r], p.c1[r], p.c2[r], p.c3[r]);
    }
    __syncthreads();
    if (x >= d.cx) return;
    // T/4 x T/4 columns of 16 bytes (4 y x 4 z) per x, a warp per column row
    for (int c = threadIdx.x >> 5; c < TB * TB; c += 8) {
        const int yb = c % TB, zb = c / TB, by = blockIdx.y * TB + yb, bz = blockIdx.z * TB + zb;
        if (by >= d.by || bz >= d.bz) continue;
        const uint4 far4 = kFused ? bplane[zb][yb] : __ldg(block_dist + ((long long)bz * d.by + by) * d.bwx + (x >> 7));
        const int far = 4 * (int)plane_count(far4, (x >> 2) & 31) - 3;
        uint32_t o[4];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            o[y] = 0u;
#pragma unroll
            for (int z = 0; z < 4; ++z) {
                const int n = (int)plane_count(plane[zb * 4 + z][yb * 4 + y], xl);
                if (n) o[y] |= (uint32_t)max(n, far) << (8 * z);
            }
        }
        reinterpret_cast<uint4*>(field)[((long long)bz * d.by + by) * d.cx + x] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

}  // namespace

cudaError_t launch_cell_minmax(const float* norm, const int n[3], uint32_t* cellq, cudaStream_t st) {
    const int pitch = cellq_pitch(n[0]);
    dim3 grid(pitch / 32, (n[1] - 1 + 8 * kCellRun - 1) / (8 * kCellRun), n[2] - 1);
    k_cell_minmax<<<grid, 256, 0, st>>>(norm, n[0], n[1], n[2], pitch, cellq);
    return cudaGetLastError();
}

cudaError_t launch_skip_field(const uint32_t* cellq, const int n[3], const uint16_t* grid, long long nbricks,
                              const float* tf, int tf_w, int tf_h, int* prefix_scratch, uint8_t* empty,
                              const SkipStore& s, cudaStream_t st) {
    const SkipDims d = skip_dims(n);
    constexpr int TC = 32 - 2 * kCellErosions, TB = 32 - 2 * kBlockErosions;
    const float* tf1 = tf_h == 1 && tf_w <= 1024 ? tf : nullptr;
    if (!tf1) k_tf_alpha_prefix<<<1, 1024, 0, st>>>(tf, tf_w, tf_h, prefix_scratch, s.limits);
    const int layers = (d.cz + 15) / 16;
    const long long per_layer = (long long)d.wx * d.by * 256;
    const long long more = (nbricks + per_layer - 1) / per_layer;
    k_cell_bits<<<dim3(d.wx, d.by, layers + (unsigned)(more < 4 ? more : 4)), 256, 0, st>>>(
        cellq, d, cellq_pitch(n[0]), s.limits, tf1, tf_w, s.cell_bits, reinterpret_cast<uint8_t*>(s.block_bits),
        layers, grid, nbricks, empty);
    const dim3 tiles(d.wx, (d.cy + TC - 1) / TC, (d.cz + TC - 1) / TC);
    if ((long long)tiles.x * tiles.y * tiles.z <= kSMs) {
        k_skip_field<true><<<tiles, 256, 0, st>>>(s.cell_bits, d, s.block_bits, nullptr, s.field);
    } else {
        k_block_dist<<<dim3(d.bwx, (d.by + TB - 1) / TB, (d.bz + TB - 1) / TB), 256, 0, st>>>(s.block_bits, d,
                                                                                            s.block_dist);
        k_skip_field<false><<<tiles, 256, 0, st>>>(s.cell_bits, d, nullptr, s.block_dist, s.field);
    }
    return cudaGetLastError();
}

int minmax_blocks(long long n) {
    long long want = (n + (long long)kReduceThreads * 16 - 1) / ((long long)kReduceThreads * 16);
    if (want < 1) want = 1;
    if (want > kSMs * 8) want = kSMs * 8;
    return (int)want;
}

cudaError_t launch_minmax_partials(const void* data, vr_dtype dt, long long n, float* partials, int nblocks,
                                   cudaStream_t st) {
    if (dt == VR_F32)
        k_minmax_partials_f32<<<nblocks, kReduceThreads, 0, st>>>((const float*)data, n, partials);
    else
        k_minmax_partials_u16<<<nblocks, kReduceThreads, 0, st>>>((const uint16_t*)data, n, partials);
    return cudaGetLastError();
}

cudaError_t launch_minmax_final(const float* partials, int nblocks, float* out2, cudaStream_t st) {
    k_minmax_final<<<1, 1024, 0, st>>>(partials, nblocks, out2);
    return cudaGetLastError();
}

cudaError_t launch_normalize(const void* raw, vr_dtype dt, long long n, const float* minmax2, VolConst* vc,
                             float* norm, cudaStream_t st) {
    const int blocks = kSMs * 8;
    if (dt == VR_F32)
        k_normalize<float><<<blocks, 256, 0, st>>>((const float*)raw, n, minmax2, vc, norm);
    else
        k_normalize<uint16_t><<<blocks, 256, 0, st>>>((const uint16_t*)raw, n, minmax2, vc, norm);
    return cudaGetLastError();
}

cudaError_t launch_make_bricks(const float* norm, const int n[3], const int nb[3], float* bricks, cudaStream_t st) {
    // nb: storage bricks, at most 256^3 = 2^24, so pieces / 256 fits the grid
    const long long pieces = (long long)nb[0] * nb[1] * nb[2] * kBrickPieces;
    k_make_bricks<<<(unsigned)((pieces + 255) / 256), 256, 0, st>>>(norm, n[0], n[1], n[2], nb[0], nb[1], pieces,
                                                                    reinterpret_cast<float4*>(bricks));
    return cudaGetLastError();
}

cudaError_t launch_brick_minmax(const float* norm, const int n[3], const int nb[3], int bs, uint16_t* grid,
                                cudaStream_t st) {
    const dim3 ctas((nb[0] + (32 >> bs) - 1) / (32 >> bs), nb[1], nb[2]);
    switch (bs) {
        case 2: k_brick_minmax<2><<<ctas, 256, 0, st>>>(norm, n[0], n[1], n[2], nb[0], grid); break;
        case 4: k_brick_minmax<4><<<ctas, 256, 0, st>>>(norm, n[0], n[1], n[2], nb[0], grid); break;
        default: k_brick_minmax<3><<<ctas, 256, 0, st>>>(norm, n[0], n[1], n[2], nb[0], grid); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_make_derived(const float* norm, const int n[3], const int nb[3], int bs, const float s[3],
                                float* dbricks, cudaStream_t st) {
    const long long nbr = (long long)nb[0] * nb[1] * nb[2];
    const float hx = 1.0f / s[0], hy = 1.0f / s[1], hz = 1.0f / s[2];
    const unsigned ctas = (unsigned)nbr;  // <= 512^3
    switch (bs) {
        case 2: k_make_derived<2><<<ctas, 256, 0, st>>>(norm, n[0], n[1], n[2], nb[0], nb[1], hx, hy, hz, dbricks); break;
        case 4: k_make_derived<4><<<ctas, 256, 0, st>>>(norm, n[0], n[1], n[2], nb[0], nb[1], hx, hy, hz, dbricks); break;
        default: k_make_derived<3><<<ctas, 256, 0, st>>>(norm, n[0], n[1], n[2], nb[0], nb[1], hx, hy, hz, dbricks); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_gmax(const float* norm, const int n[3], const float s[3], VolConst* vc, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(&vc->gmax, 0, sizeof(float), st);
    if (e != cudaSuccess) return e;
    dim3 grid((n[0] + 31) / 32, (n[1] + 7) / 8, (n[2] + kGmaxPlanes - 1) / kGmaxPlanes);
    k_gmax<<<grid, 256, 0, st>>>(norm, n[0], n[1], n[2], 0.5f / s[0], 0.5f / s[1], 0.5f / s[2], vc);
    return cudaGetLastError();
}

cudaError_t launch_classify(const uint16_t* grid, long long nbricks, const float* tf, int tf_w, int tf_h,
                            uint8_t* empty, int* prefix_scratch, cudaStream_t st) {
    k_tf_alpha_prefix<<<1, 1024, 0, st>>>(tf, tf_w, tf_h, prefix_scratch, nullptr);
    k_classify<<<(unsigned)((nbricks + 255) / 256), 256, 0, st>>>(grid, nbricks, prefix_scratch, tf_w, empty);
    return cudaGetLastError();
}

}  // namespace vr

// ---------------------------------------------------------------------------
// Allocation-free brick classification.
//
// Some callers cannot allocate device memory at the point where they need to
// re-classify bricks: a host that hands the GPU to this library with a fixed,
// pre-reserved memory budget, a real-time interaction thread that must not
// enter the allocator, or code running while another component holds the
// device's allocator. For them this entry point runs the same two kernels as
// vr_set_tissue_params' classification, but keeps their scratch (the
// transfer-function column prefix table) in a static device array compiled into
// the library instead of asking for memory.
#include <mutex>

namespace vr {
namespace {

constexpr int kStaticTfMaxW = 4096;  // largest table width the static scratch holds
constexpr int kStaticMaxDevices = 64;

// tf_w + 1 prefix counts; every call rewrites all the entries it reads, so
// nothing here has to start at zero. Each GPU that loads the library holds
// these 16 KB until the process exits.
static __device__ __align__(256) int g_static_prefix[kStaticTfMaxW + 1];

std::mutex g_static_mu;
// Per device: the device address of the static array and the id of the CUDA context
// it was taken in. A device reset (cudaDeviceReset) destroys the context and the
// module with it; the next call sees a new context id and looks the address up again.
int* g_static_prefix_ptr[kStaticMaxDevices] = {};
unsigned long long g_static_ctx_id[kStaticMaxDevices] = {};
// Driver entry points for the current context and its process-unique id, resolved
// through the runtime so that the library does not link the driver library itself.
typedef int (*CtxGetCurrentFn)(void**);
typedef int (*CtxGetIdFn)(void*, unsigned long long*);
CtxGetCurrentFn g_ctx_get_current = nullptr;
CtxGetIdFn g_ctx_get_id = nullptr;
std::once_flag g_ctx_fns_once;

// Id of the calling thread's current CUDA context, 0 when it cannot be told.
unsigned long long current_ctx_id() {
    std::call_once(g_ctx_fns_once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_ctx_get_current = reinterpret_cast<CtxGetCurrentFn>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_ctx_get_id = reinterpret_cast<CtxGetIdFn>(f);
        (void)cudaGetLastError();
    });
    if (!g_ctx_get_current || !g_ctx_get_id) return 0;
    void* cu = nullptr;
    unsigned long long id = 0;
    if (g_ctx_get_current(&cu) != 0 || !cu || g_ctx_get_id(cu, &id) != 0) return 0;
    return id;
}

void put_msg(char* buf, int len, const char* msg) {
    if (!buf || len <= 0) return;
    int i = 0;
    for (; i < len - 1 && msg[i]; ++i) buf[i] = msg[i];
    buf[i] = '\0';
}

}  // namespace

unsigned long long current_cuda_context() { return current_ctx_id(); }

}  // namespace vr

extern "C" vr_status vr_classify_bricks_noalloc(const unsigned short* d_grid, long long nbricks, const float* d_tf,
                                                int tf_w, int tf_h, unsigned char* d_empty, void* cuda_stream,
                                                char* h_msg, int msg_len) {
    using namespace vr;
    put_msg(h_msg, msg_len, "");
    if (!d_grid || !d_tf || !d_empty || nbricks < 1 || nbricks > (1LL << 31)) {
        put_msg(h_msg, msg_len, "classify_bricks_noalloc: NULL pointer or brick count outside [1, 2^31]");
        return VR_ERR_INVALID_ARG;
    }
    if (tf_w < 2 || tf_w > kStaticTfMaxW) {
        put_msg(h_msg, msg_len,
                "classify_bricks_noalloc: tf_w must be in [2, 4096]; the static scratch holds 4097 prefix counts");
        return VR_ERR_INVALID_ARG;
    }
    if (tf_h < 1 || tf_h > 256) {
        put_msg(h_msg, msg_len, "classify_bricks_noalloc: tf_h must be in [1, 256]");
        return VR_ERR_INVALID_ARG;
    }
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kStaticMaxDevices) {
        (void)cudaGetLastError();
        put_msg(h_msg, msg_len, "classify_bricks_noalloc: no usable current CUDA device");
        return VR_ERR_CUDA;
    }
    int* prefix = nullptr;
    {
        // once per device and CUDA context, with that device current: the device
        // address of the static array (the host-side symbol is not a device pointer).
        // A context id of 0 (no current context yet, or the driver cannot say) looks
        // the address up on every call.
        std::lock_guard<std::mutex> lock(g_static_mu);
        unsigned long long id = current_ctx_id();
        if (!g_static_prefix_ptr[dev] || id == 0 || id != g_static_ctx_id[dev]) {
            int* p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress((void**)&p, g_static_prefix);
            if (e != cudaSuccess || !p) {
                (void)cudaGetLastError();
                put_msg(h_msg, msg_len, "classify_bricks_noalloc: cudaGetSymbolAddress of the static scratch failed");
                return VR_ERR_CUDA;
            }
            if (id == 0) id = current_ctx_id();  // the lookup made the primary context current
            g_static_prefix_ptr[dev] = p;
            g_static_ctx_id[dev] = id;
        }
        prefix = g_static_prefix_ptr[dev];
    }
    const cudaError_t e = launch_classify(reinterpret_cast<const uint16_t*>(d_grid), nbricks, d_tf, tf_w, tf_h,
                                          reinterpret_cast<uint8_t*>(d_empty), prefix, (cudaStream_t)cuda_stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        put_msg(h_msg, msg_len, cudaGetErrorString(e));
        return VR_ERR_CUDA;
    }
    return VR_OK;
}
