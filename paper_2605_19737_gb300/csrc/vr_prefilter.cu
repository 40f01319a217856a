// vr_prefilter.cu -- optional pre-filters of the normalised volume (the
// lightweight smoothing or median compute passes proposed in Sec. 5.3 against
// low-SNR and impulsive artefacts), applied before bricking and morphology.
//
// k_median3: exact 14th smallest of the 27 clamp-to-edge neighbours by a pruned
// selection network, sharing the sorted triples of a column among the voxels around it.
#include "vr_internal.cuh"

namespace vr {

namespace {

// Floats as signed integers in the same order (-0 below +0); every NaN above all numbers.
__device__ __forceinline__ int order_key(float x) {
    const int b = __float_as_int(x);
    return x != x ? 0x7fffffff : b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float key_value(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }

__device__ __forceinline__ void cswap(int& a, int& b) {
    const int lo = min(a, b);
    b = max(a, b);
    a = lo;
}
__device__ __forceinline__ void sort3(int& a, int& b, int& c) {
    cswap(a, b);
    cswap(b, c);
    cswap(a, b);
}

// Sorts v[0..8], whose triples 0-2, 3-5, 6-8 are sorted already: the last 16 comparators
// of Floyd's 25-comparator network (Knuth, TAOCP 3, 5.3.4). Outputs the caller does not
// use drop out of the code.
__device__ __forceinline__ void merge9(int v[9]) {
    cswap(v[0], v[3]);
    cswap(v[3], v[6]);
    cswap(v[0], v[3]);
    cswap(v[1], v[4]);
    cswap(v[4], v[7]);
    cswap(v[1], v[4]);
    cswap(v[2], v[5]);
    cswap(v[5], v[8]);
    cswap(v[2], v[5]);
    cswap(v[1], v[3]);
    cswap(v[5], v[7]);
    cswap(v[2], v[6]);
    cswap(v[4], v[6]);
    cswap(v[2], v[4]);
    cswap(v[2], v[3]);
    cswap(v[5], v[6]);
}

// The 14th smallest of 27 given as three sorted rows: L, M, H of 9, the sorted lows, mids
// and highs of nine sorted columns, so that L[c] <= M[c] <= H[c]. An element (r, c) of
// that doubly sorted 3 x 9 array has (r + 1)(c + 1) - 1 elements certainly below and
// (3 - r)(9 - c) - 1 above; only L[5..8], M[2..6] and H[0..3] can have 13 of each, seven
// of the others lie below and seven above: the answer is the 7th smallest of those 13.
__device__ __forceinline__ int median_of_rows(const int L[9], const int M[9], const int H[9]) {
    int y[8] = {L[5], L[6], L[7], L[8], H[0], H[1], H[2], H[3]};
    cswap(y[0], y[4]);  // Batcher's odd-even merge of the two sorted fours
    cswap(y[1], y[5]);
    cswap(y[2], y[6]);
    cswap(y[3], y[7]);
    cswap(y[2], y[4]);
    cswap(y[3], y[5]);
    cswap(y[1], y[2]);
    cswap(y[3], y[4]);
    cswap(y[5], y[6]);
    // 7th smallest of sorted M[2..6] and y[0..7]: min over i of max(i-th of M, (7 - i)-th of y)
    int m = y[6];
    m = min(m, max(M[2], y[5]));
    m = min(m, max(M[3], y[4]));
    m = min(m, max(M[4], y[3]));
    m = min(m, max(M[5], y[2]));
    return min(m, max(M[6], y[1]));
}

// A warp owns 30 voxels of kMedRows rows (lanes 0 and 31 hold the x neighbours) and
// walks along z: per plane each lane loads its kMedRows + 2 rows, sorts every column's
// triple along z once, every output row sorts the triples of three columns along y, and
// the x neighbours' nine values come by shuffle. ~150 minimum / maximum operations per
// voxel, bound by the ALU pipe (half-rate min/max); counting each of the 27 ranks by 26
// comparisons took 478 us for 181x217x181, this 76 us.
// With 14 or more NaNs among the 27 there is no 14th smallest number: the result is then
// the (-1, -1, -1) neighbour.
constexpr int kMedRows = 4;
__global__ void __launch_bounds__(128) k_median3(const float* __restrict__ in, float* __restrict__ out, int nx, int ny,
                                                 int nz, int planes) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int x = blockIdx.x * 30 - 1 + lane;
    const int y0 = (blockIdx.y * 4 + wid) * kMedRows;
    const int z0 = blockIdx.z * planes, z1 = min(z0 + planes, nz);
    if (y0 >= ny) return;
    const long long plane = (long long)nx * ny;
    int off[kMedRows + 2];  // clamped rows, from the start of a plane
#pragma unroll
    for (int r = 0; r < kMedRows + 2; ++r)
        off[r] = min(max(y0 - 1 + r, 0), ny - 1) * nx + min(max(x, 0), nx - 1);
    int p[kMedRows + 2], c[kMedRows + 2];  // the planes below and at z
    {
        const float* a = in + max(z0 - 1, 0) * plane;
        const float* b = in + z0 * plane;
#pragma unroll
        for (int r = 0; r < kMedRows + 2; ++r) {
            p[r] = order_key(__ldg(a + off[r]));
            c[r] = order_key(__ldg(b + off[r]));
        }
    }
    for (int z = z0; z < z1; ++z) {
        const float* a = in + min(z + 1, nz - 1) * plane;
        int l[kMedRows + 2], m[kMedRows + 2], h[kMedRows + 2];
#pragma unroll
        for (int r = 0; r < kMedRows + 2; ++r) h[r] = order_key(__ldg(a + off[r]));
#pragma unroll
        for (int r = 0; r < kMedRows + 2; ++r) {
            l[r] = p[r];
            m[r] = c[r];
            p[r] = c[r];
            c[r] = h[r];
            sort3(l[r], m[r], h[r]);
        }
#pragma unroll
        for (int r = 0; r < kMedRows; ++r) {
            int L[9], M[9], H[9];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                L[3 + q] = l[r + q];
                M[3 + q] = m[r + q];
                H[3 + q] = h[r + q];
            }
            sort3(L[3], L[4], L[5]);
            sort3(M[3], M[4], M[5]);
            sort3(H[3], H[4], H[5]);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                L[q] = __shfl_up_sync(0xffffffffu, L[3 + q], 1);
                M[q] = __shfl_up_sync(0xffffffffu, M[3 + q], 1);
                H[q] = __shfl_up_sync(0xffffffffu, H[3 + q], 1);
                L[6 + q] = __shfl_down_sync(0xffffffffu, L[3 + q], 1);
                M[6 + q] = __shfl_down_sync(0xffffffffu, M[3 + q], 1);
                H[6 + q] = __shfl_down_sync(0xffffffffu, H[3 + q], 1);
            }
            merge9(L);
            merge9(M);
            merge9(H);
            const int k = median_of_rows(L, M, H);
            const int y = y0 + r;
            if (lane >= 1 && lane <= 30 && x < nx && y < ny)
                out[z * plane + (long long)y * nx + x] =
                    k != 0x7fffffff
                        ? key_value(k)
                        : __ldg(in + max(z - 1, 0) * plane + (long long)max(y - 1, 0) * nx + max(x - 1, 0));
        }
    }
}

}  // namespace

cudaError_t launch_median3(const float* in, float* out, const int n[3], cudaStream_t st) {
    const unsigned tx = (n[0] + 29) / 30, ty = (n[1] + 4 * kMedRows - 1) / (4 * kMedRows);
    const int planes = march_planes((long long)tx * ty, n[2], 8, 16);
    k_median3<<<dim3(tx, ty, (n[2] + planes - 1) / planes), 128, 0, st>>>(in, out, n[0], n[1], n[2], planes);
    return cudaGetLastError();
}

}  // namespace vr
