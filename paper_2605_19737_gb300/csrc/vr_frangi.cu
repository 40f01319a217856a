// vr_frangi.cu -- per-volume multi-scale Hessian vesselness (the multi-scale
// Hessian analysis with vesselness measures that Sec. 1 mentions, read as the
// bright-vessel response of Frangi et al., MICCAI 1998), computed once per
// volume like the paper's morphology compute shader (Sec. 2.3).
//
// For each scale sigma (voxels):
//   1. separable Gaussian smoothing, sampled normalised weights exp(-x^2/2s^2)
//      on [-R, R], R = ceil(4 sigma), clamp-to-edge, x then y then z;
//   2. Hessian of the smoothed volume by the central second / mixed differences
//      of Sec. 2.3 in voxel units, times sigma^2 (scale normalisation);
//   3. pass A: S = ||lambda|| = ||H||_F (Frobenius norm) reduced to max_v S;
//   4. pass B: the Hessian again, its eigenvalues by cyclic Jacobi rotations in
//      FP32 sorted |l1|<=|l2|<=|l3|, c = max S / 2 and
//      V_sigma = 0 if l2 > 0 or l3 > 0, else
//      (1 - exp(-Ra^2/2a^2)) exp(-Rb^2/2b^2) (1 - exp(-S^2/2c^2)),
//      Ra = |l2|/|l3|, Rb = |l1|/sqrt|l2 l3|, a = b = 1/2;
//   V = max over scales.
// The smoothing passes stream the volume through shared-memory tiles; the
// Hessian/eigen passes are ALU.
#include <math.h>

#include "vr_internal.cuh"

namespace vr {

namespace {

constexpr int kMaxRadius = 32;

struct GaussParams {
    float w[2 * kMaxRadius + 1];
    int R;
};

// The 1D Gaussian passes (clamp-to-edge). Each block stages its input span, halo
// included, in shared memory once, so that every voxel is read from L2/HBM about
// once per pass instead of once per tap; every output sums its 2R+1 taps in the
// order t = -R .. R with one fmaf each.
constexpr int kGaussRow = 256;  // x pass: outputs per block (one row segment)
constexpr int kGaussCol = 64;   // y / z passes: outputs per column, 32 columns per block

// kN consecutive outputs of a thread from a staged span, at(i) its i-th value: every
// staged value is read from shared memory once and used by all the outputs it reaches,
// each of which adds its taps in the order t = -R .. R with one fmaf each (one LDS per
// output and tap bound these passes before: x / y / z pass of 256x256x176 at R = 12 56 /
// 47 / 47 -> 21 / 26 / 26 us). kR > 0 is the radius known at compile time (the loop unrolls, weights
// become constant operands); kR = 0 reads it from G.R and keeps the kN values in a ring
// of registers, so that a tap is one LDS, one constant load and kN fmaf.
template <int kR, int kN, class At>
__device__ __forceinline__ void gauss_taps(const At& at, const GaussParams& G, float acc[kN]) {
#pragma unroll
    for (int n = 0; n < kN; ++n) acc[n] = 0.0f;
    if (kR > 0) {
#pragma unroll
        for (int i = 0; i < kN + 2 * kR; ++i) {
            const float v = at(i);
#pragma unroll
            for (int n = 0; n < kN; ++n)
                if (i - n >= 0 && i - n <= 2 * kR) acc[n] = fmaf(G.w[i - n], v, acc[n]);
        }
    } else {
        const int last = 2 * G.R;
        float v[kN];  // v[i % kN] = value i, i in [t, t + kN)
#pragma unroll
        for (int i = 0; i < kN; ++i) v[i] = at(i);
        for (int t0 = 0; t0 <= last; t0 += kN) {
#pragma unroll
            for (int q = 0; q < kN; ++q) {
                const int t = t0 + q;
                if (t > last) break;
                const float w = G.w[t];
#pragma unroll
                for (int n = 0; n < kN; ++n) acc[n] = fmaf(w, v[(q + n) % kN], acc[n]);
                if (t < last) v[q] = at(t + kN);
            }
        }
    }
}

// x pass: a warp stages 256 + 2R values of one row, lane l computes outputs 8 l .. 8 l + 7
// and the row is written back through shared memory. One pad float per 8 keeps the lanes'
// strided reads on different banks.
constexpr int kXOut = kGaussRow / 32;
template <int kR>
__global__ void __launch_bounds__(256) k_gauss_x(const float* __restrict__ in, float* __restrict__ out, int nx,
                                                 long long rows, const __grid_constant__ GaussParams G) {
    constexpr int kSpan = kGaussRow + 2 * (kR ? kR : kMaxRadius);
    __shared__ float s[8][kSpan + kSpan / 8 + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, R = kR ? kR : G.R;
    const long long row = (long long)blockIdx.x * 8 + wid;
    if (row >= rows) return;
    const int x0 = blockIdx.y * kGaussRow;
    const float* src = in + row * nx;
    float* sp = s[wid];
#pragma unroll
    for (int k = 0; k < (kSpan + 31) / 32; ++k) {  // loads issued back to back
        const int i = lane + 32 * k;
        if (i < kGaussRow + 2 * R) sp[i + (i >> 3)] = __ldg(src + min(max(x0 - R + i, 0), nx - 1));
    }
    __syncwarp();
    float acc[kXOut];
    float* mine = sp + 9 * lane;  // padded place of value 8 lane
    gauss_taps<kR, kXOut>([&](int i) { return mine[i + (i >> 3)]; }, G, acc);
    __syncwarp();
#pragma unroll
    for (int n = 0; n < kXOut; ++n) mine[n] = acc[n];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kXOut; ++k) {
        const int i = lane + 32 * k;
        if (x0 + i < nx) out[row * nx + x0 + i] = sp[i + (i >> 3)];
    }
}

// y or z pass: block = 32 consecutive x times kGaussCol outputs along the pass
// axis (extent na, element stride `stride`); blockIdx.z indexes the remaining axis
// (offset `other` elements per step). 256 threads: 32 columns x 8 runs of 8 outputs.
template <int kR>
__global__ void __launch_bounds__(256) k_gauss_col(const float* __restrict__ in, float* __restrict__ out, int nx,
                                                   int na, long long stride, long long other,
                                                   const __grid_constant__ GaussParams G) {
    __shared__ float s[kGaussCol + 2 * (kR ? kR : kMaxRadius)][32];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int x = blockIdx.x * 32 + tx;
    const int a0 = blockIdx.y * kGaussCol;
    const long long base = (long long)blockIdx.z * other + x;
    const bool col = x < nx;
    const int R = kR ? kR : G.R;
#pragma unroll
    for (int k = 0; k < (kGaussCol + 2 * (kR ? kR : kMaxRadius) + 7) / 8; ++k) {  // loads issued back to back
        const int i = ty + 8 * k;
        if (i < kGaussCol + 2 * R)
            s[i][tx] = col ? __ldg(in + base + (long long)min(max(a0 - R + i, 0), na - 1) * stride) : 0.0f;
    }
    __syncthreads();
    const int o0 = ty * (kGaussCol / 8);
    if (!col || a0 + o0 >= na) return;
    float acc[kGaussCol / 8];
    gauss_taps<kR, kGaussCol / 8>([&](int i) { return s[o0 + i][tx]; }, G, acc);
#pragma unroll
    for (int n = 0; n < kGaussCol / 8; ++n)
        if (a0 + o0 + n < na) out[base + (long long)(a0 + o0 + n) * stride] = acc[n];
}

// x, then y, then z: in -> out (x) -> tmp (y) -> out (z).
template <int kR>
void gauss_passes_r(const float* in, float* out, float* tmp, const int n[3], const GaussParams& G, cudaStream_t st) {
    const long long plane = (long long)n[0] * n[1];
    const long long rows = (long long)n[1] * n[2];  // <= 2^22
    k_gauss_x<kR><<<dim3((unsigned)((rows + 7) / 8), (n[0] + kGaussRow - 1) / kGaussRow), 256, 0, st>>>(in, out, n[0],
                                                                                                      rows, G);
    k_gauss_col<kR><<<dim3((n[0] + 31) / 32, (n[1] + kGaussCol - 1) / kGaussCol, n[2]), 256, 0, st>>>(
        out, tmp, n[0], n[1], (long long)n[0], plane, G);
    k_gauss_col<kR><<<dim3((n[0] + 31) / 32, (n[2] + kGaussCol - 1) / kGaussCol, n[1]), 256, 0, st>>>(
        tmp, out, n[0], n[2], plane, (long long)n[0], G);
}

// Radii 4, 8 and 12 (sigma = 1, 2, 3) are unrolled; others take the generic loop.
void gauss_passes(const float* in, float* out, float* tmp, const int n[3], const GaussParams& G, cudaStream_t st) {
    switch (G.R) {
        case 4: gauss_passes_r<4>(in, out, tmp, n, G, st); break;
        case 8: gauss_passes_r<8>(in, out, tmp, n, G, st); break;
        case 12: gauss_passes_r<12>(in, out, tmp, n, G, st); break;
        default: gauss_passes_r<0>(in, out, tmp, n, G, st); break;
    }
}

// Scale-normalised Hessians (xx yy zz xy xz yz) of the smoothed volume, clamp-to-edge:
// a CTA owns a 32 x 8 column of voxels and walks planes z0 .. z1 - 1. Each plane (with
// its one-voxel border) is staged in shared memory once, loaded a plane ahead; a thread
// reads the nine in-plane neighbours it needs and keeps those of the planes below and
// above in registers: 9 shared reads and 340 / 256 x (planes + 2) / planes global loads per voxel (1.5
// in walks of 16 planes) instead of 19 loads (pass A of 256x256x176: 64 -> 36 us).
// emit(z, H) is called by every thread of the CTA for every plane.
// A short volume gets shorter walks (march_planes): with 16 planes per CTA 42x41x62 had 48
// CTAs, each a chain of 18 plane loads, and took 162 us for two scales (now 94).
constexpr int kTileX = 32, kTileY = 8;
struct PlaneTile {
    float v[2][kTileY + 2][kTileX + 2];
};
struct PlaneTaps {
    float c, xm, xp, ym, yp;      // centre and axis neighbours
    float mm, pm, mp, pp;         // diagonals, (x, y) signs
};

template <class F>
__device__ __forceinline__ void march_hessians(const float* __restrict__ f, int nx, int ny, int nz, float s2, int z0,
                                               int z1, PlaneTile& tile, const F& emit) {
    constexpr int kW = kTileX + 2, kAll = kW * (kTileY + 2);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const long long plane = (long long)nx * ny;
    // the (up to) two tile entries this thread loads
    const int e1 = threadIdx.x, e2 = threadIdx.x + 256;
    auto place = [&](int e) {
        const int x = min(max((int)blockIdx.x * kTileX - 1 + e % kW, 0), nx - 1);
        const int y = min(max((int)blockIdx.y * kTileY - 1 + e / kW, 0), ny - 1);
        return y * nx + x;
    };
    const int o1 = place(e1), o2 = e2 < kAll ? place(e2) : 0;
    float n1, n2 = 0.0f;
    auto fetch = [&](int z) {
        const float* p = f + min(max(z, 0), nz - 1) * plane;
        n1 = __ldg(p + o1);
        if (e2 < kAll) n2 = __ldg(p + o2);
    };
    int buf = 0;
    auto take = [&](int next) {  // stage the fetched plane, fetch plane `next`, read the taps
        float* t = &tile.v[buf][0][0];
        t[e1] = n1;
        if (e2 < kAll) t[e2] = n2;
        __syncthreads();
        fetch(next);
        const float* q = &tile.v[buf][ty + 1][tx + 1];
        buf ^= 1;
        return PlaneTaps{q[0], q[-1], q[1], q[-kW], q[kW], q[-kW - 1], q[-kW + 1], q[kW - 1], q[kW + 1]};
    };
    fetch(z0 - 1);
    PlaneTaps a = take(z0), b = take(z0 + 1);
    for (int z = z0; z < z1; ++z) {
        const PlaneTaps n = take(z + 2);
        const float c2 = 2.0f * b.c;
        float H[6];
        H[0] = s2 * (b.xp - c2 + b.xm);
        H[1] = s2 * (b.yp - c2 + b.ym);
        H[2] = s2 * (n.c - c2 + a.c);
        H[3] = 0.25f * s2 * ((b.pp - b.pm) - (b.mp - b.mm));
        H[4] = 0.25f * s2 * ((n.xp - a.xp) - (n.xm - a.xm));
        H[5] = 0.25f * s2 * ((n.yp - a.yp) - (n.ym - a.ym));
        emit(z, H);
        a = b;
        b = n;
    }
}

// ||H||_F = ||lambda|| (the Frobenius norm is invariant under the orthogonal
// similarity that diagonalises H): S without the eigen-decomposition.
__device__ __forceinline__ float hessian_norm(const float H[6]) {
    const float off = fmaf(H[3], H[3], fmaf(H[4], H[4], H[5] * H[5]));
    return sqrtf(fmaf(2.0f, off, fmaf(H[0], H[0], fmaf(H[1], H[1], H[2] * H[2]))));
}

// One Jacobi rotation of the symmetric 3x3 matrix held as its diagonal d and its
// off-diagonal entries o[0] = a01, o[1] = a02, o[2] = a12, in the plane (p, q) with
// r the third index: the angle makes a_pq exactly zero and the other entries take
// the stable updates of the classical method (tan t of the smaller angle, tau =
// s / (1 + c)); Golub & Van Loan, Sec. 8.5 (the symmetric Schur decomposition).
__device__ __forceinline__ void jacobi_rotate(float d[3], float& opq, float& orp, float& orq, int p, int q) {
    const float apq = opq;
    if (apq == 0.0f) return;
    // The rotation stays orthogonal (c = 1/sqrt(1 + t^2), s = t c) however t is
    // rounded, so t comes from the fast reciprocal; an inexact angle leaves a
    // residual a_pq of a few ulp, which is dropped at the float resolution of H.
    const float theta = 0.5f * __fdividef(d[q] - d[p], apq);
    // t = sign(theta) / (|theta| + sqrt(theta^2 + 1)), with |theta| capped at 1e18
    // (then t ~ 5e-19: a_pq is negligible) so that theta^2 + 1 stays finite and
    // its square root can be taken as r * rsqrt(r)
    const float at = fminf(fabsf(theta), 1e18f);
    const float r = fmaf(at, at, 1.0f);
    float t = __fdividef(1.0f, fmaf(r, rsqrtf(r), at));
    if (theta < 0.0f) t = -t;
    const float c = rsqrtf(fmaf(t, t, 1.0f)), s = t * c, tau = __fdividef(s, 1.0f + c);
    d[p] = fmaf(-t, apq, d[p]);
    d[q] = fmaf(t, apq, d[q]);
    opq = 0.0f;
    const float rp = orp, rq = orq;
    orp = fmaf(-s, fmaf(tau, rp, rq), rp);
    orq = fmaf(s, fmaf(-tau, rq, rp), rq);
}

// Eigenvalues sorted by |lambda| ascending (ties by lambda ascending).
__device__ __forceinline__ void eig3_sorted(const float H[6], float l[3]) {
    float d[3] = {H[0], H[1], H[2]};
    float o01 = H[3], o02 = H[4], o12 = H[5];
    // cyclic sweeps (planes 01, 02, 12) until the off-diagonal part is below float
    // resolution of the diagonal (then every eigenvalue is within that of the
    // diagonal entry, Weyl's inequality; quadratic convergence: 2-3 sweeps), at most 8
#pragma unroll 1
    for (int sweep = 0; sweep < 8; ++sweep) {
        const float off = fabsf(o01) + fabsf(o02) + fabsf(o12);
        if (off <= 6e-8f * (fabsf(d[0]) + fabsf(d[1]) + fabsf(d[2]))) break;
        jacobi_rotate(d, o01, o02, o12, 0, 1);  // r = 2: a20 = o02, a21 = o12
        jacobi_rotate(d, o02, o01, o12, 0, 2);  // r = 1: a10 = o01, a12 = o12
        jacobi_rotate(d, o12, o01, o02, 1, 2);  // r = 0: a01 = o01, a02 = o02
    }
    l[0] = d[0];
    l[1] = d[1];
    l[2] = d[2];
    auto before = [](float u, float v) { return fabsf(u) < fabsf(v) || (fabsf(u) == fabsf(v) && u < v); };
    if (before(l[1], l[0])) { const float t = l[0]; l[0] = l[1]; l[1] = t; }
    if (before(l[2], l[1])) { const float t = l[1]; l[1] = l[2]; l[2] = t; }
    if (before(l[1], l[0])) { const float t = l[0]; l[0] = l[1]; l[1] = t; }
}

// Pass A of a scale: the maximum over voxels of S = ||H|| (block maxima folded
// into smax with an integer atomicMax on the non-negative float bits).
__global__ void __launch_bounds__(256) k_frangi_smax(const float* __restrict__ sm, int nx, int ny, int nz, float s2,
                                                     int planes, float* __restrict__ smax) {
    __shared__ PlaneTile tile;
    const int x = blockIdx.x * kTileX + (threadIdx.x & 31), y = blockIdx.y * kTileY + (threadIdx.x >> 5);
    const bool in = x < nx && y < ny;
    const int z0 = blockIdx.z * planes;
    float S = 0.0f;
    march_hessians(sm, nx, ny, nz, s2, z0, min(z0 + planes, nz), tile, [&](int, const float H[6]) {
        if (in) S = fmaxf(S, hessian_norm(H));
    });
#pragma unroll
    for (int o = 16; o; o >>= 1) S = fmaxf(S, __shfl_xor_sync(0xffffffffu, S, o));
    __shared__ float ws[8];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = S;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) S = fmaxf(S, ws[w]);
        atomicMax(reinterpret_cast<int*>(smax), __float_as_int(S));
    }
}

// Frangi response of a voxel with Hessian H and a negative trace, c = smax / 2.
__device__ __forceinline__ float vessel_response(const float H[6], float c) {
    float l[3];
    eig3_sorted(H, l);
    if (l[1] > 0.0f || l[2] > 0.0f || l[1] == 0.0f || l[2] == 0.0f) return 0.0f;
    // fast reciprocal, reciprocal square root and exponential: a few ulp on
    // factors in [0, 1], far inside the 1e-4 the response is held to
    const float Ra = __fdividef(fabsf(l[1]), fabsf(l[2]));
    const float Rb = fabsf(l[0]) * rsqrtf(fabsf(l[1] * l[2]));
    const float S = hessian_norm(H);
    // alpha = beta = 0.5: 2 alpha^2 = 2 beta^2 = 0.5
    return (1.0f - __expf(-2.0f * Ra * Ra)) * __expf(-2.0f * Rb * Rb) *
           (1.0f - __expf(-(S * S) * __fdividef(0.5f, c * c)));
}

// Pass B: per voxel the Hessian again, its eigenvalues sorted by |lambda|, and the
// Frangi response of this scale (c = smax / 2), max-combined into V.
// Bright vessels have two negative eigenvalues, so only voxels with a negative trace (half
// of a noisy volume, scattered over every warp) need the decomposition, which is nearly
// all of the pass's instructions: they are queued in shared memory and decomposed 256 at a
// time with every lane busy (256x256x176, three scales: 701 -> 516 us; what
// is left is bound by the special-function pipe, five operations per rotation). The others leave V
// as it is (V starts at zero and only grows).
__global__ void __launch_bounds__(256) k_frangi_v(const float* __restrict__ sm, int nx, int ny, int nz, float s2,
                                                  int planes, const float* __restrict__ smax,
                                                  float* __restrict__ V) {
    __shared__ PlaneTile tile;
    __shared__ float qh[6][512];
    __shared__ int qpos[512];  // z - z0 and thread of the queued voxel
    __shared__ int tail;
    const int lane = threadIdx.x & 31;
    const int x = blockIdx.x * kTileX + lane, y = blockIdx.y * kTileY + (threadIdx.x >> 5);
    const bool in = x < nx && y < ny;
    const int z0 = blockIdx.z * planes;
    const float c = 0.5f * __ldg(smax);
    if (!(c > 0.0f)) return;
    if (threadIdx.x == 0) tail = 0;
    int head = 0;  // the same in every thread; entries head .. tail - 1, modulo 512
    auto respond = [&](int e) {
        const float H[6] = {qh[0][e], qh[1][e], qh[2][e], qh[3][e], qh[4][e], qh[5][e]};
        const int z = z0 + (qpos[e] >> 8), t = qpos[e] & 255;
        const float v = vessel_response(H, c);
        if (v > 0.0f) {
            float* o = V + ((long long)z * ny + blockIdx.y * kTileY + (t >> 5)) * nx + blockIdx.x * kTileX + (t & 31);
            *o = fmaxf(*o, v);
        }
    };
    march_hessians(sm, nx, ny, nz, s2, z0, min(z0 + planes, nz), tile, [&](int z, const float H[6]) {
        const bool take = in && H[0] + H[1] + H[2] < 0.0f;
        const unsigned m = __ballot_sync(0xffffffffu, take);
        int at = 0;
        if (lane == 0) at = atomicAdd(&tail, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (take) {
            const int e = (at + __popc(m & ((1u << lane) - 1u))) & 511;
#pragma unroll
            for (int q = 0; q < 6; ++q) qh[q][e] = H[q];
            qpos[e] = ((z - z0) << 8) | (int)threadIdx.x;
        }
        __syncthreads();
        if (tail - head >= 256) {
            respond((head + (int)threadIdx.x) & 511);
            head += 256;
        }
        __syncthreads();  // the queue's places and its tail are reused
    });
    if (head + (int)threadIdx.x < tail) respond((head + (int)threadIdx.x) & 511);
}

}  // namespace

cudaError_t launch_gauss3d(const float* in, float* out, float* tmp, const int n[3], float sigma, cudaStream_t st) {
    GaussParams G;
    G.R = (int)ceil(4.0 * (double)sigma);
    if (G.R > kMaxRadius || !(sigma > 0.0f)) return cudaErrorInvalidValue;
    double sum = 0.0, w[2 * kMaxRadius + 1];
    for (int i = -G.R; i <= G.R; ++i) sum += (w[i + G.R] = exp(-(double)i * i / (2.0 * (double)sigma * sigma)));
    for (int i = 0; i <= 2 * G.R; ++i) G.w[i] = (float)(w[i] / sum);
    gauss_passes(in, out, tmp, n, G, st);
    return cudaGetLastError();
}

cudaError_t launch_frangi(const float* norm, const int n[3], const float* sigmas, int n_sigmas, float* tmp_a,
                          float* tmp_b /* nvox floats */, float* smax /* n_sigmas floats */, float* V,
                          cudaStream_t st) {
    const long long nvox = (long long)n[0] * n[1] * n[2];
    cudaError_t e = cudaMemsetAsync(V, 0, sizeof(float) * nvox, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(smax, 0, sizeof(float) * n_sigmas, st);
    if (e != cudaSuccess) return e;
    const unsigned tx = (n[0] + kTileX - 1) / kTileX, ty = (n[1] + kTileY - 1) / kTileY;
    // at most 16 planes: more leave the last wave uneven
    const int planes = march_planes((long long)tx * ty, n[2], 8, 16);
    const dim3 grid(tx, ty, (n[2] + planes - 1) / planes);
    for (int si = 0; si < n_sigmas; ++si) {
        const double sg = sigmas[si];
        GaussParams G;
        G.R = (int)ceil(4.0 * sg);
        if (G.R > kMaxRadius) return cudaErrorInvalidValue;
        double sum = 0.0, w[2 * kMaxRadius + 1];
        for (int i = -G.R; i <= G.R; ++i) sum += (w[i + G.R] = exp(-(double)i * i / (2.0 * sg * sg)));
        for (int i = 0; i <= 2 * G.R; ++i) G.w[i] = (float)(w[i] / sum);
        gauss_passes(norm, tmp_a, tmp_b, n, G, st);
        const float s2 = (float)(sg * sg);
        k_frangi_smax<<<grid, 256, 0, st>>>(tmp_a, n[0], n[1], n[2], s2, planes, smax + si);
        k_frangi_v<<<grid, 256, 0, st>>>(tmp_a, n[0], n[1], n[2], s2, planes, smax + si, V);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace vr
