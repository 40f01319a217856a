// vr_backward.cu -- adjoint raymarch: gradients of a loss on the rendered image
// with respect to the transfer-function entries, the tissue uniforms
// (gamma, ka, kd, ks, opacity_scale) and the normalised voxel intensities.
//
// One thread per ray (the forward kernel's warp packets, 4 warps per CTA). Per ray:
//   1. the ray's stopping sample k_stop and the transmittance T in front of it, from
//      the forward's ray state, or by a forward re-march with the forward kernel's
//      exact arithmetic (empty bricks skipped);
//   2. reverse sweep over every sample k = k_stop .. 0, the lanes of a warp in step
//      by sample index (no skipping: the opacity entries of the transfer function
//      receive gradient from samples whose opacity is zero) with no stored samples:
//      the sample is re-evaluated, T_k = T_{k+1} / (1 - alpha_k) (exact in real
//      arithmetic and well conditioned because early termination keeps
//      1 - alpha_k >= 1 - et before the last sample), R_k = alpha_k c_k +
//      (1 - alpha_k) R_{k+1} and P_k = prod_{j>k} (1 - alpha_j) are carried
//      backwards, and
//        dL/dalpha_k = T_k (<dL/dC, c_k - R_{k+1}> + dL/dA P_k),
//        dL/dc_k     = T_k alpha_k dL/dC              (Eqs. 5-6 differentiated);
//   3. sample_adjoint / field_adjoint_scatter chain these to the parameters.
// Transfer-function gradients are accumulated per lane while its samples stay in
// one lookup cell, then added with 16-byte vector atomics into private global
// copies of the gradient (one 16-float record per cell; CTA c into copy c % n) that
// k_sum_copies gathers afterwards -- contended atomics on one table cost 10x the
// rest of the kernel, and a shared-memory table per CTA 1.6x (1D) to 1.8x (2D
// opacities) the copies. Voxel gradients: on the derived bricks, per-voxel channel
// gradients (vector atomics, neighbouring lanes in one cell merged, corner order
// rotated) and a gather pass through the stencil transposes; otherwise scalar
// global atomics on the voxels. Uniform gradients are warp-reduced first.
#include "vr_adjoint.cuh"

namespace vr {

namespace {

struct GLoad {
    const float* __restrict__ p;
    __device__ __forceinline__ float operator()(int o) const { return __ldg(p + o); }
};

// Skip-brick id in 32-bit arithmetic: dims <= 2048 give at most 512^3 = 2^27 bricks.
__device__ __forceinline__ int bidx(const VolumeDev& v, const int b[3]) {
    return (b[2] * v.nb[1] + b[1]) * v.nb[0] + b[0];
}

// Derived brick `bi` (32-bit operands: one widening multiply-add).
template <int kBS>
__device__ __forceinline__ const float4* derived_brick(const VolumeDev& v, int bi) {
    return reinterpret_cast<const float4*>(
        v.dbricks + (size_t)(unsigned)bi * (unsigned)(kBS ? der_brick_floats(kBS) : v.der_stride));
}

// Whether a sweep reads a cell's corners in parity order (derived_channels). The table's
// gradient is continuous in the sample's field, so a sweep for the table alone takes the
// faster offset order (fit step of 8 views 6.64 -> 6.07 ms; not at edge 4, whose corners
// share L1 columns). Voxel and uniform gradients jump at table knots and at |g| = 0, and a
// sum in another order puts single samples on the other side: there the order of the
// corners stays as it has been (about 2 % of the 1080p gradient, within what its runs differ).
__host__ __device__ constexpr bool parity_order(bool table_only, int bs) { return !table_only || bs == 2; }

// The sample field, from the derived bricks (voxel-wise derivatives) or by the
// per-sample stencils -- the same linear map of the voxels, either way. kHessian:
// the Hessian channels are read even without a curvature term (gamma = 0): the
// forward values do not need them then, but dL/dgamma = sum dL/dw kappa / kappa_ref
// does.
// bi: the skip brick of the sample's cell (derived bricks); sbi, base: its storage
// brick and the stencil origin in it (intensity bricks).
template <bool kDerived, bool kHessian, bool kParity, int kBS>
__device__ __forceinline__ void eval_field(const VolumeDev& v, const TissueDev& tp, int bi, long long sbi,
                                           const int i0[3], int base, const float f[3], const float is[3],
                                           float fld[10]) {
    if (kDerived) {
        const float4* brick = derived_brick<kBS>(v, bi);
        const int m = (1 << (kBS ? kBS : v.bs)) - 1;
        const DerLayout d = kBS ? der_layout(kBS) : v.der;
        derived_channels<kParity, 0, 4>(brick, d, i0[0] & m, i0[1] & m, i0[2] & m, f[0], f[1], f[2], fld);
        if (kHessian)
            derived_channels<kParity, 4, 6>(brick, d, i0[0] & m, i0[1] & m, i0[2] & m, f[0], f[1], f[2], fld + 4);
        else
            load_hessian<kParity>(tp, brick, d, i0[0] & m, i0[1] & m, i0[2] & m, f, fld);
    } else {
        field_eval(GLoad{v.bricks + sbi * kBrickVox}, base, f[0], f[1], f[2], fld);
        scale_field(fld, is);
    }
}

// Adjoint of the derived-field interpolation: the sample's field gradient dfs (I, g, H in the
// derived channels' mm units), trilinearly weighted, into the per-voxel channel
// gradients of the cell's 8 corners -- up to three vector reductions per corner,
// the Hessian ones only when the sample has Hessian gradients (a curvature term):
// without one that removes two thirds of the reduction traffic (8-view 512^2
// backward 36 -> 27 ms).
// Per-voxel channel gradients in three planes: (I, gx, gy, gz) float4 [nvox],
// (Hxx, Hyy, Hzz, Hxy) float4 [nvox], (Hxz, Hyz) float2 [nvox]. Every vector
// reduction then covers one aligned 16- or 8-byte piece, and x-neighbouring voxels'
// pieces share sectors (1080p backward 16.2 -> 14.1 ms against 48-byte records).
// Corner order: a warp's reduction to one address is applied one lane at a time
// (one L1 wavefront per lane: 32 lanes on one address cost 32 wavefronts, on 32
// consecutive addresses one), and the lanes of a warp that scatter in the same
// step are often in the same cell. Each lane therefore starts at the corner given
// by its rank among the lanes in its cell, so that up to 8 of them hit 8 different
// voxels in each reduction instruction. The rank only orders the additions.
// Before that, horizontally neighbouring lanes 2m and 2m + 1 whose samples lie in
// the same cell merge: the even lane receives the odd one's fractions and field
// gradient (13 shuffles) and adds both samples' weighted gradients in each
// reduction, the odd lane issues none (1080p backward 12.1 -> 10.4 ms; at 512^2, where
// fewer neighbours share a cell, within 1 %); lanes left unmerged then pair the same
// way with their vertical neighbour, lane ^ ymask (the packet width): 10.4 -> 10.3 ms.
// A lane adds at most two samples.
// Float index of voxel p's channel ch (0..9).
__device__ __forceinline__ long long chan_index(long long p, long long nvox, int ch) {
    return ch < 4 ? 4 * p + ch : (ch < 8 ? 4 * nvox + 4 * p + (ch - 4) : 8 * nvox + 2 * p + (ch - 8));
}

__device__ __forceinline__ void scatter_channels(float* __restrict__ dgrad, const int n[3], const int i0[3],
                                                 const float f[3], const float dfs[10], int ymask) {
    const long long nvox = (long long)n[0] * n[1] * n[2];
    bool any = false, hess = false;
#pragma unroll
    for (int q = 0; q < 4; ++q) any |= dfs[q] != 0.0f;
#pragma unroll
    for (int q = 4; q < 10; ++q) hess |= dfs[q] != 0.0f;
    if (!any && !hess) return;
    const long long nxy = (long long)n[0] * n[1];
    const long long p0 = (long long)i0[2] * nxy + (long long)i0[1] * n[0] + i0[0];
    // lanes 2m and 2m + 1 that scatter into the same cell: the even lane adds both
    // samples' weighted gradients, the odd one issues nothing
    const unsigned act = __activemask();
    const int lane = threadIdx.x & 31;
    const unsigned lo = (unsigned)p0, hi = (unsigned)(p0 >> 32);
    const unsigned plo = __shfl_xor_sync(act, lo, 1), phi = __shfl_xor_sync(act, hi, 1);
    float pf[3], pd[10];
#pragma unroll
    for (int q = 0; q < 3; ++q) pf[q] = __shfl_xor_sync(act, f[q], 1);
#pragma unroll
    for (int q = 0; q < 10; ++q) pd[q] = __shfl_xor_sync(act, dfs[q], 1);
    int phess_v = __shfl_xor_sync(act, (int)hess, 1);
    bool merged = ((act >> (lane ^ 1)) & 1u) && plo == lo && phi == hi;
    if (merged && (lane & 1)) return;
    // second round: lanes left unmerged pair with their vertical neighbour lane ^ ymask
    {
        const unsigned act2 = __activemask();
        const unsigned qlo = __shfl_xor_sync(act2, lo, ymask), qhi = __shfl_xor_sync(act2, hi, ymask);
        const int qfree = __shfl_xor_sync(act2, (int)!merged, ymask);
        float qf[3], qd[10];
#pragma unroll
        for (int q = 0; q < 3; ++q) qf[q] = __shfl_xor_sync(act2, f[q], ymask);
#pragma unroll
        for (int q = 0; q < 10; ++q) qd[q] = __shfl_xor_sync(act2, dfs[q], ymask);
        const int qhess = __shfl_xor_sync(act2, (int)hess, ymask);
        const bool my = !merged && qfree && ((act2 >> (lane ^ ymask)) & 1u) && qlo == lo && qhi == hi;
        if (my && (lane & ymask)) return;
        if (my) {
            merged = true;
#pragma unroll
            for (int q = 0; q < 3; ++q) pf[q] = qf[q];
#pragma unroll
            for (int q = 0; q < 10; ++q) pd[q] = qd[q];
            phess_v = qhess;
        }
    }
    const bool h = hess || (merged && phess_v);
    const unsigned same = __match_any_sync(__activemask(), lo);
    const int rot = __popc(same & ((1u << lane) - 1u)) & 7;
    // instruction i scatters corner i ^ rot: per axis the two factors and offsets
    // are swapped once when that bit of rot is set, so that every corner's weight,
    // ((dx ? fx : 1 - fx) * (dy ? ...)) * (dz ? ...), and address are fixed registers
    const bool sx = rot & 1, sy = (rot >> 1) & 1, sz = (rot >> 2) & 1;
    const float gx = 1.0f - f[0], gy = 1.0f - f[1], gz = 1.0f - f[2];
    const float ax[2] = {sx ? f[0] : gx, sx ? gx : f[0]}, ay[2] = {sy ? f[1] : gy, sy ? gy : f[1]},
                az[2] = {sz ? f[2] : gz, sz ? gz : f[2]};
    const float qx = 1.0f - pf[0], qy = 1.0f - pf[1], qz = 1.0f - pf[2];
    const float bx2[2] = {sx ? pf[0] : qx, sx ? qx : pf[0]}, by2[2] = {sy ? pf[1] : qy, sy ? qy : pf[1]},
                bz2[2] = {sz ? pf[2] : qz, sz ? qz : pf[2]};
    const int nx = n[0], nxy32 = n[0] * n[1];  // < 2^23 for dims <= 2048
    const int ox[2] = {sx ? 1 : 0, sx ? 0 : 1}, oy[2] = {sy ? nx : 0, sy ? 0 : nx},
              oz[2] = {sz ? nxy32 : 0, sz ? 0 : nxy32};
    float4* const c0 = reinterpret_cast<float4*>(dgrad + chan_index(p0, nvox, 0));
    float4* const c1 = reinterpret_cast<float4*>(dgrad + chan_index(p0, nvox, 4));
    float2* const c2 = reinterpret_cast<float2*>(dgrad + chan_index(p0, nvox, 8));
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int ix = i & 1, iy = (i >> 1) & 1, iz = i >> 2;
        const float w = (ax[ix] * ay[iy]) * az[iz];
        const float pw = merged ? (bx2[ix] * by2[iy]) * bz2[iz] : 0.0f;
        if (w == 0.0f && pw == 0.0f) continue;
        const int off = ox[ix] + oy[iy] + oz[iz];
        float4 g0;
        mul2(w, w, dfs[0], dfs[1], g0.x, g0.y);
        mul2(w, w, dfs[2], dfs[3], g0.z, g0.w);
        fma2(pw, pd[0], pd[1], g0.x, g0.y);
        fma2(pw, pd[2], pd[3], g0.z, g0.w);
        atomicAdd(c0 + off, g0);
        if (h) {
            float4 g1;
            float2 g2;
            mul2(w, w, dfs[4], dfs[5], g1.x, g1.y);
            mul2(w, w, dfs[6], dfs[7], g1.z, g1.w);
            mul2(w, w, dfs[8], dfs[9], g2.x, g2.y);
            fma2(pw, pd[4], pd[5], g1.x, g1.y);
            fma2(pw, pd[6], pd[7], g1.z, g1.w);
            fma2(pw, pd[8], pd[9], g2.x, g2.y);
            atomicAdd(c1 + off, g1);
            atomicAdd(c2 + off, g2);
        }
    }
}

// dL/dI from the channel gradients: the transpose of the derived channels' clamp-to-edge
// difference stencils (I; g_a = (I[p+a] - I[p-a]) / (2 s_a); H_aa = (I[p+a] - 2 I[p] +
// I[p-a]) / s_a^2; H_ab = the four (p +- a +- b) corners / (4 s_a s_b)).
// Along one axis the transposed first difference of a channel G at voxel v is
// d(G)[v] = G[v-1] - G[v+1] and the transposed second difference s(G)[v] = G[v-1] - 2 G[v]
// + G[v+1], where at the ends, whose clamped neighbour is the end voxel itself, a missing
// G[v-1] reads -G[v] in d and G[v] in s (and a missing G[v+1] likewise): the sources of
// voxel 0 are p = 0 (its "-1" neighbour) and p = 1.
// Separably, with the planes' sums
//   A = I + d_x(gx) / 2sx + d_y(gy) / 2sy + s_x(Hxx) / sx^2 + s_y(Hyy) / sy^2 + d_x d_y(Hxy) / 4 sx sy
//   D = gz / 2sz + d_x(Hxz) / 4 sx sz + d_y(Hyz) / 4 sy sz,    S = Hzz / sz^2
// the voxel is A + d_z(D) + s_z(S). A CTA owns 32 x 8 columns and walks a run of planes: the
// ten channels of a plane (with their one-voxel border) go through shared memory once and D
// and S of three planes stay in registers: 340 / 256 x (planes + 2) / planes loads per value, 1.55
// in walks of twelve planes, most of the repeated ones from L2, instead of 28 scattered loads per
// voxel (181x217x181: 291 -> 117 us; 312 MB is each value read and each voxel written once).
constexpr int kVoxTileY = 8;
__global__ void __launch_bounds__(256) k_channels_to_voxels(const float* __restrict__ G, int nx, int ny, int nz,
                                                            float sx, float sy, float sz, int planes,
                                                            float* __restrict__ dvol) {
    constexpr int kW = 34, kH = kVoxTileY + 2, kAll = kW * kH;
    // per plane: (I, gx, gy, gz), (Hxx, Hyy, Hzz, Hxy), (Hxz, Hyz)
    __shared__ float4 t0[kAll], t1[kAll];
    __shared__ float2 t2[kAll];
    const long long nvox = (long long)nx * ny * nz, plane = (long long)nx * ny;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int x = blockIdx.x * 32 + tx, y = blockIdx.y * kVoxTileY + ty;
    const int z0 = blockIdx.z * planes, z1 = min(z0 + planes, nz);
    const bool in = x < nx && y < ny;
    const float4* G0 = reinterpret_cast<const float4*>(G);
    const float4* G1 = reinterpret_cast<const float4*>(G + 4 * nvox);
    const float2* G2 = reinterpret_cast<const float2*>(G + 8 * nvox);
    const float cx = 0.5f / sx, cy = 0.5f / sy, cz = 0.5f / sz;
    const float qx = 1.0f / (sx * sx), qy = 1.0f / (sy * sy), qz = 1.0f / (sz * sz);
    const float mxy = 0.25f / (sx * sy), mxz = 0.25f / (sx * sz), myz = 0.25f / (sy * sz);
    const int c = (ty + 1) * kW + tx + 1;
    // the entries this thread stages, clamped into the volume (a clamped border value is
    // replaced by the end rules below)
    auto place = [&](int e) {
        const int gx = min(max((int)blockIdx.x * 32 - 1 + e % kW, 0), nx - 1);
        const int gy = min(max((int)blockIdx.y * kVoxTileY - 1 + e / kW, 0), ny - 1);
        return (long long)gy * nx + gx;
    };
    const int e1 = threadIdx.x, e2 = threadIdx.x + 256;
    const long long o1 = place(e1), o2 = e2 < kAll ? place(e2) : 0;
    // end rules: the clamped border entry is the end voxel's own value, wanted as it is in
    // s and with the opposite sign in d
    const float lx = x > 0 ? 1.0f : -1.0f, rx = x < nx - 1 ? 1.0f : -1.0f;
    const float ly = y > 0 ? 1.0f : -1.0f, ry = y < ny - 1 ? 1.0f : -1.0f;
    float Am = 0.0f, Dp = 0.0f, Dm = 0.0f, Sp = 0.0f, Sm = 0.0f;  // A, D, S of plane z - 1; D, S of plane z - 2
    for (int z = z0 - 1; z <= z1; ++z) {
        const long long zo = (long long)min(max(z, 0), nz - 1) * plane;
        __syncthreads();
        t0[e1] = __ldg(G0 + zo + o1);
        t1[e1] = __ldg(G1 + zo + o1);
        t2[e1] = __ldg(G2 + zo + o1);
        if (e2 < kAll) {
            t0[e2] = __ldg(G0 + zo + o2);
            t1[e2] = __ldg(G1 + zo + o2);
            t2[e2] = __ldg(G2 + zo + o2);
        }
        __syncthreads();
        const float4 a = t0[c], h = t1[c];
        const float hxx = t1[c - 1].x - 2.0f * h.x + t1[c + 1].x, hyy = t1[c - kW].y - 2.0f * h.y + t1[c + kW].y;
        const float gx = lx * t0[c - 1].y - rx * t0[c + 1].y, gy = ly * t0[c - kW].z - ry * t0[c + kW].z;
        const float xy = ly * (lx * t1[c - kW - 1].w - rx * t1[c - kW + 1].w) -
                         ry * (lx * t1[c + kW - 1].w - rx * t1[c + kW + 1].w);
        const float A = a.x + cx * gx + cy * gy + qx * hxx + qy * hyy + mxy * xy;
        float D = cz * a.w + mxz * (lx * t2[c - 1].x - rx * t2[c + 1].x) + myz * (ly * t2[c - kW].y - ry * t2[c + kW].y);
        const float S = qz * h.z;
        if (z < 0 || z > nz - 1) D = -D;  // the plane past an end is the end plane, with d's sign
        // voxel z - 1: A + (D[z-2] - D[z]) + (S[z-2] - 2 S[z-1] + S[z])
        if (z > z0 && in) dvol[(long long)(z - 1) * plane + (long long)y * nx + x] = Am + (Dm - D) + (Sm - 2.0f * Sp + S);
        Am = A;
        Dm = Dp;
        Dp = D;
        Sm = Sp;
        Sp = S;
    }
}

// The sample of the reverse sweep at fractions f of cell i0: its field and optics. No
// skipping: a sample in empty space has alpha = 0, but its lookup still gives the opacity
// entries it reads a non-zero gradient. bs: log2 of the skip-brick edge.
template <bool kDerived, bool kLazyHessian, bool kNoHessian, bool k2D, bool kParity, int kBS>
__device__ __forceinline__ void sweep_eval(const VolumeDev& v, const TissueDev& tp, const float4* __restrict__ tf,
                                           const int i0[3], const float f[3], const float dir[3], const float is[3],
                                           float inv_gmax, float fld[10], SampleOptics& so) {
    const int bs = kBS ? kBS : v.bs, bc[3] = {i0[0] >> bs, i0[1] >> bs, i0[2] >> bs};
    const int bi = bidx(v, bc);
    int base;
    const long long sbi = storage_brick(v, i0, base);
    const float vval = v.vbricks ? value_eval(GLoad{v.vbricks + sbi * kBrickVox}, base, f[0], f[1], f[2]) : 0.f;
    if (kLazyHessian) {
        // I and the gradient, the table lookup, then the Hessian, which without
        // a curvature term only dL/dgamma needs -- and not at a zero opacity
        // entry (dL/dw = 0 there, and w = 1 whatever kappa)
        const float4* brick = derived_brick<kBS>(v, bi);
        const int m = (1 << bs) - 1;
        const DerLayout d = kBS ? der_layout(kBS) : v.der;
        derived_channels<kParity, 0, 4>(brick, d, i0[0] & m, i0[1] & m, i0[2] & m, f[0], f[1], f[2], fld);
        optics_tf<k2D ? 2 : 1>(fld, vval, tp, tf, inv_gmax, so);
        if (!kNoHessian && so.c.w != 0.0f) {
            derived_channels<kParity, 4, 6>(brick, d, i0[0] & m, i0[1] & m, i0[2] & m, f[0], f[1], f[2], fld + 4);
        } else {
#pragma unroll
            for (int q = 4; q < 10; ++q) fld[q] = 0.0f;
        }
        optics_rest(fld, dir, tp, so);
    } else {
        eval_field<kDerived, true, kParity, kBS>(v, tp, bi, sbi, i0, base, f, is, fld);
        optics_core<k2D ? 2 : 1>(fld, vval, dir, tp, tf, inv_gmax, so);
    }
}

// dL/dalpha of a sample with transmittance Tk in front of it, the colour R and
// transmittance P of everything behind it.
__device__ __forceinline__ float sweep_dalpha(const SampleOptics& so, const float4& g4, float Tk, float R0, float R1,
                                              float R2, float P) {
    return Tk * (fmaf(g4.x, so.col[0] - R0, fmaf(g4.y, so.col[1] - R1, g4.z * (so.col[2] - R2))) + g4.w * P);
}

// Zero opacity entry: alpha = 0 exactly, so only the table's opacity entries at the
// lookup receive a gradient (the one-sided derivative of the clamp at 0); colour, uniforms
// and field gradients are all zero.
template <bool k2D>
__device__ __forceinline__ void sweep_apply_empty(const TissueDev& tp, const SampleOptics& so, float da,
                                                  TfGradSink<k2D>& sink) {
    if (tp.alpha_exp > 0.0f) da *= tp.alpha_exp;
    const float dr[4] = {0.f, 0.f, 0.f,
                         (so.raw >= 0.0f && so.raw <= 1.0f) ? da * tp.opacity_scale * so.mg * so.wk : 0.0f};
    if (!k2D)
        sink.add_cell(so.j, 1.0f - so.t, so.t, 0.0f, 0.0f, dr);
    else
        sink.add_cell(so.k * tp.tf_w + so.j, (1.0f - so.q) * (1.0f - so.t), (1.0f - so.q) * so.t,
                      so.q * (1.0f - so.t), so.q * so.t, dr);
}

// Any other sample: table, uniform and (unless kTfOnly) voxel gradients. `pair`: the lane
// distance whose lane the channel scatter tries to merge with after its neighbour.
template <bool kDerived, bool kTfOnly, bool k2D>
__device__ __forceinline__ void sweep_apply(const BackwardLaunch& B, const float fld[10], const SampleOptics& so,
                                            const int i0[3], const float f[3], const float dir[3], const float is[3],
                                            float inv_gmax, float da, float Tk, const float4& g4, int pair,
                                            TfGradSink<k2D>& sink, ParamGrad& dp) {
    const VolumeDev& v = B.r.vol;
    const float ta = Tk * so.alpha;
    const float dc[3] = {ta * g4.x, ta * g4.y, ta * g4.z};
    float dfs[10];
    sample_adjoint(fld, so, dir, B.r.tp, inv_gmax, da, dc, sink, dp, dfs);
    if (kTfOnly) return;
    if (kDerived && B.dgrad) {
        scatter_channels(B.dgrad, v.n, i0, f, dfs, pair);
    } else if (B.dvol) {
        const int x0 = i0[0] - 1, y0 = i0[1] - 1, z0 = i0[2] - 1;
        const int nx = v.n[0], ny = v.n[1], nz = v.n[2];
        float* dv = B.dvol;
        field_adjoint_scatter(dfs, is, f[0], f[1], f[2], [&](int a, int b, int c, float g) {
            if (g == 0.0f) return;
            const int x = min(max(x0 + a, 0), nx - 1), y = min(max(y0 + b, 0), ny - 1),
                      z = min(max(z0 + c, 0), nz - 1);
            atomicAdd(dv + ((long long)z * ny + y) * nx + x, g);
        });
    }
}

// Uniform gradients of a warp: one double-precision addition per warp and parameter
// (float additions of thousands of warps lost 1e-6 of the sum).
__device__ __forceinline__ void add_param_grads(const ParamGrad& dp, double* __restrict__ dparams) {
    float pv[5] = {dp.gamma, dp.ka, dp.kd, dp.ks, dp.os};
#pragma unroll
    for (int e = 0; e < 5; ++e) {
#pragma unroll
        for (int o = 16; o; o >>= 1) pv[e] += __shfl_xor_sync(0xffffffffu, pv[e], o);
    }
    if ((threadIdx.x & 31) == 0 && dparams) {
#pragma unroll
        for (int e = 0; e < 5; ++e)
            if (pv[e] != 0.0f) atomicAdd(dparams + e, (double)pv[e]);
    }
}

// 4 resident CTAs per SM (<= 128 registers): measured 1 ms faster at 1080p than
// the 3 that the unbounded register count allows. The sweep re-evaluates every sample
// and is bound by instructions and registers (16 warps at 55-60 % issue), so what a
// launch does not need is compiled out:
// Derived bricks without a curvature term (gamma = 0): with kLazyHessian a sample
// reads the Hessian only when its opacity entry is non-zero (for dL/dgamma); with
// kNoHessian, when no uniform gradient is wanted, never.
// kTfOnly: neither uniform nor voxel gradients are wanted (a transfer-function fit): no
// field adjoint, no scatter. k2D: whether the table has two dimensions; a 1D table's
// sink and lookup keep 16 registers less, and the kernel for a 1D table alone fits five
// CTAs (96 registers). Forward + backward, without / with both: fit step of 8 views of
// the 128^3 head at 512^2 9.53 -> 6.86 ms (1.9 of it the forward), 4 such views with
// every gradient 6.71 -> 5.91, 1080p of the 181x217x181 head (2D) 11.63 -> 11.43, its
// table alone at 2 x 700x600 6.48 -> 5.43. (6 CTAs for the 1D table alone: 2 % slower; 5
// for 1D with every gradient: 5 % slower; 5 for the 2D table alone: 2 % slower.)
// kBS: log2 of the skip-brick edge (2, 3, 4), fixed at compile time.
template <bool kDerived, bool kLazyHessian, bool kNoHessian, bool kTfOnly, bool k2D, int kBS>
__global__ void __launch_bounds__(128, kTfOnly && !k2D ? 5 : 4) k_render_backward(const __grid_constant__ BackwardLaunch B) {
    const RenderLaunch& L = B.r;
    const size_t ncell = (size_t)L.tp.tf_w * L.tp.tf_h * kTfCellFloats;
    // one of n_copies private global copies of the gradient, so that CTAs working on
    // the same hot entries do not serialise on one address
    const int cta = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    TfGradSink<k2D> sink(B.dtf_copies + (size_t)(cta % B.n_copies) * ncell);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    int di, dj;
    tile_pixel(L.packet_w, __ffs(tile_packets_x(L.packet_w, 4)) - 1, w, l, di, dj);
    const int i = blockIdx.x * 16 + di;
    const int j = blockIdx.y * 8 + dj;
    const int cam = blockIdx.z;
    const bool inside = i < L.W && j < L.H;
    const VolumeDev& v = L.vol;
    const float4* tf = reinterpret_cast<const float4*>(L.tf);
    const float gmax = __ldg(&v.vc->gmax);
    const float inv_gmax = gmax > 0.0f ? 1.0f / gmax : 0.0f;
    const float is[3] = {1.0f / v.s[0], 1.0f / v.s[1], 1.0f / v.s[2]};
    // the reverse sweep divides by 1 - alpha: stop where A reaches 1 even when early termination is off
    const float et = fminf(L.tp.et_threshold, 1.0f);
    ParamGrad dp{0.f, 0.f, 0.f, 0.f, 0.f};

    RayDev r;
    const bool hit = inside && setup_ray(L.cams[cam], L.rc, i, j, v.n, v.s, r);
    float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
    int kstop = -1;  // the ray's last sample (-1: none)
    float Tk = 1.0f;
    if (hit) {
        const long long pix = ((long long)(L.cam_offset + cam) * L.H + j) * L.W + i;
        g4 = __ldg(reinterpret_cast<const float4*>(B.dl_drgba) + pix);
        // 1. the ray's last sample and the transmittance in front of it: recorded by the
        // forward render (ray_state), or re-marched forward here
        kstop = r.ns - 1;
        if (L.ray_state) {
            const float2 st = __ldg(L.ray_state + pix);
            kstop = __float_as_int(st.x);
            Tk = st.y;
            if (!VR_CHECK(L.tp.status, kstop >= -1 && kstop < r.ns)) kstop = -1;  // a state of another image
        } else {
            float A = 0.f, A_prev = 0.f;
            int k = 0, klast = -1;
            while (k < r.ns) {
                int i0[3], bc[3];
                float f[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    sample_cell(r, q, k, v.n[q], i0[q], f[q]);
                    bc[q] = i0[q] >> kBS;
                }
                if (!VR_CHECK(L.tp.status, (unsigned)i0[0] <= (unsigned)(v.n[0] - 2) &&
                                               (unsigned)i0[1] <= (unsigned)(v.n[1] - 2) &&
                                               (unsigned)i0[2] <= (unsigned)(v.n[2] - 2)))
                    break;
                const int bi = bidx(v, bc);
                if (L.skip && __ldg(v.empty + bi)) {
                    k = brick_exit_k(r, bc, 1 << kBS, k, r.ns);
                    continue;
                }
                int base;
                const long long sbi = storage_brick(v, i0, base);
                float fld[10];
                eval_field<kDerived, false, parity_order(kTfOnly, kBS), kBS>(v, L.tp, bi, sbi, i0, base, f, is, fld);
                const float vval =
                    v.vbricks ? value_eval(GLoad{v.vbricks + sbi * kBrickVox}, base, f[0], f[1], f[2]) : 0.f;
                float alpha, col[3];
                sample_optics(fld, vval, r.dir, L.tp, tf, inv_gmax, alpha, col);
                const float wgt = (1.0f - A) * alpha;  // as the forward kernel composites
                A_prev = A;
                A += wgt;
                klast = k;
                if (A >= et) {
                    kstop = k;
                    break;
                }
                ++k;
            }
            // transmittance before the stopping sample (1 when no sample had opacity)
            Tk = (klast == kstop) ? 1.0f - A_prev : 1.0f - A;
        }
    }
    {
            float Tk1 = Tk, R0 = 0.f, R1 = 0.f, R2 = 0.f, P = 1.0f;
            // 2. reverse sweep, the lanes of a warp in step: at iteration kr every lane
            // whose ray reaches that far works on its sample kr, so neighbouring rays sit
            // at nearly the same depth and their reads and reductions hit the same cells
            const int kmax = __reduce_max_sync(0xffffffffu, kstop);
            // the position of sample kr, u0 + kr du, carried down by exact integer steps
            long long U[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) U[q] = hit ? r.u0[q] + (long long)kmax * r.du[q] : 0ll;
            for (int kr = kmax; kr >= 0; --kr, U[0] -= r.du[0], U[1] -= r.du[1], U[2] -= r.du[2]) {
                if (kr > kstop) continue;
                int i0[3];
                float f[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) cell_at(U[q], v.n[q], i0[q], f[q]);
                if (!VR_CHECK(L.tp.status, (unsigned)i0[0] <= (unsigned)(v.n[0] - 2) &&
                                               (unsigned)i0[1] <= (unsigned)(v.n[1] - 2) &&
                                               (unsigned)i0[2] <= (unsigned)(v.n[2] - 2)))
                    continue;
                float fld[10];
                SampleOptics so;
                sweep_eval<kDerived, kLazyHessian, kNoHessian, k2D, parity_order(kTfOnly, kBS), kBS>(
                    v, L.tp, tf, i0, f, r.dir, is, inv_gmax, fld, so);
                const float alpha = so.alpha;
                // T_k = T_{k+1} / (1 - alpha_k); Tk still holds T_{k+1} here, which a zero
                // alpha leaves unchanged (x / 1 = x), so the division is skipped then
                if (kr != kstop && alpha != 0.0f) Tk = Tk1 / (1.0f - alpha);
                const float da = sweep_dalpha(so, g4, Tk, R0, R1, R2, P);
                if (so.c.w == 0.0f) {
                    sweep_apply_empty(L.tp, so, da, sink);
                    Tk1 = Tk;
                    continue;
                }
                sweep_apply<kDerived, kTfOnly>(B, fld, so, i0, f, r.dir, is, inv_gmax, da, Tk, g4, L.packet_w, sink,
                                               dp);
                R0 = fmaf(alpha, so.col[0], (1.0f - alpha) * R0);
                R1 = fmaf(alpha, so.col[1], (1.0f - alpha) * R1);
                R2 = fmaf(alpha, so.col[2], (1.0f - alpha) * R2);
                P *= (1.0f - alpha);
                Tk1 = Tk;
            }
    }
    sink.flush();
    if (kTfOnly) return;
    add_param_grads(dp, B.dparams);
}

// The sweep with G lanes per ray (G = L.lanes, a power of two up to 16), for launches
// with too few rays to fill the chip and a recorded ray state: lane g evaluates sample
// kb - g, every lane of the ray then repeats the recurrences of T, R and P over the G
// samples in the sweep's order on shuffled opacities and colours, keeping the values at
// its own sample, and applies its sample's adjoint. Time falls with the serial chain
// (backward_lanes has the figures). 3 CTAs per SM (168 registers) where the field's
// adjoint is wanted: up to 10 % faster than 4 with their spills; 4 for the table alone.
template <bool kLazyHessian, bool kNoHessian, bool kTfOnly, bool k2D, int kBS>
__global__ void __launch_bounds__(128, kTfOnly ? 4 : 3) k_backward_lanes(const __grid_constant__ BackwardLaunch B) {
    const RenderLaunch& L = B.r;
    const size_t ncell = (size_t)L.tp.tf_w * L.tp.tf_h * kTfCellFloats;
    const int cta = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    TfGradSink<k2D> sink(B.dtf_copies + (size_t)(cta % B.n_copies) * ncell);
    const int G = L.lanes, lane = threadIdx.x & 31, g = lane & (G - 1), first = lane & ~(G - 1);
    const int ray = lane / G, pw = L.packet_w;
    const int i = (blockIdx.x * 4 + (threadIdx.x >> 5)) * pw + (ray & (pw - 1));
    const int j = blockIdx.y * L.packet_h + ray / pw;
    const int cam = blockIdx.z;
    const VolumeDev& v = L.vol;
    const float4* tf = reinterpret_cast<const float4*>(L.tf);
    const float gmax = __ldg(&v.vc->gmax);
    const float inv_gmax = gmax > 0.0f ? 1.0f / gmax : 0.0f;
    const float is[3] = {1.0f / v.s[0], 1.0f / v.s[1], 1.0f / v.s[2]};
    ParamGrad dp{0.f, 0.f, 0.f, 0.f, 0.f};
    RayDev r;
    float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
    int kstop = -1;
    float Tk = 1.0f;
    const bool hit = i < L.W && j < L.H && setup_ray(L.cams[cam], L.rc, i, j, v.n, v.s, r);
    if (hit) {
        const long long pix = ((long long)(L.cam_offset + cam) * L.H + j) * L.W + i;
        g4 = __ldg(reinterpret_cast<const float4*>(B.dl_drgba) + pix);
        const float2 st = __ldg(L.ray_state + pix);
        kstop = __float_as_int(st.x);
        Tk = st.y;
        if (!VR_CHECK(L.tp.status, kstop >= -1 && kstop < r.ns)) kstop = -1;  // a state of another image
    }
    const int kmax = __reduce_max_sync(0xffffffffu, kstop);
    long long U[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) U[q] = hit ? r.u0[q] + (long long)(kmax - g) * r.du[q] : 0ll;
    float Tk1 = Tk, R0 = 0.f, R1 = 0.f, R2 = 0.f, P = 1.0f;
    for (int kb = kmax; kb >= 0; kb -= G) {
        const int kr = kb - g;
        bool on = kr >= 0 && kr <= kstop;
        int i0[3] = {0, 0, 0};
        float f[3] = {0.f, 0.f, 0.f}, fld[10];
        SampleOptics so;
        so.alpha = so.c.w = so.col[0] = so.col[1] = so.col[2] = 0.0f;
        if (on) {
#pragma unroll
            for (int q = 0; q < 3; ++q) cell_at(U[q], v.n[q], i0[q], f[q]);
            on = VR_CHECK(L.tp.status, (unsigned)i0[0] <= (unsigned)(v.n[0] - 2) &&
                                           (unsigned)i0[1] <= (unsigned)(v.n[1] - 2) &&
                                           (unsigned)i0[2] <= (unsigned)(v.n[2] - 2));
            if (on)
                sweep_eval<true, kLazyHessian, kNoHessian, k2D, parity_order(kTfOnly, kBS), kBS>(
                    v, L.tp, tf, i0, f, r.dir, is, inv_gmax, fld, so);
        }
        const unsigned shaded = __ballot_sync(0xffffffffu, on && so.c.w != 0.0f);
        // the recurrences over the samples kb, kb - 1, ...; a sample of zero opacity entry
        // leaves T, R and P as they are
        float myT = 1.0f, myR0 = 0.f, myR1 = 0.f, myR2 = 0.f, myP = 1.0f;
        for (int h = 0; h < G; ++h) {
            const int src = first + h;
            const float a = __shfl_sync(0xffffffffu, so.alpha, src);
            const float c0 = __shfl_sync(0xffffffffu, so.col[0], src), c1 = __shfl_sync(0xffffffffu, so.col[1], src),
                        c2 = __shfl_sync(0xffffffffu, so.col[2], src);
            const bool sh = (shaded >> src) & 1u;
            if (sh && kb - h != kstop && a != 0.0f) Tk = Tk1 / (1.0f - a);
            if (h == g) {
                myT = Tk;
                myR0 = R0, myR1 = R1, myR2 = R2, myP = P;
            }
            if (sh) {
                R0 = fmaf(a, c0, (1.0f - a) * R0);
                R1 = fmaf(a, c1, (1.0f - a) * R1);
                R2 = fmaf(a, c2, (1.0f - a) * R2);
                P *= (1.0f - a);
                Tk1 = Tk;
            }
        }
        if (on) {
            const float da = sweep_dalpha(so, g4, myT, myR0, myR1, myR2, myP);
            if (so.c.w == 0.0f)
                sweep_apply_empty(L.tp, so, da, sink);
            else
                sweep_apply<true, kTfOnly>(B, fld, so, i0, f, r.dir, is, inv_gmax, da, myT, g4, G, sink, dp);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) U[q] -= (long long)G * r.du[q];
    }
    sink.flush();
    if (!kTfOnly) add_param_grads(dp, B.dparams);
}

// Brick-synchronous variant of the reverse sweep. Phase 1 (the forward
// re-march) is per lane as above. In phase 2 the warp repeatedly picks the
// farthest brick (largest per-axis brick distance from the eye) that a lane's
// next reverse sample lies in; the lanes in that brick sweep their samples in
// it back to front, adding voxel gradients into a 12^3 shared-memory block with
// shared-memory atomics; the warp then adds the touched part of the block to the
// global gradient and clears it. Each lane still sweeps its own samples in
// strictly decreasing order, so every sample sees exactly the arithmetic of
// k_render_backward; only the order of the floating-point additions into the
// voxel gradient differs.
__device__ __forceinline__ unsigned far_key(const int b[3], const int e[3]) {
    const unsigned dx = min(abs(b[0] - e[0]), 1023), dy = min(abs(b[1] - e[1]), 1023), dz = min(abs(b[2] - e[2]), 1023);
    return (dz << 20) | (dy << 10) | dx;
}

template <bool k2D>
__global__ void __launch_bounds__(128) k_render_backward_staged(const __grid_constant__ BackwardLaunch B) {
    extern __shared__ float smem[];
    const RenderLaunch& L = B.r;
    const size_t ncell = (size_t)L.tp.tf_w * L.tp.tf_h * kTfCellFloats;
    const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
    float* acc = smem + warp * kBrickVox;  // this warp's 12^3 block
    for (int e = l; e < kBrickVox; e += 32) acc[e] = 0.0f;
    __syncthreads();
    const int cta = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    TfGradSink<k2D> sink(B.dtf_copies + (size_t)(cta % B.n_copies) * ncell);
    const int i = blockIdx.x * 16 + (warp & 1) * 8 + (l & 7);
    const int j = blockIdx.y * 8 + (warp >> 1) * 4 + (l >> 3);
    const int cam = blockIdx.z;
    const bool inside = i < L.W && j < L.H;
    const VolumeDev& v = L.vol;
    const float4* tf = reinterpret_cast<const float4*>(L.tf);
    const float gmax = __ldg(&v.vc->gmax);
    const float inv_gmax = gmax > 0.0f ? 1.0f / gmax : 0.0f;
    const float is[3] = {1.0f / v.s[0], 1.0f / v.s[1], 1.0f / v.s[2]};
    const float et = fminf(L.tp.et_threshold, 1.0f);
    const CamDev& cd = L.cams[cam];
    int eb[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) eb[q] = (int)floorf((cd.eye[q] / v.s[q] - 0.5f) / (float)kCells);
    ParamGrad dp{0.f, 0.f, 0.f, 0.f, 0.f};

    RayDev r;
    bool live = inside && setup_ray(cd, L.rc, i, j, v.n, v.s, r);
    float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
    int kr = -1;
    float Tk = 1.0f, Tk1 = 1.0f, R0 = 0.f, R1 = 0.f, R2 = 0.f, P = 1.0f;
    int kstop = -1;
    if (live) {
        const long long pix = ((long long)(L.cam_offset + cam) * L.H + j) * L.W + i;
        g4 = __ldg(reinterpret_cast<const float4*>(B.dl_drgba) + pix);
        float A = 0.f, A_prev = 0.f;
        int k = 0, klast = -1;
        kstop = r.ns - 1;
        while (k < r.ns) {
            int i0[3], bc[3];
            float f[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                sample_cell(r, q, k, v.n[q], i0[q], f[q]);
                bc[q] = i0[q] >> 3;
            }
            if (!VR_CHECK(L.tp.status, (unsigned)i0[0] <= (unsigned)(v.n[0] - 2) &&
                                           (unsigned)i0[1] <= (unsigned)(v.n[1] - 2) &&
                                           (unsigned)i0[2] <= (unsigned)(v.n[2] - 2)))
                break;
            const int bi = bidx(v, bc);
            if (L.skip && __ldg(v.empty + bi)) {
                k = brick_exit_k(r, bc, kCells, k, r.ns);
                continue;
            }
            const int base = ((i0[2] - kCells * bc[2]) * kEdge + (i0[1] - kCells * bc[1])) * kEdge +
                             (i0[0] - kCells * bc[0]);
            float fld[10];
            field_eval(GLoad{v.bricks + (long long)bi * kBrickVox}, base, f[0], f[1], f[2], fld);
            scale_field(fld, is);
            const float vval = v.vbricks ? value_eval(GLoad{v.vbricks + (long long)bi * kBrickVox}, base, f[0], f[1], f[2]) : 0.f;
            float alpha, col[3];
            sample_optics(fld, vval, r.dir, L.tp, tf, inv_gmax, alpha, col);
            A_prev = A;
            A += (1.0f - A) * alpha;
            klast = k;
            if (A >= et) {
                kstop = k;
                break;
            }
            ++k;
        }
        Tk = (klast == kstop) ? 1.0f - A_prev : 1.0f - A;
        Tk1 = Tk;
        kr = kstop;
    }
    const float dC[3] = {g4.x, g4.y, g4.z};
    while (true) {
        // brick of this lane's next reverse sample
        int i0[3] = {0, 0, 0}, bc[3] = {0, 0, 0};
        float f[3] = {0.f, 0.f, 0.f};
        if (live) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                sample_cell(r, q, kr, v.n[q], i0[q], f[q]);
                bc[q] = i0[q] >> 3;
            }
        }
        const unsigned key = live ? far_key(bc, eb) + 1u : 0u;
        const unsigned mk = __reduce_max_sync(0xffffffffu, key);
        if (mk == 0u) break;
        const int leader = __ffs(__ballot_sync(0xffffffffu, key == mk)) - 1;
        int sc[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) sc[q] = __shfl_sync(0xffffffffu, bc[q], leader);
        int lo_t[3] = {kEdge, kEdge, kEdge}, hi_t[3] = {-1, -1, -1};  // touched local range
        if (live && bc[0] == sc[0] && bc[1] == sc[1] && bc[2] == sc[2]) {
            const int bi = bidx(v, sc);
            while (true) {
                const int base = ((i0[2] - kCells * sc[2]) * kEdge + (i0[1] - kCells * sc[1])) * kEdge +
                                 (i0[0] - kCells * sc[0]);
                // the 4^3 stencil and its adjoint touch base + a + 12 b + 144 c, a, b, c in [0, 3]
                if (!VR_CHECK(L.tp.status, base >= 0 && base + 3 * (1 + kEdge + kEdge * kEdge) < kBrickVox)) {
                    live = false;
                    break;
                }
                float fld[10];
                field_eval(GLoad{v.bricks + (long long)bi * kBrickVox}, base, f[0], f[1], f[2], fld);
                scale_field(fld, is);
                const float vval =
                    v.vbricks ? value_eval(GLoad{v.vbricks + (long long)bi * kBrickVox}, base, f[0], f[1], f[2]) : 0.f;
                SampleOptics so;
                optics_core(fld, vval, r.dir, L.tp, tf, inv_gmax, so);
                const float alpha = so.alpha, col[3] = {so.col[0], so.col[1], so.col[2]};
                if (kr != kstop) Tk = Tk1 / (1.0f - alpha);
                const float da = Tk * (fmaf(dC[0], col[0] - R0, fmaf(dC[1], col[1] - R1, dC[2] * (col[2] - R2))) +
                                       g4.w * P);
                const float ta = Tk * alpha;
                const float dc[3] = {ta * dC[0], ta * dC[1], ta * dC[2]};
                float dfs[10];
                sample_adjoint(fld, so, r.dir, L.tp, inv_gmax, da, dc, sink, dp, dfs);
                if (B.dvol) {
                    const int lx = i0[0] - kCells * sc[0], ly = i0[1] - kCells * sc[1], lz = i0[2] - kCells * sc[2];
                    lo_t[0] = min(lo_t[0], lx), lo_t[1] = min(lo_t[1], ly), lo_t[2] = min(lo_t[2], lz);
                    hi_t[0] = max(hi_t[0], lx + 3), hi_t[1] = max(hi_t[1], ly + 3), hi_t[2] = max(hi_t[2], lz + 3);
                    field_adjoint_scatter(dfs, is, f[0], f[1], f[2], [&](int a, int b, int c, float g) {
                        if (g != 0.0f) atomicAdd(acc + base + (c * kEdge + b) * kEdge + a, g);
                    });
                }
                R0 = fmaf(alpha, col[0], (1.0f - alpha) * R0);
                R1 = fmaf(alpha, col[1], (1.0f - alpha) * R1);
                R2 = fmaf(alpha, col[2], (1.0f - alpha) * R2);
                P *= (1.0f - alpha);
                Tk1 = Tk;
                if (--kr < 0) {
                    live = false;
                    break;
                }
                int b2[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    sample_cell(r, q, kr, v.n[q], i0[q], f[q]);
                    b2[q] = i0[q] >> 3;
                }
                if (b2[0] != sc[0] || b2[1] != sc[1] || b2[2] != sc[2]) break;
            }
        }
        if (B.dvol) {
            // add the touched box of the block to the global gradient (clamped voxel
            // indices: apron cells outside the volume belong to the edge voxel), clear it
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                lo_t[q] = __reduce_min_sync(0xffffffffu, lo_t[q]);
                hi_t[q] = __reduce_max_sync(0xffffffffu, hi_t[q]);
            }
            __syncwarp();
            if (hi_t[0] >= 0) {
                const int ex = hi_t[0] - lo_t[0] + 1, ey = hi_t[1] - lo_t[1] + 1, ez = hi_t[2] - lo_t[2] + 1;
                const int cnt = ex * ey * ez;
                const int nx = v.n[0], ny = v.n[1], nz = v.n[2];
                for (int e = l; e < cnt; e += 32) {
                    const int ax = lo_t[0] + e % ex, ay = lo_t[1] + (e / ex) % ey, az = lo_t[2] + e / (ex * ey);
                    const int o = (az * kEdge + ay) * kEdge + ax;
                    const float g = acc[o];
                    if (g != 0.0f) {
                        acc[o] = 0.0f;
                        const int x = min(max(kCells * sc[0] - 1 + ax, 0), nx - 1);
                        const int y = min(max(kCells * sc[1] - 1 + ay, 0), ny - 1);
                        const int z = min(max(kCells * sc[2] - 1 + az, 0), nz - 1);
                        atomicAdd(B.dvol + ((long long)z * ny + y) * nx + x, g);
                    }
                }
            }
            __syncwarp();
        }
    }
    sink.flush();
    add_param_grads(dp, B.dparams);
}

// dtf[e] += the sum over copies [16 g, 16 g + 16) of entry e's share of the cells
// around it, one thread per (float e, g): enough threads for a small table with many
// copies (dtf is zeroed before). Entry (j, k) is corner 00 of cell (j, k), 01 of
// (j - 1, k), 10 of (j, k - 1) and 11 of (j - 1, k - 1), where those cells exist (a
// cell's j < w - 1 and, in a 2D table, k < h - 1); in a cell record the opacity of
// corner q is float q, its RGB floats 4 + 3 q .. 6 + 3 q (1D: 2 + 3 q .. 4 + 3 q).
constexpr int kCopiesPerThread = 16;
// The first five threads also round the uniform gradients' double sums.
__global__ void __launch_bounds__(256) k_sum_copies(const float* __restrict__ copies, int n_copies, int w, int h,
                                                   float* __restrict__ out, const double* __restrict__ dparams,
                                                   float* __restrict__ out_params) {
    if (out_params && blockIdx.x == 0 && threadIdx.x < 5) out_params[threadIdx.x] = (float)dparams[threadIdx.x];
    const long long n = 4ll * w * h;
    const long long stride = (long long)w * h * kTfCellFloats;
    const long long groups = (n_copies + kCopiesPerThread - 1) / kCopiesPerThread;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n * groups;
         t += (long long)gridDim.x * blockDim.x) {
        const long long e = t % n;
        const int ch = (int)(e & 3), entry = (int)(e >> 2), j = entry % w, k = entry / w;
        const int c0 = (int)(t / n) * kCopiesPerThread;
        const int c1 = min(c0 + kCopiesPerThread, n_copies);
        // (cell key, float in its record) of each corner this entry is
        int off[4], m = 0;
        const bool kin = h == 1 || k < h - 1;  // row k holds cells
        auto slot = [&](int q) { return ch == 3 ? q : (h > 1 ? 4 : 2) + 3 * q + ch; };
        if (j < w - 1 && kin) off[m++] = entry * kTfCellFloats + slot(0);
        if (j >= 1 && kin) off[m++] = (entry - 1) * kTfCellFloats + slot(1);
        if (h > 1 && k >= 1 && j < w - 1) off[m++] = (entry - w) * kTfCellFloats + slot(2);
        if (h > 1 && k >= 1 && j >= 1) off[m++] = (long long)(entry - w - 1) * kTfCellFloats + slot(3);
        float acc = 0.0f;
        for (int c = c0; c < c1; ++c)
            for (int u = 0; u < m; ++u) acc += __ldg(copies + (size_t)c * stride + off[u]);
        if (acc != 0.0f) atomicAdd(out + e, acc);
    }
}

}  // namespace

cudaError_t launch_channels_to_voxels(const float* dgrad, const int n[3], const float s[3], float* dvol,
                                      cudaStream_t st) {
    const unsigned tx = (n[0] + 31) / 32, ty = (n[1] + kVoxTileY - 1) / kVoxTileY;
    const int planes = march_planes((long long)tx * ty, n[2], 4, 12);
    k_channels_to_voxels<<<dim3(tx, ty, (n[2] + planes - 1) / planes), 256, 0, st>>>(dgrad, n[0], n[1], n[2], s[0],
                                                                                   s[1], s[2], planes, dvol);
    return cudaGetLastError();
}

cudaError_t launch_sum_copies(const float* copies, int n_copies, int tf_w, int tf_h, float* dtf,
                              const double* dparams, float* out_params, cudaStream_t st) {
    const long long n = 4ll * tf_w * tf_h;
    const long long blocks = (n * ((n_copies + kCopiesPerThread - 1) / kCopiesPerThread) + 255) / 256;
    k_sum_copies<<<(unsigned)(blocks < kSMs * 8 ? blocks : kSMs * 8), 256, 0, st>>>(copies, n_copies, tf_w, tf_h,
                                                                               dtf, dparams, out_params);
    return cudaGetLastError();
}

template <bool k2D, int kBS>
void launch_backward_bs(const BackwardLaunch& B, dim3 grid, cudaStream_t st) {
    const RenderLaunch& L = B.r;
    const bool tf_only = !B.dparams && !B.dvol && !B.dgrad;
    if (!L.vol.dbricks)
        k_render_backward<false, false, false, false, k2D, kBS><<<grid, 128, 0, st>>>(B);
    else if (L.tp.gk == 0.0f && tf_only)
        k_render_backward<true, true, true, true, k2D, kBS><<<grid, 128, 0, st>>>(B);
    else if (L.tp.gk == 0.0f && !B.dparams)
        k_render_backward<true, true, true, false, k2D, kBS><<<grid, 128, 0, st>>>(B);
    else if (L.tp.gk == 0.0f)
        k_render_backward<true, true, false, false, k2D, kBS><<<grid, 128, 0, st>>>(B);
    else if (tf_only)
        k_render_backward<true, false, false, true, k2D, kBS><<<grid, 128, 0, st>>>(B);
    else
        k_render_backward<true, false, false, false, k2D, kBS><<<grid, 128, 0, st>>>(B);
}

template <bool k2D>
void launch_backward_table(const BackwardLaunch& B, dim3 grid, cudaStream_t st) {
    switch (B.r.vol.bs) {
        case 2: launch_backward_bs<k2D, 2>(B, grid, st); break;
        case 4: launch_backward_bs<k2D, 4>(B, grid, st); break;
        default: launch_backward_bs<k2D, 3>(B, grid, st); break;
    }
}

template <bool k2D, int kBS>
void launch_backward_lanes_bs(const BackwardLaunch& B, dim3 grid, cudaStream_t st) {
    const bool tf_only = !B.dparams && !B.dvol && !B.dgrad;
    if (B.r.tp.gk == 0.0f && tf_only)
        k_backward_lanes<true, true, true, k2D, kBS><<<grid, 128, 0, st>>>(B);
    else if (B.r.tp.gk == 0.0f && !B.dparams)
        k_backward_lanes<true, true, false, k2D, kBS><<<grid, 128, 0, st>>>(B);
    else if (B.r.tp.gk == 0.0f)
        k_backward_lanes<true, false, false, k2D, kBS><<<grid, 128, 0, st>>>(B);
    else if (tf_only)
        k_backward_lanes<false, false, true, k2D, kBS><<<grid, 128, 0, st>>>(B);
    else
        k_backward_lanes<false, false, false, k2D, kBS><<<grid, 128, 0, st>>>(B);
}

template <bool k2D>
void launch_backward_lanes(const BackwardLaunch& B, dim3 grid, cudaStream_t st) {
    switch (B.r.vol.bs) {
        case 2: launch_backward_lanes_bs<k2D, 2>(B, grid, st); break;
        case 4: launch_backward_lanes_bs<k2D, 4>(B, grid, st); break;
        default: launch_backward_lanes_bs<k2D, 3>(B, grid, st); break;
    }
}

// Lanes per ray of a backward launch with that many rays. One lane per ray fills the
// chip at 152 SMs x 16 warps x 32 = 78 k rays. Forward + backward with every gradient,
// measured us at 1 / 2 / 4 / 8 / 16 lanes (128^3 head, 1D table; 181x217x181 head, 2D):
//    64 x 64    1017 / 541 / 366 / 285 / 252     96 x 96   1886 / 1095 /  834 /  739 /  732
//   128 x 128    854 / 522 / 393 / 387 / 412    160 x 160  1870 / 1233 / 1102 / 1023 / 1058
//   256 x 256    864 / 820 / 800 / 886 / 1069   256 x 256  2394 / 1850 / 1694 / 1716 / 1889
//   384 x 384   1217 / 1370 / 1462 / 1679       400 x 300  2621 / 2118 / 2018 / 2126
int backward_lanes(long long rays) {
    return rays <= 6000 ? 16 : rays <= 28000 ? 8 : rays <= 90000 ? 4 : rays <= 122880 ? 2 : 1;
}

// Shape of a launch with several lanes per ray: rays per warp across and down.
dim3 lanes_shape(RenderLaunch& L, int lanes) {
    const int rays = 32 / lanes;
    L.lanes = lanes;
    L.packet_w = rays >= 8 ? 4 : (rays >= 4 ? 2 : 1);
    L.packet_h = rays / L.packet_w;
    return dim3((L.W + 4 * L.packet_w - 1) / (4 * L.packet_w), (L.H + L.packet_h - 1) / L.packet_h, L.n_cams);
}

cudaError_t launch_render_backward(const BackwardLaunch& B, bool staged, cudaStream_t st) {
    const RenderLaunch& L = B.r;
    const int lanes = backward_lanes((long long)L.W * L.H * L.n_cams);
    if (lanes > 1 && !staged && L.ray_state && L.vol.dbricks) {
        BackwardLaunch C = B;
        const dim3 shape = lanes_shape(C.r, lanes);
        if (L.tp.tf_h > 1)
            launch_backward_lanes<true>(C, shape, st);
        else
            launch_backward_lanes<false>(C, shape, st);
        return cudaGetLastError();
    }
    dim3 grid((L.W + 15) / 16, (L.H + 7) / 8, L.n_cams);
    if (staged) {
        const int smem = 4 * kBrickBytes;
        auto kernel = L.tp.tf_h > 1 ? k_render_backward_staged<true> : k_render_backward_staged<false>;
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        kernel<<<grid, 128, smem, st>>>(B);
        return cudaGetLastError();
    }
    if (L.tp.tf_h > 1)
        launch_backward_table<true>(B, grid, st);
    else
        launch_backward_table<false>(B, grid, st);
    return cudaGetLastError();
}

}  // namespace vr
