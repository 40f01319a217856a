// vr_march.cuh -- the per-lane front-to-back march of one ray (Sec. 2.4, Eqs. 4-6)
// over the bricked volume, shared by the single-view and batched forward kernels.
#pragma once

#include "vr_sample.cuh"

namespace vr {

struct GlobalLoad {
    const float* __restrict__ p;
    __device__ __forceinline__ float operator()(int o) const { return __ldg(p + o); }
};

// Skip-brick id in 32-bit arithmetic: dims <= 2048 give at most 512^3 = 2^27 bricks.
__device__ __forceinline__ int brick_index(const VolumeDev& v, const int b[3]) {
    return (b[2] * v.nb[1] + b[1]) * v.nb[0] + b[0];
}


__device__ __forceinline__ void add_counters(vr_counters* ctr, unsigned rays, unsigned dense, unsigned evald,
                                             unsigned staged, unsigned shaded, unsigned interp) {
    const unsigned r = __reduce_add_sync(0xffffffffu, rays);
    const unsigned d = __reduce_add_sync(0xffffffffu, dense);
    const unsigned e = __reduce_add_sync(0xffffffffu, evald);
    const unsigned s = __reduce_add_sync(0xffffffffu, staged);
    const unsigned h = __reduce_add_sync(0xffffffffu, shaded);
    const unsigned ip = __reduce_add_sync(0xffffffffu, interp);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&ctr->rays, (unsigned long long)r);
        atomicAdd(&ctr->dense_samples, (unsigned long long)d);
        atomicAdd(&ctr->evaluated_samples, (unsigned long long)e);
        atomicAdd(&ctr->bricks_staged, (unsigned long long)s);
        atomicAdd(&ctr->shaded_samples, (unsigned long long)h);
        atomicAdd(&ctr->interpolated_samples, (unsigned long long)ip);
    }
}

// Opacity and colour of the sample at fractions f of cell i0. False when its
// transfer-function opacity is exactly zero (derived path): it adds nothing.
// The Hessian loads are issued before that test so that they overlap the table lookup
// (measured: equal at 1080p, 2-3 % faster on the 8-view and batched workloads than
// loading them after it).
template <bool kDerived, int kBS>
__device__ __forceinline__ bool eval_sample(const VolumeDev& v, const TissueDev& tp, const float4* __restrict__ tf,
                                            const float f[3], const int i0[3], const float dir[3],
                                            float inv_gmax, const float is[3], float& alpha, float col[3]) {
    int base = 0, sbi = 0;
    if (!kDerived || v.vbricks) sbi = storage_brick(v, i0, base);
    const float vval =
        v.vbricks ? value_eval(GlobalLoad{v.vbricks + (size_t)sbi * kBrickVox}, base, f[0], f[1], f[2]) : 0.0f;
    float fld[10];
    if (kDerived) {
        // derived brick of the cell, and the cell's place in it; I and the gradient (one
        // load per corner), the Hessian (two), then the transfer function
        const int bs = kBS ? kBS : v.bs, B = 1 << bs;
        const DerLayout dl = kBS ? der_layout(kBS) : v.der;
        const int bc[3] = {i0[0] >> bs, i0[1] >> bs, i0[2] >> bs};
        const float4* dbrick = reinterpret_cast<const float4*>(
            v.dbricks + (size_t)(unsigned)brick_index(v, bc) * (unsigned)(kBS ? der_brick_floats(kBS) : v.der_stride));
        const int lx = i0[0] & (B - 1), ly = i0[1] & (B - 1), lz = i0[2] & (B - 1);
        derived_channels<false, 0, 4>(dbrick, dl, lx, ly, lz, f[0], f[1], f[2], fld);
        load_hessian<false>(tp, dbrick, dl, lx, ly, lz, f, fld);
        SampleOptics o;
        optics_tf(fld, vval, tp, tf, inv_gmax, o);
        if (o.c.w == 0.0f) return false;
        optics_rest(fld, dir, tp, o);
        alpha = o.alpha;
        col[0] = o.col[0];
        col[1] = o.col[1];
        col[2] = o.col[2];
    } else {
        field_eval(GlobalLoad{v.bricks + (size_t)sbi * kBrickVox}, base, f[0], f[1], f[2], fld);
        scale_field(fld, is);
        sample_optics(fld, vval, dir, tp, tf, inv_gmax, alpha, col);
    }
    return true;
}

// Front-to-back march of one ray (Eqs. 4-6) over the bricked volume in HBM/L2.
// Shared by the single-view and batched kernels.
// Empty space: a sample whose cell is empty under the transfer function has opacity
// exactly 0 (its intensity lies in the range of the cell's 8 corners) and adds nothing.
// The skip field holds, per cell, the distance to the nearest cell that may have
// opacity, so one byte load both tests the cell and leaps over empty space; it needs no
// brick state in registers. With skip the volume has a field.
// The lanes of a warp walk in step: all at the same sample index k, advancing together
// by the smallest leap any lane may take. Neighbouring rays then sit at the same
// depth and their corner loads share cells; a lane that leapt alone would lose step for
// the rest of its ray. Measured (1080p of the 181x217x181 head / vessel 256x256x176 at
// 1080p / 540p of the head): single steps over empty cells inside bricks 2.15 / 0.367 /
// 0.811 ms, each lane leaping for itself 2.16 / 0.134 / 0.90, warps in step 1.81 / 0.130
// / 0.72. Bound by latency: ~0.45 issue slots used, two L1 round trips (byte, corners)
// and the table's per sample.
// With kState it also returns the ray's last sample index (kstop) and the
// transmittance in front of that sample (t_last), which the adjoint sweep starts from.
// kBS: log2 of the skip-brick edge in cells, fixed at compile time (2, 3, 4), or 0 to
// take the volume's at run time (batches that mix sizes); a fixed size keeps the
// brick and cell index arithmetic in immediates (the run-time form measured 4-10 %
// slower).
// Called by whole warps; a lane without a ray passes r.ns = 0.
constexpr unsigned kRayEnded = 0x7fffffffu;  // above any advance
template <bool kDerived, bool kState, int kBS>
__device__ __forceinline__ void march_gather(const VolumeDev& v, const TissueDev& tp, const float4* __restrict__ tf,
                                             const RayDev& r, int skip, float inv_gmax, const float is[3],
                                             float4& out, int* klast_out, float* t_last) {
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, A = 0.f;
    float A_prev = 0.f;  // kState: A before the last evaluated sample
    int klast = -1;      // kState: last evaluated sample
    int k1 = -1;         // kState: first sample with A >= 1 (where the adjoint sweep must start
    float T1 = 1.f;      // when early termination is off) and the transmittance in front of it
    int k = 0;
    // the position of sample k, u0 + k du, carried by exact integer additions
    long long U[3] = {r.u0[0], r.u0[1], r.u0[2]};
    auto step = [&]() {
#pragma unroll
        for (int q = 0; q < 3; ++q) U[q] += r.du[q];
        ++k;
    };
    auto leap = [&](int m) {
#pragma unroll
        for (int q = 0; q < 3; ++q) U[q] += (long long)m * r.du[q];
        k += m;
    };
    int ns = r.ns;  // samples of this ray, cut to the stopping one when it terminates early
    while (true) {
        int i0[3] = {0, 0, 0};
        unsigned adv = kRayEnded;
        if (k < ns) {
#pragma unroll
            for (int q = 0; q < 3; ++q) i0[q] = cell_index_at(U[q], v.n[q]);
            adv = 0u;
            if (!VR_CHECK(tp.status, (unsigned)i0[0] <= (unsigned)(v.n[0] - 2) &&
                                         (unsigned)i0[1] <= (unsigned)(v.n[1] - 2) &&
                                         (unsigned)i0[2] <= (unsigned)(v.n[2] - 2)))
                adv = 1u;
            else if (skip)
                adv = __ldg(v.skipf + skip_index(i0[0], i0[1], i0[2], v.skip_cx, v.skip_by));
        }
        const unsigned m = __reduce_min_sync(0xffffffffu, adv);  // a distance in cells
        if (m) {
            if (m == kRayEnded) break;
            leap((int)((float)(m - 1u) * tp.leap_per_cell) + 1);
            continue;
        }
        if (adv) {
            step();
            continue;
        }
        float alpha, col[3], f[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) f[q] = cell_frac_at(U[q], v.n[q]);
        if (!eval_sample<kDerived, kBS>(v, tp, tf, f, i0, r.dir, inv_gmax, is, alpha, col)) {
            step();
            continue;
        }
        const float wgt = (1.0f - A) * alpha;  // Eqs. 5-6
        fma2v(col[0], col[1], wgt, wgt, C0, C1);
        C2 = fmaf(col[2], wgt, C2);
        if (kState) {
            A_prev = A;
            klast = k;
        }
        A += wgt;
        if (kState && k1 < 0 && A >= 1.0f) {
            k1 = k;
            T1 = 1.0f - A_prev;
        }
        if (A >= tp.et_threshold) {
            ns = k + 1;
        }
        step();
    }
    out = make_float4(C0, C1, C2, A);
    if (kState) {
        // the adjoint sweep starts at the first sample with A >= min(et, 1): the stopping
        // sample, or (early termination off) the first that made A reach 1
        const int kl = ns - 1;
        *klast_out = k1 >= 0 ? k1 : kl;
        *t_last = k1 >= 0 ? T1 : ((klast == kl) ? 1.0f - A_prev : 1.0f - A);  // samples after klast: alpha 0
    }
}

// The same march, the same image and ray state, for launches that want sample counters or
// whose volume has no skip field. Evaluated samples are defined by the skip bricks (samples
// outside bricks classified empty), so a lane walks brick by brick and sample by sample, and
// leaps over empty bricks by itself. With a curvature term the lanes with the lowest sample index
// go first, so that those that have left an empty brick are waited for and the corner loads share
// cells; without one a sample is too cheap to wait for (counted, us each for itself / lowest
// first: 181x217x181 head with curvature 430^2 737 / 696, by stencils 256^2 520 / 421; 128^3 head
// without 960x540 233 / 267). Called by whole warps.
template <bool kDerived, bool kState, int kBS>
__device__ __forceinline__ void march_count(const VolumeDev& v, const TissueDev& tp, const float4* __restrict__ tf,
                                            const RayDev& r, int skip, float inv_gmax, const float is[3], float4& out,
                                            unsigned& dense, unsigned& evald, unsigned& shaded, unsigned& interp,
                                            int* klast_out = nullptr, float* t_last = nullptr) {
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, A = 0.f, A_prev = 0.f, T1 = 1.f;
    int klast = -1, k1 = -1, k = 0, ns = r.ns;
    unsigned ne = 0, nsh = 0, nip = 0;
    const int bs = kBS ? kBS : v.bs;
    int cur = -1;  // the brick whose flag `empty` is
    bool empty = false;
    long long U[3] = {r.u0[0], r.u0[1], r.u0[2]};
    auto advance = [&](int m) {
#pragma unroll
        for (int q = 0; q < 3; ++q) U[q] += m == 1 ? r.du[q] : (long long)m * r.du[q];
        k += m;
    };
    const bool in_order = tp.gk != 0.0f;
    while (true) {
        if (in_order) {
            const unsigned mine = k < ns ? (unsigned)k : kRayEnded, low = __reduce_min_sync(0xffffffffu, mine);
            if (low == kRayEnded) break;
            if (mine != low) continue;
        } else if (k >= ns) {
            break;
        }
        int i0[3], bc[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            i0[q] = cell_index_at(U[q], v.n[q]);
            bc[q] = i0[q] >> bs;
        }
        if (!VR_CHECK(tp.status, (unsigned)bc[0] < (unsigned)v.nb[0] && (unsigned)bc[1] < (unsigned)v.nb[1] &&
                                     (unsigned)bc[2] < (unsigned)v.nb[2])) {
            advance(1);
            continue;
        }
        if (skip) {
            const int bi = brick_index(v, bc);
            if (bi != cur) {
                cur = bi;
                empty = __ldg(v.empty + bi) != 0;
            }
            if (empty) {
                advance(brick_exit_k_at(r, U, bc, 1 << bs, k, ns) - k);
                continue;
            }
            if (v.skipf && __ldg(v.skipf + skip_index(i0[0], i0[1], i0[2], v.skip_cx, v.skip_by))) {
                ++ne;
                advance(1);
                continue;
            }
        }
        ++nip;
        ++ne;
        float alpha, col[3], f[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) f[q] = cell_frac_at(U[q], v.n[q]);
        if (eval_sample<kDerived, kBS>(v, tp, tf, f, i0, r.dir, inv_gmax, is, alpha, col)) {
            ++nsh;
            const float wgt = (1.0f - A) * alpha;  // Eqs. 5-6
            fma2v(col[0], col[1], wgt, wgt, C0, C1);
            C2 = fmaf(col[2], wgt, C2);
            if (kState) {
                A_prev = A;
                klast = k;
            }
            A += wgt;
            if (kState && k1 < 0 && A >= 1.0f) {
                k1 = k;
                T1 = 1.0f - A_prev;
            }
            if (A >= tp.et_threshold) ns = k + 1;
        }
        advance(1);
    }
    out = make_float4(C0, C1, C2, A);
    dense = (unsigned)ns;
    evald = ne;
    shaded = nsh;
    interp = nip;
    if (kState) {  // as march_gather
        const int kl = ns - 1;
        *klast_out = k1 >= 0 ? k1 : kl;
        *t_last = k1 >= 0 ? T1 : ((klast == kl) ? 1.0f - A_prev : 1.0f - A);
    }
}

// march_gather without counters or ray state, for the batch kernel: the byte of the next
// sample's cell is loaded before this sample is evaluated, so that one of the dependent
// round trips per sample is hidden. 32 views of four heads without a curvature term 8.25 -> 7.87 ms, 8 views with one
// 2.31 -> 2.28 (a single 120x100 view 88 -> 90 us);
// the single-view kernels lose by it (1080p with curvature 1.876 -> 1.884 ms, skip bricks
// of edge 4 0.778 -> 0.787: those are bound by the L1 data stage, not by latency).
template <bool kDerived, int kBS>
__device__ __forceinline__ void march_ahead(const VolumeDev& v, const TissueDev& tp, const float4* __restrict__ tf,
                                            const RayDev& r, int skip, float inv_gmax, const float is[3],
                                            float4& out) {
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, A = 0.f;
    const int bs = kBS ? kBS : v.bs;
    long long U[3] = {r.u0[0], r.u0[1], r.u0[2]};
    int k = 0, ns = r.ns;
    auto leap = [&](int m) {
#pragma unroll
        for (int q = 0; q < 3; ++q) U[q] += (long long)m * r.du[q];
        k += m;
    };
    // how far the ray may advance from sample k (cells; samples when there is no field), 0
    // when the sample is to be evaluated
    auto look = [&]() -> unsigned {
        if (k >= ns) return kRayEnded;
        int i0[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) i0[q] = cell_index_at(U[q], v.n[q]);
        if (!VR_CHECK(tp.status, (unsigned)i0[0] <= (unsigned)(v.n[0] - 2) &&
                                     (unsigned)i0[1] <= (unsigned)(v.n[1] - 2) &&
                                     (unsigned)i0[2] <= (unsigned)(v.n[2] - 2)))
            return 1u;
        if (!skip) return 0u;
        if (v.skipf) return __ldg(v.skipf + skip_index(i0[0], i0[1], i0[2], v.skip_cx, v.skip_by));
        const int bc[3] = {i0[0] >> bs, i0[1] >> bs, i0[2] >> bs};
        return __ldg(v.empty + brick_index(v, bc)) ? (unsigned)(brick_exit_k_at(r, U, bc, 1 << bs, k, ns) - k) : 0u;
    };
    unsigned adv = look();
    while (true) {
        const unsigned m = __reduce_min_sync(0xffffffffu, adv);
        if (m) {
            if (m == kRayEnded) break;
            leap(v.skipf ? (int)((float)(m - 1u) * tp.leap_per_cell) + 1 : (int)m);
            adv = look();
            continue;
        }
        const bool here = adv == 0u;
        int i0[3];
        float f[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) cell_at(U[q], v.n[q], i0[q], f[q]);
        leap(1);
        adv = look();
        float alpha, col[3];
        if (!here || !eval_sample<kDerived, kBS>(v, tp, tf, f, i0, r.dir, inv_gmax, is, alpha, col)) continue;
        const float wgt = (1.0f - A) * alpha;  // Eqs. 5-6
        fma2v(col[0], col[1], wgt, wgt, C0, C1);
        C2 = fmaf(col[2], wgt, C2);
        A += wgt;
        if (A >= tp.et_threshold) {
            ns = k;
            adv = kRayEnded;
        }
    }
    out = make_float4(C0, C1, C2, A);
}

// The same march with G lanes per ray (G a power of two up to 32, the lanes of a ray
// consecutive): lane g evaluates sample kb + g, then the G samples are composited in
// order, every lane of the ray repeating the one sequence of operations of
// march_gather on the values it gets by shuffle -- the image is the same bit for bit.
// For launches with too few rays to fill the chip the time is the serial chain of one
// ray, and this shortens it by almost G (64^3 at 128x128: 90 -> 29 us at G = 8); a
// filled chip gains nothing and pays the shuffles (4 per sample slot).
template <bool kDerived, bool kState, int G, int kBS>
__device__ __forceinline__ void march_lanes(const VolumeDev& v, const TissueDev& tp, const float4* __restrict__ tf,
                                            const RayDev& r, int skip, float inv_gmax, const float is[3],
                                            float4& out, int* klast_out, float* t_last) {
    const int lane = threadIdx.x & 31, g = lane & (G - 1), first = lane & ~(G - 1);
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, A = 0.f;
    float A_prev = 0.f, T1 = 1.f;
    int klast = -1, k1 = -1, kb = 0, ns = r.ns;
    long long U[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) U[q] = r.u0[q] + (long long)g * r.du[q];
    while (true) {
        int i0[3] = {0, 0, 0};
        unsigned adv = kRayEnded;
        if (kb + g < ns) {
#pragma unroll
            for (int q = 0; q < 3; ++q) i0[q] = cell_index_at(U[q], v.n[q]);
            adv = 0u;
            if (!VR_CHECK(tp.status, (unsigned)i0[0] <= (unsigned)(v.n[0] - 2) &&
                                         (unsigned)i0[1] <= (unsigned)(v.n[1] - 2) &&
                                         (unsigned)i0[2] <= (unsigned)(v.n[2] - 2)))
                adv = 1u;
            else if (skip && v.skipf)
                adv = __ldg(v.skipf + skip_index(i0[0], i0[1], i0[2], v.skip_cx, v.skip_by));
        }
        const unsigned m = __reduce_min_sync(0xffffffffu, adv);
        int next = G;  // samples to move on
        if (m) {
            if (m == kRayEnded) break;
            // every sample up to kb + G - 1 is empty, and from the last of them a leap follows
            next = G - 1 + (int)((float)(m - 1u) * tp.leap_per_cell) + 1;
        } else {
            float alpha = 0.0f, col[3] = {0.f, 0.f, 0.f};
            bool shaded = false;
            if (adv == 0u) {
                float f[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) f[q] = cell_frac_at(U[q], v.n[q]);
                shaded = eval_sample<kDerived, kBS>(v, tp, tf, f, i0, r.dir, inv_gmax, is, alpha, col);
            }
            const unsigned live = __ballot_sync(0xffffffffu, shaded);
#pragma unroll
            for (int h = 0; h < G; ++h) {
                const int src = first + h;
                const float a = __shfl_sync(0xffffffffu, alpha, src);
                const float c0 = __shfl_sync(0xffffffffu, col[0], src), c1 = __shfl_sync(0xffffffffu, col[1], src),
                            c2 = __shfl_sync(0xffffffffu, col[2], src);
                if (((live >> src) & 1u) && kb + h < ns) {
                    const float wgt = (1.0f - A) * a;  // Eqs. 5-6
                    fma2v(c0, c1, wgt, wgt, C0, C1);
                    C2 = fmaf(c2, wgt, C2);
                    if (kState) {
                        A_prev = A;
                        klast = kb + h;
                    }
                    A += wgt;
                    if (kState && k1 < 0 && A >= 1.0f) {
                        k1 = kb + h;
                        T1 = 1.0f - A_prev;
                    }
                    if (A >= tp.et_threshold) ns = kb + h + 1;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) U[q] += (long long)next * r.du[q];
        kb += next;
    }
    out = make_float4(C0, C1, C2, A);
    if (kState) {
        const int kl = ns - 1;
        *klast_out = k1 >= 0 ? k1 : kl;
        *t_last = k1 >= 0 ? T1 : ((klast == kl) ? 1.0f - A_prev : 1.0f - A);
    }
}

}  // namespace vr
