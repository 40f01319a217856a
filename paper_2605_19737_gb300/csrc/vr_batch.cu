// vr_batch.cu -- batched persistent forward raymarch over many views (uneven
// volumes x cameras) from one work queue, one launch (optionally graph-captured).
#include "vr_march.cuh"

namespace vr {

namespace {

// Batched persistent renderer: every warp pulls packet_w x packet_h ray packets
// from one work queue spanning all views (each view: its own volume, uniforms,
// transfer function, camera, output and size). A packet's view is found by
// binary search over the views' packet prefix sums. kAllDerived: every view's
// volume has derived bricks, so only that path is compiled in and the kernel is
// held to 72 registers (measured: 110 Gsamples/s on the 256-view batch, against
// 102 at 64 registers); otherwise each view takes its own path at run time.
template <bool kAllDerived, bool kCount, int kBS>
__device__ __forceinline__ void batch_body(const BatchLaunch& B) {
    const int lane = threadIdx.x & 31;
    unsigned rays_hit = 0, dense_tot = 0, eval_tot = 0, shade_tot = 0, interp_tot = 0;
    while (true) {
        unsigned item = 0;
        if (lane == 0) item = atomicAdd(B.work_counter, 1u);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= (unsigned)B.n_work) break;
        int lo = 0, hi = B.n_views - 1;  // last view with prefix <= item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((unsigned)__ldg(B.packet_prefix + mid) <= item) lo = mid;
            else hi = mid - 1;
        }
        const ViewDev& vw = B.views[lo];
        const int local = (int)item - __ldg(B.packet_prefix + lo);
        const int npx = (vw.W + B.packet_w - 1) / B.packet_w;
        const int px = local % npx, py = local / npx;
        if (!VR_CHECK(vw.tp.status, local >= 0 && py * B.packet_h < vw.H)) continue;
        const int i = px * B.packet_w + lane % B.packet_w, j = py * B.packet_h + lane / B.packet_w;
        const bool inside = i < vw.W && j < vw.H;
        const VolumeDev& v = vw.vol;
        const float gmax = __ldg(&v.vc->gmax);
        const float inv_gmax = gmax > 0.0f ? 1.0f / gmax : 0.0f;
        const float is[3] = {1.0f / v.s[0], 1.0f / v.s[1], 1.0f / v.s[2]};
        RayDev r;
        const bool hit = inside && setup_ray(vw.cam, vw.rc, i, j, v.n, v.s, r);
        float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
        unsigned dense = 0, evald = 0, shaded = 0, interp = 0;
        if (!hit) r.ns = 0;
        const float4* tf = reinterpret_cast<const float4*>(vw.tf);
        if (kAllDerived || v.dbricks) {
            if (kCount)
                march_count<true, false, kBS>(v, vw.tp, tf, r, B.skip, inv_gmax, is, out, dense, evald, shaded, interp);
            else
                march_ahead<true, kBS>(v, vw.tp, tf, r, B.skip, inv_gmax, is, out);
        } else {
            if (kCount)
                march_count<false, false, kBS>(v, vw.tp, tf, r, B.skip, inv_gmax, is, out, dense, evald, shaded, interp);
            else
                march_ahead<false, kBS>(v, vw.tp, tf, r, B.skip, inv_gmax, is, out);
        }
        if (inside) reinterpret_cast<float4*>(vw.out)[(long long)j * vw.W + i] = out;
        if (kCount) {
            rays_hit += hit ? 1u : 0u;
            dense_tot += dense;
            eval_tot += evald;
            shade_tot += shaded;
            interp_tot += interp;
        }
    }
    if (kCount && B.counters) add_counters(B.counters, rays_hit, dense_tot, eval_tot, 0u, shade_tot, interp_tot);
}

// kBS: the skip-brick size shared by every view, or 0 when the views mix sizes.
// kFew: a batch of few packets takes 128 registers, for more loads in flight per warp: the
// three planes of the derived bricks cost a sparse ray twice the lines that records did, and
// the warps wait for them. The line (batch_few) lies at 28 packets per SM without curvature,
// which reads one plane of the three, and at 170 with it (181x217x181 head, us at 72 -> 128
// registers, by packets per SM; with curvature 64^2 (0.8) 1686 -> 770, 400x300 (25) 791 -> 550,
// 16 views of 130x100 (43) 2062 -> 1275, of 260x200 (171) 2849 -> 2583, of 400x300 (395) 4150 ->
// 4270; without 64^2 478 -> 347, 400x300 408 -> 348, 430^2 (38) 422 -> 486).
template <bool kCount, bool kFew, int kBS>
__global__ void __maxnreg__(kFew ? 128 : 72) k_render_batch_derived(const __grid_constant__ BatchLaunch B) {
    batch_body<true, kCount, kBS>(B);
}

template <bool kCount>
__global__ void __launch_bounds__(256, 3) k_render_batch_mixed(const __grid_constant__ BatchLaunch B) {
    batch_body<false, kCount, 0>(B);
}

template <bool kCount, bool kFew>
void launch_derived(const BatchLaunch& B, int ctas, int threads, int bs, cudaStream_t st) {
    if (bs == 2)
        k_render_batch_derived<kCount, kFew, 2><<<ctas, threads, 0, st>>>(B);
    else if (bs == 3)
        k_render_batch_derived<kCount, kFew, 3><<<ctas, threads, 0, st>>>(B);
    else if (bs == 4)
        k_render_batch_derived<kCount, kFew, 4><<<ctas, threads, 0, st>>>(B);
    else
        k_render_batch_derived<kCount, kFew, 0><<<ctas, threads, 0, st>>>(B);
}

template <bool kCount>
void launch_variant(const BatchLaunch& B, int ctas, int threads, BatchKind kind, int bs, cudaStream_t st) {
    if (kind == BatchKind::kMixed)
        k_render_batch_mixed<kCount><<<ctas, threads, 0, st>>>(B);
    else if (kind == BatchKind::kFew)
        launch_derived<kCount, true>(B, ctas, threads, bs, st);
    else
        launch_derived<kCount, false>(B, ctas, threads, bs, st);
}

}  // namespace

BatchKind batch_kind(int packets, bool all_derived, bool curved) {
    if (!all_derived) return BatchKind::kMixed;
    return packets <= (curved ? 170 : 28) * kSMs ? BatchKind::kFew : BatchKind::kMany;
}

cudaError_t batch_ctas_per_sm(int warps_per_block, BatchKind kind, int* per_sm) {
    // every variant of a kind is held to the same registers, so one answers for all
    auto kernel = kind == BatchKind::kMixed ? k_render_batch_mixed<false>
                  : kind == BatchKind::kFew ? k_render_batch_derived<false, true, 3>
                                            : k_render_batch_derived<false, false, 3>;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kernel, warps_per_block * 32, 0);
}

cudaError_t launch_render_batch(const BatchLaunch& B, int warps_per_block, int ctas, BatchKind kind, int bs,
                                cudaStream_t st) {
    if (B.counters || !B.skip)  // without skipping there is nothing to look ahead for either
        launch_variant<true>(B, ctas, warps_per_block * 32, kind, bs, st);
    else
        launch_variant<false>(B, ctas, warps_per_block * 32, kind, bs, st);
    return cudaGetLastError();
}

}  // namespace vr
