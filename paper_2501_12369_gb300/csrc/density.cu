// Adaptive density control of the 3DGS optimisation pipeline the paper keeps (Sec. 4 block
// diagram): per-step statistics of the visible splats, then periodically clone, split and prune,
// and the opacity reset.
//
// Statistics (k_densify_stats): the view-space mean gradient in normalised device units
// (pixel gradient x (W/2, H/2)), its norm added to accum, 1 added to count, the largest screen
// radius kept -- for splats with radius > 0.
//
// Densification is a stable three-way stream compaction.  For every splat a fixed float32
// sequence decides: avg = accum / count; grow = avg >= threshold; split = grow and max scale >
// dense_scale; clone = grow and not split; a candidate survives the prune unless its opacity,
// screen radius or world scale crosses a limit (clones and children start with radius 0;
// children carry scales / div).  k_densify_count counts the survivors, kept clones and kept
// split parents of each block, k_densify_offsets scans the block counts, and k_densify_scatter
// writes, in index order within each segment, [survivors | clones | two children per split
// parent].  Survivors keep their Adam moments; clones and children start from zero.  Children's
// means are parent + R(q) (s * z) for the caller's standard-normal draws z.
#include <type_traits>

#include "kernels.cuh"

namespace darb {
namespace {

constexpr int kDenThreads = 256;
constexpr int kDenItems = 8;
constexpr int kDenTile = kDenThreads * kDenItems;

struct DenCfg {
    float thr, dense, min_op, max_screen, max_world, div, log_div;
};

struct Flags {
    bool surv, clone, split;  // survivor, kept clone, split parent with kept children
};

__device__ __forceinline__ bool survives(float opac, float smax, float radius, const DenCfg &c) {
    bool ok = opac >= c.min_op;
    if (c.max_screen > 0.0f) ok = ok && radius <= c.max_screen;
    if (c.max_world > 0.0f) ok = ok && smax <= c.max_world;
    return ok;
}

__device__ __forceinline__ Flags classify(int i, const float *__restrict__ scales, const float *__restrict__ opac,
                                          const float *__restrict__ accum, const float *__restrict__ count,
                                          const int *__restrict__ max_radius, const DenCfg &c) {
    const float cnt = count[i];
    const float avg = cnt > 0.0f ? __fdiv_rn(accum[i], cnt) : 0.0f;
    const float s0 = scales[3 * (size_t)i], s1 = scales[3 * (size_t)i + 1], s2 = scales[3 * (size_t)i + 2];
    const float smax = fmaxf(fmaxf(s0, s1), s2);
    const float o = opac[i];
    const bool grow = avg >= c.thr;
    const bool split = grow && smax > c.dense;
    const bool clone = grow && !split;
    Flags f;
    f.surv = !split && survives(o, smax, (float)max_radius[i], c);
    f.clone = clone && survives(o, smax, 0.0f, c);
    const float cmax = fmaxf(fmaxf(__fdiv_rn(s0, c.div), __fdiv_rn(s1, c.div)), __fdiv_rn(s2, c.div));
    f.split = split && survives(o, cmax, 0.0f, c);
    return f;
}

// 3 counts of up to kDenThreads packed in 10-bit fields of one word
__device__ __forceinline__ uint32_t pack(const Flags &f) {
    return (f.surv ? 1u : 0u) | (f.clone ? 1u << 10 : 0u) | (f.split ? 1u << 20 : 0u);
}

template <int NT>
__device__ __forceinline__ uint32_t block_scan_packed(uint32_t v, uint32_t *s_w, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < NT / 32 ? s_w[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < NT / 32) s_w[lane] = w;
    }
    __syncthreads();
    const uint32_t excl = (warp > 0 ? s_w[warp - 1] : 0u) + x - v;
    total = s_w[NT / 32 - 1];
    __syncthreads();
    return excl;
}

__global__ void __launch_bounds__(256)
k_densify_stats(const float4 *__restrict__ grad2d, const int *__restrict__ radius, int n, float half_w, float half_h,
                float *__restrict__ accum, float *__restrict__ count, int *__restrict__ max_radius) {
    pdl_entry();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const int r = radius[i];
    if (r <= 0) return;
    const float4 g = grad2d[3 * (size_t)i];
    const float gx = __fmul_rn(g.x, half_w), gy = __fmul_rn(g.y, half_h);
    const float norm = __fsqrt_rn(__fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)));
    accum[i] = __fadd_rn(accum[i], norm);
    count[i] = __fadd_rn(count[i], 1.0f);
    max_radius[i] = max(max_radius[i], r);
}

// Latency-bound (28 bytes a splat, 1M splats): two splats a thread, so that the whole set is in
// flight at once, and the three counts summed once per CTA.  24.8 us with a block scan per 256
// splats, 23 us with eight splats a thread and one sum, 15.2 us so.
constexpr int kCountThreads = 1024;
__global__ void __launch_bounds__(kCountThreads)
k_densify_count(int n, const float *__restrict__ scales, const float *__restrict__ opac,
                const float *__restrict__ accum, const float *__restrict__ count, const int *__restrict__ max_radius,
                DenCfg c, uint32_t *__restrict__ blk) {
    pdl_entry();
    __shared__ uint32_t s_c[3];
    if (threadIdx.x < 3) s_c[threadIdx.x] = 0;
    __syncthreads();
    uint32_t sum[3] = {0, 0, 0};
#pragma unroll
    for (int j = 0; j < kDenTile / kCountThreads; ++j) {
        const int i = blockIdx.x * kDenTile + j * kCountThreads + threadIdx.x;
        if (i < n) {
            const Flags f = classify(i, scales, opac, accum, count, max_radius, c);
            sum[0] += f.surv;
            sum[1] += f.clone;
            sum[2] += f.split;
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t w = __reduce_add_sync(0xffffffffu, sum[k]);
        if ((threadIdx.x & 31) == 0 && w) atomicAdd(&s_c[k], w);
    }
    __syncthreads();
    if (threadIdx.x < 3) blk[3 * (size_t)blockIdx.x + threadIdx.x] = s_c[threadIdx.x];
}

// One CTA: exclusive offsets of the three block counts; segment bases; n_out.
__global__ void __launch_bounds__(1024)
k_densify_offsets(int nb, uint32_t *__restrict__ blk, uint32_t *__restrict__ n_out) {
    pdl_entry();
    __shared__ uint32_t s_w[32];
    uint32_t carry[3] = {0, 0, 0};
    for (int f = 0; f < 3; ++f) {
        for (int c0 = 0; c0 < nb; c0 += 1024) {
            const int b = c0 + threadIdx.x;
            const uint32_t v = b < nb ? blk[3 * (size_t)b + f] : 0u;
            uint32_t tot;
            const uint32_t ex = block_scan_packed<1024>(v, s_w, tot);
            if (b < nb) blk[3 * (size_t)b + f] = carry[f] + ex;
            carry[f] += tot;
        }
    }
    if (threadIdx.x == 0) {
        n_out[0] = carry[0] + carry[1] + 2 * carry[2];
        n_out[1] = carry[0];             // clone segment starts here
        n_out[2] = carry[0] + carry[1];  // children start here
    }
}

struct DenIO {
    darb_train_params in, out;
    darb_adam_state sin, sout;
};

// Splats per scatter CTA: a quarter of a counted block, so that 1M splats give 1954 CTAs.
constexpr int kScatSplats = 512;
constexpr int kScatPer = kDenTile / kScatSplats;  // scatter CTAs per counted block
constexpr int kScatItems = kScatSplats / kDenThreads;
constexpr int kScatUnroll = 4;  // loads in flight per thread and array

// Rows [out0, out0 + rows) of dst from the rows i0 + list[r >> SHIFT] of src, W floats a row, by the
// whole CTA with consecutive lanes on consecutive words; 16-byte words where rows are multiples
// of 16 bytes and both arrays are aligned (the moments need not be).
template <int W, int SHIFT>
__device__ __forceinline__ void copy_rows(const float *__restrict__ src, float *__restrict__ dst, int i0, uint32_t out0,
                                          const uint16_t *list, int rows) {
    auto walk = [&](auto *s, auto *d, auto per) {
        constexpr int P = decltype(per)::value;
        const int total = rows * P;
        for (int b = threadIdx.x; b < total; b += kDenThreads * kScatUnroll) {
            typename std::remove_const<typename std::remove_reference<decltype(*s)>::type>::type v[kScatUnroll];
#pragma unroll
            for (int u = 0; u < kScatUnroll; ++u) {
                const int t = b + u * kDenThreads;
                if (t < total) {
                    const int r = t / P;
                    v[u] = s[(size_t)(i0 + list[r >> SHIFT]) * P + (t - r * P)];
                }
            }
#pragma unroll
            for (int u = 0; u < kScatUnroll; ++u) {
                const int t = b + u * kDenThreads;
                if (t < total) d[(size_t)out0 * P + t] = v[u];
            }
        }
    };
    if constexpr (W % 4 == 0) {
        if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0) {
            walk(reinterpret_cast<const float4 *>(src), reinterpret_cast<float4 *>(dst),
                 std::integral_constant<int, W / 4>{});
            return;
        }
    }
    walk(src, dst, std::integral_constant<int, W>{});
}

template <int W>
__device__ __forceinline__ void zero_rows(float *__restrict__ dst, uint32_t out0, int rows) {
    for (int t = threadIdx.x; t < rows * W; t += kDenThreads) dst[(size_t)out0 * W + t] = 0.0f;
}

template <int K3>
__device__ __forceinline__ void zero_moments(const darb_adam_state &s, uint32_t out0, int rows) {
    zero_rows<3>(s.m_means, out0, rows);
    zero_rows<3>(s.v_means, out0, rows);
    zero_rows<3>(s.m_scales, out0, rows);
    zero_rows<3>(s.v_scales, out0, rows);
    zero_rows<4>(s.m_quats, out0, rows);
    zero_rows<4>(s.v_quats, out0, rows);
    zero_rows<1>(s.m_opac, out0, rows);
    zero_rows<1>(s.v_opac, out0, rows);
    zero_rows<K3>(s.m_sh, out0, rows);
    zero_rows<K3>(s.v_sh, out0, rows);
}

// One CTA takes kScatSplats consecutive splats.  Its first output row in each segment is the
// counted block's offset plus the counts of the block's splats before it, which it classifies
// again (28 bytes a splat, mostly from L2; a table of finer offsets would need a larger
// workspace).  It lists its survivors, clones and split parents in shared memory; the rows of
// each list are consecutive in the output, so every array is then copied as one flat range.
// HBM-bound: with one thread copying each row, 32 lanes wrote 32 different rows at a time and the
// kernel took 1250 us (1M splats, SH degree 3, 1.46 GB), now 277 us (0.78 of the measured copy rate).
template <int K3>
__global__ void __launch_bounds__(kDenThreads)
k_densify_scatter(int n, DenIO io, const float *__restrict__ accum, const float *__restrict__ count,
                  const int *__restrict__ max_radius, const float *__restrict__ normals, DenCfg c,
                  const uint32_t *__restrict__ blk, const uint32_t *__restrict__ n_out) {
    pdl_entry();
    __shared__ uint32_t s_w[kDenThreads / 32];
    __shared__ uint32_t s_before[3];
    __shared__ uint16_t s_list[3][kScatSplats];
    const int block = blockIdx.x / kScatPer, sub = blockIdx.x % kScatPer;
    const int i0 = block * kDenTile + sub * kScatSplats;
    if (i0 >= n) return;  // uniform over the CTA
    if (threadIdx.x < 3) s_before[threadIdx.x] = blk[3 * (size_t)block + threadIdx.x];
    __syncthreads();
    uint32_t before[3] = {0, 0, 0};
    for (int j = 0; j < sub * kScatItems; ++j) {  // the block's splats before this CTA's (all below n)
        const Flags f = classify(block * kDenTile + j * kDenThreads + (int)threadIdx.x, io.in.scales, io.in.opacities,
                                 accum, count, max_radius, c);
        before[0] += f.surv;
        before[1] += f.clone;
        before[2] += f.split;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t w = __reduce_add_sync(0xffffffffu, before[k]);
        if ((threadIdx.x & 31) == 0 && w) atomicAdd(&s_before[k], w);
    }
    uint32_t cnt[3] = {0, 0, 0};
    for (int j = 0; j < kScatItems; ++j) {
        const int l = j * kDenThreads + (int)threadIdx.x, i = i0 + l;
        Flags f{false, false, false};
        if (i < n) f = classify(i, io.in.scales, io.in.opacities, accum, count, max_radius, c);
        uint32_t tot;
        const uint32_t ex = block_scan_packed<kDenThreads>(pack(f), s_w, tot);
        if (f.surv) s_list[0][cnt[0] + (ex & 1023u)] = (uint16_t)l;
        if (f.clone) s_list[1][cnt[1] + ((ex >> 10) & 1023u)] = (uint16_t)l;
        if (f.split) s_list[2][cnt[2] + (ex >> 20)] = (uint16_t)l;
        cnt[0] += tot & 1023u;
        cnt[1] += (tot >> 10) & 1023u;
        cnt[2] += tot >> 20;
    }
    __syncthreads();
    const darb_train_params &a = io.in, &b = io.out;
    auto params = [&](uint32_t out0, const uint16_t *list, int rows, auto shift) {  // what every copied row keeps
        constexpr int S = decltype(shift)::value;
        copy_rows<K3, S>(a.sh, b.sh, i0, out0, list, rows);
        copy_rows<4, S>(a.quats, b.quats, i0, out0, list, rows);
        copy_rows<1, S>(a.opacity_logits, b.opacity_logits, i0, out0, list, rows);
        copy_rows<1, S>(a.opacities, b.opacities, i0, out0, list, rows);
        if (S == 0) {  // children's are computed below
            copy_rows<3, S>(a.means, b.means, i0, out0, list, rows);
            copy_rows<3, S>(a.log_scales, b.log_scales, i0, out0, list, rows);
            copy_rows<3, S>(a.scales, b.scales, i0, out0, list, rows);
        }
    };
    const std::integral_constant<int, 0> one{};
    const std::integral_constant<int, 1> two{};
    if (cnt[0]) {  // survivors keep their moments
        const uint32_t o = s_before[0];
        const int rows = (int)cnt[0];
        const uint16_t *l = s_list[0];
        params(o, l, rows, one);
        copy_rows<K3, 0>(io.sin.m_sh, io.sout.m_sh, i0, o, l, rows);
        copy_rows<K3, 0>(io.sin.v_sh, io.sout.v_sh, i0, o, l, rows);
        copy_rows<3, 0>(io.sin.m_means, io.sout.m_means, i0, o, l, rows);
        copy_rows<3, 0>(io.sin.v_means, io.sout.v_means, i0, o, l, rows);
        copy_rows<3, 0>(io.sin.m_scales, io.sout.m_scales, i0, o, l, rows);
        copy_rows<3, 0>(io.sin.v_scales, io.sout.v_scales, i0, o, l, rows);
        copy_rows<4, 0>(io.sin.m_quats, io.sout.m_quats, i0, o, l, rows);
        copy_rows<4, 0>(io.sin.v_quats, io.sout.v_quats, i0, o, l, rows);
        copy_rows<1, 0>(io.sin.m_opac, io.sout.m_opac, i0, o, l, rows);
        copy_rows<1, 0>(io.sin.v_opac, io.sout.v_opac, i0, o, l, rows);
    }
    if (cnt[1]) {
        const uint32_t o = n_out[1] + s_before[1];
        params(o, s_list[1], (int)cnt[1], one);
        zero_moments<K3>(io.sout, o, (int)cnt[1]);
    }
    if (cnt[2]) {  // two children a parent
        const uint32_t o = n_out[2] + 2 * s_before[2];
        const int rows = 2 * (int)cnt[2];
        params(o, s_list[2], rows, two);
        zero_moments<K3>(io.sout, o, rows);
        for (int t = threadIdx.x; t < rows; t += kDenThreads) {
            const int i = i0 + s_list[2][t >> 1], ch = t & 1;
            const size_t r = (size_t)o + t;
            // rotation of the normalised quaternion (w, x, y, z)
            const float4 q = reinterpret_cast<const float4 *>(a.quats)[i];
            const float inv = rsqrtf(q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w);
            const float w = q.x * inv, x = q.y * inv, y = q.z * inv, z = q.w * inv;
            const float R[3][3] = {{1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y)},
                                   {2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x)},
                                   {2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)}};
            const float *zz = normals + (size_t)6 * i + 3 * ch;
            const float v[3] = {a.scales[3 * (size_t)i] * zz[0], a.scales[3 * (size_t)i + 1] * zz[1],
                                a.scales[3 * (size_t)i + 2] * zz[2]};
            for (int k = 0; k < 3; ++k) {
                b.means[3 * r + k] = a.means[3 * (size_t)i + k] + (R[k][0] * v[0] + R[k][1] * v[1] + R[k][2] * v[2]);
                const float ls = __fsub_rn(a.log_scales[3 * (size_t)i + k], c.log_div);
                b.log_scales[3 * r + k] = ls;
                b.scales[3 * r + k] = expf(ls);
            }
        }
    }
}

__global__ void __launch_bounds__(256)
k_reset_opacity(int n, float cap, float *__restrict__ logits, float *__restrict__ opac) {
    pdl_entry();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const float l = fminf(logits[i], cap);
    logits[i] = l;
    opac[i] = 1.0f / (1.0f + expf(-l));
}

}  // namespace

size_t densify_workspace_bytes(int n) {
    const size_t nb = ((size_t)n + kDenTile - 1) / kDenTile;
    return 256 + ((3 * nb * 4 + 255) & ~(size_t)255) + 256;
}

cudaError_t launch_densify_stats(const float *grad2d, const int *radius, int n, int W, int H, float *accum,
                                 float *count, int *max_radius, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    launch_k(k_densify_stats, (n + 255) / 256, 256, 0, st, reinterpret_cast<const float4 *>(grad2d), radius, n, 0.5f * W,
             0.5f * H, accum, count, max_radius);
    return cudaGetLastError();
}

cudaError_t launch_densify(const darb_train_params &in, const darb_adam_state &sin, const float *accum,
                           const float *count, const int *max_radius, const float *normals,
                           const darb_densify_cfg &cfg, void *workspace, const darb_train_params &out,
                           const darb_adam_state &sout, uint32_t *n_out, cudaStream_t st) {
    const int n = in.n;
    unsigned char *w = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(workspace) + 255) &
                                                         ~(uintptr_t)255);
    uint32_t *blk = reinterpret_cast<uint32_t *>(w + 256);
    const int nb = (n + kDenTile - 1) / kDenTile;
    DenCfg c{cfg.grad_threshold, cfg.dense_scale, cfg.min_opacity, cfg.max_screen_radius, cfg.max_world_scale,
             cfg.split_scale_div, (float)std::log((double)cfg.split_scale_div)};
    if (nb == 0) return cudaMemsetAsync(n_out, 0, 3 * sizeof(uint32_t), st);
    launch_k(k_densify_count, nb, kCountThreads, 0, st, n, in.scales, in.opacities, accum, count, max_radius, c, blk);
    launch_k(k_densify_offsets, 1, 1024, 0, st, nb, blk, n_out);
    const DenIO io{in, out, sin, sout};
    auto scatter = [&](auto kernel) {
        launch_k(kernel, nb * kScatPer, kDenThreads, 0, st, n, io, accum, count, max_radius, normals, c, blk, n_out);
    };
    switch (in.sh_degree) {
    case 0: scatter(k_densify_scatter<3>); break;
    case 1: scatter(k_densify_scatter<12>); break;
    case 2: scatter(k_densify_scatter<27>); break;
    default: scatter(k_densify_scatter<48>); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_reset_opacity(const darb_train_params &p, float max_opacity, cudaStream_t st) {
    if (p.n == 0) return cudaSuccess;
    const float cap = (float)std::log((double)max_opacity / (1.0 - (double)max_opacity));
    launch_k(k_reset_opacity, (p.n + 255) / 256, 256, 0, st, p.n, cap, p.opacity_logits, p.opacities);
    return cudaGetLastError();
}

}  // namespace darb
