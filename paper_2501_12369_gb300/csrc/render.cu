// Step 4 and its backward: per-pixel front-to-back compositing over each tile's depth-sorted
// splat run (paper Sec. 4.1 "alpha blending ... similar to 3DGS", Eq. HalfCosine and
// Eq. 2DSplattedFunction; forward and backward listings of Sec. B).
//
// A CTA takes a tile (backward) or a square of one (forward).  Each thread owns PIX pixels of one
// column, so every splat record loaded from shared memory serves PIX pixels and dx is shared.  The
// tile's run is consumed in batches of NT records (NT = threads): each thread gathers one splat's
// record (mean, conic, opacity, colour) into shared memory, then every thread walks the batch.  A
// CTA-wide vote ends the loop once every pixel of the CTA has stopped (T < 1e-4) -- the early
// termination of 3DGS.
//
// The support test uses the fixed FP32 sequence conic_q(), and alpha / the kernel value are
// computed by the same inline code in forward and backward, so the backward re-takes exactly
// the forward's decisions when it replays a pixel from its last contributor.
#include <type_traits>

#include "kernels.cuh"

namespace darb {

namespace {

struct Bg {
    float r, g, b;
};

constexpr int kMaxDevicesRender = 64;


// The forward's CTA composites a SUB x SUB square of a tile (the squares of a tile walk the same
// list), PIX pixels a thread.  A warp covers a compact block (LX columns, LY * PIX rows), because it
// walks until its last pixel has stopped and neighbouring pixels stop at about the same record; a
// thread's pixels share their column, so that dx is shared.
template <int TILE_, int SUB_, int PIX_>
struct FwdShape {
    static constexpr int TILE = TILE_, SUB = SUB_, PIX = PIX_;
    static constexpr int NT = SUB * SUB / PIX;  // threads per CTA = records per batch
    static constexpr int PARTS = (TILE / SUB) * (TILE / SUB);
    static constexpr int LX = SUB == 16 && PIX == 4 ? 16 : 8, LY = 32 / LX;
    static constexpr int BH = LY * PIX, BX = SUB / LX;  // rows of a warp's block, blocks side by side
    static_assert(BH <= SUB && SUB % BH == 0, "blocks tile the square");
    __device__ static int column() { return (int)((threadIdx.x >> 5) % BX) * LX + (int)(threadIdx.x & 31) % LX; }
    __device__ static int row(int k) {
        return (int)((threadIdx.x >> 5) / BX) * BH + (int)(threadIdx.x & 31) / LX + k * LY;
    }
};
// 16 x 16 squares (8 x 8 in 8-pixel tiles, one warp) of two pixels a thread.  A CTA holds its place
// until its slowest warp has stopped, so small squares cost less although each gathers its records
// again: Gaussian, 1M splats, 1080p, 32-pixel tiles: 169 us with the whole tile as one CTA of four
// pixels a thread, 152 with squares of 16 and four pixels, 148 with two, 162 with squares of 8;
// 8-pixel tiles 155 us with one pixel a thread, 118 with two.
template <int TILE> struct FwdOf { using S = FwdShape<TILE, TILE == 8 ? 8 : 16, 2>; };
// The batched launch takes four pixels a thread (2026 us against 2096 for 16 views of 1M splats:
// its views' lists are short and half the warps then fetch items and records).
template <int TILE> struct BatchOf { using S = FwdShape<TILE, TILE == 8 ? 8 : 16, TILE == 8 ? 2 : 4>; };

// Arithmetic on a pair of values (the packed two-lane FP32 instructions of sm_100+, which round each lane
// as the scalar form does).
struct Pair {
    using T = float2;
    static __device__ __forceinline__ T dup(float a) { return make_float2(a, a); }
    static __device__ __forceinline__ T mul(T a, T b) { return __fmul2_rn(a, b); }
    static __device__ __forceinline__ T add(T a, T b) { return __fadd2_rn(a, b); }
    static __device__ __forceinline__ T fma(T a, T b, T c) { return __ffma2_rn(a, b, c); }
    static __device__ __forceinline__ float &at(T &v, int l) { return l ? v.y : v.x; }
};

// q = dx (A dx + 2B dy) + (C dy) dy as a fixed FP32 sequence, for a record (B2 = 2B, exact) and a pair of
// pixels of one column.  Forward and backward both call it, so that they take the same support
// decision.
__device__ __forceinline__ float2 conic_q(float2 dx, float2 dy, float2 A, float2 B2, float2 C) {
    using V = Pair;
    const float2 g = V::fma(A, dx, V::mul(B2, dy));
    return V::fma(dx, g, V::mul(V::mul(C, dy), dy));
}

// The profile F of a pair of values: the multiplications in front of the special functions, and the whole
// sinc series (sin(x)/x >= 0 on the main lobe, x^2 = pi^2 q / 9), on the pair, the other kernels by lane.
template <int KIND>
__device__ __forceinline__ float2 kernel_F_pair(float2 q, const KernelSpec &ks) {
    using V = Pair;
    float2 r = q;
    if constexpr (KIND == DARB_GAUSSIAN || KIND == DARB_HALF_COSINE) {
        r = V::mul(q, V::dup(KIND == DARB_GAUSSIAN ? -kHalfLog2e : kPi / 18.0f));
#pragma unroll
        for (int l = 0; l < 2; ++l) V::at(r, l) = KIND == DARB_GAUSSIAN ? ex2_ftz(V::at(r, l)) : __cosf(V::at(r, l));
    } else if constexpr (KIND == DARB_PARABOLA) {
        r = V::fma(q, V::dup(-1.0f / 9.0f), V::dup(1.0f));
    } else if constexpr (KIND == DARB_MOD_SINC) {
        const float2 u = V::mul(q, V::dup(kPi * kPi / 9.0f));
        r = V::fma(u, V::dup(1.0f / 1307674368000.0f), V::dup(-1.0f / 6227020800.0f));
        r = V::fma(r, u, V::dup(1.0f / 39916800.0f));
        r = V::fma(r, u, V::dup(-1.0f / 362880.0f));
        r = V::fma(r, u, V::dup(1.0f / 5040.0f));
        r = V::fma(r, u, V::dup(-1.0f / 120.0f));
        r = V::fma(r, u, V::dup(1.0f / 6.0f));
        r = V::fma(r, V::mul(u, V::dup(-1.0f)), V::dup(1.0f));
#pragma unroll
        for (int l = 0; l < 2; ++l) V::at(r, l) = fmaxf(V::at(r, l), 0.0f);
    } else {
#pragma unroll
        for (int l = 0; l < 2; ++l) V::at(r, l) = kernel_F<KIND>(V::at(q, l), ks);
    }
    return r;
}

// Records walked per step of the forward: their alphas do not depend on the transmittance, so a
// step's alphas overlap; a batch is padded with records of opacity 0 to whole steps.
// Steps of 4 records and few resident threads (512 an SM, up to 128 registers) for the plain forward:
// overlap within a warp pays more than more warps (157 us against 169 at steps of 2 and 768
// threads, 188 at steps of 1 and 1024, Gaussian).  The L1 forward is a training step's, whose
// dense scenes stop after some 20 records: steps of 2 and 1024 threads, as its CTAs mostly wait on
// their gathers.  The batched launch: 2 and 768.
constexpr int kStepPlain = 4, kStepL1 = 2, kStepBatch = 2;
constexpr int kThreadsPlain = 512, kThreadsL1 = 1024, kThreadsBatch = 768;  // resident per SM at least

// A batch of staged records: the 9 floats of a splat in two float4s and a float, so that a thread
// reads a record in 3 shared-memory loads.
template <int NT>
struct FwdSmem {
    float4 a[NT];  // x, y, A, 2B
    float4 b[NT];  // C, opacity, red, green
    float c[NT];   // blue
};

// Where a tile's results go; t_final, last and n_contrib may be null (not written).
struct FwdSink {
    float *image;
    float *t_final;
    uint32_t *last;
    uint32_t *n_contrib;
    Bg bg;
};

// The L1 image loss (Sec. 4.2) taken in the forward's epilogue, where each pixel's colour is
// in registers: dL/dC = sign(C - target) / count per channel, and the block's sum of
// |C - target| / count added to *loss (zeroed by the caller).  FP32 additions in memory round at
// the size of the whole sum, so there should be few: the CTAs of a cluster of kL1Cluster hand their sums
// to its first one, which adds them at once (1 020 additions for 1080p in 32-pixel tiles instead of
// 8 160, whose error reached 2e-6 of the loss).  Only the first CTA waits for the others.
struct L1Out {
    const float *target;
    float *dL;
    float *loss;
    float inv_count;
};
constexpr unsigned kL1Cluster = 8;

struct L1Smem {
    uint64_t full;  // mbarrier of the cluster's first CTA: one arrival from each of the others
    float part[kL1Cluster];
};

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// Before the compositing: the barrier is there and the cluster's CTAs run once l1_cluster_add waits.
__device__ __forceinline__ void l1_cluster_begin(L1Smem &sm) {
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&sm.full)), "r"(kL1Cluster - 1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}

// Adds the cluster's sums to *loss; `sum` is thread 0's.
__device__ __forceinline__ void l1_cluster_add(L1Smem &sm, float sum, const L1Out &l1) {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (threadIdx.x != 0) return;
    const unsigned rank = blockIdx.x % kL1Cluster;
    if (rank != 0) {
        asm volatile(
            "{\n\t"
            ".reg .b32 part, full;\n\t"
            "mapa.shared::cluster.u32 part, %0, 0;\n\t"
            "mapa.shared::cluster.u32 full, %1, 0;\n\t"
            "st.shared::cluster.f32 [part], %2;\n\t"
            "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [full];\n\t"
            "}" ::"r"(smem_addr(&sm.part[rank])), "r"(smem_addr(&sm.full)), "f"(sum)
            : "memory");
        return;
    }
    unsigned long long t0, now;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (;;) {
        unsigned done;
        asm volatile(
            "{\n\t"
            ".reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t"
            "}" : "=r"(done) : "r"(smem_addr(&sm.full)) : "memory");
        if (done) break;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
        if (now - t0 > 60000000000ull) {  // a minute: the other CTAs never came; the loss says so
            atomicAdd(l1.loss, __int_as_float(0x7fc00000));
            return;
        }
    }
#pragma unroll
    for (unsigned c = 1; c < kL1Cluster; ++c) sum += sm.part[c];
    atomicAdd(l1.loss, sum * l1.inv_count);
}

// One tile of one view, by the whole CTA.  sink() is called once, after the compositing loop,
// so the output pointers need not stay live in registers across it.  With L1 the epilogue also
// takes the sum of the L1 loss over the square's pixels (thread 0's *l1_sum).  AUX: the outputs
// beside the image and T that the caller may ask for (0: none, 1: last, 2: last and n_contrib).
//
// The body is branch-free and keeps few instructions on the ALU pipe (compares, selects, minimum),
// which runs at half the rate of the FP32 pipe and bound it before.  For every (pixel, record),
// with the support and alpha tests in `use`:
//   a = use ? alpha : 0;  t' = t (1 - a);  blend = use and t' >= 1e-4
//   w = blend ? a t : 0;  T = blend ? t' : T;  t = t'
// t runs on past the stop, where it stays below 1e-4 as every factor is at most 1, so a stopped
// pixel needs no flag of its own, and the chain from record to record is one multiplication.  A
// record that does not blend leaves t, T and the colours exactly as they are.  q >= 0 and
// q <= q_lim are one unsigned comparison (q is never -0: it ends in an addition to +0 or more).
// Pairs of records instead of pairs of pixels as the packed lanes (no value then needs duplicating)
// took as many instructions and more registers (189 us against 175 at the time).
template <int KIND, class S, int AUX, int STEP, bool L1 = false, class SinkFn>
__device__ __forceinline__ void render_tile_fwd(int item, FwdSmem<S::NT> &sm,
                                                const uint2 *__restrict__ ranges,
                                                const uint32_t *__restrict__ values,
                                                const float2 *__restrict__ mean2d,
                                                const float4 *__restrict__ conic_o, const float *__restrict__ rgb,
                                                int W, int H, int tiles_x, float qmax, int strict,
                                                const KernelSpec &ks, SinkFn sink, const L1Out &l1 = L1Out{},
                                                float *s_l1 = nullptr, float *l1_sum = nullptr) {
    constexpr int TILE = S::TILE, NT = S::NT, PIX = S::PIX, L = 2, NV = PIX / L;  // NV pairs
    using V = Pair;
    using VT = V::T;
    static_assert(PIX % L == 0, "whole pairs");
    static_assert(NT % STEP == 0, "a full batch is whole steps");
    const int tile = item / S::PARTS, part = item % S::PARTS;
    const int px = (tile % tiles_x) * TILE + part % (TILE / S::SUB) * S::SUB + S::column();
    const int y0 = (tile / tiles_x) * TILE + part / (TILE / S::SUB) * S::SUB;
    const float fpx = (float)px + 0.5f;
    const uint2 r = ranges[tile];
    const int start = (int)r.x, end = (int)r.y;
    const uint32_t qlim = __float_as_uint(support_limit(qmax, strict));

    VT t[NV], Tf[NV], C0[NV], C1[NV], C2[NV], nfpy[NV];
    uint32_t count[PIX], lastp[PIX];
    auto all_stopped = [&] {
        float m = 0.0f;
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int l = 0; l < L; ++l) m = fmaxf(m, V::at(t[v], l));
        return m < kTMin;
    };
    // The square, by steps of ST records.  Where a colour was not finite, which a weight of 0 does not take out of
    // a sum, once more, record by record, with the colours of what does not blend masked.  (The flag kept in shared
    // memory, or looked at in every batch, cost 3% of the Gaussian's 182 us, this 0.6%.)
    bool odd = false;  // whether this thread gathered such a colour
    auto composite = [&](auto steps, auto masked) {
        constexpr int ST = decltype(steps)::value;
        constexpr bool MASKED = decltype(masked)::value;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            Tf[v] = V::dup(1.0f);
            C0[v] = C1[v] = C2[v] = V::dup(0.0f);
#pragma unroll
            for (int l = 0; l < L; ++l) {
                const int py = y0 + S::row(v * L + l);
                V::at(nfpy[v], l) = -((float)py + 0.5f);
                V::at(t[v], l) = px < W && py < H ? 1.0f : 0.0f;  // pixels outside the image have stopped
                count[v * L + l] = lastp[v * L + l] = 0;
            }
        }
        for (int b0 = start; b0 < end; b0 += NT) {
            const bool stopped = all_stopped();
            if (__syncthreads_count(stopped) == NT) break;
            const int nb = min(NT, end - b0), i = threadIdx.x;
            if (i < nb) {
                const uint32_t id = values[b0 + i];
                const float2 xy = mean2d[id];
                const float4 co = conic_o[id];
                const float c0 = rgb[3 * (size_t)id], c1 = rgb[3 * (size_t)id + 1], c2 = rgb[3 * (size_t)id + 2];
                sm.a[i] = make_float4(xy.x, xy.y, co.x, 2.0f * co.y);
                sm.b[i] = make_float4(co.z, co.w, c0, c1);
                sm.c[i] = c2;
                if (!MASKED) odd |= !isfinite(c0 + c1 + c2);
            } else if (i < nb + ST) {  // the last step's padding
                sm.a[i] = sm.b[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                sm.c[i] = 0.0f;
            }
            __syncthreads();
            if (stopped) continue;
            const uint32_t pos0 = (uint32_t)(b0 - start + 1);
            for (int j0 = 0; j0 < nb; j0 += ST) {
#pragma unroll
                for (int u = 0; u < ST; ++u) {
                    const float4 pa = sm.a[j0 + u], pb = sm.b[j0 + u];
                    const float pc = sm.c[j0 + u];
                    const VT dx = V::dup(__fsub_rn(pa.x, fpx)), y = V::dup(pa.y), A = V::dup(pa.z), B2 = V::dup(pa.w);
                    const VT Cc = V::dup(pb.x), o = V::dup(pb.y), r0 = V::dup(pb.z), r1 = V::dup(pb.w), r2 = V::dup(pc);
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const VT dy = V::add(y, nfpy[v]);
                        VT q = conic_q(dx, dy, A, B2, Cc);
                        VT a = V::mul(o, kernel_F_pair<KIND>(q, ks));
                        bool use[L];
#pragma unroll
                        for (int l = 0; l < L; ++l) {
                            const float alpha = fminf(kAlphaMax, V::at(a, l));
                            use[l] = __float_as_uint(V::at(q, l)) <= qlim && alpha >= kAlphaMin;
                            V::at(a, l) = use[l] ? alpha : 0.0f;
                        }
                        VT w = V::mul(a, t[v]);
                        t[v] = V::mul(t[v], V::fma(a, V::dup(-1.0f), V::dup(1.0f)));
#pragma unroll
                        for (int l = 0; l < L; ++l) {
                            const float tn = V::at(t[v], l);
                            const bool blend = use[l] && tn >= kTMin;
                            V::at(w, l) = blend ? V::at(w, l) : 0.0f;
                            V::at(Tf[v], l) = blend ? tn : V::at(Tf[v], l);
                            if (AUX >= 2) count[v * L + l] += blend ? 1u : 0u;
                            if (AUX >= 1) lastp[v * L + l] = blend ? pos0 + (uint32_t)(j0 + u) : lastp[v * L + l];
                        }
                        if constexpr (MASKED) {  // per lane: what blends has a weight above 0
#pragma unroll
                            for (int l = 0; l < L; ++l) {
                                if (V::at(w, l) == 0.0f) continue;
                                V::at(C0[v], l) = fmaf(pb.z, V::at(w, l), V::at(C0[v], l));
                                V::at(C1[v], l) = fmaf(pb.w, V::at(w, l), V::at(C1[v], l));
                                V::at(C2[v], l) = fmaf(pc, V::at(w, l), V::at(C2[v], l));
                            }
                        } else {
                            C0[v] = V::fma(r0, w, C0[v]);
                            C1[v] = V::fma(r1, w, C1[v]);
                            C2[v] = V::fma(r2, w, C2[v]);
                        }
                    }
                }
                if (all_stopped()) break;
            }
        }
    };
    composite(std::integral_constant<int, STEP>{}, std::false_type{});
    if (__syncthreads_or(odd))
        composite(std::integral_constant<int, 1>{}, std::true_type{});
    const size_t plane = (size_t)W * H;
    const FwdSink o = sink();
    float acc = 0.0f;  // the pixels' |C - target| (with L1)
#pragma unroll
    for (int k = 0; k < PIX; ++k) {
        const int py = y0 + S::row(k);
        if (!(px < W && py < H)) continue;
        const size_t pix = (size_t)py * W + px;
        const float T = V::at(Tf[k / L], k % L);
        const float c[3] = {fmaf(T, o.bg.r, V::at(C0[k / L], k % L)), fmaf(T, o.bg.g, V::at(C1[k / L], k % L)),
                            fmaf(T, o.bg.b, V::at(C2[k / L], k % L))};
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            if (o.image) o.image[ch * plane + pix] = c[ch];
            if constexpr (L1) {
                const float d = c[ch] - l1.target[ch * plane + pix];
                l1.dL[ch * plane + pix] = d > 0.0f ? l1.inv_count : (d < 0.0f ? -l1.inv_count : 0.0f);
                acc += fabsf(d);
            }
        }
        if (o.t_final) o.t_final[pix] = T;
        if (AUX >= 1 && o.last) o.last[pix] = lastp[k];
        if (AUX >= 2 && o.n_contrib) o.n_contrib[pix] = count[k];
    }
    if constexpr (L1) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if ((threadIdx.x & 31) == 0) s_l1[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            float sum = 0.0f;
            for (int w = 0; w < S::NT / 32; ++w) sum += s_l1[w];
            *l1_sum = sum;
        }
    }
}

template <int KIND, int TILE, int AUX, bool L1>
__global__ void __launch_bounds__(FwdOf<TILE>::S::NT, (L1 ? kThreadsL1 : kThreadsPlain) / FwdOf<TILE>::S::NT)
k_render_fwd(const uint2 *__restrict__ ranges, const uint32_t *__restrict__ values,
             const float2 *__restrict__ mean2d, const float4 *__restrict__ conic_o,
             const float *__restrict__ rgb, int W, int H, int tiles_x, float qmax, int strict, KernelSpec ks, Bg bg,
             float *__restrict__ image, float *__restrict__ t_final, uint32_t *__restrict__ last,
             uint32_t *__restrict__ n_contrib, int n_items, L1Out l1) {
    using S = typename FwdOf<TILE>::S;
    __shared__ FwdSmem<S::NT> sm;
    __shared__ float s_l1[L1 ? (S::NT + 31) / 32 : 1];
    auto tile = [&](float *l1_sum) {
        render_tile_fwd<KIND, S, AUX, L1 ? kStepL1 : kStepPlain, L1>(
            blockIdx.x, sm, ranges, values, mean2d, conic_o, rgb, W, H, tiles_x, qmax, strict, ks,
            [&] { return FwdSink{image, t_final, last, n_contrib, bg}; }, l1, s_l1, l1_sum);
    };
    if constexpr (L1) {
        __shared__ L1Smem s_cluster;
        l1_cluster_begin(s_cluster);
        pdl_entry();
        float sum = 0.0f;
        if ((int)blockIdx.x < n_items) tile(&sum);  // the grid is whole clusters
        l1_cluster_add(s_cluster, sum, l1);
    } else {
        pdl_entry();
        tile(nullptr);
    }
}

// Several views in one persistent launch: CTAs take items (a square of a tile of a view) from a
// device counter (numbered view-major; views[v].tile_begin is the first tile of view v) until all
// are done, so small and large views share the GPU without per-view launches or tails.
template <int KIND, int TILE, int AUX>
__global__ void __launch_bounds__(BatchOf<TILE>::S::NT, kThreadsBatch / BatchOf<TILE>::S::NT)
k_render_fwd_batch(const BatchView *__restrict__ views, int n_views, int total_tiles, uint32_t *__restrict__ queue,
                   float qmax, int strict, KernelSpec ks) {
    pdl_entry();
    using S = typename BatchOf<TILE>::S;
    __shared__ FwdSmem<S::NT> sm;
    __shared__ int s_item, s_view;
    for (;;) {
        if (threadIdx.x == 0) {
            const int item = (int)atomicAdd(queue, 1u), t = item / S::PARTS;
            int v = 0;
            if (t < total_tiles) {  // last view whose first tile is <= t
                int lo = 0, hi = n_views - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (views[mid].tile_begin <= t) lo = mid; else hi = mid - 1;
                }
                v = lo;
            }
            s_item = item;
            s_view = v;
        }
        __syncthreads();
        const int item = s_item, v = s_view;
        if (item / S::PARTS >= total_tiles) break;
        const BatchView &bv = views[v];
        render_tile_fwd<KIND, S, AUX, kStepBatch>(
            item - bv.tile_begin * S::PARTS, sm, bv.ranges, bv.values, bv.mean2d, bv.conic_o, bv.rgb, bv.W, bv.H,
            bv.tiles_x, qmax, strict, ks, [&] {
                const BatchView &b = views[v];
                return FwdSink{b.image, b.t_final, b.last, b.n_contrib, Bg{b.bg[0], b.bg[1], b.bg[2]}};
            });
        __syncthreads();  // the CTA is done with s_item and the staging arrays
    }
}

// The raised cosine with a q_max past its main lobe (q <= 6.25), as a caller may set it: there F rises again,
// and the derivative's series has ended.
constexpr int kRaisedCosineWide = kNumKernels;
constexpr float kRaisedCosineEnd = 6.5f;

// dF/dq of a pair of values, F the profile there.  Where F gives it, from F; the sinc's from the
// derivative of its series (to u^7, the next term below 1e-8 on the main lobe) and the raised cosine's
// from the sinc's series, which need no sine, cosine, root or division and are nearer the derivative than their
// quotient (the raised cosine's to 4e-7 of its value for q <= 4, where __sinf left 1.7e-5).
template <int KIND>
__device__ __forceinline__ float2 kernel_dF2(float2 q, float2 F) {
    auto dup = [](float a) { return make_float2(a, a); };
    if constexpr (KIND == DARB_GAUSSIAN) {
        return __fmul2_rn(F, dup(-0.5f));
    } else if constexpr (KIND == DARB_HALF_COSINE) {
        const float2 x = __fmul2_rn(q, dup(kPi / 18.0f));
        return __fmul2_rn(make_float2(__sinf(x.x), __sinf(x.y)), dup(-(kPi / 18.0f)));
    } else if constexpr (KIND == DARB_MOD_SINC) {
        // sum over k of (-1)^k k u^(k - 1) / (2k + 1)!, k = 1 .. 8, times du/dq
        constexpr float a = kPi * kPi / 9.0f;
        const float2 u = __fmul2_rn(q, dup(a));
        float2 r = __ffma2_rn(u, dup(8.0f / 355687428096000.0f), dup(-7.0f / 1307674368000.0f));
        r = __ffma2_rn(r, u, dup(6.0f / 6227020800.0f));
        r = __ffma2_rn(r, u, dup(-5.0f / 39916800.0f));
        r = __ffma2_rn(r, u, dup(4.0f / 362880.0f));
        r = __ffma2_rn(r, u, dup(-3.0f / 5040.0f));
        r = __ffma2_rn(r, u, dup(2.0f / 120.0f));
        r = __ffma2_rn(r, u, dup(-1.0f / 6.0f));
        return __fmul2_rn(r, dup(a));
    } else if constexpr (KIND == DARB_INV_QUADRIC) {
        return __fmul2_rn(F, __fmul2_rn(F, dup(-1.0f)));
    } else if constexpr (KIND == DARB_INV_MULTIQUADRIC) {
        return __fmul2_rn(__fmul2_rn(F, F), __fmul2_rn(F, dup(-0.5f)));
    } else if constexpr (KIND == DARB_PARABOLA) {
        return dup(-1.0f / 9.0f);
    } else if constexpr (KIND == kRaisedCosineWide) {
        constexpr float k = kPi / 2.5f;
        auto d = [](float v) { return -0.25f * k * __sinf(k * sqrt_newton(v)) / sqrt_newton(v); };
        const float2 z = __ffma2_rn(q, dup(k * k * k * k / 24.0f), dup(-0.25f * k * k));  // the limit at q = 0
        return make_float2(q.x < 1e-6f ? z.x : d(q.x), q.y < 1e-6f ? z.y : d(q.y));
    } else {
        // raised cosine: -(k^2/4) sin(x)/x, x^2 = u = k^2 q, k = pi/2.5, by the series to u^8 / 17! (the next
        // term is below 1e-8 at x = pi)
        constexpr float kk = kPi * kPi / 6.25f;
        const float2 u = __fmul2_rn(q, dup(kk));
        float2 r = __ffma2_rn(u, dup(1.0f / 355687428096000.0f), dup(-1.0f / 1307674368000.0f));
        r = __ffma2_rn(r, u, dup(1.0f / 6227020800.0f));
        r = __ffma2_rn(r, u, dup(-1.0f / 39916800.0f));
        r = __ffma2_rn(r, u, dup(1.0f / 362880.0f));
        r = __ffma2_rn(r, u, dup(-1.0f / 5040.0f));
        r = __ffma2_rn(r, u, dup(1.0f / 120.0f));
        r = __ffma2_rn(r, u, dup(-1.0f / 6.0f));
        r = __ffma2_rn(r, u, dup(1.0f));
        return __fmul2_rn(r, dup(-0.25f * kk));
    }
}

// Warp sums of v[0..7] by halving exchanges (4 + 2 + 1 shuffles move half of the remaining
// values to the partner lane, then 2 more finish the sum): afterwards lane 4i (and its
// neighbours 4i+1..4i+3) holds the sum of v[i].  v[8] is summed by a plain butterfly into r8.
// 14 shuffles for 9 values instead of 45.
__device__ __forceinline__ float warp_sum8(const float (&v)[9], int lane, float &r8) {
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    float a[4], b[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float send = b4 ? v[i] : v[i + 4];
        a[i] = (b4 ? v[i + 4] : v[i]) + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float send = b3 ? a[i] : a[i + 2];
        b[i] = (b3 ? a[i + 2] : a[i]) + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    float c = (b2 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, b2 ? b[0] : b[1], 4);
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    c += __shfl_xor_sync(0xffffffffu, c, 1);
    r8 = v[8];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) r8 += __shfl_xor_sync(0xffffffffu, r8, off);
    return c;  // the sum of v[4 b4 + 2 b3 + b2] = v[lane >> 2]
}

// Whether the ellipse {q <= qmax} of a record may reach the block of pixel centres [xl, xh] x
// [yl, yh] (relative to its centre): the least q over the rectangle, which lies on an edge that faces
// the centre, against qmax with a margin of 5%.  The margin covers the rounding of q, whose
// relative error grows with the conic's cancellation 1 / (1 - B^2 / (A C)); above 1e4 (or for a
// conic that is not positive definite in FP32) every record is kept.
__device__ __forceinline__ bool may_reach(float A, float B, float C, float xl, float xh, float yl, float yh, float qmax) {
    const float ac = A * C, det = ac - B * B;
    if (!(det * 1e4f > ac)) return true;
    const float ex = xl > 0.0f ? xl : xh, ey = yl > 0.0f ? yl : yh;  // the facing edges, where one faces
    const bool fx = xl > 0.0f || xh < 0.0f, fy = yl > 0.0f || yh < 0.0f;
    if (!fx && !fy) return true;
    float m = 3.0e38f;
    if (fx) {
        const float dy = fminf(fmaxf(__fdividef(-B * ex, C), yl), yh);
        m = A * ex * ex + (2.0f * B * ex + C * dy) * dy;
    }
    if (fy) {
        const float dx = fminf(fmaxf(__fdividef(-B * ey, A), xl), xh);
        m = fminf(m, A * dx * dx + (2.0f * B * dx + C * ey) * ey);
    }
    return !(m > 1.05f * qmax);
}

// a + b - fl(a + b), exactly (Knuth's two-sum).
__device__ __forceinline__ float add_error(float a, float b) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

// The conic's three sums take up what their additions in memory lost, which k_render_bwd keeps in the
// last three floats of a row for splats of kManyTiles tiles or more; these are zero again.  Bound by latency
// (tile counts, rows, stores): 10 us for 3M splats, four a thread (15 with one, 20 for every visible splat).
// Fewer than kManyTiles additions cost no more than the last rounding of the sum itself.
constexpr uint32_t kManyTiles = 8;
__global__ void __launch_bounds__(256)
k_fold_conic(int n, const uint32_t *__restrict__ tiles, float4 *__restrict__ grad2d) {
    pdl_entry();
    const int i0 = 4 * (blockIdx.x * 256 + threadIdx.x);
    if (i0 >= n) return;
    uint32_t t[4] = {0, 0, 0, 0};
    if (i0 + 4 <= n) {
        const uint4 t4 = *reinterpret_cast<const uint4 *>(tiles + i0);
        t[0] = t4.x, t[1] = t4.y, t[2] = t4.z, t[3] = t4.w;
    } else {
        for (int k = 0; i0 + k < n; ++k) t[k] = tiles[i0 + k];
    }
    float4 *row = grad2d + 3 * (size_t)i0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (t[k] < kManyTiles) continue;
        float *g = reinterpret_cast<float *>(row + 3 * k);
        const float4 lo = row[3 * k + 2];
        const float hi[3] = {g[2], g[3], g[4]}, lost[3] = {lo.y, lo.z, lo.w};
        if (lost[0] == 0.0f && lost[1] == 0.0f && lost[2] == 0.0f) continue;
#pragma unroll
        for (int u = 0; u < 3; ++u)
            if (isfinite(hi[u])) g[2 + u] = hi[u] + lost[u];  // a sum that is not finite lost nothing
        row[3 * k + 2] = make_float4(lo.x, 0.0f, 0.0f, 0.0f);
    }
}

// Backward: replay each pixel back to front from its last contributor.  With T_k the
// transmittance in front of splat k and S the colour composited behind it (background
// included), dC/dalpha_k = c_k T_k - S / (1 - alpha_k) and dC/dc_k = alpha_k T_k.  Only the
// projection of S on the pixel's upstream gradient g is needed: g . dC/dalpha_k =
// T_k (g . c_k) - (g . S) / (1 - alpha_k), and g . S grows by (g . c_k) alpha_k T_k per splat,
// so each pixel carries the scalar g . S instead of three colour channels.
//
// A CTA of NW warps takes a tile, a warp of it a block of LX x (32 / LX * PIX) pixels, PIX of one
// column a lane.  The warps walk the tile's run independently, 32 records at a
// time: each lane gathers one, keeps it if its ellipse may reach the block, and the kept ones are
// compacted in the warp's shared memory.  The pair body is branch-free (a pair that does not
// contribute has alpha 0 and leaves T, g . S and every sum as they are) and runs on pairs of pixels
// with the packed two-lane FP32 instructions.  The gradients w.r.t. centre and conic come from three sums
// over a lane's column instead of five products a pair: s, s b and s b^2 (s = dL/dF dF/dq, b the pixel's
// distance from the column's middle, a constant), with the record's dx, dy and conic at the middle applied
// once per lane and record.  A dx and B dy, which nearly cancel along a thin ellipse, meet before anything is
// summed over lanes: with sums of s dx and s dy over the tile, combined at its end, the centre's gradient of
// an ellipse of 560 x 4 pixels was off by up to 4e-6 of the sum of its terms' magnitudes, now by 2e-7.
//
// The sums are kept per warp in shared memory for a window of kWindow records, added over the CTA at
// the window's end, and leave through one set of vector atomics per (tile, record): a near splat
// that covers the image then sums as few FP32 terms in memory as there are tiles.  A set per
// block instead took 114 us where this takes 122, but made the error of such sums 2.7 times as
// large.  Windows of 64 cost 1% more; of 96 in CTAs of eight warps, within 48 KB.
//
// The conic's gradients go on to the covariance through -K G K, which cancels by a thin splat's aspect
// ratio squared, so the rounding of the additions in memory, in whatever order they come, showed in the
// quaternions' and scales' gradients: two equal steps at 3M splats, 1080p differed by 4e-6 in the second
// moments (mean over ten views, up to 3e-4).  Each addition of the conic's three therefore returns the sum
// it met, and what it lost to rounding is added to one of the row's three spare floats, which k_fold_conic puts
// back: two equal steps then agree to 3e-10.  A step went from 1339 to 1353 us.
//
// Bound by the FP32 and ALU pipes of the pair body.  Launch, 300k splats, 1245 x 825, 16-pixel tiles, against
// a thread per pixel column of the tile with scalar arithmetic and a list of kept records for the
// whole CTA: sinc 217 -> 122 us, Gaussian 367 -> 225, half-cosine 100 -> 64; sinc with 32-pixel tiles
// 273 -> 135, 8-pixel 237 -> 120; 20k splats 142 -> 84, at 333 x 207 167 -> 67.  (Before the two points above,
// which take 3% and the second launch's 4 us.)
template <int KIND, int LX, int PIX, int NW>
__global__ void __launch_bounds__(32 * NW, (PIX == 2 ? 28 : NW == 8 ? 24 : 20) / NW)
k_render_bwd(const uint2 *__restrict__ ranges, const uint32_t *__restrict__ values,
             const float2 *__restrict__ mean2d, const float4 *__restrict__ conic_o,
             const float *__restrict__ rgb, const uint32_t *__restrict__ tiles, int W, int H, int tiles_x, int tile,
             float qmax, int strict, KernelSpec ks, Bg bg, const float *__restrict__ t_final,
             const uint32_t *__restrict__ last, const float *__restrict__ dL_dimage, float4 *__restrict__ grad2d) {
    pdl_entry();
    static_assert(PIX == 2 || PIX == 4, "one or two pairs of pixels a lane");
    constexpr int LY = 32 / LX, BH = LY * PIX, NV = PIX / 2, kWindow = NW == 8 ? 96 : 128;
    struct WarpSmem {
        float4 a[32], b[32];      // x, y, A, 2B; C, opacity, red, green
        float c[32];              // blue
        int pos[32];
        float sum[kWindow * 9];
    };
    __shared__ WarpSmem smem[NW];
    __shared__ int s_last[NW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    WarpSmem &sm = smem[warp];
    const int t = blockIdx.x, start = (int)ranges[t].x;
    const uint32_t qlim = __float_as_uint(support_limit(qmax, strict));
    const size_t plane = (size_t)W * H;
    auto dup = [](float a) { return make_float2(a, a); };
    auto emit = [&](uint32_t id, float o, bool many, const float (&s)[9]) {  // a record's sums to its gradients
        bool any = false;
#pragma unroll
        for (int u = 0; u < 9; ++u) any |= s[u] != 0.0f;
        if (!any) return;
        float4 *gp = grad2d + 3 * (size_t)id;
        const float4 x = make_float4(2.0f * o * s[0], 2.0f * o * s[1], o * s[2], 2.0f * o * s[3]);
        const float4 y = make_float4(o * s[4], s[5], s[6], s[7]);
        if (many) {
            const float4 p = atomicAdd(gp, x), q = atomicAdd(gp + 1, y);
            atomicAdd(gp + 2, make_float4(s[8], add_error(p.z, x.z), add_error(p.w, x.w), add_error(q.x, y.x)));
        } else {
            atomicAdd(gp, x);
            atomicAdd(gp + 1, y);
            atomicAdd(reinterpret_cast<float *>(gp + 2), s[8]);
        }
    };
    const int x0 = (t % tiles_x) * tile + warp % (tile / LX) * LX, y0 = (t / tiles_x) * tile + warp / (tile / LX) * BH;
    const int px = x0 + lane % LX;
    const float fpx = (float)px + 0.5f;
    const float fmid = (float)(y0 + lane / LX) + 0.5f + 0.5f * (PIX - 1) * LY;  // the middle of the lane's column
    float2 nfpy[NV], T[NV], GS[NV], g0[NV], g1[NV], g2[NV];
    int my_last[PIX], nlast = 0;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const int py = y0 + lane / LX + (2 * v + l) * LY;
            float tt = 1.0f, a0 = 0.0f, a1 = 0.0f, a2 = 0.0f;
            int ml = 0;
            if (px < W && py < H) {
                const size_t pix = (size_t)py * W + px;
                tt = t_final[pix];
                ml = (int)last[pix];
                a0 = dL_dimage[pix];
                a1 = dL_dimage[plane + pix];
                a2 = dL_dimage[2 * plane + pix];
            }
            const float gs = tt * fmaf(a2, bg.b, fmaf(a1, bg.g, a0 * bg.r));
            (l ? nfpy[v].y : nfpy[v].x) = -((float)py + 0.5f);
            (l ? T[v].y : T[v].x) = tt;
            (l ? GS[v].y : GS[v].x) = gs;
            (l ? g0[v].y : g0[v].x) = a0;
            (l ? g1[v].y : g1[v].x) = a1;
            (l ? g2[v].y : g2[v].x) = a2;
            my_last[2 * v + l] = ml;
            nlast = max(nlast, ml);
        }
    }
    nlast = (int)__reduce_max_sync(0xffffffffu, (unsigned)nlast);
    if (lane == 0) s_last[warp] = nlast;
    // an upstream gradient or a record that is not finite reaches only what blended: where some value is large
    // enough for a product of two to overflow, the pairs that did not blend are masked
    auto tame = [](float x) { return fabsf(x) < 1e15f; };
    bool odd = false;
#pragma unroll
    for (int v = 0; v < NV; ++v)
        odd |= !(tame(g0[v].x) && tame(g0[v].y) && tame(g1[v].x) && tame(g1[v].y) && tame(g2[v].x) && tame(g2[v].y));
    odd = __any_sync(0xffffffffu, odd);
    __syncthreads();
    int top = nlast;
#pragma unroll
    for (int w = 0; w < NW; ++w) top = max(top, s_last[w]);
#pragma unroll 1
    for (int win = top > 0 ? (top - 1) / kWindow * kWindow : -1; win >= 0; win -= kWindow) {
        const int end = min(top - win, kWindow);
        for (int i = lane; i < 9 * end; i += 32) sm.sum[i] = 0.0f;
        int bstart;
        for (int bend = min(nlast, win + kWindow); bend > win; bend = bstart) {
            bstart = max(bend - 32, win);
            const int pos = bend - 1 - lane;  // lane 0 the last record: the walk goes back to front
            bool keep = false;
            uint32_t id = 0;
            float2 xy;
            float4 co;
            if (pos >= bstart) {
                id = values[start + pos];
                xy = mean2d[id];
                co = conic_o[id];
                keep = may_reach(co.x, co.y, co.z, (float)x0 + 0.5f - xy.x, (float)(x0 + LX) - 0.5f - xy.x,
                                 (float)y0 + 0.5f - xy.y, (float)(y0 + BH) - 0.5f - xy.y, qmax);
            }
            const uint32_t kept = __ballot_sync(0xffffffffu, keep);
            const int n = __popc(kept);
            bool wild = false;
            if (keep) {
                const int slot = __popc(kept & ((1u << lane) - 1u));
                const float c0 = rgb[3 * (size_t)id], c1 = rgb[3 * (size_t)id + 1], c2 = rgb[3 * (size_t)id + 2];
                sm.a[slot] = make_float4(xy.x, xy.y, co.x, 2.0f * co.y);
                sm.b[slot] = make_float4(co.z, co.w, c0, c1);
                sm.c[slot] = c2;
                sm.pos[slot] = pos;
                wild = !(tame(c0) && tame(c1) && tame(c2) && tame(co.x) && tame(co.y) && tame(co.z) && tame(xy.x) && tame(xy.y));
            }
            wild = __any_sync(0xffffffffu, wild);
            __syncwarp();
            auto walk = [&](int j, auto masked) {
                const float4 ra = sm.a[j], rb = sm.b[j];
                const float rc = sm.c[j];
                const int rpos = sm.pos[j];
                const float dx1 = __fsub_rn(ra.x, fpx);
                const float2 dx = dup(dx1), y = dup(ra.y), A = dup(ra.z), B2 = dup(ra.w), Cc = dup(rb.x), o = dup(rb.y);
                const float2 c0 = dup(rb.z), c1 = dup(rb.w), c2 = dup(rc);
                float2 sq[NV], SF = dup(0.0f), W0 = dup(0.0f), W1 = dup(0.0f), W2 = dup(0.0f);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const float2 dy = __fadd2_rn(y, nfpy[v]);
                    const float2 qr = conic_q(dx, dy, A, B2, Cc);
                    // outside the support the profile is taken at its limit: finite, so that the pair's zero
                    // weight leaves the sums alone (as unsigned words negative values lie above the limit too)
                    const uint32_t q0 = __float_as_uint(qr.x), q1 = __float_as_uint(qr.y);
                    const float2 q = make_float2(__uint_as_float(min(q0, qlim)), __uint_as_float(min(q1, qlim)));
                    float2 F, dF;
                    if constexpr (KIND == DARB_GENERIC) {  // costly: skipped where no lane is in the support
                        F = dF = dup(0.0f);
                        if (__any_sync(0xffffffffu, q0 <= qlim || q1 <= qlim)) {
                            generic_both(q.x, ks, F.x, dF.x);
                            generic_both(q.y, ks, F.y, dF.y);
                        }
                    } else {
                        F = kernel_F_pair<KIND == kRaisedCosineWide ? DARB_RAISED_COSINE : KIND>(q, ks);
                        dF = kernel_dF2<KIND>(q, F);
                    }
                    const float2 of = __fmul2_rn(o, F);
                    const float al0 = fminf(kAlphaMax, of.x), al1 = fminf(kAlphaMax, of.y);
                    const bool u0 = rpos < my_last[2 * v] && q0 <= qlim && al0 >= kAlphaMin;
                    const bool u1 = rpos < my_last[2 * v + 1] && q1 <= qlim && al1 >= kAlphaMin;
                    const float2 a = make_float2(u0 ? al0 : 0.0f, u1 ? al1 : 0.0f);
                    const float2 om = __ffma2_rn(a, dup(-1.0f), dup(1.0f));
                    const float2 iom = make_float2(rcp_ftz(om.x), rcp_ftz(om.y));
                    const float2 Tk = __fmul2_rn(T[v], iom);
                    float2 h0 = g0[v], h1 = g1[v], h2 = g2[v];
                    if constexpr (decltype(masked)::value) {
                        if (!u0) h0.x = h1.x = h2.x = 0.0f;
                        if (!u1) h0.y = h1.y = h2.y = 0.0f;
                    }
                    float2 gc = __ffma2_rn(h2, c2, __ffma2_rn(h1, c1, __fmul2_rn(h0, c0)));
                    if constexpr (decltype(masked)::value) gc = make_float2(u0 ? gc.x : 0.0f, u1 ? gc.y : 0.0f);
                    const float2 dal = __ffma2_rn(Tk, gc, __fmul2_rn(__fmul2_rn(GS[v], dup(-1.0f)), iom));
                    const float2 w = __fmul2_rn(a, Tk);
                    GS[v] = __ffma2_rn(gc, w, GS[v]);
                    T[v] = Tk;
                    W0 = __ffma2_rn(w, h0, W0);
                    W1 = __ffma2_rn(w, h1, W1);
                    W2 = __ffma2_rn(w, h2, W2);
                    // the alpha clamp has zero derivative
                    const float2 da = make_float2(u0 && !(of.x > kAlphaMax) ? dal.x : 0.0f,
                                                  u1 && !(of.y > kAlphaMax) ? dal.y : 0.0f);
                    SF = __ffma2_rn(F, da, SF);
                    sq[v] = __fmul2_rn(dF, da);
                }
                // the column's sums of s, s b and s b^2; with dy = dym - b, dym at the column's middle, the
                // centre's from e = K d there, and the conic's
                constexpr float h = 0.5f * LY;
                const float top = sq[0].x, bottom = sq[NV - 1].y;
                float t0 = top + bottom, t1 = (PIX - 1) * h * (bottom - top), t2 = (PIX - 1) * (PIX - 1) * h * h * t0;
                if constexpr (NV == 2) {
                    const float in0 = sq[0].y, in1 = sq[1].x, in = in0 + in1;
                    t1 = fmaf(h, in1 - in0, t1);
                    t2 = fmaf(h * h, in, t2);
                    t0 += in;
                }
                const float dym = __fsub_rn(ra.y, fmid);
                const float B = 0.5f * ra.w, r0 = fmaf(dym, t0, -t1);
                const float2 KB = make_float2(B, rb.x), e = __ffma2_rn(make_float2(ra.z, B), dx, __fmul2_rn(KB, dup(dym)));
                const float2 u = __ffma2_rn(e, dup(t0), __fmul2_rn(KB, dup(-t1)));
                const float2 xs = __fmul2_rn(make_float2(t0 * dx1, r0), dx);
                float sums[9] = {u.x, u.y, xs.x, xs.y, fmaf(dym, r0, fmaf(-dym, t1, t2)),
                                 SF.x + SF.y, W0.x + W0.y, W1.x + W1.y, W2.x + W2.y};
                if (decltype(masked)::value && t0 == 0.0f && t1 == 0.0f && t2 == 0.0f)
                    sums[0] = sums[1] = sums[2] = sums[3] = sums[4] = 0.0f;
                float r8;
                float r = warp_sum8(sums, lane, r8);
                // lanes 0, 4, .. 28 hold the first eight sums, every lane the ninth: lane 1 takes that
                r = lane == 1 ? r8 : r;
                if ((lane & 3) == 0 || lane == 1) {
                    const int u = lane == 1 ? 8 : lane >> 2;
                    sm.sum[9 * (rpos - win) + u] += r;
                }
            };
            if (odd || wild)
                for (int j = 0; j < n; ++j) walk(j, std::true_type{});
            else
                for (int j = 0; j < n; ++j) walk(j, std::false_type{});
            __syncwarp();
        }
        __syncthreads();
        for (int i = threadIdx.x; i < end; i += 32 * NW) {
            float s[9];
#pragma unroll
            for (int u = 0; u < 9; ++u) s[u] = 0.0f;
#pragma unroll
            for (int w = 0; w < NW; ++w)
#pragma unroll
                for (int u = 0; u < 9; ++u) s[u] += smem[w].sum[9 * i + u];
            const uint32_t id = values[start + win + i];
            emit(id, conic_o[id].w, tiles[id] >= kManyTiles, s);
        }
        if (win > 0) __syncthreads();
    }
}

template <int KIND, int TILE>
cudaError_t fwd_t(int n_tiles, const uint2 *ranges, const uint32_t *values, const float2 *mean2d,
                  const float4 *conic_o, const float *rgb, const Cam &cam, int tiles_x, float qmax, int strict,
                  const KernelSpec &ks, float *image, float *t_final, uint32_t *last, uint32_t *n_contrib,
                  const L1Out &l1, cudaStream_t st) {
    using S = typename FwdOf<TILE>::S;
    const int items = n_tiles * S::PARTS;
    const unsigned cluster = l1.target ? kL1Cluster : 1;
    auto go = [&](auto kernel) {
        launch_cluster(kernel, (items + cluster - 1) / cluster * cluster, cluster, S::NT, 0, st, ranges, values, mean2d,
                       conic_o, rgb, cam.W, cam.H, tiles_x, qmax, strict, ks, Bg{cam.bg[0], cam.bg[1], cam.bg[2]},
                       image, t_final, last, n_contrib, items, l1);
    };
    if (!l1.target) go(k_render_fwd<KIND, TILE, 2, false>);
    else if (n_contrib) go(k_render_fwd<KIND, TILE, 2, true>);
    else go(k_render_fwd<KIND, TILE, 1, true>);
    return cudaGetLastError();
}

template <int KIND, int TILE, int LX, int PIX>
cudaError_t bwd_t(int n_tiles, const uint2 *ranges, const uint32_t *values, const float2 *mean2d,
                  const float4 *conic_o, const float *rgb, const uint32_t *tiles, const Cam &cam, int tiles_x, float qmax,
                  int strict, const KernelSpec &ks, const float *t_final, const uint32_t *last, const float *dL, float *grad2d,
                  cudaStream_t st) {
    constexpr int NW = TILE / LX * (TILE / (32 / LX * PIX));
    launch_k(k_render_bwd<KIND, LX, PIX, NW>, n_tiles, 32 * NW, 0, st,
             ranges, values, mean2d, conic_o, rgb, tiles, cam.W, cam.H, tiles_x, TILE, qmax, strict, ks,
             Bg{cam.bg[0], cam.bg[1], cam.bg[2]}, t_final, last, dL, reinterpret_cast<float4 *>(grad2d));
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_render_fwd(int kind, int tile, int tiles_x, int tiles_y, const uint32_t *ranges,
                              const uint32_t *values, const float2 *mean2d, const float4 *conic_o,
                              const float *rgb, const Cam &cam, float qmax, int strict, const KernelSpec &ks,
                              float *image, float *t_final, uint32_t *last, uint32_t *n_contrib,
                              cudaStream_t st, const float *l1_target, float *l1_dL, float *l1_loss) {
    const int n_tiles = tiles_x * tiles_y;
    if (n_tiles == 0) return cudaSuccess;
    const uint2 *rg = reinterpret_cast<const uint2 *>(ranges);
    const L1Out l1{l1_target, l1_dL, l1_loss, 1.0f / (3.0f * (float)cam.W * (float)cam.H)};
#define FWD_ARGS (n_tiles, rg, values, mean2d, conic_o, rgb, cam, tiles_x, qmax, strict, ks, image, t_final, last, n_contrib, l1, st)
#define FWD_CALL(K, T) fwd_t<K, T> FWD_ARGS
    if (tile == 8) {
        switch (kind) {
        case 0: return FWD_CALL(0, 8); case 1: return FWD_CALL(1, 8); case 2: return FWD_CALL(2, 8);
        case 3: return FWD_CALL(3, 8); case 4: return FWD_CALL(4, 8); case 5: return FWD_CALL(5, 8);
        case 6: return FWD_CALL(6, 8); default: return FWD_CALL(7, 8);
        }
    } else if (tile == 16) {
        switch (kind) {
        case 0: return FWD_CALL(0, 16); case 1: return FWD_CALL(1, 16); case 2: return FWD_CALL(2, 16);
        case 3: return FWD_CALL(3, 16); case 4: return FWD_CALL(4, 16); case 5: return FWD_CALL(5, 16);
        case 6: return FWD_CALL(6, 16); default: return FWD_CALL(7, 16);
        }
    } else {
        switch (kind) {
        case 0: return FWD_CALL(0, 32); case 1: return FWD_CALL(1, 32); case 2: return FWD_CALL(2, 32);
        case 3: return FWD_CALL(3, 32); case 4: return FWD_CALL(4, 32); case 5: return FWD_CALL(5, 32);
        case 6: return FWD_CALL(6, 32); default: return FWD_CALL(7, 32);
        }
    }
#undef FWD_CALL
#undef FWD_ARGS
}

namespace {

template <int KIND, int TILE, int AUX>
cudaError_t fwd_batch_aux(const BatchView *views, int n_views, int total_tiles, uint32_t *queue, float qmax, int strict,
                          const KernelSpec &ks, int max_ctas, cudaStream_t st) {
    constexpr int NT = BatchOf<TILE>::S::NT;
    static int per_sm[kMaxDevicesRender] = {};  // resident CTAs per SM, once per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int occ = (dev >= 0 && dev < kMaxDevicesRender) ? per_sm[dev] : 0;
    if (occ == 0) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_render_fwd_batch<KIND, TILE, AUX>, NT, 0);
        if (e != cudaSuccess) return e;
        occ = occ > 0 ? occ : 1;
        if (dev >= 0 && dev < kMaxDevicesRender) per_sm[dev] = occ;
    }
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    long long grid = (long long)sms * occ;
    if (max_ctas > 0 && grid > max_ctas) grid = max_ctas;
    const long long items = (long long)total_tiles * BatchOf<TILE>::S::PARTS;
    if (grid > items) grid = items;
    e = launch_zero(st, queue, sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    launch_k(k_render_fwd_batch<KIND, TILE, AUX>, (int)grid, NT, 0, st, views, n_views, total_tiles, queue, qmax, strict,
             ks);
    return cudaGetLastError();
}

template <int KIND, int TILE>
cudaError_t fwd_batch_t(const BatchView *views, int n_views, int total_tiles, bool aux, uint32_t *queue, float qmax,
                        int strict, const KernelSpec &ks, int max_ctas, cudaStream_t st) {
    return aux ? fwd_batch_aux<KIND, TILE, 2>(views, n_views, total_tiles, queue, qmax, strict, ks, max_ctas, st)
               : fwd_batch_aux<KIND, TILE, 0>(views, n_views, total_tiles, queue, qmax, strict, ks, max_ctas, st);
}

}  // namespace

cudaError_t launch_render_fwd_batch(int kind, int tile, const BatchView *views, int n_views, int total_tiles, bool aux,
                                    uint32_t *queue, float qmax, int strict, const KernelSpec &ks, int max_ctas,
                                    cudaStream_t st) {
    if (total_tiles == 0 || n_views == 0) return cudaSuccess;
#define FB_CALL(K, T) fwd_batch_t<K, T>(views, n_views, total_tiles, aux, queue, qmax, strict, ks, max_ctas, st)
    if (tile == 8) {
        switch (kind) {
        case 0: return FB_CALL(0, 8); case 1: return FB_CALL(1, 8); case 2: return FB_CALL(2, 8);
        case 3: return FB_CALL(3, 8); case 4: return FB_CALL(4, 8); case 5: return FB_CALL(5, 8);
        case 6: return FB_CALL(6, 8); default: return FB_CALL(7, 8);
        }
    } else if (tile == 16) {
        switch (kind) {
        case 0: return FB_CALL(0, 16); case 1: return FB_CALL(1, 16); case 2: return FB_CALL(2, 16);
        case 3: return FB_CALL(3, 16); case 4: return FB_CALL(4, 16); case 5: return FB_CALL(5, 16);
        case 6: return FB_CALL(6, 16); default: return FB_CALL(7, 16);
        }
    } else {
        switch (kind) {
        case 0: return FB_CALL(0, 32); case 1: return FB_CALL(1, 32); case 2: return FB_CALL(2, 32);
        case 3: return FB_CALL(3, 32); case 4: return FB_CALL(4, 32); case 5: return FB_CALL(5, 32);
        case 6: return FB_CALL(6, 32); default: return FB_CALL(7, 32);
        }
    }
#undef FB_CALL
}

cudaError_t launch_render_bwd(int kind, int n, const uint32_t *tiles, int tile, int tiles_x, int tiles_y, const uint32_t *ranges,
                              const uint32_t *values, const float2 *mean2d, const float4 *conic_o,
                              const float *rgb, const Cam &cam, float qmax, int strict, const KernelSpec &ks,
                              const float *t_final, const uint32_t *last, const float *dL_dimage,
                              float *grad2d, cudaStream_t st) {
    const int n_tiles = tiles_x * tiles_y;
    if (n_tiles == 0) return cudaSuccess;
    const uint2 *rg = reinterpret_cast<const uint2 *>(ranges);
    // 16 x 8 blocks (four pixels a lane), but 16 x 4 in 16-pixel tiles where the image has fewer than 48
    // blocks of 16 x 8 per SM: the chip is then not full, and a warp's time is its own chain.  Measured
    // (sinc, 20k and 300k splats): 333 x 207 115 -> 67 and 132 -> 79 us, 640 x 360 72 -> 47 and 84 -> 63, 960 x
    // 540 70 -> 57 and 86 -> 78, 1280 x 720 (47 blocks per SM) 77 -> 71 and 112 -> 112; 1245 x 825 (54)
    // 84 -> 77 and 122 -> 124, 1080p 120 -> 120 and 194 -> 210.  In 32-pixel tiles the CTAs of sixteen warps
    // that 16 x 4 blocks need were slower at every size (333 x 207: 148 -> 163, 960 x 540: 86 -> 109).
    const bool few = (long long)n_tiles * (tile * tile / 128) < 48ll * kGridSms;
#define BWD_ARGS n_tiles, rg, values, mean2d, conic_o, rgb, tiles, cam, tiles_x, qmax, strict, ks, t_final, last, dL_dimage, grad2d, st
#define BWD_CALL(K) (tile == 8 ? bwd_t<K, 8, 8, 2>(BWD_ARGS) : tile == 32 ? bwd_t<K, 32, 16, 4>(BWD_ARGS) \
                     : few ? bwd_t<K, 16, 16, 2>(BWD_ARGS) : bwd_t<K, 16, 16, 4>(BWD_ARGS))
    cudaError_t e;
    switch (kind) {
    case 0: e = BWD_CALL(0); break; case 1: e = BWD_CALL(1); break; case 3: e = BWD_CALL(3); break;
    case DARB_RAISED_COSINE: e = qmax > kRaisedCosineEnd ? BWD_CALL(kRaisedCosineWide) : BWD_CALL(2); break;
    case 4: e = BWD_CALL(4); break; case 5: e = BWD_CALL(5); break; case 6: e = BWD_CALL(6); break; default: e = BWD_CALL(7);
    }
    if (e != cudaSuccess || n == 0 || !tiles) return e;
    launch_k(k_fold_conic, (n + 1023) / 1024, 256, 0, st, n, tiles, reinterpret_cast<float4 *>(grad2d));
    return cudaGetLastError();
#undef BWD_CALL
#undef BWD_ARGS
}

}  // namespace darb
