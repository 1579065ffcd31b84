// Training-step kernels: the L1 photometric loss term (paper Sec. 4.2) and the Adam update of
// the 3DGS optimiser (Sec. 5: original 3DGS hyper-parameters, opacity learning rate 0.02).
// Both are elementwise and HBM-bound; float4 accesses where the layout allows.
#include <algorithm>

#include "kernels.cuh"

namespace darb {

namespace {

__global__ void __launch_bounds__(256)
k_l1_loss(const float *__restrict__ image, const float *__restrict__ target, int count, float inv_count,
          float *__restrict__ dL, float *__restrict__ loss) {
    pdl_entry();
    __shared__ float s_warp[8];
    float acc = 0.0f;
    auto sgn = [inv_count](float d) { return d > 0.0f ? inv_count : (d < 0.0f ? -inv_count : 0.0f); };
    const int tid = blockIdx.x * 256 + threadIdx.x, stride = gridDim.x * 256;
    // float4 lanes when all three buffers are 16-byte aligned, then the ragged end one by one
    const bool vec = ((reinterpret_cast<uintptr_t>(image) | reinterpret_cast<uintptr_t>(target) |
                       reinterpret_cast<uintptr_t>(dL)) & 15) == 0;
    const int n4 = vec ? count >> 2 : 0;
    for (int i = tid; i < n4; i += stride) {
        const float4 a = reinterpret_cast<const float4 *>(image)[i], b = reinterpret_cast<const float4 *>(target)[i];
        const float d0 = a.x - b.x, d1 = a.y - b.y, d2 = a.z - b.z, d3 = a.w - b.w;
        reinterpret_cast<float4 *>(dL)[i] = make_float4(sgn(d0), sgn(d1), sgn(d2), sgn(d3));
        acc += (fabsf(d0) + fabsf(d1)) + (fabsf(d2) + fabsf(d3));
    }
    for (int i = 4 * n4 + tid; i < count; i += stride) {
        const float d = image[i] - target[i];
        dL[i] = sgn(d);
        acc += fabsf(d);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.0f;
        for (int w = 0; w < 8; ++w) s += s_warp[w];
        atomicAdd(loss, s * inv_count);
    }
}

// The whole Adam step of a training state in one launch: each block takes kAdamBlock consecutive floats
// of one parameter group (the groups' blocks one after the other), float4 lanes, the loads of a
// thread's lanes issued before the first update.  HBM-bound; as a launch per group (and scalar lanes
// for the SH rows whose length is no multiple of 4) the small groups ran at half the copy rate
// and a small state was five launches: 243 -> 232 us at 1M splats,
// degree 3 (1684 B a splat; part of the gradients is still in L2); with the gradients before it, degree 2 320 -> 220 us, degree 0 111 -> 101.
constexpr int kAdamThreads = 256, kAdamLanes = 2;
constexpr int kAdamBlock = kAdamThreads * kAdamLanes * 4;  // floats per block

// ACT: 0 = identity, 1 = exp (log-scale -> scale), 2 = sigmoid (logit -> opacity).  For ACT != 0 the
// incoming gradient is w.r.t. the activated value and `act` holds that value; the raw gradient is
// g * d(act)/d(raw), and `act` is refreshed after the step.
template <int ACT>
__device__ __forceinline__ void adam_elem(float &p, float g, float &m, float &v, float lr, const AdamConsts &c,
                                          float &act) {
    if (ACT == 1) g *= act;
    if (ACT == 2) g *= act * (1.0f - act);
    adam_apply(p, g, m, v, lr, c);
    if (ACT == 1) act = expf(p);
    if (ACT == 2) act = 1.0f / (1.0f + expf(-p));
}

template <int ACT, class LrOf>
__device__ __forceinline__ void adam_group(long long count, long long block, float *__restrict__ p,
                                           const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
                                           float *__restrict__ act, LrOf lr_of, const AdamConsts &c) {
    const long long n4 = count >> 2, j0 = block * (kAdamBlock / 4) + threadIdx.x;
    float4 P[kAdamLanes], G[kAdamLanes], M[kAdamLanes], V[kAdamLanes], A[kAdamLanes];
#pragma unroll
    for (int u = 0; u < kAdamLanes; ++u) {
        const long long j = j0 + u * kAdamThreads;
        if (j < n4) {
            P[u] = reinterpret_cast<float4 *>(p)[j];
            G[u] = reinterpret_cast<const float4 *>(g)[j];
            M[u] = reinterpret_cast<float4 *>(m)[j];
            V[u] = reinterpret_cast<float4 *>(v)[j];
            A[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ACT) A[u] = reinterpret_cast<float4 *>(act)[j];
        }
    }
#pragma unroll
    for (int u = 0; u < kAdamLanes; ++u) {
        const long long j = j0 + u * kAdamThreads;
        if (j < n4) {
            float lr[4];
            lr_of(4 * j, lr);
            adam_elem<ACT>(P[u].x, G[u].x, M[u].x, V[u].x, lr[0], c, A[u].x);
            adam_elem<ACT>(P[u].y, G[u].y, M[u].y, V[u].y, lr[1], c, A[u].y);
            adam_elem<ACT>(P[u].z, G[u].z, M[u].z, V[u].z, lr[2], c, A[u].z);
            adam_elem<ACT>(P[u].w, G[u].w, M[u].w, V[u].w, lr[3], c, A[u].w);
            reinterpret_cast<float4 *>(p)[j] = P[u];
            reinterpret_cast<float4 *>(m)[j] = M[u];
            reinterpret_cast<float4 *>(v)[j] = V[u];
            if (ACT) reinterpret_cast<float4 *>(act)[j] = A[u];
        }
    }
    // the ragged end (count % 4 floats), by the group's first block
    if (block == 0 && threadIdx.x < (unsigned)(count & 3)) {
        const long long i = (n4 << 2) + threadIdx.x;
        float lr[4], pp = p[i], mm = m[i], vv = v[i], a = ACT ? act[i] : 0.f;
        lr_of(i, lr);
        adam_elem<ACT>(pp, g[i], mm, vv, lr[0], c, a);
        p[i] = pp;
        m[i] = mm;
        v[i] = vv;
        if (ACT) act[i] = a;
    }
}

__host__ __device__ constexpr long long adam_blocks(long long count) { return (count + kAdamBlock - 1) / kAdamBlock; }

template <int DEG>
__global__ void __launch_bounds__(kAdamThreads)
k_adam(long long n, darb_train_params P, darb_splat_grads G, darb_adam_state A, AdamConsts c) {
    pdl_entry();
    constexpr int ROW = 3 * (DEG + 1) * (DEG + 1);
    auto same = [](float lr) {
        return [lr](long long, float (&r)[4]) { r[0] = r[1] = r[2] = r[3] = lr; };
    };
    const float dc = c.lr_sh_dc, rest = c.lr_sh_rest;
    // the SH rows first, the bulk of the bytes; their first 3 floats are the DC term
    long long b = blockIdx.x;
    if (b < adam_blocks(ROW * n)) {
        adam_group<0>(ROW * n, b, P.sh, G.dsh, A.m_sh, A.v_sh, nullptr, [=](long long f, float (&r)[4]) {
            const int pos = (int)(f % ROW);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q = pos + u >= ROW ? (pos + u) % ROW : pos + u;  // a float4 straddles rows of 3 and 27
                r[u] = q < 3 ? dc : rest;
            }
        }, c);
        return;
    }
    b -= adam_blocks(ROW * n);
    if (b < adam_blocks(4 * n)) {
        adam_group<0>(4 * n, b, P.quats, G.dquats, A.m_quats, A.v_quats, nullptr, same(c.lr_quats), c);
        return;
    }
    b -= adam_blocks(4 * n);
    if (b < adam_blocks(3 * n)) {
        adam_group<0>(3 * n, b, P.means, G.dmeans, A.m_means, A.v_means, nullptr, same(c.lr_means), c);
        return;
    }
    b -= adam_blocks(3 * n);
    if (b < adam_blocks(3 * n)) {
        adam_group<1>(3 * n, b, P.log_scales, G.dscales, A.m_scales, A.v_scales, P.scales, same(c.lr_scales), c);
        return;
    }
    b -= adam_blocks(3 * n);
    adam_group<2>(n, b, P.opacity_logits, G.dopacities, A.m_opac, A.v_opac, P.opacities, same(c.lr_opacities), c);
}

int grid_for(long long count) {
    long long b = (count + 255) / 256;
    return (int)(b < kGridSms * 16 ? (b > 0 ? b : 1) : kGridSms * 16);
}

}  // namespace

namespace {

struct ZeroRegion {
    void *p;
    size_t bytes;
};

__global__ void __launch_bounds__(256) k_zero(ZeroRegion r0, ZeroRegion r1, ZeroRegion r2) {
    pdl_entry();
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    const ZeroRegion rs[3] = {r0, r1, r2};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const ZeroRegion r = rs[k];
        if (!r.p || r.bytes == 0) continue;
        if ((reinterpret_cast<uintptr_t>(r.p) & 15) == 0 && (r.bytes & 15) == 0) {
            uint4 *q = reinterpret_cast<uint4 *>(r.p);
            for (size_t i = tid; i < r.bytes / 16; i += stride) q[i] = make_uint4(0, 0, 0, 0);
        } else {
            uint32_t *q = reinterpret_cast<uint32_t *>(r.p);
            for (size_t i = tid; i < r.bytes / 4; i += stride) q[i] = 0u;
        }
    }
}

}  // namespace

cudaError_t launch_zero(cudaStream_t st, void *p0, size_t b0, void *p1, size_t b1, void *p2, size_t b2) {
    const size_t words = (b0 + b1 + b2) / 16 + 1;
    const int blocks = (int)std::min<size_t>((words + 255) / 256, kGridSms * 8);
    launch_k(k_zero, blocks, 256, 0, st, ZeroRegion{p0, b0}, ZeroRegion{p1, b1}, ZeroRegion{p2, b2});
    return cudaGetLastError();
}

cudaError_t launch_l1_loss(const float *image, const float *target, int count, float *dL, float *loss,
                           cudaStream_t st) {
    cudaError_t e = launch_zero(st, loss, sizeof(float));
    if (e != cudaSuccess) return e;
    if (count == 0) return cudaSuccess;
    launch_k(k_l1_loss, grid_for((count + 3) / 4), 256, 0, st, image, target, count, 1.0f / (float)count, dL, loss);
    return cudaGetLastError();
}

cudaError_t launch_adam(const darb_train_params &p, const darb_splat_grads &g, const darb_adam_state &s,
                        const darb_adam_config &c, cudaStream_t st) {
    const long long n = p.n;
    if (n == 0) return cudaSuccess;
    const AdamConsts ac = make_adam_consts(c);
    const long long row = 3ll * (p.sh_degree + 1) * (p.sh_degree + 1);
    const long long blocks = adam_blocks(row * n) + adam_blocks(4 * n) + 2 * adam_blocks(3 * n) + adam_blocks(n);
    auto go = [&](auto kernel) { launch_k(kernel, (unsigned)blocks, kAdamThreads, 0, st, n, p, g, s, ac); };
    switch (p.sh_degree) {
    case 0: go(k_adam<0>); break;
    case 1: go(k_adam<1>); break;
    case 2: go(k_adam<2>); break;
    default: go(k_adam<3>); break;
    }
    return cudaGetLastError();
}

}  // namespace darb
