// The paper's image loss (Sec. 4.2): L = (1 - lambda) L1 + lambda (1 - SSIM), with the SSIM of
// the 3DGS work it builds on -- per channel, an 11 x 11 Gaussian window (sigma 1.5, normalised)
// over zero-padded images, C1 = 0.01^2, C2 = 0.03^2 -- averaged over channels and pixels.
//
// Two kernels over 32 x 32 output tiles of one channel with a 5-pixel halo, both blurs separable in
// shared memory, every thread 8 consecutive outputs along x and 4 along y (an input is read from
// shared memory once for all the outputs it reaches):
//   k_ssim_fwd  stages (x, y) pairs, blurs the four moments that SSIM needs (x, y, (x - y)^2, xy), and
//               writes per pixel the partial derivatives of SSIM w.r.t. the local moments m_x, s_xx,
//               s_xy, plus the block sums of SSIM and |x - y|;
//   k_ssim_bwd  blurs those three maps (the window is symmetric, so the blur is its own adjoint)
//               and forms dL/dx = (1 - lambda) sign(x - y) / N - lambda (G*d_m + 2x G*d_sxx +
//               y G*d_sxy) / N, N = 3HW; its first CTA also writes the loss.
// With A1 = 2 m_x m_y + C1, A2 = 2 (s_xy - m_x m_y) + C2, B1 = m_x^2 + m_y^2 + C1,
// B2 = s_xx - m_x^2 + s_yy - m_y^2 + C2 and SSIM = A1 A2 / (B1 B2):
//   d_m = 2 m_y (A2 - A1) / (B1 B2) - 2 m_x SSIM (1/B1 - 1/B2),  d_sxx = -SSIM / B2,
//   d_sxy = 2 A1 / (B1 B2).
// s_xx and s_yy enter B2 only as their sum, which is the variance of x - y and twice s_xy: B2 = A2 + var(x - y),
// and B1 = A1 + (m_x - m_y)^2.  What A2 lost to cancellation B2 then shares, and SSIM is near their
// quotient: on images that are nearly equal the gradient's error against 64 bits is 0.6 to 0.95 of what the five
// moments gave, where the sum x^2 + y^2 gave 0.9 to 1.24.
// The forward is bound by issue slots and shared memory (70% and 55% busy), the backward by latency.
// The quantities blurred under one tap weight lie side by side in shared memory, so they load as the
// operands of the packed two-lane FMA; columns lie in four planes (column mod 4), which keeps both
// passes' accesses nearly free of bank conflicts (with rows of pairs they were 42% of the
// wavefronts: 58 and 70 us).  1920 x 1080: 67 us and 59 us with five scalar moments, 51 and 57 now.
#include <algorithm>

#include "kernels.cuh"

namespace darb {
namespace {

constexpr int kSsimFwdCtas = 4, kSsimBwdCtas = 3;  // resident CTAs per SM (5 and 6: 114 and 130 us against 109)
constexpr int kSsimR = 5;
constexpr int kSsimTs = 32;
constexpr int kSsimIn = kSsimTs + 2 * kSsimR;  // 42
constexpr int kSsimThreads = 256;
constexpr int kSsimRb = 4;  // outputs per thread along y (register blocking)
constexpr int kSsimTaps = 2 * kSsimR + 1;
constexpr float kSsimC1 = 0.01f * 0.01f;
constexpr float kSsimC2 = 0.03f * 0.03f;
static_assert(kSsimTs % kSsimRb == 0 && (kSsimTs / kSsimRb) * kSsimTs == kSsimThreads, "one vertical group per thread");

// Shared-memory planes: column c of a row lies in plane c % 4 at c / 4, 42 staged columns in rows of 11
// entries, 32 blurred ones in rows of 9.  The x pass has consecutive lanes on consecutive rows: the odd
// row lengths put them in different banks.  The staging and the y pass have consecutive lanes on
// consecutive columns: the planes are padded so that four planes' neighbouring entries do not
// meet in a bank, for entries of 4, 8 and 16 bytes (plane = 8 mod 32, 4 mod 16, 2 mod 8 entries).
// Outputs of a thread along x (8: one round of 168 threads; 4 took 116 us against 109), groups of a row.
constexpr int kRbX = 8, kGroups = kSsimTs / kRbX;
constexpr int kInRow = 11, kOutRow = 9;
constexpr int plane_pad(int rows_entries, int mod, int want) {
    int p = rows_entries;
    while (p % mod != want) ++p;
    return p;
}
template <class T>
constexpr int kInPlane = sizeof(T) == 4 ? plane_pad(kSsimIn * kInRow, 32, 8) : plane_pad(kSsimIn * kInRow, 16, 4);
template <class T>
constexpr int kOutPlane = sizeof(T) == 4   ? plane_pad(kSsimIn * kOutRow, 32, 8)
                          : sizeof(T) == 8 ? plane_pad(kSsimIn * kOutRow, 16, 4)
                                           : plane_pad(kSsimIn * kOutRow, 8, 2);

// The taps twice over: an operand of the packed FMA.  The window is symmetric.
struct Window {
    float2 g[kSsimR + 1];
    __device__ __forceinline__ float2 at(int k) const { return g[k <= kSsimR ? k : kSsimTaps - 1 - k]; }
};

Window make_window() {
    Window w;
    double sum = 0.0, v[kSsimTaps];
    for (int k = -kSsimR; k <= kSsimR; ++k) {
        v[k + kSsimR] = std::exp(-(double)(k * k) / (2.0 * 1.5 * 1.5));
        sum += v[k + kSsimR];
    }
    for (int k = 0; k <= kSsimR; ++k) w.g[k].x = w.g[k].y = (float)(v[k] / sum);
    return w;
}

__device__ __forceinline__ float2 fma_tap(float2 g, float2 v, float2 acc) { return __ffma2_rn(g, v, acc); }
__device__ __forceinline__ float fma_tap(float2 g, float v, float acc) { return fmaf(g.x, v, acc); }

// An asynchronous copy of N bytes to shared memory, zeros where !in (src is then not read).
template <int N>
__device__ __forceinline__ void copy_async(void *dst, const void *src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(N), "r"(in ? N : 0)
                 : "memory");
}

// One output tile of one channel.
struct SsimTile {
    int x0, y0;
    size_t off;
    __device__ SsimTile(int t, int tiles_x, int tiles_y, size_t plane) {
        const int ch = t / (tiles_x * tiles_y), r = t - ch * (tiles_x * tiles_y);
        y0 = r / tiles_x * kSsimTs;
        x0 = (r - r / tiles_x * tiles_x) * kSsimTs;
        off = (size_t)ch * plane;
    }
};

// Starts the copies of a tile's halo, zeros outside the image: a warp takes every eighth row, columns
// lane and lane + 32.  copy(plane, entry, offset, in) starts one element's.
template <class Copy>
__device__ __forceinline__ void stage_halo(const SsimTile &t, int W, int H, Copy copy) {
    constexpr int NW = kSsimThreads / 32, R = (kSsimIn + NW - 1) / NW;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gx = t.x0 - kSsimR + lane;
    const bool in0 = gx >= 0 && gx < W, in1 = gx + 32 < W;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int r = warp + u * NW, gy = t.y0 - kSsimR + r, j = r * kInRow + (lane >> 2);
        if (r >= kSsimIn) break;
        const bool row = gy >= 0 && gy < H;
        const size_t p = t.off + (size_t)gy * W + gx;
        copy(lane & 3, j, row && in0 ? p : 0, row && in0);
        if (lane < kSsimIn - 32) copy(lane & 3, j + 8, row && in1 ? p + 32 : 0, row && in1);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// out[i] = sum over k of g[k] in(i + k) for N consecutive outputs of a quantity (or a pair of
// them), each sum in tap order; in(t) is called once for every input.
template <int N, class V, class In>
__device__ __forceinline__ void blur(const Window &win, In in, V (&out)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) out[i] = V{};
#pragma unroll
    for (int t = 0; t < N + kSsimTaps - 1; ++t) {
        const V v = in(t);
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (t - i >= 0 && t - i < kSsimTaps) out[i] = fma_tap(win.at(t - i), v, out[i]);
    }
}

// Forward: the four local moments by separable blurs (x along rows, then y along columns), then the
// derivative maps and the block sums.
__global__ void __launch_bounds__(kSsimThreads, kSsimFwdCtas)
k_ssim_fwd(const float *__restrict__ x, const float *__restrict__ y, int W, int H, Window win,
           float2 *__restrict__ d_m_sxx, float *__restrict__ d_sxy, double *__restrict__ sums) {
    pdl_entry();
    __shared__ float2 sxy[4 * kInPlane<float2>];
    __shared__ float4 h[4 * kOutPlane<float4>];  // blurred along x: x, y, (x - y)^2, xy
    __shared__ float s_part[2][kSsimThreads / 32];
    const int tiles_x = (W + kSsimTs - 1) / kSsimTs, tiles_y = (H + kSsimTs - 1) / kSsimTs;
    const size_t plane = (size_t)W * H;
    const SsimTile tile(blockIdx.x, tiles_x, tiles_y, plane);
    {  // the halo tile: as stage_halo, by loads through registers (all issued before the first store)
        constexpr int NW = kSsimThreads / 32, R = (kSsimIn + NW - 1) / NW;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int gx = tile.x0 - kSsimR + lane;
        const bool in0 = gx >= 0 && gx < W, in1 = lane < kSsimIn - 32 && gx + 32 < W;
        float2 v[R][2];
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const int r = warp + u * NW, gy = tile.y0 - kSsimR + r;
            const bool row = r < kSsimIn && gy >= 0 && gy < H;
            const size_t p = tile.off + (size_t)gy * W + gx;
            v[u][0] = v[u][1] = make_float2(0.0f, 0.0f);
            if (row && in0) v[u][0] = make_float2(x[p], y[p]);
            if (row && in1) v[u][1] = make_float2(x[p + 32], y[p + 32]);
        }
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const int r = warp + u * NW, j = (lane & 3) * kInPlane<float2> + r * kInRow + (lane >> 2);
            if (r < kSsimIn) {
                sxy[j] = v[u][0];
                if (lane < kSsimIn - 32) sxy[j + 8] = v[u][1];
            }
        }
    }
    __syncthreads();
    // along x: item = (group of kRbX columns, row)
    for (int item = threadIdx.x; item < kSsimIn * kGroups; item += kSsimThreads) {
        const int g = item / kSsimIn, r = item - g * kSsimIn;
        const float2 *row = sxy + r * kInRow + g * (kRbX / 4);
        float2 xy[kRbX], sp[kRbX];
#pragma unroll
        for (int i = 0; i < kRbX; ++i) xy[i] = sp[i] = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < kRbX + kSsimTaps - 1; ++k) {
            const float2 v = row[(k & 3) * kInPlane<float2> + (k >> 2)];
            const float d = v.x - v.y;
            const float2 p = make_float2(d * d, v.x * v.y);
#pragma unroll
            for (int i = 0; i < kRbX; ++i)
                if (k - i >= 0 && k - i < kSsimTaps) {
                    xy[i] = fma_tap(win.at(k - i), v, xy[i]);
                    sp[i] = fma_tap(win.at(k - i), p, sp[i]);
                }
        }
#pragma unroll
        for (int i = 0; i < kRbX; ++i)
            h[(i & 3) * kOutPlane<float4> + r * kOutRow + g * (kRbX / 4) + (i >> 2)] =
                make_float4(xy[i].x, xy[i].y, sp[i].x, sp[i].y);
    }
    __syncthreads();
    // along y: thread = (column, group of four rows)
    const int c = threadIdx.x % kSsimTs, r0 = (threadIdx.x / kSsimTs) * kSsimRb;
    const float4 *col = h + (c & 3) * kOutPlane<float4> + (c >> 2);
    float2 m[kSsimRb], q[kSsimRb];
#pragma unroll
    for (int i = 0; i < kSsimRb; ++i) m[i] = q[i] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k < kSsimRb + kSsimTaps - 1; ++k) {
        const float4 v = col[(r0 + k) * kOutRow];
#pragma unroll
        for (int i = 0; i < kSsimRb; ++i)
            if (k - i >= 0 && k - i < kSsimTaps) {
                m[i] = fma_tap(win.at(k - i), make_float2(v.x, v.y), m[i]);
                q[i] = fma_tap(win.at(k - i), make_float2(v.z, v.w), q[i]);
            }
    }
    float ssim_sum = 0.0f, l1_sum = 0.0f;
#pragma unroll
    for (int i = 0; i < kSsimRb; ++i) {
        const int r = r0 + i, gy = tile.y0 + r, gx = tile.x0 + c;
        if (gx >= W || gy >= H) continue;
        const float mx = m[i].x, my = m[i].y;
        const float md = mx - my;
        const float A1 = 2.0f * mx * my + kSsimC1;
        const float A2 = 2.0f * fmaf(-mx, my, q[i].y) + kSsimC2;
        const float B1 = fmaf(md, md, A1);
        const float B2 = fmaf(-md, md, q[i].x) + A2;
        const float iB = __frcp_rn(B1 * B2), iB1 = iB * B2, iB2 = iB * B1;  // one reciprocal for both
        const float sv = A1 * A2 * iB;
        const size_t p = tile.off + (size_t)gy * W + gx;
        d_m_sxx[p] = make_float2(2.0f * my * (A2 - A1) * iB - 2.0f * mx * sv * (iB1 - iB2), -sv * iB2);
        d_sxy[p] = 2.0f * A1 * iB;
        ssim_sum += sv;
        const int cc = c + kSsimR;
        const float2 v = sxy[(cc & 3) * kInPlane<float2> + (r + kSsimR) * kInRow + (cc >> 2)];
        l1_sum += fabsf(v.x - v.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ssim_sum += __shfl_xor_sync(0xffffffffu, ssim_sum, o);
        l1_sum += __shfl_xor_sync(0xffffffffu, l1_sum, o);
    }
    if ((threadIdx.x & 31) == 0) {
        s_part[0][threadIdx.x >> 5] = ssim_sum;
        s_part[1][threadIdx.x >> 5] = l1_sum;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        float sum = 0.0f;
        for (int w = 0; w < kSsimThreads / 32; ++w) sum += s_part[threadIdx.x][w];
        atomicAdd(&sums[threadIdx.x], (double)sum);
    }
}

// A few CTAs per SM walk the tiles a grid apart and copy the next tile's halo while they blur the
// present one: with a CTA per tile each waited for its own loads (8 of 15 stalled warps).
// Backward: blurs the three derivative maps (the window is symmetric, so the blur is its own
// adjoint) with the same blocking, then forms dL/dx.
__global__ void __launch_bounds__(kSsimThreads, kSsimBwdCtas)
k_ssim_bwd(const float *__restrict__ x, const float *__restrict__ y, int W, int H, Window win,
           const float2 *__restrict__ d_m_sxx, const float *__restrict__ d_sxy, float lam,
           const double *__restrict__ sums, float *__restrict__ dL, float *__restrict__ loss) {
    pdl_entry();
    extern __shared__ __align__(16) unsigned char smem[];
    struct Smem {
        float2 a[2][4 * kInPlane<float2>], ha[4 * kOutPlane<float2>];  // d_m, d_sxx
        float b[2][4 * kInPlane<float>], hb[4 * kOutPlane<float>];     // d_sxy
    };
    Smem &sm = *reinterpret_cast<Smem *>(smem);
    const int tiles_x = (W + kSsimTs - 1) / kSsimTs, tiles_y = (H + kSsimTs - 1) / kSsimTs;
    const int tiles = 3 * tiles_x * tiles_y;
    const size_t plane = (size_t)W * H;
    const double n = 3.0 * (double)plane;
    const float inv_n = (float)(1.0 / n);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const double ssim = sums[0] / n, l1 = sums[1] / n;
        loss[0] = (float)((1.0 - lam) * l1 + lam * (1.0 - ssim));
        loss[1] = (float)ssim;
    }
    const int c = threadIdx.x % kSsimTs, r0 = (threadIdx.x / kSsimTs) * kSsimRb;
    auto start = [&](int t, int buf) {
        stage_halo(SsimTile(t, tiles_x, tiles_y, plane), W, H, [&](int q, int j, size_t p, bool in) {
            copy_async<8>(&sm.a[buf][q * kInPlane<float2> + j], d_m_sxx + p, in);
            copy_async<4>(&sm.b[buf][q * kInPlane<float> + j], d_sxy + p, in);
        });
    };
    start(blockIdx.x, 0);
    int buf = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, buf ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // the tile has arrived, and every thread is done with the tile before
        if (t + (int)gridDim.x < tiles) start(t + gridDim.x, buf ^ 1);
        const SsimTile tile(t, tiles_x, tiles_y, plane);
        // the images' own pixels, on their way while the maps are blurred
        float xv[kSsimRb], yv[kSsimRb];
#pragma unroll
        for (int i = 0; i < kSsimRb; ++i) {
            const int gy = tile.y0 + r0 + i, gx = tile.x0 + c;
            const bool in = gx < W && gy < H;
            const size_t p = tile.off + (size_t)gy * W + gx;
            xv[i] = in ? x[p] : 0.0f;
            yv[i] = in ? y[p] : 0.0f;
        }
        const float2 *ia = sm.a[buf];
        const float *ib = sm.b[buf];
        for (int item = threadIdx.x; item < kSsimIn * kGroups; item += kSsimThreads) {
            const int g = item / kSsimIn, r = item - g * kSsimIn;
            const int j = r * kInRow + g * (kRbX / 4), o = r * kOutRow + g * (kRbX / 4);
            float2 oa[kRbX];
            float ob[kRbX];
            blur(win, [&](int k) { return ia[(k & 3) * kInPlane<float2> + j + (k >> 2)]; }, oa);
            blur(win, [&](int k) { return ib[(k & 3) * kInPlane<float> + j + (k >> 2)]; }, ob);
#pragma unroll
            for (int i = 0; i < kRbX; ++i) {
                sm.ha[(i & 3) * kOutPlane<float2> + o + (i >> 2)] = oa[i];
                sm.hb[(i & 3) * kOutPlane<float> + o + (i >> 2)] = ob[i];
            }
        }
        __syncthreads();
        const float2 *ca = sm.ha + (c & 3) * kOutPlane<float2> + (c >> 2);
        const float *cb = sm.hb + (c & 3) * kOutPlane<float> + (c >> 2);
        float2 a[kSsimRb];
        float b[kSsimRb];
        blur(win, [&](int k) { return ca[(r0 + k) * kOutRow]; }, a);
        blur(win, [&](int k) { return cb[(r0 + k) * kOutRow]; }, b);
#pragma unroll
        for (int i = 0; i < kSsimRb; ++i) {
            const int gy = tile.y0 + r0 + i, gx = tile.x0 + c;
            if (gx >= W || gy >= H) continue;
            const float d = xv[i] - yv[i];
            const float sgn = d > 0.0f ? 1.0f : (d < 0.0f ? -1.0f : 0.0f);
            const float dssim = (a[i].x + 2.0f * xv[i] * a[i].y + yv[i] * b[i]) * inv_n;
            dL[tile.off + (size_t)gy * W + gx] = (1.0f - lam) * sgn * inv_n - lam * dssim;
        }
    }
}

// Dynamic shared memory of k_ssim_bwd.
constexpr size_t kSsimBwdSmem = (2 * kInPlane<float2> + kOutPlane<float2>) * 4 * 8 +
                                (2 * kInPlane<float> + kOutPlane<float>) * 4 * 4;

}  // namespace

size_t l1_dssim_workspace_bytes(int W, int H) {
    const size_t maps = 3 * (size_t)3 * W * H * sizeof(float);
    return 256 + ((maps + 255) & ~(size_t)255) + 256;
}

cudaError_t launch_l1_dssim(const float *image, const float *target, int W, int H, float lam, void *workspace,
                            float *dL, float *loss, cudaStream_t st) {
    unsigned char *w = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(workspace) + 255) &
                                                         ~(uintptr_t)255);
    double *sums = reinterpret_cast<double *>(w);
    float *maps = reinterpret_cast<float *>(w + 256);
    const size_t n = (size_t)3 * W * H;
    cudaError_t e = launch_zero(st, sums, 2 * sizeof(double));
    if (e != cudaSuccess) return e;
    static const Window win = make_window();
    const long long tiles = 3ll * ((W + kSsimTs - 1) / kSsimTs) * ((H + kSsimTs - 1) / kSsimTs);
    const unsigned walkers = (unsigned)std::min<long long>(tiles, (long long)kSsimBwdCtas * kGridSms);
    e = cudaFuncSetAttribute(k_ssim_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSsimBwdSmem);
    if (e != cudaSuccess) return e;
    launch_k(k_ssim_fwd, (unsigned)tiles, kSsimThreads, 0, st, image, target, W, H, win,
             reinterpret_cast<float2 *>(maps), maps + 2 * n, sums);
    launch_k(k_ssim_bwd, walkers, kSsimThreads, kSsimBwdSmem, st, image, target, W, H, win,
             reinterpret_cast<const float2 *>(maps), maps + 2 * n, lam, sums, dL, loss);
    return cudaGetLastError();
}

}  // namespace darb
