// k x k median filter (Sec. 3.1.5) and the U-/V-disparity maps (Sec. 3.2).
#include "sgm_internal.cuh"

namespace sgm {
namespace {

// ---------------------------------------------------------------------------
// Median.  A 64 x 8 tile plus a (k-1)/2 halo with clamped (replicated)
// borders is staged in shared memory.  A thread takes two neighbouring pixels,
// whose windows it keeps as packed 16-bit pairs: one packed minimum and one
// packed maximum order an element of both windows.  The median comes from
// repeated elimination: of any (k*k + 3)/2 of the elements the smallest and the
// largest cannot be the median of all, so they are dropped, the next element
// joins, and so on down to three.  Bound by those minima and maxima (2 x 132
// per pixel pair for 5 x 5); a Batcher sort of each pixel's window took 17.3 us on
// 1280 x 720, this 14.5.  Invalid pixels (0xFF) take part and sort above every
// valid disparity.
// ---------------------------------------------------------------------------

constexpr int kMX = 32, kMY = 8;

__device__ __forceinline__ void cmpswap2(uint32_t &a, uint32_t &b) {
    uint32_t lo, hi;
    asm("min.u16x2 %0, %1, %2;" : "=r"(lo) : "r"(a), "r"(b));
    asm("max.u16x2 %0, %1, %2;" : "=r"(hi) : "r"(a), "r"(b));
    a = lo;
    b = hi;
}

// Median of the N elements v[0..N-1] (both halves apart).
template <int N>
__device__ __forceinline__ uint32_t median_of(uint32_t (&v)[N]) {
    constexpr int M = (N + 3) / 2;
    // the set is v[0 .. n-1]; the smallest goes to its front, the largest to its end
#pragma unroll
    for (int s = 0; s <= M - 3; s++) {
        const int n = M - s;  // v[0 .. n-1], where v[0] is the element that joined
#pragma unroll
        for (int i = 0; i < n / 2; i++) cmpswap2(v[i], v[n - 1 - i]);
#pragma unroll
        for (int i = 1; i < (n + 1) / 2; i++) cmpswap2(v[0], v[i]);
#pragma unroll
        for (int i = n / 2; i < n - 1; i++) cmpswap2(v[i], v[n - 1]);
        if (n > 3) {  // drop both: the next element takes the front's place, the set shrinks at the end
            v[0] = v[M + s];
        }
    }
    return v[1];
}

template <int K>
__global__ void __launch_bounds__(kMX *kMY)
    median_kernel(const uint8_t *__restrict__ in, uint8_t *__restrict__ out, int W, int H) {
    wait_for_predecessor();
    constexpr int R = K / 2, TW = 2 * kMX + K - 1, TH = kMY + K - 1;
    constexpr int N = K * K, NH = (K + 1) / 2;
    __shared__ __align__(4) uint8_t tile[TH][TW];
    static_assert(TW % 2 == 0, "a thread's bytes start at an even address");
    const int x0 = blockIdx.x * 2 * kMX - R, y0 = blockIdx.y * kMY - R;
    // all of a thread's loads before its first store: their latencies overlap
    constexpr int kLoads = (TW * TH + kMX * kMY - 1) / (kMX * kMY);
    uint8_t t[kLoads];
#pragma unroll
    for (int k = 0; k < kLoads; k++) {
        const int i = threadIdx.y * kMX + threadIdx.x + k * kMX * kMY;
        const int ty = i / TW, tx = i - ty * TW;
        const int gx = min(max(x0 + tx, 0), W - 1), gy = min(max(y0 + ty, 0), H - 1);
        const long long gi = (long long)gy * W + gx;
        t[k] = i < TW * TH && in_range(gi, (long long)W * H) ? in[gi] : 0xFF;
    }
#pragma unroll
    for (int k = 0; k < kLoads; k++) {
        const int i = threadIdx.y * kMX + threadIdx.x + k * kMX * kMY;
        if (i < TW * TH) tile[i / TW][i % TW] = t[k];
    }
    __syncthreads();
    const int x = blockIdx.x * 2 * kMX + 2 * threadIdx.x, y = blockIdx.y * kMY + threadIdx.y;
    if (x >= W || y >= H) return;
    uint32_t v[N];
#pragma unroll
    for (int r = 0; r < K; r++) {
        uint32_t h[NH];  // bytes 2j, 2j + 1 of the row's K + 1
#pragma unroll
        for (int j = 0; j < NH; j++)
            h[j] = *reinterpret_cast<const uint16_t *>(&tile[threadIdx.y + r][2 * threadIdx.x + 2 * j]);
#pragma unroll
        for (int j = 0; j < K; j++)  // (byte j, byte j + 1)
            v[r * K + j] = j % 2 == 0 ? __byte_perm(h[j / 2], 0u, 0x4140) : __byte_perm(h[j / 2], h[(j + 1) / 2], 0x2421);
    }
    const uint32_t m = median_of<N>(v);
    const long long o = (long long)y * W + x;
    if (in_range(o, (long long)W * H)) out[o] = (uint8_t)(m & 0xFFu);
    if (x + 1 < W && in_range(o + 1, (long long)W * H)) out[o + 1] = (uint8_t)(m >> 16);
}

// ---------------------------------------------------------------------------
// U- and V-maps in one launch of 1024-thread CTAs.  The first ceil(W/32)
// CTAs build the U-map of a 32-column strip: 32 row phases x 32 columns walk
// the strip and bump a shared [D][32] histogram; each column's counts are
// then written once.  The remaining CTAs build the V-map of 8 rows each with
// shared [8][D] histograms.  Every output element is written exactly once,
// so no clearing is needed.
// ---------------------------------------------------------------------------

constexpr int kUVThreads = 1024, kVRows = 8;

__global__ void __launch_bounds__(kUVThreads)
    uvmap_kernel(const uint8_t *__restrict__ disp, int W, int H, int D, int ustrips,
                 uint16_t *__restrict__ umap, uint16_t *__restrict__ vmap) {
    extern __shared__ uint32_t hist[];
    wait_for_predecessor();
    if ((int)blockIdx.x < ustrips) {
        const int x0 = blockIdx.x * 32;
        const int col = threadIdx.x & 31, phase = threadIdx.x >> 5, nphase = kUVThreads / 32;
        for (int i = threadIdx.x; i < D * 32; i += kUVThreads) hist[i] = 0;
        __syncthreads();
        const int x = x0 + col;
        if (x < W) {
            for (int y = phase; y < H; y += nphase) {
                const int d = in_range((long long)y * W + x, (long long)W * H) ? disp[(size_t)y * W + x] : 0xFF;
                if (d < D && in_range(d * 32 + col, D * 32)) atomicAdd(&hist[d * 32 + col], 1u);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < D * 32; i += kUVThreads) {
            const int d = i >> 5, c = i & 31;
            if (x0 + c < W && in_range((long long)d * W + x0 + c, (long long)D * W)) umap[(size_t)d * W + x0 + c] = (uint16_t)hist[i];
        }
    } else {
        const int y0 = ((int)blockIdx.x - ustrips) * kVRows;
        for (int i = threadIdx.x; i < kVRows * D; i += kUVThreads) hist[i] = 0;
        __syncthreads();
        const int rows = min(kVRows, H - y0);
        for (int i = threadIdx.x; i < rows * W; i += kUVThreads) {
            const int r = i / W, x = i - r * W;
            const int d = in_range((long long)(y0 + r) * W + x, (long long)W * H) ? disp[(size_t)(y0 + r) * W + x] : 0xFF;
            if (d < D && in_range(r * D + d, kVRows * D)) atomicAdd(&hist[r * D + d], 1u);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < rows * D; i += kUVThreads)
            if (in_range((long long)y0 * D + i, (long long)H * D)) vmap[(size_t)y0 * D + i] = (uint16_t)hist[i];
    }
}

}  // namespace

SGM_GUARD_COUNTER(guard_hits_post)

cudaError_t launch_median(const uint8_t *in, uint8_t *out, int W, int H, int k, cudaStream_t s) {
    dim3 block(kMX, kMY), grid((W + 2 * kMX - 1) / (2 * kMX), (H + kMY - 1) / kMY);
    switch (k) {
        case 3: return launch_k(median_kernel<3>, grid, block, 0, s, in, out, W, H);
        case 5: return launch_k(median_kernel<5>, grid, block, 0, s, in, out, W, H);
        case 7: return launch_k(median_kernel<7>, grid, block, 0, s, in, out, W, H);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_uvmap(const uint8_t *disp, int W, int H, int D, uint16_t *umap, uint16_t *vmap,
                         cudaStream_t s) {
    const int ustrips = (W + 31) / 32, vblocks = (H + kVRows - 1) / kVRows;
    const size_t smem = (size_t)(D * 32 > kVRows * D ? D * 32 : kVRows * D) * sizeof(uint32_t);
    return launch_k(uvmap_kernel, dim3(ustrips + vblocks), dim3(kUVThreads), smem, s, disp, W, H, D, ustrips,
                    umap, vmap);
}

}  // namespace sgm
