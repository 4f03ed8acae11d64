// Census transform of both images of a pair (Sec. 3.1.2).
//
// One CTA covers a 32 x 8 pixel tile of one image (blockIdx.z selects left or
// right).  The tile and its (cw-1)/2, (ch-1)/2 halo are staged once in shared
// memory as 16-bit values with 256 standing for "outside the image", which is
// never darker than a centre pixel and so yields the 0 bit the border rule
// asks for.  Each thread then builds its pixel's code from shared memory.
// Bit k of a code is set iff the k-th window neighbour (raster order, centre
// skipped) is darker than the centre.  Codes of up to 32 bits are stored as
// uint32, longer ones as uint64.  HBM traffic: 1 byte read + 4/8 bytes
// written per pixel and image.
#include <type_traits>

#include "sgm_internal.cuh"

namespace sgm {
namespace {

constexpr int kBX = 32, kBY = 8;
constexpr int kRows = 4;  // rows per thread of the unrolled census kernel

// One CTA covers 32 x 32 pixels of one image; a thread computes the pixels
// of kRows consecutive rows of one column.  The tile plus halo is staged as
// bytes with 255 for "outside the image": 255 is never darker than a centre
// pixel, which gives the 0 bit the border rule asks for.  Each bit is the
// sign of I(q) - I(p), shifted into one of two 32-bit halves (two
// instructions per bit).  The thread's windows overlap: it walks the
// kRows + CH - 1 tile rows it touches from the bottom up, loads each row's CW
// bytes once, and appends them to every pixel whose window holds that row;
// every pixel thus receives its window backwards, so the first neighbour in
// raster order ends at bit 0.
template <typename CodeT, int CW, int CH, bool RECT>
__global__ void __launch_bounds__(kBX *kBY)
    census_kernel(const uint8_t *__restrict__ left, const uint8_t *__restrict__ right, int pitch,
                  int W, int H, CodeT *__restrict__ codes, RectMaps maps) {
    wait_for_predecessor();
    constexpr int TW = kBX + CW - 1, TH = kBY * kRows + CH - 1;
    constexpr int RX = CW / 2, RY = CH / 2;
    constexpr int NB = CW * CH - 1;  // bits per code
    __shared__ uint8_t tile[TH][TW];
    const uint8_t *img = blockIdx.z ? right : left;
    const uint16_t *mx = blockIdx.z ? maps.rx : maps.lx, *my = blockIdx.z ? maps.ry : maps.ly;
    const int x0 = blockIdx.x * kBX - RX, y0 = blockIdx.y * kBY * kRows - RY;
    const int tid = threadIdx.y * kBX + threadIdx.x;
    // All of a thread's tile loads are issued before any is stored, so their
    // latencies overlap instead of adding up.
    constexpr int kLoads = (TW * TH + kBX * kBY - 1) / (kBX * kBY);
    uint8_t v[kLoads];
#pragma unroll
    for (int k = 0; k < kLoads; k++) {
        const int i = tid + k * kBX * kBY;
        const int ty = i / TW, tx = i - ty * TW;
        const int gx = x0 + tx, gy = y0 + ty;
        v[k] = (i < TW * TH && gx >= 0 && gx < W && gy >= 0 && gy < H)
                   ? rect_pixel<RECT>(img, pitch, W, H, gx, gy, mx, my)
                   : 255;
    }
#pragma unroll
    for (int k = 0; k < kLoads; k++) {
        const int i = tid + k * kBX * kBY;
        if (i < TW * TH) tile[i / TW][i % TW] = v[k];
    }
    __syncthreads();
    const int x = blockIdx.x * kBX + threadIdx.x;
    if (x >= W) return;
    const int ly0 = threadIdx.y * kRows;  // first tile row of the thread's windows
    int c[kRows];
    uint32_t lo[kRows], hi[kRows];
#pragma unroll
    for (int r = 0; r < kRows; r++) {
        c[r] = tile[ly0 + r + RY][threadIdx.x + RX];
        lo[r] = hi[r] = 0u;
    }
#pragma unroll
    for (int t = kRows + CH - 2; t >= 0; t--) {  // tile row ly0 + t, bottom up
        int q[CW];
#pragma unroll
        for (int wx = 0; wx < CW; wx++) q[wx] = tile[ly0 + t][threadIdx.x + wx];
#pragma unroll
        for (int r = 0; r < kRows; r++) {
            const int wy = t - r;  // window row of tile row t for pixel r
            if (wy < 0 || wy >= CH) continue;
#pragma unroll
            for (int wx = CW - 1; wx >= 0; wx--) {
                if (wy == RY && wx == RX) continue;
                // bit index of neighbour (wy, wx) in raster order, centre skipped
                const int bit = wy * CW + wx - (wy * CW + wx > RY * CW + RX ? 1 : 0);
                const uint32_t diff = (uint32_t)(q[wx] - c[r]);
                if (bit >= 32) hi[r] = __funnelshift_l(diff, hi[r], 1);
                else lo[r] = __funnelshift_l(diff, lo[r], 1);
            }
        }
    }
    static_assert(NB <= 64, "codes hold at most 64 bits");
#pragma unroll
    for (int r = 0; r < kRows; r++) {
        const int y = blockIdx.y * kBY * kRows + ly0 + r;
        if (y >= H) break;
        CodeT code;
        if constexpr (sizeof(CodeT) == 8) code = ((uint64_t)hi[r] << 32) | lo[r];
        else code = lo[r];
        const long long ci = (long long)blockIdx.z * W * H + (long long)y * W + x;
        if (in_range(ci, 2LL * W * H)) codes[ci] = code;
    }
}

// Generic window (any odd size up to 64 bits), loops not unrolled.
template <typename CodeT, bool RECT>
__global__ void __launch_bounds__(kBX *kBY)
    census_kernel_any(const uint8_t *__restrict__ left, const uint8_t *__restrict__ right, int pitch,
                      int W, int H, int cw, int ch, CodeT *__restrict__ codes, RectMaps maps) {
    wait_for_predecessor();
    extern __shared__ uint16_t tile_any[];
    const int TW = kBX + cw - 1, TH = kBY + ch - 1;
    const int rx = cw / 2, ry = ch / 2;
    const uint8_t *img = blockIdx.z ? right : left;
    const uint16_t *mx = blockIdx.z ? maps.rx : maps.lx, *my = blockIdx.z ? maps.ry : maps.ly;
    const int x0 = blockIdx.x * kBX - rx, y0 = blockIdx.y * kBY - ry;
    const int tid = threadIdx.y * kBX + threadIdx.x;
    for (int i = tid; i < TW * TH; i += kBX * kBY) {
        int ty = i / TW, tx = i - ty * TW;
        int gx = x0 + tx, gy = y0 + ty;
        tile_any[i] = (gx >= 0 && gx < W && gy >= 0 && gy < H)
                          ? (uint16_t)rect_pixel<RECT>(img, pitch, W, H, gx, gy, mx, my)
                          : (uint16_t)256;
    }
    __syncthreads();
    const int x = blockIdx.x * kBX + threadIdx.x, y = blockIdx.y * kBY + threadIdx.y;
    if (x >= W || y >= H) return;
    const uint16_t c = tile_any[(threadIdx.y + ry) * TW + threadIdx.x + rx];
    CodeT code = 0;
    int bit = 0;
    for (int wy = 0; wy < ch; wy++)
        for (int wx = 0; wx < cw; wx++) {
            if (wy == ry && wx == rx) continue;
            code |= (CodeT)(tile_any[(threadIdx.y + wy) * TW + threadIdx.x + wx] < c) << bit;
            bit++;
        }
    const long long ci = (long long)blockIdx.z * W * H + (long long)y * W + x;
    if (in_range(ci, 2LL * W * H)) codes[ci] = code;
}

// ---------------------------------------------------------------------------
// Matching cost volume (Eq. 1): C(x,y,d) = popc(code_l(x,y) ^ code_r(x-d,y)),
// or the code width when x-d < 0, for d < D; padding slots d >= D hold
// kPadCost.  One CTA per segment of kSeg pixels of one row: the
// segment's left codes and the right codes it reaches (kSeg + Dp + 2 of them)
// are staged in shared memory.  A thread computes two words (eight
// disparities, four at either end of the range) of the folded records of
// two neighbouring pixels from two runs of five right codes read as
// aligned vectors, with consecutive threads on consecutive pixel pairs
// (conflict-free reads); the segment is transposed through a padded shared
// tile and written out with coalesced 8-byte stores (the segment's Dp-byte
// pixel records are contiguous in global memory).  popc runs on the XU pipe
// (16 per SM per clock; two per estimate for 64-bit codes), which bounds
// this kernel.
// ---------------------------------------------------------------------------

// 2 warps per 32-pixel segment: each thread computes 4 chunks for D = 128
// (measured on GB300 against 64-pixel segments: 256 threads 37.8 us, 128
// threads 35.6 us, this 35.0 us on the 1242 x 375, D = 128 cost volume).
constexpr int kCostThreads = 64, kSeg = 32;

__device__ __forceinline__ uint32_t popcnt(uint32_t v) { return __popc(v); }
__device__ __forceinline__ uint32_t popcnt(uint64_t v) { return __popcll(v); }

// Dp is a template parameter: with it at run time the loops' address and piece
// arithmetic took a fifth of the instructions (1280 x 720, D = 128, 24-bit codes: 45.0
// us; pieces stepped without a division 41.1; this 33.0).
template <typename CodeT, int Dp, bool RAGGED>
__global__ void __launch_bounds__(kCostThreads)
    cost_kernel(const CodeT *__restrict__ codes, int W, int H, int D, int nbits, uint8_t *__restrict__ cost,
                unsigned *__restrict__ job_state) {
    wait_for_predecessor();
    if (job_state && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *job_state = 0u;
    extern __shared__ __align__(16) unsigned char cost_smem[];
    constexpr int stride = Dp + 8;  // padded tile row (bytes)
    uint8_t *tile = cost_smem;                                          // [kSeg][stride]
    constexpr int tile_bytes = (kSeg * stride + 15) & ~15;
    CodeT *cl = reinterpret_cast<CodeT *>(cost_smem + tile_bytes);     // [kSeg]
    CodeT *cr = cl + kSeg;                                              // [kSeg + Dp + 2]
    const int y = blockIdx.y, x0 = blockIdx.x * kSeg;
    const int xr0 = x0 - Dp - 1;  // right code cr[i] is column xr0 + i
    const CodeT *rowl = codes + (size_t)y * W;
    const CodeT *rowr = codes + (size_t)W * H + (size_t)y * W;
    for (int i = threadIdx.x; i < kSeg; i += kCostThreads)
        cl[i] = x0 + i < W && in_range((long long)y * W + x0 + i, (long long)W * H) ? rowl[x0 + i] : 0;
    for (int i = threadIdx.x; i < kSeg + Dp + 2; i += kCostThreads) {
        const int xr = xr0 + i;
        cr[i] = (xr >= 0 && xr < W && in_range((long long)W * H + (long long)y * W + xr, 2LL * W * H)) ? rowr[xr] : 0;
    }
    __syncthreads();
    constexpr int chunks = Dp / 8;
    const bool border = x0 < Dp;  // only the first segments see x - d < 0
    // A thread takes the two words (four pairs) i of the pixel pair (px, px+1), px
    // even: the disparities 4i + e and Dp-1-4i-e, e < 4.  Column x - d of pixel px
    // sits at cr[px - d + Dp + 1], so the pair needs two runs of five codes:
    // wl[k] = cr[px + Dp - 2 - 4i + k] (pixel px uses wl[3 - e], px + 1 wl[4 - e]) and
    // wh[k] = cr[px + 2 + 4i + k] (wh[e] and wh[e + 1]); both start at an even
    // index, so the codes are read as aligned vectors of two.
    // A thread's pixel pair is the same for all its words (kCostThreads is a
    // multiple of kSeg / 2), so its two left codes are read once.
    static_assert(kCostThreads % (kSeg / 2) == 0, "one pixel pair per thread");
    const int px = 2 * (threadIdx.x % (kSeg / 2));
    auto two = [](const CodeT *p, CodeT &a, CodeT &b) {
        if constexpr (sizeof(CodeT) == 8) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p);
            a = v.x;
            b = v.y;
        } else {
            const uint2 v = *reinterpret_cast<const uint2 *>(p);
            a = v.x;
            b = v.y;
        }
    };
    CodeT a0, a1;
    two(cl + px, a0, a1);
#pragma unroll 2
    for (int i = threadIdx.x / (kSeg / 2); i < chunks; i += kCostThreads / (kSeg / 2)) {
        const CodeT *rl = cr + px + Dp - 2 - 4 * i, *rh = cr + px + 2 + 4 * i;
        CodeT wl[5], wh[5];
        two(rl, wl[0], wl[1]);
        two(rl + 2, wl[2], wl[3]);
        wl[4] = rl[4];
        two(rh, wh[0], wh[1]);
        two(rh + 2, wh[2], wh[3]);
        wh[4] = rh[4];
#pragma unroll
        for (int p = 0; p < 2; p++) {
            const CodeT a = p ? a1 : a0;
            uint32_t lo[4], hi[4];
#pragma unroll
            for (int e = 0; e < 4; e++) {
                lo[e] = popcnt(a ^ wl[3 + p - e]);
                hi[e] = popcnt(a ^ wh[p + e]);
            }
            if (RAGGED || border) {
                const int x = x0 + px + p;
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    const int dl = 4 * i + e, dh = Dp - 1 - dl;
                    if (x - dl < 0) lo[e] = (uint32_t)nbits;
                    if (x - dh < 0) hi[e] = (uint32_t)nbits;
                    if (RAGGED && dl >= D) lo[e] = kPadCost;
                    if (RAGGED && dh >= D) hi[e] = kPadCost;
                }
            }
            uint2 w;
            w.x = (hi[0] * 256u + hi[1]) * 65536u + (lo[0] * 256u + lo[1]);
            w.y = (hi[2] * 256u + hi[3]) * 65536u + (lo[2] * 256u + lo[3]);
            *reinterpret_cast<uint2 *>(tile + (px + p) * stride + 8 * i) = w;
        }
    }
    __syncthreads();
    const int npx = min(kSeg, W - x0);
    uint8_t *out = cost + ((size_t)y * W + x0) * Dp;
    // thread t copies the 8-byte pieces t, t + kCostThreads, ..: piece q of pixel p,
    // stepped along without a division per piece
    constexpr int dp = kCostThreads / chunks, dq = kCostThreads - dp * chunks;
    int p = threadIdx.x / chunks, q = threadIdx.x - p * chunks;
    while (p < npx) {
        // a record of 8 bytes starting at byte o of the W x H x Dp volume
        const long long o = ((long long)y * W + x0 + p) * Dp + 8 * q;
        if (in_range(o, (long long)W * H * Dp - 8 + 1))
            *reinterpret_cast<uint2 *>(out + p * Dp + 8 * q) = *reinterpret_cast<const uint2 *>(tile + p * stride + 8 * q);
        p += dp;
        q += dq;
        if (q >= chunks) {
            q -= chunks;
            p++;
        }
    }
}

}  // namespace

cudaError_t launch_census(const uint8_t *left, const uint8_t *right, int pitch, int W, int H,
                          int cw, int ch, int code_bytes, void *codes, const RectMaps &maps,
                          cudaStream_t s) {
    dim3 block(kBX, kBY), grid((W + kBX - 1) / kBX, (H + kBY - 1) / kBY, 2);
    const dim3 grid4((W + kBX - 1) / kBX, (H + kBY * kRows - 1) / (kBY * kRows), 2);
    const bool rect = maps.lx != nullptr;
#define SGM_CENSUS(T, CWv, CHv)                                                                                     \
    (rect ? launch_k(census_kernel<T, CWv, CHv, true>, grid4, block, 0, s, left, right, pitch, W, H, (T *)codes, maps) \
          : launch_k(census_kernel<T, CWv, CHv, false>, grid4, block, 0, s, left, right, pitch, W, H, (T *)codes, maps))
    // the usual windows unrolled (641 x 479 pair, 7 x 7: 21.2 us any-window, 10.2 unrolled)
    if (cw == 3 && ch == 3) return SGM_CENSUS(uint32_t, 3, 3);
    if (cw == 5 && ch == 5) return SGM_CENSUS(uint32_t, 5, 5);
    if (cw == 7 && ch == 5) return SGM_CENSUS(uint64_t, 7, 5);
    if (cw == 7 && ch == 7) return SGM_CENSUS(uint64_t, 7, 7);
    if (cw == 9 && ch == 7) return SGM_CENSUS(uint64_t, 9, 7);
#undef SGM_CENSUS
    const size_t smem = (size_t)(kBX + cw - 1) * (kBY + ch - 1) * sizeof(uint16_t);
    if (code_bytes == 4) {
        uint32_t *c = (uint32_t *)codes;
        return rect ? launch_k(census_kernel_any<uint32_t, true>, grid, block, smem, s, left, right, pitch, W, H, cw, ch, c, maps)
                    : launch_k(census_kernel_any<uint32_t, false>, grid, block, smem, s, left, right, pitch, W, H, cw, ch, c, maps);
    }
    uint64_t *c = (uint64_t *)codes;
    return rect ? launch_k(census_kernel_any<uint64_t, true>, grid, block, smem, s, left, right, pitch, W, H, cw, ch, c, maps)
                : launch_k(census_kernel_any<uint64_t, false>, grid, block, smem, s, left, right, pitch, W, H, cw, ch, c, maps);
}

SGM_GUARD_COUNTER(guard_hits_census)

}  // namespace sgm

namespace sgm {

// The CUDA-core kernel measured faster than the tensor-core one on GB300 for
// every D the latter supports (1242 x 375, D = 128: 31.3 against 43.1 us).
int cost_kernel_for(int) { return SGM_COST_KERNEL_CUDA_CORES; }

cudaError_t launch_cost(const void *codes, int code_bytes, int W, int H, int D, int nbits,
                        uint8_t *cost, unsigned *job_state, unsigned *status, int kernel, cudaStream_t s) {
    if (kernel == SGM_COST_KERNEL_AUTO) kernel = cost_kernel_for(D);
    if (kernel == SGM_COST_KERNEL_TENSOR_CORES)
        return launch_cost_mma(codes, code_bytes, W, H, D, nbits, cost, job_state, status, s);
    if (kernel != SGM_COST_KERNEL_CUDA_CORES) return cudaErrorInvalidValue;
    const int Dp = padded_disparities(D);
    const size_t smem = (((size_t)kSeg * (Dp + 8) + 15) & ~(size_t)15) + (size_t)(2 * kSeg + Dp + 2) * code_bytes;
    const dim3 grid((W + kSeg - 1) / kSeg, H);
    auto go = [&](auto kernel, auto *c) {
        return launch_k(kernel, grid, dim3(kCostThreads), smem, s, c, W, H, D, nbits, cost, job_state);
    };
    const bool rag = D != Dp;
    const uint32_t *c4 = (const uint32_t *)codes;
    const uint64_t *c8 = (const uint64_t *)codes;
    cudaError_t e;
#define SGM_COST(P)                                                                                       \
    case P:                                                                                               \
        if (code_bytes == 4) e = rag ? go(cost_kernel<uint32_t, P, true>, c4) : go(cost_kernel<uint32_t, P, false>, c4); \
        else e = rag ? go(cost_kernel<uint64_t, P, true>, c8) : go(cost_kernel<uint64_t, P, false>, c8);                 \
        break
    switch (Dp) {
        SGM_COST(8);
        SGM_COST(16);
        SGM_COST(32);
        SGM_COST(64);
        SGM_COST(96);
        SGM_COST(128);
        SGM_COST(160);
        SGM_COST(192);
        SGM_COST(224);
        SGM_COST(256);
        default: return cudaErrorInvalidValue;
    }
#undef SGM_COST
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace sgm
