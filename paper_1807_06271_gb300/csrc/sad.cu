// SAD matching cost (Sec. 3.1.2: the pixel-wise sum of absolute differences,
// over the 5 x 5 support region of Sec. 4.1):
//     C(x,y,d) = sum over |u| <= rw, |v| <= rh of |I_l(x+u, y+v) - I_r(x-d+u, y+v)|
// with both images read at clamped (replicated) coordinates, the maximum
// cmax = ww * wh * 255 where x - d < 0, and kPadCostWide in the padding slots
// d >= D.
//
// One CTA per segment of kSeg pixels of kRows consecutive rows.  The left
// rows (kSeg + 2 rw columns) and right rows (kSeg + Dp - 1 + 2 rw columns)
// the segment reaches, kRows + wh - 1 of each, are staged once in shared
// memory, read through the rectification maps when they are set, directly
// as the packed 16-bit pairs the arithmetic uses: (l, l) for a left pixel
// and (R[c], R[c-4]) for right column c.  For each column j of the segment
// and its halo and each 8-disparity chunk the CTA keeps the vertical sums
//     V(j, d) = sum_v |I_l(j, v) - I_r(j - d, v)|
// as four words, word k = the pair (d+k, d+k+4): the first row sums wh rows
// of absolute differences, each later row adds the row entering the window
// and subtracts the one leaving it (halves never borrow: V holds the row
// that leaves).  |a - b| = max.u16x2 - min.u16x2 (full rate on GB300).
// Each row's costs then add ww neighbouring columns of V, four packed adds
// per chunk and column (halves never carry: a cost is at most
// ww * wh * 255 <= 32766).  A thread sums a chunk and its mirror image at the
// other end of the disparity range, whose halves make up two 16-byte quarters of
// the pixel's folded record; consecutive threads write consecutive 32 bytes of the
// segment's contiguous records.
#include "sgm_internal.cuh"

namespace sgm {
namespace {

// 64 pixels x 4 rows per CTA: rows per CTA against threads measured on GB300
// (640 x 360, D = 60, 5 x 5): 8 rows 29.0 us, 16 rows 38.3, 2 rows (128
// threads) 29.0, 4 rows 27.0 us; more CTAs hide the row staging better.
//
// Bound by instruction issue and shared memory.  Two chunks per thread and the
// vertical sums in mirror order fold the records for nothing: chunks through a
// shared tile, then the records from it, and this, us: 1242 x 375, D = 128, 3 x 3
// 81.8, 70.0, 7 x 7 112.4, 101.0; 640 x 360, D = 60, 3 x 3 28.6, 24.6; 1280 x 720, D =
// 96, 7 x 7 139.3, 127.0 (chunks in their natural order 153.9: bank conflicts); halves
// exchanged between lanes 76.4, 103.6, 28.6, 133.2.  The column loop is not unrolled:
// with 54 registers instead of 40 four CTAs fit an SM instead of six (640 x 360 26.8).
constexpr int kSeg = 64, kRows = 4, kThreads = 256;

__device__ __forceinline__ uint32_t vmin2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t vmax2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// |a - b| of the pair words of one staged row for chunk (j, i), added to or
// subtracted from the chunk's four vertical-sum words.
template <bool ADD>
__device__ __forceinline__ void absdiff_row(uint4 &v, uint32_t l, const uint32_t *r) {
    const uint32_t r0 = r[0], r1 = r[-1], r2 = r[-2], r3 = r[-3];
    const uint32_t a0 = vmax2(l, r0) - vmin2(l, r0), a1 = vmax2(l, r1) - vmin2(l, r1);
    const uint32_t a2 = vmax2(l, r2) - vmin2(l, r2), a3 = vmax2(l, r3) - vmin2(l, r3);
    if (ADD) {
        v.x += a0;
        v.y += a1;
        v.z += a2;
        v.w += a3;
    } else {
        v.x -= a0;
        v.y -= a1;
        v.z -= a2;
        v.w -= a3;
    }
}

// The chunk at place r of a column's vertical sums: mirror images side by side (an
// even number of chunks, or one).
__device__ __forceinline__ int chunk_at(int r, int chunks) { return r & 1 ? chunks - 1 - (r >> 1) : r >> 1; }

// The pair of costs of the disparities (d, d + 4) at column x, with the padding and
// the columns left of the image put in.
__device__ __forceinline__ uint32_t edge_pair(uint32_t v, int d, int x, int D, uint32_t cmax) {
    const uint32_t lo = d >= D ? kPadCostWide : x - d < 0 ? cmax : (v & 0xFFFFu);
    const uint32_t hi = d + 4 >= D ? kPadCostWide : x - d - 4 < 0 ? cmax : (v >> 16);
    return lo | (hi << 16);
}

template <bool RECT>
__global__ void __launch_bounds__(kThreads)
    sad_cost_kernel(const uint8_t *__restrict__ left, const uint8_t *__restrict__ right, int pitch,
                    int W, int H, int D, int Dp, int ww, int wh, RectMaps maps,
                    uint4 *__restrict__ cost, unsigned *__restrict__ job_state) {
    extern __shared__ __align__(16) unsigned char sad_smem[];
    wait_for_predecessor();
    if (job_state && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *job_state = 0u;
    const int rw = ww / 2, rh = wh / 2;
    const int ncol = kSeg + 2 * rw;          // V columns (segment + halo)
    const int lcols = ncol, rcols = kSeg + Dp - 1 + 2 * rw;
    const int chunks = Dp / 8, mirrored = (chunks + 1) / 2;  // an even number of chunks, or one
    const int y0 = blockIdx.y * kRows, x0 = blockIdx.x * kSeg;
    const int nrows = min(kRows, H - y0);   // output rows of this CTA
    const int srows = nrows + wh - 1;       // staged rows: y0 - rh .. y0 + nrows - 1 + rh
    uint4 *V = reinterpret_cast<uint4 *>(sad_smem);                              // [ncol][chunks], chunk_at order
    uint32_t *Lp = reinterpret_cast<uint32_t *>(V + (size_t)ncol * chunks);      // [srows][lcols]: (l, l)
    uint8_t *Rb = reinterpret_cast<uint8_t *>(Lp + srows * lcols);               // [srows][rcols] bytes
    uint32_t *Rp = reinterpret_cast<uint32_t *>(Rb + ((srows * rcols + 3) & ~3));  // [srows][rcols]: (R[c], R[c-4])
    const int xl0 = x0 - rw;            // image column of left column 0
    const int xr0 = x0 - rw - (Dp - 1);  // image column of right column 0
    for (int i = threadIdx.x; i < srows * lcols; i += kThreads) {
        const int v = i / lcols, c = i - v * lcols;
        const int gy = min(max(y0 + v - rh, 0), H - 1), gx = min(max(xl0 + c, 0), W - 1);
        Lp[i] = rect_pixel<RECT>(left, pitch, W, H, gx, gy, maps.lx, maps.ly) * 0x00010001u;
    }
    for (int i = threadIdx.x; i < srows * rcols; i += kThreads) {
        const int v = i / rcols, c = i - v * rcols;
        const int gy = min(max(y0 + v - rh, 0), H - 1), gx = min(max(xr0 + c, 0), W - 1);
        Rb[i] = rect_pixel<RECT>(right, pitch, W, H, gx, gy, maps.rx, maps.ry);
    }
    __syncthreads();
    // right pairs; columns c < 4 have no c - 4 and are only read as the low half
    for (int i = threadIdx.x; i < srows * rcols; i += kThreads) {
        const int v = i / rcols, c = i - v * rcols;
        Rp[i] = Rb[i] | (c >= 4 ? (uint32_t)Rb[i - 4] << 16 : 0u);
    }
    __syncthreads();
    const uint32_t cmax = (uint32_t)(ww * wh * 255);
    const int npx = min(kSeg, W - x0);
    const bool ragged = D != Dp, border = x0 < Dp;
    for (int r = 0; r < nrows; r++) {
        // Vertical sums of output row y0 + r (staged rows r .. r + wh - 1).  Word k
        // of chunk (j, i) reads the right pair at c0 - k, c0 = j + Dp - 1 - 8i:
        // column j - d + Dp - 1 for d = 8i + k, high half 4 columns left (>= j >= 0).
        for (int it = threadIdx.x; it < ncol * chunks; it += kThreads) {
            const int j = it / chunks, i = chunk_at(it - j * chunks, chunks);
            const int c0 = j + Dp - 1 - 8 * i;
            uint4 v;
            if (r == 0) {
                v = make_uint4(0u, 0u, 0u, 0u);
                for (int q = 0; q < wh; q++) absdiff_row<true>(v, Lp[q * lcols + j], Rp + q * rcols + c0);
            } else {
                v = V[it];
                const int qin = r + wh - 1, qout = r - 1;
                absdiff_row<true>(v, Lp[qin * lcols + j], Rp + qin * rcols + c0);
                absdiff_row<false>(v, Lp[qout * lcols + j], Rp + qout * rcols + c0);
            }
            V[it] = v;
        }
        __syncthreads();
        // C(x, d) = sum over u < ww of V(x - x0 + u, d); cmax where x - d < 0.  A thread
        // sums chunk i and its mirror image m = chunks - 1 - i, whose halves make up the
        // quarters 2i and 2i + 1 of the pixel's record: the pairs 8i + e, e < 4, hold the
        // lower halves of i and the upper ones of m backwards, the pairs 8i + 4 + e what
        // remains.  Half of the lanes read m first, so that the lanes read distinct banks.
        const long long at = ((long long)(y0 + r) * W + x0) * chunks;
        const int mfirst = chunks > 1 && (threadIdx.x & 4) ? 1 : 0, step = chunks > 1 ? 1 - 2 * mfirst : 0;
        for (int it = threadIdx.x; it < npx * mirrored; it += kThreads) {
            const int px = it / mirrored, i = it - px * mirrored;
            const uint4 *v = V + px * chunks + 2 * i + mfirst;
            uint32_t a[4] = {0u, 0u, 0u, 0u}, b[4] = {0u, 0u, 0u, 0u};
#pragma unroll 1
            for (int u = 0; u < ww; u++, v += chunks) {
                const uint4 p = v[0], q = v[step];
                a[0] += p.x;
                a[1] += p.y;
                a[2] += p.z;
                a[3] += p.w;
                b[0] += q.x;
                b[1] += q.y;
                b[2] += q.z;
                b[3] += q.w;
            }
            uint32_t l[4], m[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                l[k] = mfirst ? b[k] : a[k];
                m[k] = mfirst ? a[k] : b[k];
            }
            if (ragged || border) {
                const int x = x0 + px, dm = Dp - 8 - 8 * i;
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    l[k] = edge_pair(l[k], 8 * i + k, x, D, cmax);
                    m[k] = edge_pair(m[k], dm + k, x, D, cmax);
                }
            }
            const long long o = at + px * chunks + 2 * i;
            if (in_range(o, (long long)W * H * chunks))
                cost[o] = make_uint4(__byte_perm(l[0], m[3], 0x7610), __byte_perm(l[1], m[2], 0x7610),
                                     __byte_perm(l[2], m[1], 0x7610), __byte_perm(l[3], m[0], 0x7610));
            if (chunks > 1 && in_range(o + 1, (long long)W * H * chunks))
                cost[o + 1] = make_uint4(__byte_perm(l[0], m[3], 0x5432), __byte_perm(l[1], m[2], 0x5432),
                                         __byte_perm(l[2], m[1], 0x5432), __byte_perm(l[3], m[0], 0x5432));
        }
        __syncthreads();
    }
}

// The 5 x 5 window of Sec. 4.1, all in registers.  One CTA covers kRows5 rows and
// kSegs segments of kSegLen pixels; a thread walks one segment from left to right
// with eight disparities, the four 4q + e and the four Dp-1-4q-e that make up
// quarter q of a folded record, as the packed pairs (e, e + 2).  Per column it
// takes one new pair of right pixels for either end (the other two are last
// column's), the absolute differences of its kRows5 + 4 image rows, the vertical
// sums of its kRows5 output rows (each the one above plus the row entering minus
// the row leaving), and adds the last four columns' sums, which it keeps.
// Bound by instruction issue (about 55 a column, row and quarter); the kernel
// above goes through shared memory and two barriers per row for the same
// sums.  kSegLen is 3 modulo 4 so that the segments of a warp read distinct banks.
// Measured, us, the kernel above and this one: 640 x 360, D = 60: 26.9, 21.2; 1242 x
// 375, D = 128: 85.8, 55.6; 430 x 312, D = 192: 52.1, 32.8.  4 rows took 27.0 / 68.0 /
// 41.1, segments of 31 pixels 37 / 58.8 / 37.2.
constexpr int kRows5 = 2, kSegLen = 15;
// Segments of a row that a CTA covers.
__host__ __device__ constexpr int window5_segs(int Dp) { return Dp < 32 ? 32 : 128 / (Dp / 8); }

// Whether a W x H image with Dp slots takes this kernel.  With few slots its CTAs are
// wide, and a small image has too few of them.  Measured, us, the kernel above and
// this one:
//   8 to 32 slots  320 x 240 (D = 16) 10.5, 17.0;  640 x 480 22.6, 25.1;  800 x 600 32.2, 25.6;
//                  1280 x 720 51.4, 47.2, (D = 16) 36.9, 37.0;  640 x 480 (D = 8) 16.5, 18.6
//   64 slots       320 x 240 14.6, 16.6;  350 x 250 16.5, 16.4;  300 x 300 16.4, 16.4;
//                  240 x 480 20.6, 16.5;  480 x 260 20.6, 16.7
//   more           160 x 96 (D = 96) 15.5, 14.1;  100 x 40 (D = 128) 16.4, 13.4;  60 x 64 16.5, 13.1
// An image of a third of a CTA's width leaves most of it idle: 40 x 4000 (D = 128) 49.3,
// 53.6;  16 x 1000 18.3, 18.8;  but 30 x 400 (D = 200) 22.6, 15.3.
bool window5_pays(int W, int H, int Dp) {
    const long npx = (long)W * H;
    return 3 * W > window5_segs(Dp) * kSegLen && (Dp >= 96 || npx >= (Dp == 64 ? 90000 : 400000));
}

template <bool RECT>
__global__ void __launch_bounds__(128)
    sad5_cost_kernel(const uint8_t *__restrict__ left, const uint8_t *__restrict__ right, int pitch, int W, int H, int D,
                     int Dp, RectMaps maps, uint4 *__restrict__ cost, unsigned *__restrict__ job_state) {
    extern __shared__ __align__(16) unsigned char sad_smem[];
    wait_for_predecessor();
    if (job_state && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *job_state = 0u;
    constexpr int S = kRows5 + 4;  // staged rows
    const int quarters = Dp / 8, segs = window5_segs(Dp), width = segs * kSegLen;
    const int x0 = blockIdx.x * width, y0 = blockIdx.y * kRows5;
    const int lcols = width + 8, rcols = width + 8 + Dp;
    uint32_t *Lp = reinterpret_cast<uint32_t *>(sad_smem);  // [S][lcols]: (l, l), column x0 - 2 + i
    uint32_t *Rp = Lp + S * lcols;                           // [S][rcols]: (R[c], R[c-2]), column x0 - 2 - Dp + 1 + i
#pragma unroll 4
    for (int i = threadIdx.x; i < S * lcols; i += blockDim.x) {
        const int v = i / lcols, c = i - v * lcols;
        const int gy = min(max(y0 + v - 2, 0), H - 1), gx = min(max(x0 - 2 + c, 0), W - 1);
        Lp[i] = rect_pixel<RECT>(left, pitch, W, H, gx, gy, maps.lx, maps.ly) * 0x00010001u;
    }
#pragma unroll 4
    for (int i = threadIdx.x; i < S * rcols; i += blockDim.x) {
        const int v = i / rcols, c = i - v * rcols;
        const int gy = min(max(y0 + v - 2, 0), H - 1), gx = x0 - 2 - Dp + 1 + c;
        const uint32_t a = rect_pixel<RECT>(right, pitch, W, H, min(max(gx, 0), W - 1), gy, maps.rx, maps.ry);
        const uint32_t b = rect_pixel<RECT>(right, pitch, W, H, min(max(gx - 2, 0), W - 1), gy, maps.rx, maps.ry);
        Rp[i] = a | b << 16;
    }
    __syncthreads();
    const int seg = threadIdx.x / quarters, q = threadIdx.x - seg * quarters;
    if (seg >= segs) return;
    const int xs = seg * kSegLen;  // first pixel of the segment, relative to x0
    const uint32_t cmax = 25u * 255u;
    // column j of the segment (image column x0 - 2 + xs + j): the lower disparities read the
    // right pairs at lo + j (e = 0, 2) and lo + j - 1 (e = 1, 3), the upper ones those at
    // hi + j (e = 2, 0) and hi + j + 1 (e = 3, 1)
    const uint32_t *L = Lp + xs, *lo = Rp + xs + Dp - 1 - 4 * q, *hi = Rp + xs + 4 * q + 2;
    uint32_t l1[S], h0[S];  // the pairs that column j + 1 takes over: lo + j, hi + j + 1
#pragma unroll
    for (int v = 0; v < S; v++) {
        l1[v] = lo[v * rcols - 1];
        h0[v] = hi[v * rcols];
    }
    uint32_t past[4][kRows5][4], sum4[kRows5][4];  // vertical sums of the last four columns, and their sum
#pragma unroll
    for (int r = 0; r < kRows5; r++)
#pragma unroll
        for (int k = 0; k < 4; k++) past[0][r][k] = past[1][r][k] = past[2][r][k] = past[3][r][k] = sum4[r][k] = 0u;
    const int dmax = Dp - 1 - 4 * q;  // the thread's largest disparity
    uint32_t pad[4];                  // kPadCostWide where a word holds padding
#pragma unroll
    for (int e = 0; e < 4; e++)
        pad[e] = (4 * q + e >= D ? kPadCostWide : 0u) | (dmax - e >= D ? kPadCostWide << 16 : 0u);
#pragma unroll 1
    for (int j0 = 0; j0 < kSegLen + 4; j0 += 4) {
#pragma unroll
        for (int jj = 0; jj < 4; jj++) {
            const int j = j0 + jj;
            uint32_t V[kRows5][4], first[kRows5 - 1][4];  // first: the rows that leave the later windows
#pragma unroll
            for (int v = 0; v < S; v++) {
                const uint32_t l = L[v * lcols + j];
                const uint32_t w[4] = {lo[v * rcols + j], l1[v], h0[v], hi[v * rcols + j + 1]};
                l1[v] = w[0];
                h0[v] = w[3];
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const uint32_t d = vmax2(l, w[k]) - vmin2(l, w[k]);
                    if (v < kRows5 - 1) first[v][k] = d;
                    if (v < 5) V[0][k] = v == 0 ? d : V[0][k] + d;
                    else V[v - 4][k] = V[v - 5][k] + d - first[v - 5][k];
                }
            }
            const int px = j - 4;  // the pixel whose window ends at this column
            const int x = x0 + xs + px;
#pragma unroll
            for (int r = 0; r < kRows5; r++) {
                uint32_t c[4];
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    c[k] = sum4[r][k] + V[r][k];
                    sum4[r][k] = c[k] - past[jj][r][k];
                    past[jj][r][k] = V[r][k];
                }
                if (px >= 0 && px < kSegLen && x < W && y0 + r < H) {
                    // c: (e = 0, 2), (1, 3) of the lower and (2, 0), (3, 1) of the upper disparities
                    uint32_t o[4] = {__byte_perm(c[0], c[2], 0x7610), __byte_perm(c[1], c[3], 0x7610),
                                     __byte_perm(c[0], c[2], 0x5432), __byte_perm(c[1], c[3], 0x5432)};
                    if (x < dmax) {
#pragma unroll
                        for (int e = 0; e < 4; e++) {
                            const uint32_t a = x < 4 * q + e ? cmax : o[e] & 0xFFFFu;
                            const uint32_t b = x < dmax - e ? cmax : o[e] >> 16;
                            o[e] = a | b << 16;
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 4; e++) o[e] |= pad[e];  // a cost has no bit that 0x7FFF lacks
                    const long long at = ((long long)(y0 + r) * W + x) * quarters + q;
                    if (in_range(at, (long long)W * H * quarters)) cost[at] = make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
        }
    }
}

}  // namespace

SGM_GUARD_COUNTER(guard_hits_sad)

cudaError_t launch_sad_cost(const uint8_t *left, const uint8_t *right, int pitch, int W, int H,
                            int D, int ww, int wh, const RectMaps &maps, uint16_t *cost,
                            unsigned *job_state, cudaStream_t s) {
    if (ww < 1 || wh < 1 || ww > kMaxSadWindow || wh > kMaxSadWindow)
        return cudaErrorInvalidValue;
    const int Dp = padded_disparities(D);
    if (ww == 5 && wh == 5 && window5_pays(W, H, Dp)) {
        const int width = window5_segs(Dp) * kSegLen;
        const size_t smem = (size_t)(kRows5 + 4) * (2 * (width + 8) + Dp) * sizeof(uint32_t);
        return launch_k(maps.lx ? sad5_cost_kernel<true> : sad5_cost_kernel<false>,
                        dim3((W + width - 1) / width, (H + kRows5 - 1) / kRows5), dim3(128), smem, s, left, right, pitch, W, H,
                        D, Dp, maps, reinterpret_cast<uint4 *>(cost), job_state);
    }
    const int rw = ww / 2;
    const int ncol = kSeg + 2 * rw, rcols = kSeg + Dp - 1 + 2 * rw;
    const size_t srows = (size_t)kRows + wh - 1;
    const size_t smem = (size_t)ncol * (Dp / 8) * sizeof(uint4) + srows * ncol * 4 +
                        ((srows * rcols + 3) & ~(size_t)3) + srows * rcols * 4;
    const dim3 grid((W + kSeg - 1) / kSeg, (H + kRows - 1) / kRows);
    uint4 *out = reinterpret_cast<uint4 *>(cost);
    auto kernel = maps.lx ? sad_cost_kernel<true> : sad_cost_kernel<false>;
    const cudaError_t e = allow_max_smem(kernel);
    if (e != cudaSuccess) return e;
    return launch_k(kernel, grid, dim3(kThreads), smem, s, left, right, pitch, W, H, D, Dp, ww, wh, maps, out,
                    job_state);
}

}  // namespace sgm
