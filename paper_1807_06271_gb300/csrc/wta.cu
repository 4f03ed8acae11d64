// Winner-takes-all on S = sum of the path planes (Sec. 3.1.3), the right
// disparity taken from the same S (Sec. 3.1.4) and the left-right check.
//
// One CTA per image row.  The planes share the aggregation kernel's layout
// (all planes of a pixel back to back, folded records): a pixel's disparities
// are held by Dp / 8 lanes, four pairs (d, Dp-1-d) each, so a warp covers G
// pixels at once, and every group of lanes walks a contiguous segment of the
// row from left to right.  The records of the next kStages - 1 pixels of each
// group are on their way into shared memory (16-byte asynchronous copies)
// while one is reduced: the kernel is bound by HBM, whose rate follows the bytes
// in flight, and loads into registers would wait for one another (a warp has
// few scoreboards).
//
// Sums.  The bytes of a word are added as two sums of pairs: O over the odd
// bytes (one byte-permute and an add per plane) and V over the whole words,
// whose carries cancel in V - 256 O, the even ones.  No half carries: S <= 8 *
// 255 for 8-bit planes, and the host bounds the 16-bit path costs so that their
// sum fits 16 bits.
//
// Winners.  The key of a disparity is (S << 8) | d, one byte-permute of the
// packed sums with a per-lane constant (whose top byte is 0xFF for d >= D).  The
// left winner is the minimum key over the pixel's lanes (ties go to the
// smallest d, which sits in the low bits).  The right winner of x' is the minimum
// over d of key(x' + d, d): as a lane moves one pixel to the right, the slot x -
// d of its disparity d becomes that of d + 1, so the running minima of a lane's
// four consecutive disparities move along by one register and only the one
// that falls off goes to the slot's shared-memory minimum: 2 shared atomics
// per pixel and lane instead of 8.  After a CTA barrier the row's LR check runs
// from shared memory.  HBM traffic: the planes once (npaths * Dp path costs per
// pixel) plus 1 byte written per pixel.  Measured on GB300 against one warp-wide load
// per plane and 8 shared atomics per pixel and lane: 1280 x 720, D = 128, 4
// paths 90 -> 77 us, 640 x 360, D = 60, 4 paths 24.4 -> 18.3, 1242 x 375, D =
// 128, 8 paths 80 -> 80 (477 MB at 6.0 TB/s).
#include "sgm_internal.cuh"

namespace sgm {
namespace {

// 16 warps and 3 stages: 64 KB of records in flight per CTA at 8 planes, two CTAs
// per SM.  Measured (1242 x 375 and 1280 x 720, D = 128; 640 x 360, D = 60), us: this
// 80.1 / 76.8 / 18.3; 8 warps and 4 stages 85.5 / 83.0 / 17.8; 16 and 4 (one CTA per
// SM) 80.2 / 77.5 / 16.9; 4 and 4 77.1 / 80.6 / 18.9 but 673 against 598 at 1920 x 1080.
// A row split over a cluster of 2 or 4 CTAs that merge their minima at the end
// measured 82-85 / 80-84.
//
// 16-bit records of 8 paths are 192 KB of ring at 16 warps, which leaves room for
// rows of some 6900 pixels; longer ones halve the warps (wta_warps below).  Only
// the kernels for any number of planes take the warps from the block size: the
// others lose 5 % by it (80.1 -> 86.9 at 1242 x 375).
constexpr int kMaxWarps = 16;
constexpr int kStages = 3;

// Minimum of v over the lanes of this lane's pixel (grp of the warp's G): one
// full-warp redux.sync per pixel, fed 0xFFFFFFFF by the other pixels' lanes.
template <int G>
__device__ __forceinline__ uint32_t group_min(uint32_t v, int grp) {
    if constexpr (G == 32) {
        return v;
    } else if constexpr (G == 1) {
        return __reduce_min_sync(0xffffffffu, v);
    } else {
        uint32_t m = 0;
#pragma unroll
        for (int g = 0; g < G; g++) {
            const uint32_t r = __reduce_min_sync(0xffffffffu, grp == g ? v : 0xFFFFFFFFu);
            if (grp == g) m = r;
        }
        return m;
    }
}

// The planes are read exactly once: they leave L2 first.
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ void copy16(uint32_t dst, const uint8_t *src, uint64_t pol) {
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(pol) : "memory");
}
__device__ __forceinline__ void copy8(uint32_t dst, const uint8_t *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// NP > 0: NP planes and kMaxWarps warps (compile time); NP == 0: any of both.
template <int G, bool WIDE, int NP, bool DEBUG>
__global__ void __launch_bounds__(kMaxWarps * 32)
    wta_kernel(const uint8_t *__restrict__ planes, int nplanes, int W, int H, int D, int Dp, int tol,
               uint8_t *__restrict__ disp_lr, uint8_t *__restrict__ dbg_left, uint8_t *__restrict__ dbg_right,
               uint16_t *__restrict__ dbg_sum) {
    wait_for_predecessor();
    constexpr int EB = WIDE ? 2 : 1;  // bytes per path cost
    constexpr int NQ = NP > 0 ? NP : kMaxPaths;
    const int np = NP > 0 ? NP : nplanes;
    const int rec = np * Dp * EB;  // bytes of a pixel's record
    const int lps = Dp / 8;        // lanes per pixel
    const int warps = NP > 0 ? kMaxWarps : (int)blockDim.x / 32;
    extern __shared__ __align__(16) uint8_t wta_smem[];
    uint8_t *ring = wta_smem;  // [warps][kStages][G][rec]
    uint32_t *key_right = reinterpret_cast<uint32_t *>(wta_smem + (size_t)warps * kStages * G * rec);  // slots -Dp .. W-1
    uint8_t *dl_row = reinterpret_cast<uint8_t *>(key_right + Dp + W);                                // W bytes
    const int y = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = lane / lps, li = lane - grp * lps;
    for (int i = threadIdx.x; i < Dp + W; i += warps * 32) key_right[i] = 0xFFFFFFFFu;
    __syncthreads();
    // this group's pixels [xb, xe); lanes past the last group have none
    const int seg = (W + warps * G - 1) / (warps * G);
    const int xb = min((warp * G + grp) * seg, W), xe = grp < G ? min(xb + seg, W) : xb;
    const uint64_t pol = policy_evict_first();
    const uint32_t ring_warp = (uint32_t)__cvta_generic_to_shared(ring) + (uint32_t)(warp * kStages * G * rec);
    const uint32_t ring_grp = ring_warp + (uint32_t)((grp < G ? grp : 0) * rec);
    const long long row = (long long)y * W;
    // Copies the record of pixel x into stage st; the group's lanes share it.
    auto fetch = [&](int x, int st) {
        if (x < xe) {
            const long long at = (row + x) * rec;
            const uint32_t to = ring_grp + (uint32_t)(st * G * rec);
            const long long bytes = (long long)W * H * rec;
            if (rec % 16 == 0) {
#pragma unroll
                for (int j = 0; j < (NQ * EB + 1) / 2; j++) {
                    const int o = (j * lps + li) * 16;
                    if (o < rec && in_range(at + o, bytes - 15)) copy16(to + o, planes + at + o, pol);
                }
            } else {
                for (int o = li * 8; o < rec; o += lps * 8)
                    if (in_range(at + o, bytes - 7)) copy8(to + o, planes + at + o);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // key constants of pair k: bytes d, top (lower half), d, top (upper half); top is 0xFF for d >= D
    const int k0 = 4 * li;
    uint32_t kc[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const uint32_t dl = k0 + k, dh = Dp - 1 - k0 - k;
        kc[k] = (dl & 0xFFu) | ((int)dl >= D ? 0xFF00u : 0u) | ((dh & 0xFFu) << 16) | ((int)dh >= D ? 0xFF000000u : 0u);
    }
    uint32_t tl[4], th[4];  // running right minima of the slots x - d, lower and upper disparities
#pragma unroll
    for (int k = 0; k < 4; k++) tl[k] = th[k] = 0xFFFFFFFFu;
    uint32_t *slot_lo = key_right + Dp + xb - k0, *slot_hi = key_right + Dp + xb - (Dp - 1 - k0);  // slots of pair k0
    auto flush = [&](uint32_t *slot, uint32_t key) {
        if (in_range(slot - key_right, Dp + W)) atomicMin(slot, key);
    };
#pragma unroll
    for (int s = 0; s < kStages - 1; s++) fetch(xb + s, s);
#pragma unroll 1
    for (int i = 0; i < seg; i++) {
        const int x = xb + i;
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
        __syncwarp();  // all lanes' copies of this record are there, and the one before has been read
        fetch(x + kStages - 1, (i + kStages - 1) % kStages);
        const uint32_t from = ring_grp + (uint32_t)(i % kStages * G * rec) + li * 8 * EB;
        uint32_t S[4];
        if constexpr (WIDE) {
#pragma unroll
            for (int k = 0; k < 4; k++) S[k] = 0u;
#pragma unroll
            for (int q = 0; q < NQ; q++)
                if (NP > 0 || q < np) {
                    uint32_t v[4];
                    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                                 : "r"(from + q * Dp * EB));
#pragma unroll
                    for (int k = 0; k < 4; k++) S[k] += v[k];
                }
        } else {
            uint32_t O[2] = {0u, 0u}, V[2] = {0u, 0u};
#pragma unroll
            for (int q = 0; q < NQ; q++)
                if (NP > 0 || q < np) {
                    uint32_t v[2];
                    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(from + q * Dp));
#pragma unroll
                    for (int w = 0; w < 2; w++) {
                        O[w] += __byte_perm(v[w], 0u, 0x4341);
                        V[w] += v[w];
                    }
                }
#pragma unroll
            for (int w = 0; w < 2; w++) {
                S[2 * w] = O[w];
                S[2 * w + 1] = V[w] - O[w] * 256u;
            }
        }
        uint32_t kl[4], kh[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            kl[k] = __byte_perm(S[k], kc[k], 0x5104);
            kh[k] = __byte_perm(S[k], kc[k], 0x7326);
        }
        const bool active = x < xe;
        uint32_t best = min(min(min(kl[0], kl[1]), min(kl[2], kl[3])), min(min(kh[0], kh[1]), min(kh[2], kh[3])));
        if (!active) best = 0xFFFFFFFFu;
        best = group_min<G>(best, grp);
        if (active) {
            if (li == 0 && in_range(x, W)) dl_row[x] = (uint8_t)(best & 0xFFu);
            // the slots of the pixel before: that of its pair 3 leaves downwards, the
            // upper half's pair 0 upwards
            flush(slot_lo - 4, tl[3]);
            flush(slot_hi - 1, th[0]);
            tl[3] = min(tl[2], kl[3]);
            tl[2] = min(tl[1], kl[2]);
            tl[1] = min(tl[0], kl[1]);
            tl[0] = kl[0];
            th[0] = min(th[1], kh[0]);
            th[1] = min(th[2], kh[1]);
            th[2] = min(th[3], kh[2]);
            th[3] = kh[3];
            slot_lo++;
            slot_hi++;
            if constexpr (DEBUG) {
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    uint16_t *out = dbg_sum + ((size_t)row + x) * D;
                    if (k0 + k < D) out[k0 + k] = (uint16_t)(S[k] & 0xFFFFu);
                    if (Dp - 1 - k0 - k < D) out[Dp - 1 - k0 - k] = (uint16_t)(S[k] >> 16);
                }
            }
        }
    }
    if (xb < xe) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            flush(slot_lo - 1 - k, tl[k]);
            flush(slot_hi - 1 + k, th[k]);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int xx = threadIdx.x; xx < W; xx += warps * 32) {
        const int dl = dl_row[xx];
        uint8_t v = (uint8_t)dl;
        if (tol >= 0) {
            const int xr = xx - dl;
            if (xr < 0 || !in_range(xr, W)) {
                v = SGM_INVALID;
            } else {
                const int dr = (int)(key_right[Dp + xr] & 0xFFu);
                const int diff = dl > dr ? dl - dr : dr - dl;
                if (diff > tol) v = SGM_INVALID;
            }
        }
        const size_t pix = (size_t)y * W + xx;
        if (!in_range((long long)pix, (long long)W * H)) continue;
        disp_lr[pix] = v;
        if (dbg_left) dbg_left[pix] = (uint8_t)dl;
        if (dbg_right) dbg_right[pix] = (uint8_t)(key_right[Dp + xx] & 0xFFu);
    }
}

// Shared memory of a CTA: the rings (rec bytes per warp and stage), the right minima
// and the left winners of the row.
size_t wta_smem_bytes(int W, int Dp, size_t rec, int warps) {
    return (size_t)warps * kStages * rec + (size_t)(Dp + W) * sizeof(uint32_t) + (size_t)((W + 3) & ~3);
}

// As many warps as fit a CTA's shared memory.
int wta_warps(int W, int Dp, size_t rec) {
    int warps = kMaxWarps;
    while (warps > 1 && wta_smem_bytes(W, Dp, rec, warps) > kMaxSmem) warps /= 2;
    return warps;
}

template <bool WIDE>
cudaError_t launch_wta_t(const uint8_t *planes, int nplanes, int W, int H, int D, int tol, uint8_t *disp_lr,
                         uint8_t *dbg_left, uint8_t *dbg_right, uint16_t *dbg_sum, cudaStream_t s) {
    const int Dp = padded_disparities(D);
    const int warps = wta_warps(W, Dp, (size_t)(256 / Dp) * nplanes * Dp * (WIDE ? 2 : 1));
    const bool all = warps == kMaxWarps;
    auto go = [&](auto kernel, int G) {
        const size_t smem = wta_smem_bytes(W, Dp, (size_t)G * nplanes * Dp * (WIDE ? 2 : 1), warps);
        const cudaError_t e = allow_max_smem(kernel);
        if (e != cudaSuccess) return e;
        return launch_k(kernel, dim3(H), dim3(warps * 32), smem, s, planes, nplanes, W, H, D, Dp, tol, disp_lr, dbg_left,
                        dbg_right, dbg_sum);
    };
#define SGM_WTA(G)                                                          \
    case G:                                                                 \
        if (dbg_sum) return go(wta_kernel<G, WIDE, 0, true>, G);            \
        if (all && nplanes == 8) return go(wta_kernel<G, WIDE, 8, false>, G);\
        if (all && nplanes == 4) return go(wta_kernel<G, WIDE, 4, false>, G);\
        return go(wta_kernel<G, WIDE, 0, false>, G)
    switch (256 / Dp) {  // pixels per warp
        SGM_WTA(32);
        SGM_WTA(16);
        SGM_WTA(8);
        SGM_WTA(4);
        SGM_WTA(2);
        SGM_WTA(1);
        default: return cudaErrorInvalidValue;
    }
#undef SGM_WTA
}

}  // namespace

SGM_GUARD_COUNTER(guard_hits_wta)

cudaError_t launch_wta(const uint8_t *planes, int nplanes, int W, int H, int D, bool wide,
                       int tol, uint8_t *disp_lr, uint8_t *dbg_left, uint8_t *dbg_right,
                       uint16_t *dbg_sum, cudaStream_t s) {
    if (wide) return launch_wta_t<true>(planes, nplanes, W, H, D, tol, disp_lr, dbg_left, dbg_right, dbg_sum, s);
    return launch_wta_t<false>(planes, nplanes, W, H, D, tol, disp_lr, dbg_left, dbg_right, dbg_sum, s);
}

}  // namespace sgm
