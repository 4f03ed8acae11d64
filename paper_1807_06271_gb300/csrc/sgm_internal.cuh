// Internal declarations of libsgm: handle layout and kernel launchers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sgm.h"

namespace sgm {

constexpr int kMaxPaths = 8;
constexpr int kMaxD = 255;
constexpr int kMaxW = 8192;  // the right-WTA keeps one 32-bit key per column in shared memory
constexpr int kMaxSadWindow = 15;  // largest SAD support window side (shared-memory rows of the cost kernel)

// Path directions (dx, dy), bit r of a path mask enables entry r.
__host__ __device__ constexpr int dir_dx(int r) {
    return r == 0 ? 1 : r == 1 ? -1 : r == 2 ? 0 : r == 3 ? 0 : r == 4 ? 1 : r == 5 ? -1 : r == 6 ? -1 : 1;
}
__host__ __device__ constexpr int dir_dy(int r) {
    return r == 0 ? 0 : r == 1 ? 0 : r == 2 ? 1 : r == 3 ? -1 : r == 4 ? 1 : r == 5 ? -1 : r == 6 ? 1 : -1;
}

// Number of scanlines of direction r in a W x H image.  Diagonals move along the
// short axis and wrap around the long one (where the path starts anew), so that
// all of them have the length of the short axis.
inline long scanlines_of(int r, int W, int H) {
    const int dx = dir_dx(r), dy = dir_dy(r);
    if (dy == 0) return H;
    if (dx == 0) return W;
    return W >= H ? W : H;
}

// Rectification maps of the left and right image (device, W x H each; all
// null when the images are already rectified).
// Programmatic dependent launch.  Every kernel of the pipeline is launched
// with programmatic stream serialisation, so the launch of kernel k+1 overlaps
// the end of kernel k; each kernel's first statement waits until its stream
// predecessor has completed and its memory is visible, before it reads or
// writes anything.  Kernels launched the ordinary way pass the wait at once.
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                     Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Lets a kernel that declares no shared memory of its own have all a CTA can have.
// The limit belongs to the function on the device, not to the launch: always the
// same value, as one that followed the launch's size could be lowered by another
// host thread before the launch.
constexpr size_t kMaxSmem = 227 * 1024;
template <typename... KArgs>
cudaError_t allow_max_smem(void (*kernel)(KArgs...)) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
}

struct RectMaps {
    const uint16_t *lx, *ly, *rx, *ry;
};

// Pixel (gx, gy) of the rectified image: the source image read through the
// maps (Sec. 3.1.1), 0 where a map entry leaves the source.
// Guarded builds (compiled with -DSGM_GUARDED: a test variant of the
// library, never the default).  The plane path's kernels (census, the
// CUDA-core and SAD costs, the aggregation, the WTA, the median and the U/V
// maps) check each global index they compute, and each shared index that depends
// on the image, against its buffer's extent before the access.  An index out
// of range skips the access and is counted in the translation unit's
// counter; sgm_debug_guard_hits sums the counters.  In the default build
// in_range is constant true and the checks compile away.
#ifdef SGM_GUARDED
static __device__ unsigned long long g_guard_hits;  // one per translation unit
__device__ __forceinline__ bool in_range(long long i, long long n) {
    if (i >= 0 && i < n) return true;
    atomicAdd(&g_guard_hits, 1ull);
    return false;
}
#define SGM_GUARD_COUNTER(name)                                                   \
    unsigned long long name(bool reset) {                                         \
        unsigned long long v = 0, z = 0;                                          \
        if (cudaMemcpyFromSymbol(&v, g_guard_hits, sizeof(v)) != cudaSuccess)     \
            v = ~0ull;                                                            \
        if (reset && cudaMemcpyToSymbol(g_guard_hits, &z, sizeof(z)) != cudaSuccess) \
            v = ~0ull;                                                            \
        return v;                                                                 \
    }
#else
__device__ __forceinline__ constexpr bool in_range(long long, long long) { return true; }
#define SGM_GUARD_COUNTER(name) \
    unsigned long long name(bool) { return 0; }
#endif
// Each guarded translation unit's counter (~0 when it cannot be read).
unsigned long long guard_hits_census(bool reset);
unsigned long long guard_hits_sad(bool reset);
unsigned long long guard_hits_aggregate(bool reset);
unsigned long long guard_hits_wta(bool reset);
unsigned long long guard_hits_post(bool reset);

template <bool RECT>
__device__ __forceinline__ uint8_t rect_pixel(const uint8_t *__restrict__ img, int pitch, int W,
                                              int H, int gx, int gy, const uint16_t *__restrict__ mx,
                                              const uint16_t *__restrict__ my) {
    if constexpr (!RECT) {
        const long long i = (long long)gy * pitch + gx;
        return in_range(i, (long long)pitch * H) ? img[i] : 0;
    } else {
        const long long m = (long long)gy * W + gx;
        if (!in_range(m, (long long)W * H)) return 0;
        const int sx = mx[m], sy = my[m];
        return (sx < W && sy < H) ? img[(size_t)sy * pitch + sx] : 0;
    }
}

// Disparity layout.  A pixel owns Dp slots in the cost volume and in every path
// plane: 8, 16 or the multiple of 32 that holds D; slots d >= D are padding.
// (Powers of two alone move a third more bytes at D = 192: 1920 x 1080, 8 paths,
// cost 280 -> 194 us, aggregation 1229 -> 1084.  Multiples of 16 that are not
// multiples of 32 split the 32-byte sectors of neighbouring pixels: 641 x 479,
// D = 97 in 112 slots, aggregation 91 -> 155 us, WTA 60 -> 84.)  The
// record is folded: pair k (0 <= k < Dp/2) holds the disparities (k, Dp-1-k), so
// that a pair's neighbours in both halves are the pairs k-1 and k+1, whatever
// number of consecutive pairs a lane of the aggregation kernel holds.
//   8-bit costs (census): 32-bit word w holds pairs 2w and 2w+1 as the bytes
//     2w+1  2w  Dp-2-2w  Dp-1-2w  (the upper halves in increasing order);
//   16-bit costs (SAD, "wide"): word k holds pair k, the lower half first.
inline int lanes_per_scanline(int D) {  // 8-disparity chunks of D, rounded up to a power of two
    int need = (D + 7) / 8, l = 1;
    while (l < need) l *= 2;
    return l;
}
inline int padded_disparities(int D) {
    return D <= 8 ? 8 : D <= 16 ? 16 : (D + 31) / 32 * 32;
}
// Slot (byte, or uint16 for wide) of disparity d in a pixel's record.
__host__ __device__ constexpr int fold_slot(int d, int Dp, bool wide) {
    const int hi = d >= Dp / 2, k = hi ? Dp - 1 - d : d;
    return wide ? 2 * k + hi : 4 * (k / 2) + 1 - k % 2 + 2 * hi;
}
// Cost of the padding slots.  With it they never hold a scanline's minimum nor
// help a neighbour (census bits + P2 <= 255; SAD cmax + P2 < 0x7FFF).
constexpr unsigned kPadCost = 255u, kPadCostWide = 0x7FFFu;

// Pairs of disparities a lane of the aggregation kernel holds, for the
// long-axis scanlines and for the other directions.
struct LaneConfig {
    int np_long, np_other;
};
inline int lanes_of(int D, int np) { return padded_disparities(D) / (2 * np); }

// Work list of the aggregation kernel: entry k is a set of enabled directions (the
// two of the long axis, then the up to three that move along the short axis one
// way and those that move the other way; large images take the long axis second)
// whose nlines scanlines are cut into jobs of G neighbouring scanlines (one warp
// each, G = 32 / lanes per scanline); the jobs of the directions alternate.  Job j
// belongs to entry k when jbegin[k] <= j < jbegin[k+1].
struct PathJobs {
    LaneConfig lanes;
    int n;                     // number of entries
    int ndir[3];               // directions of entry k
    int dx[3][3], dy[3][3];
    int plane[3][3];           // their output planes, numbered in this order
    int nlines[3];
    int jbegin[4];
    int klong;                 // entry of the long-axis directions (-1: none)
    int nlong;                 // their jobs
    uint32_t unit;             // always 1; see the kernel's multiply-adds
};

// Work-queue state of the aggregation kernel: word 0 counts the jobs handed out
// beyond the warps' first ones (cleared before every launch).  The rest is not used;
// the size is part of what sgm.h documents and sgm_scratch_bytes reports.
constexpr size_t kJobStateBytes = 4224;

// Builds the work list for the directions in `mask`, under the
// sgm_set_aggregation setting cpl.  many: other pairs' work runs beside it, so
// the lanes are not narrowed to shorten a small image's chains and the long axis
// comes first.
PathJobs make_path_jobs(int W, int H, int D, int mask, bool wide, int cpl, bool many = false);
// Resident 4-warp blocks per SM for a handle whose caller sets none.
int default_blocks_per_sm(const PathJobs &jobs);
// The most chunks per lane the aggregation takes for D (1 for 16-bit costs, up to 4).
int chunks_per_lane_max(int D, bool wide);
// Whether the settings above 1 change the lanes for D (they run as 1 for 96, 160, 192
// and 224 slots).
bool chunks_apply(int D, bool wide);
// Chunks-per-lane code of the mixed layout: long-axis scanlines at 1, the others at 2.
constexpr int kMixedCpl = SGM_AGG_CHUNKS_MIXED;

// One pair of a batched aggregation launch (device-resident table entry).
struct BatchAggPair {
    const void *cost;  // the pair's cost volume
    void *planes;      // its path planes
    int W, H, Dp;
    int nplanes;
    PathJobs jobs;
};

}  // namespace sgm

namespace sgm {

// Launchers (return cudaGetLastError() of the launch).
cudaError_t launch_census(const uint8_t *left, const uint8_t *right, int pitch, int W, int H,
                          int cw, int ch, int code_bytes, void *codes, const RectMaps &maps,
                          cudaStream_t s);
// The cost kernels also clear word 0 of job_state (may be null), the
// work-queue state of the aggregation kernel that follows them on the stream.
// Hamming costs of the census codes come from one of two kernels (kernel:
// SGM_COST_KERNEL_*): POPC on the CUDA cores (any D) or +-1 inner products on
// the tensor cores (Dp <= 128), which ORs 1 into *status (may be null) when its
// bounded wait for the MMA gives up.
cudaError_t launch_cost(const void *codes, int code_bytes, int W, int H, int D, int nbits,
                        uint8_t *cost, unsigned *job_state, unsigned *status, int kernel, cudaStream_t s);
bool cost_mma_supported(int D);
// stall_test != 0: the kernel's first wait is on an mbarrier nothing arrives at,
// with a 2 ms limit, so that it takes its timeout path (for tests of it).
cudaError_t launch_cost_mma(const void *codes, int code_bytes, int W, int H, int D, int nbits, uint8_t *cost,
                            unsigned *job_state, unsigned *status, cudaStream_t s, int stall_test = 0);
// The kernel SGM_COST_KERNEL_AUTO selects for D.
int cost_kernel_for(int D);
// SAD over a ww x wh window (clamped reads; rectified through maps when set) into a
// 16-bit cost volume [H][W][Dp] of folded records.
cudaError_t launch_sad_cost(const uint8_t *left, const uint8_t *right, int pitch, int W, int H,
                            int D, int ww, int wh, const RectMaps &maps, uint16_t *cost,
                            unsigned *job_state, cudaStream_t s);
// Planes are pixel-interleaved: [H][W][nplanes][Dp], entry k of `jobs` writing
// plane jobs.plane[k].  job_counter (kJobStateBytes) must have been cleared by
// the cost kernel launched before it on s.
// wide: 16-bit costs and planes (SAD), else 8-bit.  cpl: 8-disparity chunks
// per lane (1, 2 or 4, at most chunks_per_lane_max; jobs built with the same).
cudaError_t launch_aggregate(const uint8_t *cost, int W, int H, int D, int P1, int P2, bool wide,
                             const PathJobs &jobs, uint8_t *planes, int nplanes,
                             unsigned *job_counter, int blocks_per_sm, int cpl, cudaStream_t s);
// All pairs' aggregation in one persistent launch (pairs: device table of
// npairs entries; prefix: device [2][npairs + 1], the running counts of the
// pairs' long-axis jobs and of their other jobs).  job_counter as above, for
// this launch alone.  P1/P2 and the cost width are shared by the pairs.
// cpl: 1 or 4 (4 only for 8-bit costs and pairs whose D allows it).
cudaError_t launch_aggregate_batch(const BatchAggPair *pairs, int npairs, const int *prefix, int P1, int P2,
                                   bool wide, int cpl, unsigned *job_counter, int blocks_per_sm, cudaStream_t s);
// Copies a single plane ([H][W][Dp], folded records) to L ([H][W][D] uint16, natural order).
cudaError_t launch_unpermute(const uint8_t *plane, int W, int H, int D, bool wide, uint16_t *L,
                             cudaStream_t s);
cudaError_t launch_wta(const uint8_t *planes, int nplanes, int W, int H, int D, bool wide,
                       int tol, uint8_t *disp_lr, uint8_t *dbg_left, uint8_t *dbg_right,
                       uint16_t *dbg_sum, cudaStream_t s);
cudaError_t launch_median(const uint8_t *in, uint8_t *out, int W, int H, int k, cudaStream_t s);
// Host-side argument checks shared by every entry point (SGM_OK or an error status).
int validate_params(int W, int H, int D, const sgm_params *p);

cudaError_t launch_uvmap(const uint8_t *disp, int W, int H, int D, uint16_t *umap, uint16_t *vmap,
                         cudaStream_t s);

// The paper's streaming set in one top-down sweep with the cost, the paths,
// both winners and the LR check fused (sweep.cu): census codes (code_bytes 4
// or 8) of both images in, the checked map disp_lr out (dbg_left/dbg_right,
// optional, receive the raw maps).  Supported for D <= 128 and path masks
// within 0x55.  scratch: sweep_scratch_bytes(W, H, D, rows_per_cta) bytes.
// A bounded wait that gives up ORs 2 into *status (may be null).
// Returns cudaErrorCooperativeLaunchTooLarge when the grid cannot be resident at once.
bool sweep_supported(int D, int mask, int code_bytes);
bool sweep_fits(int H, int D, int code_bytes, int rows_per_cta);
size_t sweep_scratch_bytes(int W, int H, int D, int rows_per_cta);
// stall_test != 0: row 1 waits for a pixel row 0 never publishes, with a 2 ms
// limit, so that the bounded waits take their timeout path (for tests of it).
cudaError_t launch_sweep(const void *codes, int code_bytes, int W, int H, int D, int nbits, int P1, int P2,
                         int mask, int tol, uint8_t *disp_lr, uint8_t *dbg_left, uint8_t *dbg_right,
                         void *scratch, unsigned *status, int rows_per_cta, cudaStream_t s, int stall_test = 0);

}  // namespace sgm
