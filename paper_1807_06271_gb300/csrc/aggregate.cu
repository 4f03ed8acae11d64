// Semi-global path aggregation (Sec. 3.1.3, Eq. 2) over a precomputed cost
// volume (Eq. 1).
//
// Decomposition.  Every enabled direction cuts the image into independent
// scanlines.  Let W >= H (else swap the axes): rows for the horizontal
// directions, and W scanlines of H steps, one row per step, for each of the six
// others.  A diagonal that leaves the image on the left or right comes in again on
// the other side of the next row, where its path starts anew, so all of them have
// the same length.  The Dp disparities of one pixel are held by LPS lanes, NP pairs
// of disparities per lane, so one warp walks G = 32 / LPS neighbouring scanlines in
// lock-step.  The kernel is persistent: blocks_per_sm blocks of 4 warps run on
// every SM and pull jobs (one direction, G scanlines) from a work queue until it is
// empty.
//
// Sweeps.  The column and the two diagonals that go down start together, have the
// same length and stay within a few rows of one another, so a row of costs is read
// from HBM once for the three of them; the three that go up follow and start on the
// rows that were read last.  1280 x 720, D = 192, 8 paths: 0.96 GB read where
// directions one after the other read 1.18 GB (the costs are 0.18 GB), 1.37 GB
// written.  Aggregation in us, directions one after the other -> sweeps: 1242 x 375,
// D = 128, 8 paths 125 -> 116, 641 x 479, D = 97 90 -> 82, 480 x 752, D = 128 105
// -> 97, 1920 x 1080, D = 192 1147 -> 1105 (with six pairs per lane; 1053 with the
// rows between the sweeps), 1280 x 720, D = 64 168 -> 154; 640 x 360, D = 60, three of
// the six directions, 32.8 -> 34.9.
//
// Arithmetic.  The record of a pixel is folded: pair k holds the disparities
// (k, Dp-1-k), packed as two 16-bit halves, and a lane holds NP consecutive
// pairs R_0 .. R_{NP-1}.  The d-1 / d+1 neighbours of both halves of pair k
// are then the whole registers of pairs k-1 and k+1 in either order, and the
// minimum over the two does not care which is which.  Only the ends need
// other lanes: the last pair of the lane before and the first pair of the lane
// after (one shuffle each).  Before pair 0 there is nothing, so the first lane
// takes a value that changes no minimum; after the last pair comes itself with
// its halves swapped (one byte-permute with a per-lane selector serves every
// lane).  One update is
//     t = min(min(L(d-1), L(d+1), m + P2 - P1) + P1, L(d));   L' = t + C - m
// (the same minimum as min(L(d±1) + P1, L(d), m + P2)): a three-way packed
// minimum, a packed add-then-minimum and a three-input add.  Keeping L without the
// "- m" for some steps (a two-input add, m subtracted when storing) took fewer ALU
// instructions and the same time (131-135 us against 128, 1242 x 375).  m = min_d L is
// reduced within the lane, folded over the two halves, then reduced over the
// scanline's lanes: xor-shuffles for scanlines of up to 4 lanes, one full-warp
// redux.sync per scanline of the warp for wider ones.  Starting from L = 0, m = 0
// makes the first step produce L = C without a special case.
//
// Padding.  Slots d >= D hold the cost 255 (0x7FFF for 16-bit costs).  As bits
// + P2 <= 255 (cmax + P2 <= 0x7FFF), a padding slot's path cost is at least m +
// P2 at the next step, so it neither is the minimum nor helps a neighbour, and
// needs no special case either.
//
// Lanes per scanline.  One step of a scanline is a dependent chain: the update,
// the minimum over the lanes, the next update.  Fewer disparities per lane
// shorten it, more of them need fewer instructions per disparity.  The
// long-axis scanlines (rows when W >= H) are the longest chains, so they
// run with 2 pairs per lane (a scanline of D = 128 fills a warp) and the other
// directions with 4; see lane_config for small images.
//
// Pipes.  On GB300 the packed minima, byte-permutes, logic, redux.sync and
// three-input adds issue on the ALU pipe at 16 lanes per cycle (measured: 2
// cycles each and scheduler), two-input adds at 32 lanes beside it; the adds
// that could merge into three-input ones or shifts are written as multiply-adds
// by a 1 the compiler cannot see (the job table's unit field), which run on the
// FMA pipe.
//
// Memory.  Costs come through a ring of four stages of 2 to 16 steps per warp in
// shared memory, filled by 16-byte asynchronous copies: with loads into registers,
// 16 steps ahead, a third of the warps' time was waits, as a warp has few
// scoreboards and a wait for the oldest load also waited for the youngest (1242 x
// 375, 8 paths: 149 -> 128 us).  Each step stores the lane's path costs to the
// direction's plane, in the cost volume's order and width, with evict_first: the
// planes are read back only once, by the WTA kernel (without it 125 -> 135 us).  The
// planes of a sweep's directions are neighbours in a pixel's record (numbered by
// direction instead: 900 x 901, D = 96, 254 us against 243).
//
// Bound.  At D = 128 and more it is HBM: 5.1 to 5.3 TB/s of reads and writes mixed, in
// runs of a pixel's Dp bytes.  Small images are bound by the ALU pipe while all
// scanlines run and by the long axis' chain of steps after that.

#include <cuda_fp16.h>

#include <type_traits>

#include "sgm_internal.cuh"

namespace sgm {

namespace {

constexpr int kSchedulers = 608;  // warp schedulers of the GPU (152 SMs)

// Pairs per lane for a W x H image.  The base is 2 on the long axis and 4 in the
// other directions (4 and 4 above D = 128).
//
// Small images leave schedulers idle and take as long as their longest chain of
// steps, so they get narrower lanes (a step of one pair per lane and one scanline
// per warp takes 28 ns, of two and two 40, of four and four 80; with D = 128, two
// and one 31, four and two 50), as long as nearly all of their warps are resident at
// once; where both sides of the image are alike the other directions' chain is the
// longer one, and the long axis keeps 2.  Measured, aggregation in us:
//   D = 64    640 x 360, 4 paths: base 40.7, (1, 4) 36.9, (1, 2) 34.8
//             640 x 480, 4 paths: base 46.3, (1, 4) 54, (1, 2) 39.0, (2, 2) 38.6;  8 paths: 63.4, 71.7, 63.7, 56.1
//             514 x 166, 8 paths: base 32.6, (1, 4) 26.8, (1, 2) 31.0;  437 x 1032: 83.3, 73.7, 91.4
//             1280 x 720, 8 paths: base 154, (2, 2) 157
//   D = 32    246 x 269, 8 paths: base 25.5, (1, 1) 18.7;  1280 x 720: base 123.9, (1, 4) 132.9
//   D = 128   230 x 182, 8 paths: base 22.2, (2, 2) 19.5;  480 x 752: base 97.5, (2, 2) 104
//
// Four paths at D = 128 also take (2, 2) where the base leaves a second round of jobs
// nearly empty (rounds of 16 warps per SM, base): 1.03 (800 x 900) base 127, (2, 2) 107;
// 1.12 (1280 x 720) 154, 142;  1.15 (1400 x 700) 162, 143;  1.30 (1044 x 1079) 205, 181;
// 1.42 (1300 x 1080) 235, 239;  0.92 (708 x 818) 88, 94.
//
// 96 and 192 slots are 12 or 24 lanes of four pairs, which leave a quarter of every
// warp idle; 8 or 16 lanes of six fill it.  It pays where the diagonals read their
// costs from L2 and the warps, fewer by a third, still fill the chip:
//   D = 192   1920 x 1080, 8 paths: (4, 4) 1174, (4, 6) 1110;  570 x 280: 77, 72;  320 x 240: 42, 45
//             1280 x 720, 4 paths: 248, 276
//   D = 96    1784 x 799, 8 paths: (2, 4) 486, (2, 6) 460;  640 x 480: 86, 98
LaneConfig lane_config(int W, int H, int D, int mask, bool wide, int cpl, bool many) {
    const int Dp = padded_disparities(D);
    if (chunks_apply(D, wide)) {
        if (cpl == 2) return {8, 8};
        if (cpl == 4) return {16, 16};
        if (cpl == kMixedCpl) return {4, 8};
    }
    LaneConfig lc{Dp <= 128 ? 2 : 4, 4};
    if (many || Dp < 32) return lc;
    const int axis = W >= H ? 0x03 : 0x0C;  // the long-axis directions
    const int longer = W >= H ? W : H, shorter = W >= H ? H : W;
    long lines_long = 0, lines_other = 0;
    for (int r = 0; r < kMaxPaths; r++)
        if ((mask >> r) & 1) (((axis >> r) & 1) ? lines_long : lines_other) += scanlines_of(r, W, H);
    auto warps = [&](int np_long, int np_other) {
        return lines_long * lanes_of(D, np_long) / 32 + lines_other * lanes_of(D, np_other) / 32;
    };
    // One pair of 16-bit costs is stored by its index in units of 4 bytes, which must
    // stay below 2^32 (all other lanes do within the bounds of handle creation): the
    // columns of an image of 2100 x 65535 alone, say, would go beyond.
    if (wide && (long long)W * H * __builtin_popcount((unsigned)mask) * Dp / 2 >= (1ll << 32)) return lc;
    if (Dp == 32) {
        if (warps(1, 1) <= 2 * kSchedulers) return {1, 1};
        if (warps(1, 4) <= 3 * kSchedulers) return {1, 4};
        return lc;
    }
    if (Dp == 64) {
        // chain of the long axis at 2 pairs per lane against that of the others at 4
        const bool square = 56. * longer < 80. * shorter, flat = 32. * longer > 80. * shorter;
        if (warps(1, 2) <= (square ? 3. : 3.6) * kSchedulers && !flat) return {1, 2};
        if (square) return warps(2, 2) <= 12 * kSchedulers ? LaneConfig{2, 2} : lc;
        if (warps(1, 4) <= 4 * kSchedulers) return {1, 4};
        return lc;
    }
    // without diagonals, base warps that fill a second round of 16 per SM by a third at most
    const long base = warps(lc.np_long, 4);
    const bool both = (mask & (0x0F ^ axis)) == (0x0F ^ axis) && !(mask & 0xF0);
    const bool short_round = Dp == 128 && both && base > 4 * kSchedulers && base <= 5.4 * kSchedulers;
    if (short_round || (Dp <= 128 && 50. * shorter > 31. * longer && warps(2, 2) <= 4 * kSchedulers)) lc.np_other = 2;
    else if (!wide && Dp % 96 == 0 && (mask & 0xF0) && warps(lc.np_long, 6) >= 3 * kSchedulers) lc.np_other = 6;
    return lc;
}

}  // namespace

PathJobs make_path_jobs(int W, int H, int D, int mask, bool wide, int cpl, bool many) {
    PathJobs j = {};
    j.unit = 1u;
    const LaneConfig lc = lane_config(W, H, D, mask, wide, cpl, many);
    j.lanes = lc;
    const bool wide_image = W >= H;
    auto along = [&](int r) { return wide_image ? dir_dy(r) : dir_dx(r); };  // step along the short axis
    // entries: the long axis, all that moves along the short axis one way, and all that
    // moves the other way
    int planes = 0;
    // Their order: the long axis first, as its chains are the longest, unless the costs
    // are more than L2 keeps.  Then they come between the sweeps, whose warps must all
    // run at once to share them.  Measured, long axis first and second, us (8 paths): 1920
    // x 1080, D = 192 (398 MB) 1102, 1053;  1280 x 720, D = 192 (177 MB) 462, 425;  1920 x
    // 1080, D = 64 (133 MB) 386, 365;  1280 x 720, D = 128 (118 MB) 264, 258;  1500 x 500, D
    // = 128 (96 MB) 204, 210;  1242 x 375, D = 192 (89 MB) 196, 199;  900 x 700, D = 96 (60
    // MB) 157, 188.  1280 x 720, D = 128, 4 paths without diagonals: 152, 155.
    const double volume = (double)W * H * padded_disparities(D) * (wide ? 2 : 1);
    const bool sweeps_first = !many && volume >= 100e6 && (mask & 0xF0);
    j.klong = -1;
    for (int i : {sweeps_first ? 1 : 0, sweeps_first ? 0 : 1, 2}) {
        const int k = j.n;
        for (int r = 0; r < kMaxPaths; r++) {
            if (!((mask >> r) & 1) || along(r) != (i == 0 ? 0 : i == 1 ? 1 : -1)) continue;
            const int e = j.ndir[k]++;
            j.dx[k][e] = dir_dx(r);
            j.dy[k][e] = dir_dy(r);
            j.plane[k][e] = planes++;
            j.nlines[k] = (int)scanlines_of(r, W, H);
        }
        if (j.ndir[k] == 0) continue;
        const int G = 32 / lanes_of(D, i == 0 ? lc.np_long : lc.np_other);
        j.jbegin[k + 1] = j.jbegin[k] + j.ndir[k] * ((j.nlines[k] + G - 1) / G);
        j.n++;
        if (i == 0) j.nlong = j.jbegin[k + 1] - j.jbegin[k], j.klong = k;
    }
    return j;
}

// 16 resident warps per SM, or 20 where these leave the last round of short-axis
// jobs less than half full and 20 do not (the long-axis jobs outlast several rounds).
// Measured, aggregation in us at 4 and 5 blocks per SM, 8 paths:
//   rounds of 2.2 and 1.6 (1242 x 375, D = 128) 127, 116;  2.4 and 1.6 (1000 x 600, D = 128) 161, 155
//   1.5 and 0.9 (656 x 572, D = 128) 104, 114;  2.6 and 1.9 (1400 x 400, D = 128) 139, 148
//   1.1 and 0.8 (1280 x 720, D = 64) 155, 172;  2.1 and 1.5 (1920 x 1080, D = 64) 381, 393
int default_blocks_per_sm(const PathJobs &j) {
    const double others = j.jbegin[j.n] - j.nlong;
    auto rounds = [&](int blocks) { return others / (blocks * kSchedulers - j.nlong); };
    if (j.klong != 0 || 4 * kSchedulers <= j.nlong) return 4;
    const double r4 = rounds(4), r5 = rounds(5);
    return r5 > 1 && r4 - (int)r4 < 0.5 && r5 - (int)r5 > 0.5 ? 5 : 4;
}

namespace {

constexpr int kWarps = 4;
constexpr int kRingBytes = 8192, kStages = 4;  // cost ring of a warp

__device__ __forceinline__ uint32_t vmin2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// a * b + c on the FMA pipe.
__device__ __forceinline__ uint32_t mad(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

// The planes are written once and read back only by the WTA kernel, so they
// leave L2 first (evict_first).
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// Job scheduling.  Jobs are numbered in the order of the work list: long-axis
// scanlines first, as they take longest, or after one sweep from 100 MB of costs
// on (make_path_jobs).  A warp's first job is its rank: one warp of every SM and
// scheduler in turn, so that the long-axis jobs spread over all of them.  Later jobs come
// from one counter, and only when there are more jobs than warps: thousands of
// warps that start with an atomic on one address pay about 8 ns each, one after
// the other (320x240, 8 blocks per SM: 61.7 us against 26.3 with 1).
__device__ __forceinline__ int first_job(int sms) {
    const int before = blockIdx.x / sms * sms, sm = blockIdx.x - before;  // blocks of the layers before
    const int layer = min(sms, (int)gridDim.x - before);
    return before * kWarps + (int)(threadIdx.x >> 5) * layer + sm;
}

// The job after the warps' first ones, total when there is none.
__device__ __forceinline__ int next_job(unsigned *counter, int total, int lane) {
    const int warps = (int)gridDim.x * kWarps;
    int job = total;
    if (warps < total) {
        if (lane == 0) job = warps + (int)atomicAdd(counter, 1u);
        job = __shfl_sync(0xffffffffu, job, 0);
    }
    return job;
}

// The NP pairs one lane holds, as they sit in the cost volume and the planes:
// 2 bytes per pair for 8-bit costs, 4 for the 16-bit costs of SAD.  With one
// 8-bit pair per lane (kHalf) two lanes share a word; the even one stores it.
template <int NP, bool WIDE>
struct Blk {
    static constexpr bool kHalf = NP == 1 && !WIDE;
    static constexpr int kLane = WIDE ? 4 * NP : 2 * NP;  // bytes of a lane
    static constexpr int kWords = WIDE ? NP : NP == 1 ? 1 : NP / 2;
    static constexpr bool kStaged = kWords == 3;  // no vector: stored by way of shared memory
    static_assert(kWords <= 3 || kWords % 4 == 0, "a lane block is 4, 8, 12 or whole 16-byte vectors");
    uint32_t w[kWords];
};

template <int NP, bool WIDE>
__device__ __forceinline__ Blk<NP, WIDE> ld_ring(uint32_t at) {
    Blk<NP, WIDE> v;
    if constexpr (Blk<NP, WIDE>::kWords == 1) {
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v.w[0]) : "r"(at));
    } else if constexpr (Blk<NP, WIDE>::kWords == 2) {
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.w[0]), "=r"(v.w[1]) : "r"(at));
    } else if constexpr (Blk<NP, WIDE>::kStaged) {
#pragma unroll
        for (int q = 0; q < 3; q++) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v.w[q]) : "r"(at + 4 * q));
    } else {
#pragma unroll
        for (int q = 0; q < Blk<NP, WIDE>::kWords; q += 4)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(v.w[q]), "=r"(v.w[q + 1]), "=r"(v.w[q + 2]), "=r"(v.w[q + 3])
                         : "r"(at + 4 * q));
    }
    return v;
}
template <int NP, bool WIDE>
__device__ __forceinline__ void st_blk(Blk<NP, WIDE> *p, const Blk<NP, WIDE> &v, uint64_t pol) {
    if constexpr (Blk<NP, WIDE>::kWords == 1) {
        asm volatile("st.global.L1::no_allocate.L2::cache_hint.u32 [%0], %1, %2;" ::"l"(p), "r"(v.w[0]), "l"(pol)
                     : "memory");
    } else if constexpr (Blk<NP, WIDE>::kWords == 2) {
        asm volatile("st.global.L1::no_allocate.L2::cache_hint.v2.u32 [%0], {%1, %2}, %3;" ::"l"(p), "r"(v.w[0]),
                     "r"(v.w[1]), "l"(pol)
                     : "memory");
    } else {
#pragma unroll
        for (int q = 0; q < Blk<NP, WIDE>::kWords; q += 4)
            asm volatile("st.global.L1::no_allocate.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(
                             reinterpret_cast<uint32_t *>(p) + q),
                         "r"(v.w[q]), "r"(v.w[q + 1]), "r"(v.w[q + 2]), "r"(v.w[q + 3]), "l"(pol)
                         : "memory");
    }
}

// Stores 16 bytes of a step that the lanes have left in shared memory at `from`.
__device__ __forceinline__ void st_staged(uint4 *p, uint32_t from, uint64_t pol) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(from) : "memory");
    asm volatile("st.global.L1::no_allocate.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "r"(v.x),
                 "r"(v.y), "r"(v.z), "r"(v.w), "l"(pol)
                 : "memory");
}

// The cost ring of a warp: kStages stages of one block of steps each, in shared
// memory.  A step is the warp's 32 lane blocks; one asynchronous copy of the
// warp moves kCopy bytes per lane, kPer steps together (or a part of one).
template <int NP, int G, bool WIDE>
struct Ring {
    static constexpr int kStep = 32 * Blk<NP, WIDE>::kLane;                           // bytes of a step
    static constexpr bool kTiny = G >= 8 && (32 / G) * Blk<NP, WIDE>::kLane == 8;  // records of 8 bytes
    static constexpr int kCopy = kTiny ? 8 : 16;
    static constexpr int kPer = 32 * kCopy >= kStep ? 32 * kCopy / kStep : 1;     // steps of a copy
    static constexpr int kParts = 32 * kCopy >= kStep ? 1 : kStep / (32 * kCopy);  // copies of a step
    static constexpr int kFit = kRingBytes / kStages / kStep;
    static constexpr int kBlock = kFit >= 16 ? 16 : kFit > 4 ? kFit & ~3 : kFit;  // steps of a stage
    static constexpr int kBytes = kBlock * kStep;
    static constexpr int kStageOut = Blk<NP, WIDE>::kStaged ? 2 * kStep : 0;  // path costs on their way out, behind the stages
    static_assert(kStages * kBytes + kStageOut <= kRingBytes, "the ring holds the stages");
};

// Asynchronous copies of BYTES into shared memory (zeros when ok is false).
template <int BYTES>
__device__ __forceinline__ void copy_async(uint32_t dst, const void *src) {
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
template <int BYTES>
__device__ __forceinline__ void copy_or_zero(uint32_t dst, const void *src, bool ok) {
    const int n = ok ? BYTES : 0;
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// One lane's place in its scanline, fixed for a job.
struct LaneGeom {
    int grp, li;          // scanline of the warp, lane within it
    int src_up, src_dn;   // lanes that hold the neighbouring pairs (its own at the scanline's ends)
    uint32_t sel_dn;      // byte-permute selector: the lane after, or its own last pair swapped
    uint32_t sel_c;       // byte-permute selector of a lane's pair in the word it shares
    uint32_t lo_mark;     // added to the pair before the scanline's first one
    bool first;
};

// Path state of one lane: R[k] = pair k, m2 = (m, m), mQ = m2 + (P2 - P1, P2 - P1).
template <int NP>
struct PathState {
    uint32_t R[NP];
    uint32_t m2, mQ;
};

// The smaller half of x in both halves.  Non-negative half floats order like
// their bits, and the path costs stay below infinity's (0x7C00): one minimum of
// the two halves instead of a byte-permute and a minimum.
__device__ __forceinline__ uint32_t fold_min(uint32_t x) {
    const __half2 h = *reinterpret_cast<const __half2 *>(&x);
    const __half2 m = __hmin2(__low2half2(h), __high2half2(h));
    return *reinterpret_cast<const uint32_t *>(&m);
}

// One step of Eq. 2 for the lane's NP pairs with cost block b; returns the
// block to store.
template <int NP, int G, bool WIDE>
__device__ __forceinline__ Blk<NP, WIDE> path_step(PathState<NP> &st, const Blk<NP, WIDE> &b, uint32_t P1x2, uint32_t QPx2,
                                                   const LaneGeom &lg, uint32_t one) {
    constexpr int kLanes = 32 / G;                          // lanes per scanline where it is a power of two
    constexpr bool kTiny = G >= 8 && 2 * NP * kLanes == 8;  // Dp = 8: padding in both halves of a pair
    const uint32_t m2 = st.m2;
    uint32_t c[NP];
#pragma unroll
    for (int w = 0; w < NP; w += 2) {
        if constexpr (WIDE) {
            c[w] = b.w[w];
            if (NP > 1) c[NP > 1 ? w + 1 : 0] = b.w[NP > 1 ? w + 1 : 0];
        } else if constexpr (NP == 1) {
            c[0] = __byte_perm(b.w[0], 0u, lg.sel_c);
        } else {
            const uint32_t v = b.w[w / 2];
            c[w] = __byte_perm(v, 0u, 0x4341);               // bytes 1, 3
            c[w + 1] = mad(c[w], one * 0xFFFFFF00u, v);      // bytes 0, 2: v - (bytes 1, 3) * 256
        }
    }
    uint32_t before, after;
    if constexpr (G == 32) {  // one lane per scanline
        before = st.R[NP > 1 ? 1 : 0];
        after = __byte_perm(st.R[NP - 1], 0u, 0x1032);
    } else {
        before = __shfl_sync(0xffffffffu, st.R[NP - 1], lg.src_up);
        const uint32_t dn = __shfl_sync(0xffffffffu, st.R[0], lg.src_dn);
        after = __byte_perm(dn, st.R[NP - 1], lg.sel_dn);
        // the first lane got its own last pair: for NP = 2 that is a neighbour of
        // its first pair anyway, for NP = 1 the pair itself, which changes nothing;
        // otherwise it is lifted out of the way
        if constexpr (NP > 2) {
            if constexpr (WIDE) before = lg.first ? st.R[1] : before;
            else before = mad(before, one, lg.lo_mark);
        }
    }
    uint32_t n[NP];
#pragma unroll
    for (int k = 0; k < NP; k++) {
        const uint32_t l = k == 0 ? before : st.R[k - 1];
        const uint32_t r = k == NP - 1 ? after : st.R[k + 1];
        const uint32_t t = __viaddmin_u16x2(__vimin3_u16x2(l, r, st.mQ), P1x2, st.R[k]);
        n[k] = t + c[k] - m2;
    }
    Blk<NP, WIDE> out;
    if constexpr (WIDE) {
#pragma unroll
        for (int k = 0; k < NP; k++) out.w[k] = n[k];
    } else if constexpr (NP == 1) {
        out.w[0] = mad(n[0], one * 256u, __shfl_xor_sync(0xffffffffu, n[0], 1));  // of even lanes
    } else if constexpr (kTiny) {
#pragma unroll
        for (int w = 0; w < NP / 2; w++) out.w[w] = __byte_perm(n[2 * w + 1], n[2 * w], 0x6240);
    } else {
        // a padding slot above 255 carries into a padding slot of a larger
        // disparity or out of the word, as only the upper halves hold padding
#pragma unroll
        for (int w = 0; w < NP / 2; w++) out.w[w] = mad(n[2 * w], one * 256u, n[2 * w + 1]);
    }
    // the lane's minimum, folded over the halves, over the scanline's lanes
    uint32_t x = n[0];
    if constexpr (NP == 2) {
        x = vmin2(n[0], n[1]);
    } else if constexpr (NP > 2) {
        uint32_t y = __vimin3_u16x2(n[0], n[1], n[2]);
#pragma unroll
        for (int k = 3; k + 1 < NP; k += 2) y = __vimin3_u16x2(y, n[k], n[k + 1]);
        x = vmin2(y, n[NP - 1]);
    }
#pragma unroll
    for (int k = 0; k < NP; k++) st.R[k] = n[k];
    x = WIDE ? vmin2(x, __byte_perm(x, 0u, 0x1032)) : fold_min(x);
    uint32_t mn;
    if constexpr (G >= 8 || (NP >= 8 && G == 4)) {
#pragma unroll
        for (int o = 1; o < kLanes; o <<= 1) x = vmin2(x, __shfl_xor_sync(0xffffffffu, x, o));
        mn = x;
    } else if constexpr (G == 1) {
        mn = __reduce_min_sync(0xffffffffu, x);
    } else {
        // (m, m) = m * 0x10001 is monotonic in m; the other scanlines' lanes feed
        // x + 0x80008000, more than any (m, m)
        uint32_t r[G];
#pragma unroll
        for (int g = 0; g < G; g++) r[g] = __reduce_min_sync(0xffffffffu, mad(x, one, lg.grp == g ? 0u : 0x80008000u));
        if constexpr (G == 4) mn = lg.grp < 2 ? (lg.grp == 0 ? r[0] : r[1]) : (lg.grp == 2 ? r[2] : r[3]);
        else mn = lg.grp == 0 ? r[0] : r[1];
        static_assert(G == 2 || G == 4, "scanlines per warp that reduce with redux.sync");
    }
    st.m2 = mn;
    st.mQ = mad(mn, one, QPx2);
    return out;
}

// Scanline s of direction (dx, dy): its first pixel, the step before which it
// wraps (kNever: never) and what the wrap adds to the pixel index.
constexpr int kNever = 0x3FFFFFFF;
struct Walk {
    int x, y, wrap, jump;
};
__device__ __forceinline__ Walk walk_of(int dx, int dy, int s, int W, int H) {
    const bool by_rows = dx == 0 || (dy != 0 && W >= H);  // one row per step, from column s
    Walk w;
    w.x = by_rows ? s : dx > 0 ? 0 : W - 1;
    w.y = by_rows ? dy > 0 ? 0 : H - 1 : s;
    w.wrap = kNever;
    w.jump = 0;
    if (dx != 0 && dy != 0) {
        const int n = by_rows ? W : H, step = by_rows ? dx : dy;
        w.wrap = step > 0 ? n - s : s + 1;
        w.jump = -step * (by_rows ? W : H * W);
    }
    return w;
}

// One job: the G neighbouring scanlines s0 .. s0+G-1 of one direction
// (dx, dy), scanline s0 + grp for this lane's group, written to plane
// `plane` of `nplanes`.  A scanline's pixel is LPS lane blocks of NP pairs.
// FULL: the G scanlines' lanes fill the warp.
// WRAP: diagonals may be among the directions.
template <int NP, int G, bool WIDE, bool FULL, bool WRAP>
__device__ __forceinline__ void run_job(const void *__restrict__ cost_, void *__restrict__ planes_, int W, int H,
                                        int lps_, int nplanes, int dx, int dy, int plane, int nlines, int s0,
                                        uint32_t P1x2, uint32_t P2x2, uint64_t pol, uint32_t one) {
    using BT = Blk<NP, WIDE>;
    using RT = Ring<NP, G, WIDE>;
    extern __shared__ __align__(16) uint8_t agg_smem[];
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(agg_smem) + (threadIdx.x >> 5) * kRingBytes;
    const int LPS = G >= 8 || FULL ? 32 / G : lps_;
    const int lane = threadIdx.x & 31;
    LaneGeom lg;
    // Lanes beyond the last scanline repeat its last lane, in all it computes and stores.
    const int vl = FULL ? lane : min(lane, G * LPS - 1);
    lg.grp = vl / LPS;
    lg.li = vl - lg.grp * LPS;
    lg.first = lg.li == 0;
    const bool last = lg.li == LPS - 1;
    lg.src_up = lg.first ? lane : vl - 1;
    lg.src_dn = last ? lane : lane + 1;
    lg.sel_dn = last ? 0x5476u : 0x3210u;
    lg.lo_mark = lg.first ? 0x7FFF7FFFu : 0u;
    lg.sel_c = lg.li & 1 ? 0x4240u : 0x4341u;
    // Likewise scanlines beyond the last repeat it.
    const Walk wk = walk_of(dx, dy, min(s0 + lg.grp, nlines - 1), W, H);
    const int len = dx == 0 || (dy != 0 && W >= H) ? H : W;
    // block indices: cost block (x, y, li) is cost[(y*W + x)*LPS + li], plane
    // block is planes[((y*W + x)*nplanes + plane)*LPS + li] (all planes of a
    // pixel are adjacent).  They stay below 2^32 (checked at handle creation).
    const long long pix = (long long)wk.y * W + wk.x, dir = (long long)dy * W + dx;
    const int rec = LPS * BT::kLane;  // bytes of a pixel's record
    const long long cost_copies = (long long)W * H * rec / RT::kCopy;
    const long long plane_blocks = (long long)W * H * nplanes * rec / (BT::kStaged ? 16 : (int)sizeof(BT));
    // the lane block of the step to store (their count stays below 2^32, checked at
    // handle creation; 32 bits keep the address arithmetic on the FMA pipe)
    constexpr int kUnit = BT::kStaged ? 16 : (int)sizeof(BT);  // bytes of a store
    uint32_t oi = (uint32_t)(((pix * nplanes + plane) * rec + lg.li * BT::kLane) / kUnit);
    const uint32_t ostep = (uint32_t)(dir * nplanes * rec / kUnit);
    const uint32_t ojump = (uint32_t)((long long)wk.jump * nplanes * rec / kUnit);
    bool stores = !BT::kHalf || !(lg.li & 1);
    int owrap = wk.wrap;  // of the scanline this lane stores for
    if constexpr (BT::kStaged) {
        const int ogrp = lane * 16 / rec;
        const Walk ow = walk_of(dx, dy, min(s0 + ogrp, nlines - 1), W, H);
        stores = ogrp < G;
        owrap = ow.wrap;
        oi = (uint32_t)(((((long long)ow.y * W + ow.x) * nplanes + plane) * rec + lane * 16 - ogrp * rec) / 16);
    }
    // this lane's share of the copies: kCopy bytes at offset ccol of the record of
    // scanline s0 + cgrp (one per part of a step), csub steps into the copy
    const int csub = lane * RT::kCopy / RT::kStep;
    int cwrap[RT::kParts];
    bool mine[RT::kParts];  // a step's records may be shorter than the warp's copies
    uint32_t ci[RT::kParts];  // in units of kCopy bytes, below 2^32 like oi
#pragma unroll
    for (int p = 0; p < RT::kParts; p++) {
        const int unit = (p * 32 + lane) * RT::kCopy % RT::kStep;  // byte of the step
        const int cgrp = unit / rec;
        const Walk cw = walk_of(dx, dy, min(s0 + cgrp, nlines - 1), W, H);
        cwrap[p] = cw.wrap;
        mine[p] = BT::kStaged ? lane * RT::kCopy < RT::kStep : FULL || cgrp < G;
        ci[p] = (uint32_t)((((long long)cw.y * W + cw.x + csub * dir) * rec + (unit - cgrp * rec)) / RT::kCopy);
    }
    const uint32_t cjump = (uint32_t)((long long)wk.jump * rec / RT::kCopy);
    const uint32_t cadv = (uint32_t)(dir * RT::kPer * rec / RT::kCopy);
    const uint32_t ring_w = ring + lane * RT::kCopy, ring_r = ring + (vl * BT::kLane & ~3);
    using CT = typename std::conditional<RT::kCopy == 16, uint4, uint2>::type;
    const CT *__restrict__ cost = reinterpret_cast<const CT *>(cost_);
    BT *__restrict__ planes = reinterpret_cast<BT *>(planes_);
    const uint32_t out = ring + kStages * RT::kBytes;  // [2][kStep], BT::kStaged only
    // Stores the path costs of step i of a block, where ok.
    auto put = [&](int i, const BT &o, bool ok) {
        if constexpr (BT::kStaged) {
            // two buffers: a lane writes one again only after the barrier of the step
            // between, which follows every lane's read of it
            const uint32_t buf = out + (uint32_t)(i & 1) * RT::kStep;
#pragma unroll
            for (int q = 0; q < 3; q++)
                asm volatile("st.shared.u32 [%0], %1;" ::"r"(buf + lane * BT::kLane + 4 * q), "r"(o.w[q]) : "memory");
            __syncwarp();
            if (ok && in_range(oi, plane_blocks)) st_staged(reinterpret_cast<uint4 *>(planes_) + oi, buf + lane * 16, pol);
        } else {
            if (ok && in_range(oi, plane_blocks)) st_blk(planes + oi, o, pol);
        }
        oi += ostep;
    };
    // Copies block `blk` into its stage; what a scanline does not have reads as 0.
    // checked: the block may be past the end or hold a wrap.
    auto fetch = [&](int blk, auto checked) {
        const uint32_t at = ring_w + (uint32_t)(blk % kStages) * RT::kBytes;
#pragma unroll
        for (int i = 0; i < RT::kBlock; i += RT::kPer) {
#pragma unroll
            for (int p = 0; p < RT::kParts; p++) {
                const uint32_t to = at + i * RT::kStep + p * 32 * RT::kCopy;
                if constexpr (decltype(checked)::value) {
                    const int t = blk * RT::kBlock + i + csub;
                    if (WRAP && t >= cwrap[p]) {
                        ci[p] += cjump;
                        cwrap[p] = kNever;
                    }
                    const bool ok = mine[p] && t < len && in_range(ci[p], cost_copies);
                    if (!BT::kStaged || mine[p]) copy_or_zero<RT::kCopy>(to, cost + (ok ? ci[p] : 0u), ok);
                } else if (mine[p] && in_range(ci[p], cost_copies)) {
                    copy_async<RT::kCopy>(to, cost + ci[p]);
                }
                ci[p] += cadv;
            }
        }
        if constexpr (WRAP && decltype(checked)::value) {
            // a lane that copies every kPer-th step may have its first one past the
            // wrap in the next block
#pragma unroll
            for (int p = 0; p < RT::kParts; p++)
                if (cwrap[p] < (blk + 1) * RT::kBlock) {
                    ci[p] += cjump;
                    cwrap[p] = kNever;
                }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const uint32_t QPx2 = P2x2 - P1x2;
    PathState<NP> st;
#pragma unroll
    for (int k = 0; k < NP; k++) st.R[k] = 0u;
    st.m2 = 0u;
    st.mQ = QPx2;
    using Checked = std::integral_constant<bool, true>;
    using Unchecked = std::integral_constant<bool, false>;
    constexpr int B = RT::kBlock;
    __syncwarp();  // the ring of the warp's previous job has been read
#pragma unroll 1
    for (int j = 0; j < kStages - 1; j++) fetch(j, Checked());
    // Blocks of steps: nblk, the first nfull of them whole; [wrap0, wrap1) may hold a wrap.
    const int nblk = (len + B - 1) / B, nfull = len / B;
    const int wrap0 = WRAP ? min((int)__reduce_min_sync(0xffffffffu, (unsigned)wk.wrap) / B, nblk) : nblk;
    const int wrap1 = WRAP ? min((int)__reduce_max_sync(0xffffffffu, (unsigned)wk.wrap) / B + 1, nblk) : nblk;
    auto next_block = [&](int blk) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
        __syncwarp();  // every lane's copies of this block are there, and the block before has been read
        const int ahead = blk + kStages - 1;
        if (ahead < nfull && (ahead < wrap0 || ahead >= wrap1)) fetch(ahead, Unchecked());
        else fetch(ahead, Checked());
        return ring_r + (uint32_t)(blk % kStages) * RT::kBytes;
    };
    constexpr int kTail = B < 4 ? B : 4;
    static_assert(B % kTail == 0, "whole parts of a block");
    // a block in which nothing ends or wraps: no checks
    auto plain = [&](int blk) {
        const uint32_t at = next_block(blk);
        BT cur = ld_ring<NP, WIDE>(at);
#pragma unroll
        for (int i = 0; i < B; i++) {
            BT nxt = cur;
            if (i + 1 < B) nxt = ld_ring<NP, WIDE>(at + (i + 1) * RT::kStep);
            const BT o = path_step<NP, G, WIDE>(st, cur, P1x2, QPx2, lg, one);
            put(i, o, stores);
            cur = nxt;
        }
    };
    // any other, a few steps at a time: what is computed past the end is not stored
    auto special = [&](int blk) {
        const uint32_t at = next_block(blk);
#pragma unroll 1
        for (int i = 0; i < B && blk * B + i < len; i += kTail) {
            BT in[kTail];
#pragma unroll
            for (int q = 0; q < kTail; q++) in[q] = ld_ring<NP, WIDE>(at + (i + q) * RT::kStep);
#pragma unroll
            for (int q = 0; q < kTail; q++) {
                const int t = blk * B + i + q;
                if (WRAP && t == wk.wrap) {
#pragma unroll
                    for (int k = 0; k < NP; k++) st.R[k] = 0u;
                    st.m2 = 0u;
                    st.mQ = QPx2;
                }
                if (WRAP && t == owrap) oi += ojump;
                const BT o = path_step<NP, G, WIDE>(st, in[q], P1x2, QPx2, lg, one);
                put(q, o, stores && t < len);
            }
        }
    };
    int blk = 0;
    if constexpr (WRAP) {
        const int cut = min(wrap0, nfull);
#pragma unroll 1
        for (; blk < cut; blk++) plain(blk);
#pragma unroll 1
        for (; blk < wrap1; blk++) special(blk);
#pragma unroll 1
        for (; blk < nfull; blk++) plain(blk);
#pragma unroll 1
        for (; blk < nblk; blk++) special(blk);
    } else {
#pragma unroll 1
        for (; blk < nfull; blk++) plain(blk);
#pragma unroll 1
        for (; blk < nblk; blk++) special(blk);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Jobs of the long-axis entry hold NPL pairs per lane (GL scanlines per warp),
// the others NPO (GO).
template <int NPL, int GL, int NPO, int GO, bool WIDE, bool FULL>
__global__ void __launch_bounds__(kWarps * 32, 6)
    aggregate_kernel(const void *__restrict__ cost, int W, int H, int Dp, uint32_t P1x2, uint32_t P2x2,
                     const __grid_constant__ PathJobs jobs, void *__restrict__ planes, int nplanes,
                     unsigned *__restrict__ job_counter, int sms) {
    wait_for_predecessor();
    const int lane = threadIdx.x & 31;
    const int total = jobs.jbegin[jobs.n];
    const uint64_t pol = policy_evict_first();
    int job = first_job(sms);
    while (job < total) {
        int k = 0;
        while (job >= jobs.jbegin[k + 1]) k++;
        const int q = job - jobs.jbegin[k];
        const int line = q / jobs.ndir[k], e = q - line * jobs.ndir[k];
        if (k == jobs.klong)
            run_job<NPL, GL, WIDE, FULL, false>(cost, planes, W, H, Dp / (2 * NPL), nplanes, jobs.dx[k][e], jobs.dy[k][e],
                                   jobs.plane[k][e], jobs.nlines[k], line * GL, P1x2, P2x2, pol, jobs.unit);
        else
            run_job<NPO, GO, WIDE, FULL || NPO == 6, true>(cost, planes, W, H, Dp / (2 * NPO), nplanes, jobs.dx[k][e], jobs.dy[k][e],
                                   jobs.plane[k][e], jobs.nlines[k], line * GO, P1x2, P2x2, pol, jobs.unit);
        job = next_job(job_counter, total, lane);
    }
}

// Scanlines a warp walks at once.
__host__ __device__ constexpr int lines_per_warp(int Dp, int np) { return Dp / (2 * np) > 0 ? 32 / (Dp / (2 * np)) : 0; }

// Many pairs in one persistent launch.  The work list of pair p is its
// PathJobs; the two queues number all pairs' long-axis jobs (queue 0) and
// all their other jobs (queue 1) in pair order, pair p's starting at
// pfx[0][p] and pfx[1][p].  Each job runs with its pair's lanes per scanline;
// CPL == 4 adds the lanes of 16 pairs.
template <int CPL, bool WIDE>
__global__ void __launch_bounds__(kWarps * 32, 6)
    aggregate_batch_kernel(const BatchAggPair *__restrict__ pairs, int npairs, const int *__restrict__ prefix,
                           uint32_t P1x2, uint32_t P2x2, unsigned *__restrict__ job_counter, int sms) {
    wait_for_predecessor();
    extern __shared__ __align__(16) uint8_t agg_smem[];
    int *spfx = reinterpret_cast<int *>(agg_smem + kWarps * kRingBytes);  // [2][npairs + 1]
    for (int i = threadIdx.x; i < 2 * (npairs + 1); i += blockDim.x) spfx[i] = prefix[i];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int nlong = spfx[npairs], nother = spfx[npairs + 1 + npairs];
    const int total = nlong + nother;
    const uint64_t pol = policy_evict_first();
    int job = first_job(sms);
    while (job < total) {
        // the pair: binary search in the queue's prefix
        const bool lq = job < nlong;
        const int *q = lq ? spfx : spfx + npairs + 1;
        const int jq = lq ? job : job - nlong;
        int lo = 0, hi = npairs;  // q[lo] <= jq < q[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (q[mid] <= jq) lo = mid;
            else hi = mid;
        }
        const BatchAggPair &p = pairs[lo];
        const int local = lq ? jq - q[lo] : p.jobs.nlong + (jq - q[lo]);
        int k = 0;
        while (local >= p.jobs.jbegin[k + 1]) k++;
        const int ql = local - p.jobs.jbegin[k];
        const int line = ql / p.jobs.ndir[k], e = ql - line * p.jobs.ndir[k];
        auto job_as = [&](auto np, auto g) {
            constexpr int NP = decltype(np)::value, G = decltype(g)::value;
            run_job<NP, G, WIDE, (G >= 8), true>(p.cost, p.planes, p.W, p.H, p.Dp / (2 * NP), p.nplanes, p.jobs.dx[k][e],
                                 p.jobs.dy[k][e], p.jobs.plane[k][e], p.jobs.nlines[k], line * G, P1x2, P2x2, pol,
                                 p.jobs.unit);
        };
        // pairs per lane of this job, and scanlines per warp
        const int np = lq ? p.jobs.lanes.np_long : p.jobs.lanes.np_other;
#define SGM_JOB(NP, G) \
    case 64 * NP + G: job_as(std::integral_constant<int, NP>(), std::integral_constant<int, G>()); break
        switch (64 * np + lines_per_warp(p.Dp, np)) {
            SGM_JOB(2, 16);
            SGM_JOB(2, 8);
            SGM_JOB(2, 4);
            SGM_JOB(2, 2);
            SGM_JOB(2, 1);
            SGM_JOB(4, 32);
            SGM_JOB(4, 16);
            SGM_JOB(4, 8);
            SGM_JOB(4, 4);
            SGM_JOB(4, 2);
            SGM_JOB(4, 1);
            default:
                if constexpr (CPL == 4) switch (64 * np + lines_per_warp(p.Dp, np)) {
                    SGM_JOB(16, 32);
                    SGM_JOB(16, 16);
                    SGM_JOB(16, 8);
                    SGM_JOB(16, 4);
                }
        }
#undef SGM_JOB
        job = next_job(job_counter, total, lane);
    }
}

using AggKernel = void (*)(const void *, int, int, int, uint32_t, uint32_t, const PathJobs, void *, int, unsigned *, int);

// The kernel of a pair of lane widths, null when there is none.
template <bool WIDE>
AggKernel agg_kernel_t(int Dp, LaneConfig lc) {
    const bool full = (Dp & (Dp - 1)) == 0;
#define SGM_AGG_F(NPL, GL, NPO, GO, FULL)                                                                            \
    if (full == FULL && lc.np_long == NPL && lc.np_other == NPO && lines_per_warp(Dp, NPL) == GL && lines_per_warp(Dp, NPO) == GO) \
        return aggregate_kernel<NPL, GL, NPO, GO, WIDE, FULL>
#define SGM_AGG(NPL, GL, NPO, GO) SGM_AGG_F(NPL, GL, NPO, GO, true)
    SGM_AGG(2, 16, 4, 32);  // Dp = 8
    SGM_AGG(2, 8, 4, 16);   // 16
    SGM_AGG(2, 4, 4, 8);    // 32
    SGM_AGG(1, 2, 4, 8);
    SGM_AGG(1, 2, 1, 2);
    SGM_AGG(2, 2, 4, 4);    // 64
    SGM_AGG(2, 2, 2, 2);
    SGM_AGG(1, 1, 4, 4);
    SGM_AGG(1, 1, 2, 2);
    SGM_AGG_F(2, 1, 4, 2, false);  // 96
    SGM_AGG_F(2, 1, 2, 1, false);
    SGM_AGG(2, 1, 4, 2);    // 128
    SGM_AGG(2, 1, 2, 1);
    SGM_AGG_F(4, 1, 4, 1, false);  // 160, 192, 224
    SGM_AGG(4, 1, 4, 1);    // 256
    if constexpr (!WIDE) {
        SGM_AGG_F(2, 1, 6, 4, false);  // 96
        SGM_AGG_F(4, 1, 6, 2, false);  // 192
        // Dp a power of two, 16 to 256
        SGM_AGG(8, 32, 8, 32);
        SGM_AGG(8, 16, 8, 16);
        SGM_AGG(8, 8, 8, 8);
        SGM_AGG(8, 4, 8, 4);
        SGM_AGG(8, 2, 8, 2);
        SGM_AGG(4, 16, 8, 32);
        SGM_AGG(4, 8, 8, 16);
        SGM_AGG(4, 4, 8, 8);
        SGM_AGG(4, 2, 8, 4);
        SGM_AGG(4, 1, 8, 2);
        SGM_AGG(16, 32, 16, 32);
        SGM_AGG(16, 16, 16, 16);
        SGM_AGG(16, 8, 16, 8);
        SGM_AGG(16, 4, 16, 4);
    }
#undef SGM_AGG
#undef SGM_AGG_F
    return nullptr;
}
AggKernel agg_kernel(int Dp, LaneConfig lc, bool wide) {
    return wide ? agg_kernel_t<true>(Dp, lc) : agg_kernel_t<false>(Dp, lc);
}

// Plane 0 ([H][W][Dp], folded records) -> L ([H][W][D] uint16, natural order).
__global__ void unpermute_kernel(const uint8_t *__restrict__ plane, int npx, int D, int Dp, bool wide,
                                 uint16_t *__restrict__ L) {
    wait_for_predecessor();
    const size_t n = (size_t)npx * D;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t p = i / D;
        const int d = (int)(i - p * D);
        const size_t at = p * Dp + fold_slot(d, Dp, wide);
        L[i] = wide ? reinterpret_cast<const uint16_t *>(plane)[at] : plane[at];
    }
}

cudaError_t sm_count(int *sms) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e == cudaSuccess ? cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev) : e;
}

}  // namespace

bool chunks_apply(int D, bool wide) {
    const int Dp = padded_disparities(D);
    return !wide && (Dp & (Dp - 1)) == 0;  // lanes of 8 and 16 pairs come in powers of two
}

int chunks_per_lane_max(int D, bool wide) {
    const int chunks = lanes_per_scanline(D);  // 8-disparity chunks per pixel
    return wide ? 1 : (chunks >= 4 ? 4 : chunks);
}

cudaError_t launch_aggregate(const uint8_t *cost, int W, int H, int D, int P1, int P2, bool wide,
                             const PathJobs &jobs, uint8_t *planes, int nplanes,
                             unsigned *job_counter, int blocks_per_sm, int cpl, cudaStream_t s) {
    if (jobs.jbegin[jobs.n] == 0) return cudaSuccess;
    if (cpl != 1 && cpl != 2 && cpl != 4 && cpl != kMixedCpl) return cudaErrorInvalidValue;
    if ((cpl == kMixedCpl ? 2 : cpl) > chunks_per_lane_max(D, wide)) return cudaErrorInvalidValue;
    int sms = 0;
    const cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    // no more blocks than the jobs fill
    const int wanted = sms * (blocks_per_sm > 0 ? blocks_per_sm : 2), filled = (jobs.jbegin[jobs.n] + kWarps - 1) / kWarps;
    const int blocks = filled < sms ? sms : filled < wanted ? filled : wanted;  // whole layers
    const int Dp = padded_disparities(D);
    const LaneConfig lc = jobs.lanes;
    const uint32_t P1x2 = (uint32_t)P1 * 0x00010001u, P2x2 = (uint32_t)P2 * 0x00010001u;
    auto kernel = agg_kernel(Dp, lc, wide);
    if (!kernel) return cudaErrorInvalidValue;
    return launch_k(kernel, dim3(blocks), dim3(kWarps * 32), kWarps * kRingBytes, s, (const void *)cost, W, H, Dp, P1x2,
                    P2x2, jobs, (void *)planes, nplanes, job_counter, sms);
}

cudaError_t launch_aggregate_batch(const BatchAggPair *pairs, int npairs, const int *prefix, int P1, int P2,
                                   bool wide, int cpl, unsigned *job_counter, int blocks_per_sm, cudaStream_t s) {
    if (npairs <= 0) return cudaSuccess;
    int sms = 0;
    const cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    const int blocks = sms * (blocks_per_sm > 0 ? blocks_per_sm : 2);
    const uint32_t P1x2 = (uint32_t)P1 * 0x00010001u, P2x2 = (uint32_t)P2 * 0x00010001u;
    const size_t smem = kWarps * kRingBytes + sizeof(int) * 2 * (size_t)(npairs + 1);
    auto kernel = wide ? aggregate_batch_kernel<1, true>
                       : cpl == 4 ? aggregate_batch_kernel<4, false> : aggregate_batch_kernel<1, false>;
    const cudaError_t ea = allow_max_smem(kernel);
    if (ea != cudaSuccess) return ea;
    return launch_k(kernel, dim3(blocks), dim3(kWarps * 32), smem, s, pairs, npairs, prefix, P1x2, P2x2, job_counter, sms);
}

SGM_GUARD_COUNTER(guard_hits_aggregate)

cudaError_t launch_unpermute(const uint8_t *plane, int W, int H, int D, bool wide, uint16_t *L,
                             cudaStream_t s) {
    const int npx = W * H;
    const size_t n = (size_t)npx * D;
    const size_t want = (n + 255) / 256;
    const int blocks = (int)(want < 4096 ? want : 4096);
    unpermute_kernel<<<blocks, 256, 0, s>>>(plane, npx, D, padded_disparities(D), wide, L);
    return cudaGetLastError();
}

}  // namespace sgm
