// quality.cu -- event-video quality metrics (Sec. 4.2): the frame error of
// the mapped event frames, and the distance from every event to the nearest
// event of the same polarity in the other video, behind the polarity-aware
// F1 score and chamfer distance.
//
// Two event videos of one scene differ by little: most events have their
// counterpart in the same voxel and nearly all within a few.  So both videos are
// first packed into bit masks (one bit per voxel, polarity and video: 1/2 byte
// per voxel and rows padded to 32 columns, which stays in L2), events whose own bit is set in the target are
// counted by AND and population count, and only the rest search the target's
// rows around them ring by ring until no nearer event can exist.  Events
// without a neighbour in two rings and 15 columns are listed and searched for by a warp
// each through a coarse grid of cells, in a bounded number of steps.  Sets (polarity and
// direction) with more of them than the list holds, or with one that is not found
// in time, are matched by an exact squared Euclidean
// distance transform on the integer lattice (x, y, t), separable by axis:
//   rows (x): the input is binary, so a warp sweeps each row left to right
//     with a max-scan of event columns and right to left with a min-scan;
//   columns (y, then t): F'(u) = min_i (u - i)^2 + F(i) is the lower
//     envelope of parabolas rooted at the finite sites i of the line, built
//     in one forward sweep with integer separation points
//     floor((u^2 - i^2 + F(u) - F(i)) / (2 (u - i))) and read back in one
//     backward sweep (Meijster, Roerdink and Hesselink 2000; Felzenszwalb
//     and Huttenlocher 2012).  One thread owns one line at a time.  All
//     arithmetic is integer, so the result is exact.
// Every way gives the same integers: a distance is the minimum over the same events.
#include <algorithm>
#include <climits>
#include <utility>

#include "quality.h"

namespace mcev {
namespace {

constexpr int32_t QINF = 1 << 30;
constexpr int QBLOCK = 256;
constexpr int SMEM_BUDGET = 220 * 1024;

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// block-wide sums of three counters and one double, one atomic per nonzero
// value per block (slots < 0 are skipped)
__device__ void block_flush(unsigned long long u0, unsigned long long u1, unsigned long long u2, double d0,
                            unsigned long long* acc, int s0, int s1, int s2, int sd) {
    __shared__ unsigned long long p0[QBLOCK / 32], p1[QBLOCK / 32], p2[QBLOCK / 32];
    __shared__ double pd[QBLOCK / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    u0 = warp_sum(u0);
    u1 = warp_sum(u1);
    u2 = warp_sum(u2);
    d0 = warp_sum(d0);
    if (lane == 0) {
        p0[wid] = u0;
        p1[wid] = u1;
        p2[wid] = u2;
        pd[wid] = d0;
    }
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        u0 = warp_sum(lane < nw ? p0[lane] : 0ull);
        u1 = warp_sum(lane < nw ? p1[lane] : 0ull);
        u2 = warp_sum(lane < nw ? p2[lane] : 0ull);
        d0 = warp_sum(lane < nw ? pd[lane] : 0.0);
        if (lane == 0) {
            if (s0 >= 0 && u0) atomicAdd(acc + s0, u0);
            if (s1 >= 0 && u1) atomicAdd(acc + s1, u1);
            if (s2 >= 0 && u2) atomicAdd(acc + s2, u2);
            if (sd >= 0 && d0 != 0.0) atomicAdd(reinterpret_cast<double*>(acc + sd), d0);
        }
    }
}

// ---------------------------------------------------------------- event bits + frame error
// bytes of w (4 voxels) equal to v, as 4 bits
__device__ __forceinline__ uint32_t eq_bits(uint32_t w, uint32_t v) {
    return ((__vcmpeq4(w, v) & 0x01010101u) * 0x10204080u) >> 28;
}

// The 32 voxels from p on (n of them in the row; the rest read as 0) as eight
// 4-byte words, whatever the alignment: aligned words and a funnel shift, byte
// loads where an aligned word would reach outside [lo, hi).
__device__ __forceinline__ void load32(const int8_t* p, int n, const int8_t* lo, const int8_t* hi, uint32_t v[8]) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(p);
    if (n == 32 && (at & 15) == 0) {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(p)), y = __ldg(reinterpret_cast<const uint4*>(p) + 1);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
        return;
    }
    const int8_t* base = reinterpret_cast<const int8_t*>(at & ~(uintptr_t)3);
    if (n == 32 && base >= lo && base + 36 <= hi) {
        const uint32_t* q = reinterpret_cast<const uint32_t*>(base);
        const uint32_t sh = 8u * (uint32_t)(at & 3);
        uint32_t w = __ldg(q);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t x = __ldg(q + k + 1);
            v[k] = __funnelshift_r(w, x, sh);
            w = x;
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        uint32_t w = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * k + j < n) w |= (uint32_t)(uint8_t)p[4 * k + j] << (8 * j);
        v[k] = w;
    }
}

__device__ __forceinline__ void pack32(const uint32_t v[8], uint32_t& pos, uint32_t& neg, uint32_t& bad) {
    pos = neg = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t ep = eq_bits(v[k], 0x01010101u), en = eq_bits(v[k], 0xFFFFFFFFu);
        pos |= ep << (4 * k);
        neg |= en << (4 * k);
        bad |= (ep | en | eq_bits(v[k], 0u)) ^ 0xFu;
    }
}

// One thread packs 32 voxels of a row of both videos and tallies them: 2 B read and
// 1/2 B written per voxel (rows are padded to whole words).  1280x720x100 in 68 us, 3.4
// TB/s, half of the measured copy rate (6.67 TB/s): the compares and logic that pack the
// bytes keep the ALU pipe 81 % busy.  The tally alone, one voxel at a time, took 75 us.
__global__ void __launch_bounds__(QBLOCK) k_pack(const int8_t* __restrict__ a, const int8_t* __restrict__ b, int W,
                                                 int ww, int64_t n_words, int64_t n, uint32_t* __restrict__ masks,
                                                 unsigned long long* acc) {
    unsigned long long sq = 0;
    unsigned long long cnt[QSETS] = {0, 0, 0, 0};
    uint32_t bad = 0;
    const int64_t nth = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_words; i += nth) {
        const int64_t row = i / ww;
        const int x0 = (int)(i - row * ww) * 32;
        const int64_t at = row * W + x0;
        const int len = min(32, W - x0);
        uint32_t v[8], m[QSETS];
        load32(a + at, len, a, a + n, v);
        pack32(v, m[0], m[1], bad);
        load32(b + at, len, b, b + n, v);
        pack32(v, m[2], m[3], bad);
#pragma unroll
        for (int s = 0; s < QSETS; ++s) {
            masks[s * n_words + i] = m[s];
            cnt[s] += __popc(m[s]);
        }
        // (a - b)^2: 4 where the signs are opposite, 1 where one of them is zero
        sq += 4 * __popc((m[0] & m[3]) | (m[1] & m[2])) + __popc((m[0] | m[1]) ^ (m[2] | m[3]));
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(acc + QACC_BAD, 1ull);
    block_flush(sq, cnt[0], cnt[1], 0.0, acc, QACC_SQ, QACC_COUNT, QACC_COUNT + 1, -1);
    __syncthreads();
    block_flush(cnt[2], cnt[3], 0ull, 0.0, acc, QACC_COUNT + 2, QACC_COUNT + 3, -1, -1);
}

// ---------------------------------------------------------------- window search
// the masks' geometry
struct QGrid {
    int W, H, T, ww;
    int64_t n_words;      // per mask
};
constexpr int QNEAR = 15;     // columns of the first search's window
constexpr int QRINGS = 2;      // its rings (a 1280x720x100 call at 1 / 2 / 3 / 5 rings: 0.80 / 0.81 / 0.89 / 1.14 ms)
constexpr int QSETTLED = (QRINGS + 1) * (QRINGS + 1);   // what it has not looked at is this far away at least
// cells of the far search: 32 columns (a mask word) x 8 rows x 8 frames; a warp
// reads a cell row's 64 rows two per lane
constexpr int QCELL = 8;
__device__ __forceinline__ int set_target(int set) { return set ^ 2; }   // the other video, same polarity
// The searches drop set s from here on; the transform matches all of it anew.
__device__ __forceinline__ void leave_to_edt(unsigned long long* acc, int s) {
    if (!(*(volatile unsigned long long*)(acc + QACC_EDT) >> s & 1ull)) atomicOr(acc + QACC_EDT, 1ull << s);
}

// squared column distance from x to the nearest set bit of the row within
// QNEAR columns, or QINF
__device__ __forceinline__ int32_t row_near(const uint32_t* __restrict__ row, int ww, int x) {
    const int start = x - QNEAR;
    const int w = start >> 5;      // floor
    const uint32_t lo = w >= 0 ? __ldg(row + w) : 0u, hi = w + 1 < ww ? __ldg(row + w + 1) : 0u;
    const uint32_t bits = __funnelshift_r(lo, hi, (uint32_t)(start & 31));
    // bit k = column start + k; x is bit QNEAR
    const uint32_t left = bits & ((2u << QNEAR) - 1u), right = (bits >> QNEAR) & ((2u << QNEAR) - 1u);
    int32_t d = QINF;
    if (left) d = QNEAR - (31 - __clz(left));
    if (right) d = min(d, __ffs(right) - 1);
    return d < QINF ? d * d : QINF;
}

// the same without a column limit, looking no further than d2 < best
__device__ __forceinline__ int32_t row_wide(const uint32_t* __restrict__ row, int ww, int x, int32_t best) {
    const int w0 = x >> 5, bx = x & 31;
    uint32_t m = __ldg(row + w0);
    const uint32_t left = m & (uint32_t)((2ull << bx) - 1ull), right = m & (0xFFFFFFFFu << bx);
    int32_t d = QINF;
    if (left) d = bx - (31 - __clz(left));
    if (right) d = min(d, __ffs(right) - 1 - bx);
    if (d < QINF) best = min(best, d * d);
    for (int w = w0 - 1; w >= 0; --w) {
        const int edge = x - (32 * w + 31);        // distance of the word's nearest column
        if (edge * edge >= best) break;
        m = __ldg(row + w);
        if (m) {
            const int e = edge + __clz(m);
            best = min(best, e * e);
            break;
        }
    }
    for (int w = w0 + 1; w < ww; ++w) {
        const int edge = 32 * w - x;
        if (edge * edge >= best) break;
        m = __ldg(row + w);
        if (m) {
            const int e = edge + __ffs(m) - 1;
            best = min(best, e * e);
            break;
        }
    }
    return best;
}

// One warp takes 32 mask words of all four sets.  Events with the target's
// bit set have distance 0; the others are listed in shared memory, so that the
// lanes share them evenly, and each searches its target rows ring by ring
// (ring r: rows with max(|dy|, |dt|) = r, at least r^2 away).  Bound by the
// latency of the mask words' loads (72 % from L2; 11 of 32 lanes active): 212 us on
// 1280x720x100.
constexpr int QWARPS = 4;
__global__ void __launch_bounds__(32 * QWARPS) k_search(QGrid G, const uint32_t* __restrict__ masks, int tau2,
                                                       int32_t* __restrict__ d2_a, int32_t* __restrict__ d2_b,
                                                       uint64_t* __restrict__ far_list, int64_t far_cap,
                                                       unsigned long long* acc) {
    __shared__ uint16_t todo[QWARPS][2048];     // word << 5 | bit, + set << 10; a voxel is in at most 2 sets
    __shared__ uint32_t hist[QSETS][QSETTLED + 1];
    for (int i = threadIdx.x; i < QSETS * (QSETTLED + 1); i += blockDim.x) (&hist[0][0])[i] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    // no event to search for, or none that is worth it: earlier blocks have left the set to
    // the transform (which counts it anew)
    const unsigned edt = (unsigned)*(volatile unsigned long long*)(acc + QACC_EDT);
    bool lacks[QSETS];
#pragma unroll
    for (int s = 0; s < QSETS; ++s) lacks[s] = acc[QACC_COUNT + set_target(s)] == 0 || (edt >> s & 1u) != 0;
    unsigned long long matched[QSETS] = {0, 0, 0, 0}, none[QSETS] = {0, 0, 0, 0};
    const int64_t chunks = (G.n_words + 31) / 32;
    for (int64_t c = (int64_t)blockIdx.x * QWARPS + wib; c < chunks; c += (int64_t)gridDim.x * QWARPS) {
        const int64_t i = 32 * c + lane;
        const bool in = i < G.n_words;
        uint32_t m[QSETS];
#pragma unroll
        for (int s = 0; s < QSETS; ++s) m[s] = in ? __ldg(masks + s * G.n_words + i) : 0u;
        const int64_t row0 = 32 * c / G.ww;          // row of the chunk's first word
        const int word0 = (int)(32 * c - row0 * G.ww);
        // this lane's word in voxels
        const int off = word0 + lane;
        const int64_t vox = (row0 + off / G.ww) * G.W + 32 * (off % G.ww);
        int at = 0;
#pragma unroll
        for (int s = 0; s < QSETS; ++s) {
            int32_t* d2 = s < 2 ? d2_a : d2_b;
            uint32_t q = m[s];
            if (lacks[s]) {
                none[s] += __popc(q);
                if (d2)
                    for (; q; q &= q - 1) d2[vox + __ffs(q) - 1] = -2;
            }
            uint32_t same = q & m[set_target(s)];
            matched[s] += __popc(same);
            q ^= same;
            if (d2)
                for (; same; same &= same - 1) d2[vox + __ffs(same) - 1] = 0;
            if (lacks[s]) q = 0;
            if (!__any_sync(0xffffffffu, q != 0)) continue;
            const int k = __popc(q);
            int v = k;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += y;
            }
            for (int p = at + v - k; q; q &= q - 1, ++p)
                todo[wib][p] = (uint16_t)(s << 10 | lane << 5 | (__ffs(q) - 1));
            at += __shfl_sync(0xffffffffu, v, 31);
        }
        __syncwarp();
        for (int e = lane; e < at; e += 32) {
            const int id = todo[wib][e];
            const int s = id >> 10, o = word0 + ((id >> 5) & 31), dr = o / G.ww;
            const int x = 32 * (o - dr * G.ww) + (id & 31);
            const int64_t row = row0 + dr;
            const int t = (int)(row / G.H), y = (int)(row - (int64_t)t * G.H);
            const uint32_t* M = masks + set_target(s) * G.n_words;
            int32_t best = QINF;
            for (int r = 0; r <= QRINGS && r * r < best; ++r) {
                for (int dt = -r; dt <= r; ++dt) {
                    const int tt = t + dt;
                    if (tt < 0 || tt >= G.T) continue;
                    const int step = (dt == -r || dt == r) ? 1 : 2 * r;   // a ring's inner frames have two rows
                    for (int dy = -r; dy <= r; dy += step) {
                        const int yy = y + dy;
                        const int32_t d = dy * dy + dt * dt;
                        if (yy < 0 || yy >= G.H || d >= best) continue;
                        const int32_t dx = row_near(M + ((int64_t)tt * G.H + yy) * G.ww, G.ww, x);
                        if (dx < QINF) best = min(best, dx + d);
                    }
                }
            }
            // (what was not looked at is at least QRINGS + 1 rings or QNEAR + 1 columns away)
            const int64_t voxel = row * G.W + x;
            if (best <= QSETTLED) {
                if (best <= tau2) ++matched[0 + s];
                atomicAdd(&hist[s][best], 1u);
                int32_t* d2 = s < 2 ? d2_a : d2_b;
                if (d2) d2[voxel] = best;
            } else {
                bool listed = false;
                if ((int64_t)*(volatile unsigned long long*)(acc + QACC_FAR) <= far_cap) {
                    const unsigned long long k = atomicAdd(acc + QACC_FAR, 1ull);
                    listed = (int64_t)k < far_cap;
                    if (listed) far_list[k] = (uint64_t)s << 60 | (uint64_t)voxel;
                }
                if (!listed) leave_to_edt(acc, s);
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int s = 0; s < QSETS; ++s) {
        unsigned long long* as = acc + QACC_SET + s * QSET_WORDS;
        block_flush(matched[s], none[s], 0ull, 0.0, as, QSET_MATCH, QSET_NONE, -1, -1);
        __syncthreads();
        for (int b = threadIdx.x; b <= QSETTLED; b += blockDim.x)
            if (b > 0 && hist[s][b]) atomicAdd(as + QSET_HIST + b, (unsigned long long)hist[s][b]);
    }
}

// One bit per cell, [set][cell row][word]: whether the set has an event in it.  One
// warp per cell row and 32 words; nothing to do when no event is listed.
__global__ void __launch_bounds__(QBLOCK) k_cells(QGrid G, const uint32_t* __restrict__ masks,
                                                  uint32_t* __restrict__ cells, const unsigned long long* acc) {
    if (acc[QACC_FAR] == 0) return;
    const unsigned edt = (unsigned)acc[QACC_EDT];
    const int lane = threadIdx.x & 31;
    const int sw = (G.ww + 31) / 32, cy_n = (G.H + QCELL - 1) / QCELL, ct_n = (G.T + QCELL - 1) / QCELL;
    const int64_t per_set = (int64_t)cy_n * ct_n * sw, n = QSETS * per_set;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n; k += nw) {
        const int64_t set = k / per_set, rest = k - set * per_set, cr = rest / sw;
        if (edt >> set_target((int)set) & 1u) continue;     // (no event looks for this set's any more)
        const int word = (int)(rest - cr * sw) * 32 + lane;
        const int ct = (int)(cr / cy_n), cy = (int)(cr - (int64_t)ct * cy_n);
        uint32_t any = 0;
        if (word < G.ww) {
#pragma unroll
            for (int j = 0; j < QCELL * QCELL; ++j) {
                const int t = ct * QCELL + j / QCELL, y = cy * QCELL + j % QCELL;
                if (t < G.T && y < G.H) any |= __ldg(masks + set * G.n_words + ((int64_t)t * G.H + y) * G.ww + word);
            }
        }
        const uint32_t bits = __ballot_sync(0xffffffffu, any != 0);
        if (lane == 0) cells[k] = bits;
    }
}

// least column distance from x to an occupied cell of a cell row, or QINF
__device__ __forceinline__ int32_t cells_near(const uint32_t* __restrict__ row, int sw, int x) {
    const int c = x >> 5, w0 = c >> 5, b0 = c & 31;
    int32_t d = QINF;
    for (int w = w0; w >= 0; --w) {
        uint32_t m = __ldg(row + w);
        if (w == w0) m &= (uint32_t)((2ull << b0) - 1ull);
        if (m) {
            d = max(0, x - (32 * (32 * w + 31 - __clz(m)) + 31));
            break;
        }
    }
    for (int w = w0; w < sw; ++w) {
        uint32_t m = __ldg(row + w);
        if (w == w0) m &= 0xFFFFFFFFu << b0;
        if (m) {
            d = min(d, max(0, 32 * (32 * w + __ffs(m) - 1) - x));
            break;
        }
    }
    return d;
}

// The listed events, one warp each.  The warp's lanes look at the cell rows of a
// ring around the event (ring r is at least 8 (r - 1) + 1 frames or rows away);
// an occupied cell bounds the distance from above and below, and of those that
// could hold a nearer event the nearest is searched first, its 64 rows two per
// lane.  Bound by the dependent loads of one event after the other and some 4000
// instructions each.  Events differ widely in cost, so the blocks are small and up
// to five times as many as are resident (20 of 64 threads, 48 registers, no
// spills): whole quality calls of 1280x720x100, two videos, 0.79 and 0.71 ms with 8
// blocks of 256 threads per SM, 0.72 and 0.66 ms with 40, 0.69 and 0.62 ms with 100
// blocks of 64, the same with 300 or with a cursor on the device; 0.72 and
// 0.65 ms with 40 registers.  Lane s adds up what its warp found for set s: one
// addition per warp to the set's words instead of one per event.
//
// The transform costs the same wherever the events are, this search the more the
// farther they are.  An event may take 512 steps (a step: 32 cell rows of a ring, or the
// search of one cell row; more where rows are wider than 2048), and all events together
// `budget` beyond their first 64 (most take 10 to 30, the farthest of a video a
// hundred or two).  An event that is not settled then leaves its set to the
// transform, and the set's other events are skipped.  Whole calls / four transforms:
// 80000 events of 1280x720x100 500 rows from the other video's 1.53 / 3.96 ms, opposite ends
// of 64x64x8192 4.35 / 5.46, 250000 events of 16384x16384x1 against one in a corner 13.8 /
// 55.1.  (With 128 steps and no common budget one 1280x720x100 drifting grating in fifteen went
// to the transform for an event of 130 steps, 0.67 -> 2.03 ms.)  A search without the bound or
// the rings' clipping took 258 us of a benchmark call, this one 282; with every ring clipped
// and the budget looked at in every step it took 303.
constexpr int FWARPS = 2;
constexpr int FSTEPS = 448;      // beyond the first 64
__global__ void __launch_bounds__(32 * FWARPS, 20) k_search_far(QGrid G, const uint32_t* __restrict__ masks,
                                                                const uint32_t* __restrict__ cells, int tau2,
                                                                int32_t* __restrict__ d2_a, int32_t* __restrict__ d2_b,
                                                                const uint64_t* __restrict__ far_list, int64_t far_cap,
                                                                int64_t budget, unsigned long long* acc) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t n = min((int64_t)acc[QACC_FAR], far_cap);
    const int sw = (G.ww + 31) / 32, cy_n = (G.H + QCELL - 1) / QCELL, ct_n = (G.T + QCELL - 1) / QCELL;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    unsigned long long closed = 0, matched = 0;      // of the set whose number the lane has
    double sum = 0.0;
    unsigned edt = (unsigned)acc[QACC_EDT];          // sets left to the transform: lane 0's view counts
    for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n; k += nw) {
        const uint64_t id = far_list[k];
        const int s = (int)(id >> 60);
        const unsigned skip = __shfl_sync(full, edt, 0);
        if (lane == 0) edt = (unsigned)*(volatile unsigned long long*)(acc + QACC_EDT);   // for the next event
        if (skip >> s & 1u) continue;
        const int64_t voxel = (int64_t)(id & ((1ull << 60) - 1ull));
        const int64_t row = voxel / G.W;
        const int x = (int)(voxel - row * G.W);
        const int t = (int)(row / G.H), y = (int)(row - (int64_t)t * G.H);
        const uint32_t* M = masks + set_target(s) * G.n_words;
        const uint32_t* C = cells + (int64_t)set_target(s) * cy_n * ct_n * sw;
        const int cy0 = y / QCELL, ct0 = t / QCELL;
        const int r_end = max(max(cy0, cy_n - 1 - cy0), max(ct0, ct_n - 1 - ct0));
        int32_t best = QINF;
        int left = 64, paid = 0;       // steps in hand, and those taken beyond the first 64
        const int cost = 1 + (G.ww >> 6);
        // this lane's cell row, if it has one in the video: bounds first, then the searches
        auto look = [&](bool in, int cy, int ct) {
            int32_t bound = QINF;      // no event of the cell row is nearer,
            int32_t within = QINF;     // and one of them is nearer than this
            if (in) {
                const int dy = max(0, max(cy * QCELL - y, y - (cy * QCELL + QCELL - 1)));
                const int dt = max(0, max(ct * QCELL - t, t - (ct * QCELL + QCELL - 1)));
                const int32_t d = dy * dy + dt * dt;
                if (d < best) {
                    const int32_t dx = cells_near(C + ((int64_t)ct * cy_n + cy) * sw, sw, x);
                    if (dx < QINF) {
                        const int uy = max(abs(cy * QCELL - y), abs(cy * QCELL + QCELL - 1 - y));
                        const int ut = max(abs(ct * QCELL - t), abs(ct * QCELL + QCELL - 1 - t));
                        bound = d + dx * dx;
                        within = uy * uy + ut * ut + (dx + 31) * (dx + 31) + 1;
                    }
                }
            }
            left -= cost;
            best = min(best, __reduce_min_sync(full, within));
            while (true) {
                const int32_t first = __reduce_min_sync(full, bound);
                if (first >= best) break;
                const int src = __ffs(__ballot_sync(full, bound == first)) - 1;
                const int yy = __shfl_sync(full, cy, src) * QCELL + (lane & (QCELL - 1));
                const int tt0 = __shfl_sync(full, ct, src) * QCELL + lane / QCELL;
                if (lane == src) bound = QINF;
                left -= cost;
                int32_t got = best;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const int tt = tt0 + half * (QCELL / 2);
                    const int32_t d = (yy - y) * (yy - y) + (tt - t) * (tt - t);
                    if (yy < G.H && tt < G.T && d < got)
                        got = row_wide(M + ((int64_t)tt * G.H + yy) * G.ww, G.ww, x, got - d) + d;
                }
                best = min(best, __reduce_min_sync(full, got));
            }
        };
        auto ring_is_nearer = [&](int r) {
            const int ring = QCELL * (r - 1) + 1;
            return r == 0 || ring * ring < best;
        };
        // the rings of up to 32 cell rows, one lane each wherever they lie: two full sides
        // of 2r + 1 cell rows, then pairs
        int r = 0;
        for (; r <= min(r_end, 4) && ring_is_nearer(r); ++r) {
            const int side = 2 * r + 1;
            int cy, ct;
            if (lane < 2 * side) {
                ct = ct0 + (lane < side ? -r : r);
                cy = cy0 + (lane < side ? lane : lane - side) - r;
            } else {
                const int p = lane - 2 * side;
                ct = ct0 + (p >> 1) - r + 1;
                cy = cy0 + ((p & 1) ? r : -r);
            }
            look(lane < (r == 0 ? 1 : 8 * r) && cy >= 0 && cy < cy_n && ct >= 0 && ct < ct_n, cy, ct);
        }
        // larger rings: only the cell rows within the video, in the same order
        for (; r <= r_end && paid <= FSTEPS && ring_is_nearer(r); ++r) {
            const int y0 = max(cy0 - r, 0), ny = min(cy0 + r, cy_n - 1) - y0 + 1;
            const int t0 = max(ct0 - r + 1, 0), nt = max(min(ct0 + r - 1, ct_n - 1) - t0 + 1, 0);
            const bool low = cy0 >= r, high = cy0 + r < cy_n;
            const int first_rows = ct0 >= r ? ny : 0;
            const int sides = first_rows + (ct0 + r < ct_n ? ny : 0);
            const int rows = sides + nt * ((int)low + (int)high);
            for (int j0 = 0; j0 < rows; j0 += 32) {
                // (a look takes at most 33 steps, so it is enough to pay here)
                if (left < 0) {
                    const int more = (63 - left) & ~63;
                    left += more;
                    paid += more;
                    int stop = 0;
                    if (lane == 0)
                        stop = (int64_t)atomicAdd(acc + QACC_STEPS, (unsigned long long)more) >= budget ||
                               (*(volatile unsigned long long*)(acc + QACC_EDT) >> s & 1ull) != 0;
                    if (__shfl_sync(full, stop, 0)) paid = FSTEPS + 1;
                    if (paid > FSTEPS) break;
                }
                const int j = j0 + lane;
                int cy, ct;
                if (j < sides) {
                    ct = ct0 + (j < first_rows ? -r : r);
                    cy = y0 + (j < first_rows ? j : j - first_rows);
                } else {
                    const int p = j - sides;
                    const bool both = low && high;
                    ct = t0 + (both ? p >> 1 : p);
                    cy = (both ? (p & 1) != 0 : high) ? cy0 + r : cy0 - r;
                }
                look(j < rows, cy, ct);
            }
        }
        if (paid > FSTEPS) {
            if (lane == 0) leave_to_edt(acc, s);
            continue;
        }
        // (the set's target has events, so one was found)
        if (lane != s) continue;
        ++closed;
        matched += best <= tau2;
        if (best < QHIST) atomicAdd(acc + QACC_SET + s * QSET_WORDS + QSET_HIST + best, 1ull);
        else sum += sqrt((double)best);
        int32_t* d2 = s < 2 ? d2_a : d2_b;
        if (d2) d2[voxel] = best;
    }
    if (closed == 0) return;                         // (lanes from QSETS on, and warps without an event)
    unsigned long long* as = acc + QACC_SET + lane * QSET_WORDS;
    if (matched) atomicAdd(as + QSET_MATCH, matched);
    if (sum != 0.0) atomicAdd(reinterpret_cast<double*>(as + QSET_SUM), sum);
}

// ---------------------------------------------------------------- rows: 1-D distance to the nearest event
// One warp per row; `left` (shared) keeps the column of the nearest event at
// or left of each x between the two sweeps.  The first block also clears what the
// searches left in the set's accumulators.
__global__ void k_edt_rows(const int8_t* __restrict__ v, int W, int64_t rows, int pol, int32_t* __restrict__ out,
                           unsigned long long* acc) {
    extern __shared__ int32_t q_left[];
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < QSET_WORDS; i += blockDim.x) acc[i] = 0;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    int32_t* left = q_left + (size_t)wib * W;
    for (int64_t r = (int64_t)blockIdx.x * wpb + wib; r < rows; r += (int64_t)gridDim.x * wpb) {
        const int8_t* src = v + r * W;
        int32_t* dst = out + r * W;
        int carry = -1;
        for (int x0 = 0; x0 < W; x0 += 32) {
            const int x = x0 + lane;
            int idx = (x < W && src[x] == pol) ? x : -1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, idx, o);
                if (lane >= o) idx = max(idx, y);
            }
            idx = max(idx, carry);
            if (x < W) left[x] = idx;
            carry = __shfl_sync(0xffffffffu, idx, 31);
        }
        carry = INT_MAX;
        for (int x0 = (W - 1) & ~31; x0 >= 0; x0 -= 32) {
            const int x = x0 + lane;
            int idx = (x < W && src[x] == pol) ? x : INT_MAX;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_down_sync(0xffffffffu, idx, o);
                if (lane + o < 32) idx = min(idx, y);
            }
            idx = min(idx, carry);
            if (x < W) {
                const int l = left[x];
                int32_t d = QINF;
                if (l >= 0) d = (x - l) * (x - l);
                if (idx != INT_MAX) d = min(d, (idx - x) * (idx - x));
                dst[x] = d;
            }
            carry = __shfl_sync(0xffffffffu, idx, 0);
        }
    }
}

// ---------------------------------------------------------------- columns: lower envelope of parabolas
constexpr int COL_PREFETCH = 16;

__device__ __forceinline__ int32_t floordiv32(int32_t a, int32_t b) {  // b > 0
    const int32_t q = a / b;
    return (a % b != 0 && a < 0) ? q - 1 : q;
}

// Line `line` = (outer, inner x): elements base + u * step, u = 0..L-1,
// base = outer * outer_stride + x.  The envelope is a stack of sites (site s,
// interval start t, site value f); its top lives in registers, the entries
// below it in global memory, entry (depth k, thread g) at k * G + g for the
// G threads of the launch, packed as (s | t << 16, f).  A thread owns one
// stack and walks lines g, g + G, ...; keeping the stacks out of shared
// memory lets every SM run at full occupancy, which hides the latency of the
// sweeps (stacks in shared memory held a 720-long line pass to 39 threads
// per SM and ran 6.7x slower).  The forward sweep loads 16 elements ahead.
// Every quantity fits in int32: extents <= 16384 keep squared distances
// <= 3 * 16383^2 < 2^30.
__global__ void __launch_bounds__(256) k_edt_cols(const int32_t* __restrict__ in, int32_t* __restrict__ out,
                                                    int64_t n_lines, int W, int64_t outer_stride, int64_t step, int L,
                                                    int2* __restrict__ stack) {
    const int64_t G = (int64_t)gridDim.x * blockDim.x;
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t line = g; line < n_lines; line += G) {
        const int64_t x = line % W, outer = line / W;
        const int32_t* src = in + outer * outer_stride + x;
        int32_t* dst = out + outer * outer_stride + x;
        int depth = 0;
        int32_t top_s = 0, top_t = 0, top_f = 0;
        for (int u0 = 0; u0 < L; u0 += COL_PREFETCH) {
            int32_t buf[COL_PREFETCH];
#pragma unroll
            for (int j = 0; j < COL_PREFETCH; ++j)
                buf[j] = u0 + j < L ? __ldg(src + (int64_t)(u0 + j) * step) : QINF;
#pragma unroll
            for (int j = 0; j < COL_PREFETCH; ++j) {
                const int32_t u = u0 + j, fu = buf[j];
                if (fu >= QINF) continue;
                while (depth > 0) {
                    const int32_t f_site = (top_t - top_s) * (top_t - top_s) + top_f;
                    const int32_t f_new = (top_t - u) * (top_t - u) + fu;
                    if (f_site <= f_new) break;
                    if (--depth > 0) {
                        const int2 e = stack[(int64_t)(depth - 1) * G + g];
                        top_s = e.x & 0xFFFF;
                        top_t = (int32_t)((uint32_t)e.x >> 16);
                        top_f = e.y;
                    }
                }
                if (depth == 0) {
                    depth = 1;
                    top_s = u;
                    top_t = 0;
                    top_f = fu;
                } else {
                    const int32_t w = 1 + floordiv32(u * u - top_s * top_s + fu - top_f, 2 * (u - top_s));
                    if (w < L) {
                        stack[(int64_t)(depth - 1) * G + g] = make_int2(top_s | (top_t << 16), top_f);
                        ++depth;
                        top_s = u;
                        top_t = w;
                        top_f = fu;
                    }
                }
            }
        }
        for (int32_t u = L - 1; u >= 0; --u) {
            int32_t d = QINF;
            if (depth > 0) {
                d = (u - top_s) * (u - top_s) + top_f;
                if (u == top_t && --depth > 0) {
                    const int2 e = stack[(int64_t)(depth - 1) * G + g];
                    top_s = e.x & 0xFFFF;
                    top_t = (int32_t)((uint32_t)e.x >> 16);
                    top_f = e.y;
                }
            }
            dst[(int64_t)u * step] = d;
        }
    }
}

// ---------------------------------------------------------------- matching of one polarity
__device__ __forceinline__ void match_one(int32_t d, int64_t i, int32_t* d2_out, int tau2, uint32_t* hist,
                                          unsigned long long& matched, unsigned long long& none, double& sum) {
    if (d >= QINF) {
        ++none;
        if (d2_out) d2_out[i] = -2;
    } else {
        matched += d <= tau2;
        if (d >= QHIST) sum += sqrt((double)d);
        else if (d > 0) atomicAdd(hist + d, 1u);
        if (d2_out) d2_out[i] = d;
    }
}

// vec: the query video is 4-byte aligned (the distance volume always is), so
// each thread takes 4 voxels per step with one 4-byte and one 16-byte load.
// Distances are tallied per squared value in a shared histogram.
__global__ void __launch_bounds__(QBLOCK) k_match(const int8_t* __restrict__ qv, const int32_t* __restrict__ d2,
                                                  int64_t n, int pol, int tau2, int vec, int32_t* __restrict__ d2_out,
                                                  unsigned long long* acc) {
    __shared__ uint32_t hist[QHIST];
    for (int b = threadIdx.x; b < QHIST; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    unsigned long long matched = 0, none = 0;
    double sum = 0.0;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nth = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if (vec) {
        const int64_t n4 = n >> 2;
        const int32_t* q4 = reinterpret_cast<const int32_t*>(qv);
        const int4* d4 = reinterpret_cast<const int4*>(d2);
        for (int64_t i = tid; i < n4; i += nth) {
            const int32_t qw = __ldg(q4 + i);
            if (qw == 0) continue;      // no event among the 4 voxels
            bool any = false;
#pragma unroll
            for (int k = 0; k < 4; ++k) any |= (int)(int8_t)(qw >> (8 * k)) == pol;
            if (!any) continue;
            const int4 dv = __ldg(d4 + i);
            const int32_t ds[4] = {dv.x, dv.y, dv.z, dv.w};
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((int)(int8_t)(qw >> (8 * k)) == pol)
                    match_one(ds[k], 4 * i + k, d2_out, tau2, hist, matched, none, sum);
        }
        done = n4 << 2;
    }
    for (int64_t i = done + tid; i < n; i += nth)
        if (qv[i] == pol) match_one(__ldg(d2 + i), i, d2_out, tau2, hist, matched, none, sum);
    block_flush(matched, none, 0ull, sum, acc, QSET_MATCH, QSET_NONE, -1, QSET_SUM);   // synchronises the block
    for (int b = threadIdx.x; b < QHIST; b += blockDim.x)
        if (hist[b]) atomicAdd(acc + QSET_HIST + b, (unsigned long long)hist[b]);
}

// Blocks of 256 threads for the column kernel: enough for every line, at
// most 8 per SM, and no more than the stack scratch holds.
int stack_blocks(int64_t n_lines, int L, int sms) {
    const int64_t by_lines = (n_lines + 255) / 256;
    const int64_t by_sms = (int64_t)sms * 8;
    const int64_t by_mem = QUALITY_STACK_BYTES / (8 * (int64_t)L * 256);
    return (int)std::max<int64_t>(1, std::min(by_lines, std::min(by_sms, by_mem)));
}

int grid_of(int64_t work, int per_block, int sms, int per_sm) {
    const int64_t need = (work + per_block - 1) / per_block;
    const int64_t cap = (int64_t)sms * per_sm;
    return (int)(need < 1 ? 1 : (need < cap ? need : cap));
}

}  // namespace

int64_t quality_stack_bytes(int32_t W, int32_t H, int32_t T, int sms) {
    const int64_t lines[2] = {(int64_t)T * W, (int64_t)H * W}, len[2] = {H, T};
    int64_t need = 0;
    for (int ax = 0; ax < 2; ++ax) {
        if (len[ax] < 2) continue;
        const int b = stack_blocks(lines[ax], (int)len[ax], sms);
        need = std::max<int64_t>(need, (int64_t)b * 256 * len[ax] * 8);
    }
    return need;
}

int64_t quality_mask_bytes(int32_t W, int32_t H, int32_t T) {
    return 4ll * QSETS * ((W + 31) / 32) * H * T;
}

int64_t quality_cell_bytes(int32_t W, int32_t H, int32_t T) {
    const int64_t sw = ((W + 31) / 32 + 31) / 32;
    return 4 * QSETS * sw * ((H + QCELL - 1) / QCELL) * ((T + QCELL - 1) / QCELL);
}

// Far events the list holds.  Their search takes 1.3 ms per 80000 events of some
// 100 steps each at 1280x720x100 (all four sets by the transform: 4 to 10 ms) and a
// tenth of that for events a few cells away, so the list may hold this many before the
// transform is the better bet; small videos' events have few cells to look at.
// Unrelated random videos, whole calls with a list of voxels / 1024 + 1024, this one and four
// transforms: 10^-3 events per voxel 1280x720x100 6.11 / 0.70 / 5.81 ms, 203x199x31 0.43 /
// 0.09 / 0.37; 10^-2 8.26 / 8.16 / 7.95 (more than either holds) and 0.64 / 0.12 / 0.57.
int64_t quality_far_cap(int32_t W, int32_t H, int32_t T) { return (int64_t)W * H * T / 512 + 16384; }

cudaError_t launch_quality(const QualityArgs& A, int sms, cudaStream_t st, int* launches) {
    const int64_t n = (int64_t)A.W * A.H * A.T;
    QGrid G{A.W, A.H, A.T, (A.W + 31) / 32, 0};
    G.n_words = (int64_t)G.ww * A.H * A.T;
    cudaError_t e = cudaMemsetAsync(A.acc, 0, QACC_WORDS * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    if (A.d2_a && (e = cudaMemsetAsync(A.d2_a, 0xff, n * sizeof(int32_t), st)) != cudaSuccess) return e;
    if (A.d2_b && (e = cudaMemsetAsync(A.d2_b, 0xff, n * sizeof(int32_t), st)) != cudaSuccess) return e;
    const int64_t far_cap = quality_far_cap(A.W, A.H, A.T);
    k_pack<<<grid_of(G.n_words, QBLOCK, sms, 8), QBLOCK, 0, st>>>(A.a, A.b, A.W, G.ww, G.n_words, n, A.masks, A.acc);
    k_search<<<grid_of(G.n_words, 32 * QWARPS, sms, 32), 32 * QWARPS, 0, st>>>(G, A.masks, A.tau2, A.d2_a, A.d2_b,
                                                                            A.far_list, far_cap, A.acc);
    k_cells<<<sms * 8, QBLOCK, 0, st>>>(G, A.masks, A.cells, A.acc);
    k_search_far<<<grid_of(n / 1024 + 1024, FWARPS, sms, 100), 32 * FWARPS, 0, st>>>(G, A.masks, A.cells, A.tau2, A.d2_a,
                                                                             A.d2_b, A.far_list, far_cap, n / 8 + 65536,
                                                                                       A.acc);
    *launches += 4;
    return cudaGetLastError();
}

cudaError_t launch_quality_edt(const QualityArgs& A, int set, int sms, cudaStream_t st, int* launches) {
    static bool attrs[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attrs[dev]) {
        if ((e = cudaFuncSetAttribute(k_edt_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET)) !=
            cudaSuccess)
            return e;
        if (dev >= 0 && dev < 64) attrs[dev] = true;
    }
    const int64_t W = A.W, H = A.H, T = A.T, n = W * H * T;
    const int dir = set >> 1, pol = (set & 1) ? -1 : 1;
    const int8_t* target = dir ? A.a : A.b;
    const int8_t* query = dir ? A.b : A.a;
    int32_t* d2_out = dir ? A.d2_b : A.d2_a;
    unsigned long long* acc = A.acc + QACC_SET + set * QSET_WORDS;
    // rows: warps per block bounded by the shared budget (W ints per warp)
    const int wpb = (int)std::max<int64_t>(1, std::min<int64_t>(8, SMEM_BUDGET / (4 * W)));
    int32_t* cur = A.vol0;
    int32_t* other = A.vol1;
    k_edt_rows<<<grid_of(H * T, wpb, sms, 16), 32 * wpb, (size_t)wpb * W * 4, st>>>(target, (int)W, H * T, pol, cur,
                                                                                  acc);
    ++*launches;
    // column passes along y, then t
    const int64_t lines[2] = {T * W, H * W}, ostride[2] = {H * W, W}, stp[2] = {W, H * W};
    const int64_t len[2] = {H, T};
    for (int ax = 0; ax < 2; ++ax) {
        if (len[ax] < 2) continue;
        const int L = (int)len[ax];
        const int blocks = stack_blocks(lines[ax], L, sms);
        k_edt_cols<<<blocks, 256, 0, st>>>(cur, other, lines[ax], (int)W, ostride[ax], stp[ax], L,
                                            reinterpret_cast<int2*>(A.stack));
        ++*launches;
        std::swap(cur, other);
    }
    const int qvec = (reinterpret_cast<uintptr_t>(query) & 3) == 0;
    k_match<<<grid_of(n / 4 + 1, QBLOCK, sms, 8), QBLOCK, 0, st>>>(query, cur, n, pol, A.tau2, qvec, d2_out, acc);
    ++*launches;
    return cudaGetLastError();
}

}  // namespace mcev
