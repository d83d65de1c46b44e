// kernels.h -- host-callable launchers of the renderer's kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "layout.h"

namespace mcev {

enum { MODE_REFERENCE = 0, MODE_DETECT = 1, MODE_MEAN = 2 };
enum { VAR_ONE_TAILED = 0, VAR_TWO_TAILED = 1, VAR_MEAN_ONLY = 2, VAR_UNIFORM = 3 };
enum { SE_PAPER = 0, SE_WELCH = 1 };

struct StatsArgs {
    PixStats cur, ref;
    const float* tcrit;   // critical t per test round r, n = spp_min + r * spp_batch
    int8_t* events;
    int32_t* spp_out;
    float* mean_out;
    float eps, C;
    int32_t spp_r;        // samples per pixel traced this round
    int32_t sub;          // batch size: the round's samples are merged and tested in batches of `sub`
    int64_t k_base;       // samples taken before this round
    int32_t spp_min, spp_batch, spp_max;
    int32_t mode, variant, se_mode;
    int64_t n_total;      // per-pixel array length, checked only by the allocation-free entry point
};

// The paths of one chunk: spp_r samples, from number k_base on, of consecutive
// entries of a pixel queue from j0 on.
struct Chunk {
    const int32_t* queue;
    int64_t j0, k_base;
    int32_t n_paths, spp_r;
};

// State of the device-resident round loop of one call (device memory): the
// round's pixel queue and sizes, the current chunk, and what was done.  The
// control kernel advances it after every chunk; the first traversal launch and
// the statistics kernel read their sizes from it instead of from launch arguments.
struct RoundCtl {
    int32_t* queue[2];        // ping-pong pixel queues; queue[qi] is this round's
    int64_t Q;                // pixels queued this round
    int64_t n_done;           // samples every queued pixel already has (k_base)
    int64_t j0, nj;           // current chunk: first queue entry, pixels
    int64_t per_chunk;        // pixels per chunk this round
    int64_t paths;            // samples traced by finished rounds
    int64_t stats_pix;        // pixel visits of the statistics kernel
    int32_t spp_r, sub;       // samples per pixel this round; batch size of its tests
    int32_t qi, rounds, iters;
    int32_t status;           // RC_OK, RC_TIMEOUT (a bound ran out), RC_CAP (undecided at spp_max)
    unsigned long long t_start;  // %globaltimer (ns) when the loop started
};
enum { RC_OK = 0, RC_TIMEOUT = 1, RC_CAP = 2 };

// Bounds and schedule of a device-resident round loop.
struct RoundPlan {
    int64_t cap;              // wavefront paths per chunk
    int64_t Q0;               // pixels queued in the first round
    int32_t spp_min, spp_batch, spp_max, window_max;
    int32_t max_iters;        // chunks after which the loop gives up (RC_TIMEOUT)
    int32_t uniform;          // 1: no pixel is decided before spp_max (VAR_UNIFORM)
    unsigned long long timeout_ns;  // wall-clock bound of the loop (RC_TIMEOUT)
};

// Batches of `sub` samples that a round after the first traces per undecided
// pixel (q pixels with n_done samples each), merged and tested in order; the
// samples a pixel draws after its decision are traced in vain.  A pixel that
// needed n_done samples will hardly stop at the very next test, so a round may
// add a quarter of what its pixels already have, and in any case as many
// batches as make 2^20 paths (five path lengths of the 152 SMs' resident lanes:
// below that a round costs its launches' latency, not its paths); at most what
// fills the wavefront.  Filling the wavefront always (32M paths) traced 20 % of
// a sphere-field frame's paths and 85 % of a 346x260 frame's in vain.  Frame
// times filling the wavefront / at a half, a quarter, an eighth with 2^18 paths:
// sphere field 211 / 200 / 192 / 191 ms, 346x260 with 12 moving spheres 15.7 /
// 13.0 / 13.8 / 13.8 ms, terrain 773 / 773 / 773 / 784 ms, eight jobs 136 / 132 /
// 132 / 137 ms; at a quarter with 2^17, 2^19, 2^20, 2^21 paths the 346x260 frame
// takes 14.8, 12.9, 12.2, 12.5 ms.
constexpr int64_t ROUND_FILL = (int64_t)1 << 20;
// Uniform sampling (`uniform`) decides at the cap only, traces nothing in vain and
// fills the wavefront: sphere field 346x260 to 1024 samples 57.3 (19 rounds) -> 48.5 ms (5),
// 128x96 to 2048 20.0 -> 15.7, 640x480 to 4096 659 -> 650, terrain 640x360 328 -> 322.
MCEV_HD inline int64_t round_window(int64_t cap, int64_t q, int64_t sub, int64_t n_done, int64_t spp_max,
                                    int64_t window_max, bool uniform) {
    const int64_t left = (spp_max - n_done + sub - 1) / sub;
    const int64_t per_batch = q * sub;
    const int64_t fill = (ROUND_FILL + per_batch - 1) / per_batch;
    int64_t m = n_done / (4 * sub);
    if (m < fill) m = fill;
    if (uniform || m > cap / per_batch) m = cap / per_batch;
    if (m > left) m = left;
    if (m > window_max) m = window_max;
    return m < 1 ? 1 : m;
}

// `jobs`: device job table of a batched render, or nullptr for a single
// context (then the frame / settings / state arguments are used).  `rc`:
// sizes from the device-resident round loop instead of the arguments.
// `wide`: the scenes' BLAS use the compressed 8-wide layout (Node8)
// Traversal kernel variant (the `trav` argument of the launchers): the BLAS
// layout, and whether the frame has two or more moving instances under a
// TLAS (frames with at most one run kernels without the TLAS loop).
enum { TRAV_WIDE = 1, TRAV_TLAS = 2 };

// closest hits of bounce `depth` (ray queue ecur; at depth 0 the camera rays of
// chunk `ch`, or of the round loop's) and, with scur >= 0, the
// shadow rays that shade(scur) left, in one launch
cudaError_t launch_trace(const DevScene& sc, const DevFrame& fr, const DevParams& P, const Wave& w, int ecur, int scur,
                         int depth, const Chunk& ch, int64_t max_n, int32_t* err, int sms, cudaStream_t st,
                         const Job* jobs, int trav, const RoundCtl* rc);
// hits of bounce `depth` (ray queue cur), queueing the rays that go on unless it is the last
cudaError_t launch_shade(const DevScene& sc, const DevFrame& fr, const DevParams& P, const Wave& w, int cur,
                         int depth, bool last, int64_t max_n, int sms, cudaStream_t st, const Job* jobs);
cudaError_t launch_stats(const Wave& w, const StatsArgs& A, const int32_t* queue, int64_t j0, int64_t n_pix,
                         int32_t* next_queue, int sms, cudaStream_t st, const Job* jobs, const RoundCtl* rc = nullptr);
// appends the pixels that launch_stats left undecided to the next round's queue
// (the device-resident loop's control kernel does it itself)
cudaError_t launch_requeue(const Wave& w, const int32_t* queue, int64_t j0, int64_t n_pix, int32_t* next_queue,
                           cudaStream_t st);
// device-resident round loop: start state (and, with W > 0, queue 0 = the pixels of a W x H image)
cudaError_t launch_round_init(RoundCtl* rc, const Wave& w, const RoundPlan& plan, int32_t* q0, int32_t* q1,
                              int W, int H, int sms, cudaStream_t st);
// after a chunk: next chunk or round, or the end of the loop (condition 0)
cudaError_t launch_round_next(RoundCtl* rc, const Wave& w, const RoundPlan& plan, cudaGraphConditionalHandle h,
                              cudaStream_t st);
// out[i] += (float)acc[i] for i < n (the adjoint's FP64 emission accumulator)
cudaError_t launch_add_f64(float* out, const double* acc, int n, cudaStream_t st);
cudaError_t launch_fill_entries(int32_t* q, int W, int H, int job, int sms, cudaStream_t st);
cudaError_t launch_write_samples(const Wave& w, int64_t out0, int64_t n_paths, float* L_out, uint32_t* sig_out,
                                 int sms, cudaStream_t st);
// every pixel of a W x H image, in tiles
cudaError_t launch_pixel_queue(int32_t* q, int W, int H, int sms, cudaStream_t st);

}  // namespace mcev
