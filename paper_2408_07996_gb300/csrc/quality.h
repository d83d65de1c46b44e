// quality.h -- launchers of the event-video quality kernels (Sec. 4.2 metrics).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mcev {

// Squared distances below QHIST are counted per value (the host sums
// count * sqrt(d^2)); only the rare longer ones take a double square root on
// the device, whose FP64 rate is low.
constexpr int QHIST = 1024;

// One query set: the events of one polarity of one video, matched against the
// other video's events of that polarity.  Set 2 * dir + (polarity < 0), dir 0:
// events of a against b, dir 1: events of b against a.
constexpr int QSETS = 4;

// accumulator slots (unsigned 64-bit words; the distance sums are doubles)
enum {
    QACC_SQ = 0,        // sum over voxels of (a - b)^2
    QACC_BAD = 1,       // nonzero if a value outside {-1, 0, 1} was seen
    QACC_COUNT = 2,     // events per set's query: a+, a-, b+, b-
    QACC_FAR = 6,       // events listed for the far search
    QACC_EDT = 7,       // bit s: set s is left to the exact transform
    QACC_STEPS = 8,     // steps of the far search beyond the first 64 of an event
    QACC_SET = 9,       // per set: QSET_WORDS
    QSET_MATCH = 0,     // events within sqrt(tau2)
    QSET_NONE = 1,      // events whose polarity the other video lacks
    QSET_SUM = 2,       // double: sum of the distances with d^2 >= QHIST
    QSET_HIST = 3,      // counts per squared distance 1..QHIST-1 (index = d^2)
    QSET_WORDS = 3 + QHIST,
    QACC_WORDS = QACC_SET + QSETS * QSET_WORDS
};

struct QualityArgs {
    const int8_t* a;
    const int8_t* b;
    int32_t W, H, T;
    int32_t tau2;
    int32_t* d2_a;               // optional per-voxel squared distances of a's events (else NULL)
    int32_t* d2_b;
    uint32_t* masks;             // quality_mask_bytes() of scratch: events as bits, a+, a-, b+, b-
    uint32_t* cells;             // quality_cell_bytes() of scratch: occupied cells of the masks
    uint64_t* far_list;          // quality_far_cap() entries: events whose nearest is not in the window
    unsigned long long* acc;     // QACC_WORDS words
    // exact transform of the sets in QACC_EDT (launch_quality_edt)
    int32_t* vol0;               // scratch volumes, W*H*T int32 each
    int32_t* vol1;
    void* stack;                 // quality_stack_bytes() of scratch for long-line envelopes
};

int64_t quality_mask_bytes(int32_t W, int32_t H, int32_t T);
int64_t quality_cell_bytes(int32_t W, int32_t H, int32_t T);
int64_t quality_far_cap(int32_t W, int32_t H, int32_t T);

// Upper bound on the envelope-stack scratch of long column passes (enough
// for every resident thread at lines of up to ~1000; longer lines run fewer
// threads).
constexpr int64_t QUALITY_STACK_BYTES = (int64_t)1 << 31;

// Stack scratch one exact transform of a W x H x T video needs.
int64_t quality_stack_bytes(int32_t W, int32_t H, int32_t T, int sms);

// Largest extent per axis: keeps every squared lattice distance below 2^30.
constexpr int32_t QUALITY_MAX_EXTENT = 16384;

// Frame error, event bits and the searches, enqueued on `st`; returns the
// first launch error.  `launches` is increased by the number of kernels.
cudaError_t launch_quality(const QualityArgs& A, int sms, cudaStream_t st, int* launches);

// Clears set `set`'s accumulators and matches it by an exact distance
// transform (the distances may be any).
cudaError_t launch_quality_edt(const QualityArgs& A, int set, int sms, cudaStream_t st, int* launches);

}  // namespace mcev
