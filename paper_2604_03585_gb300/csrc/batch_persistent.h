// Host interface of the one-launch ragged batch kernel (batch_persistent.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sar {

// One strip as the kernel sees it.  Range lines are raw rows of n_range
// samples; azimuth lines are image rows of n_az samples, transformed at
// length l_az (zero-padded when n_az < l_az).
struct BStrip {
    const float2 *raw;       // [n_az][n_range], read only
    float2 *image;           // [n_range][n_az]
    const float2 *filt_r, *tw_r;   // range class: filter in register order, twiddles
    const float2 *filt_a, *tw_a;   // azimuth class
    int32_t n_range, n_az, l_az;
    int32_t expect;          // range lines that must be done before an azimuth item runs (n_az)
};

// One work item: `nlines` consecutive lines (line0 ...) of one strip, of one
// kind.  Range lines are azimuth rows; azimuth lines are range bins.
struct BItem {
    int32_t kind;            // 0 range, 1 azimuth
    int32_t strip;
    int32_t line0, nlines;
};

constexpr int kBatchThreads = 512;       // one block per SM
constexpr int kLongLines = 4;            // lines of a range item at least: a 32-byte sector of the image row
constexpr int kBatchScratch = 3 * 16384; // samples of one block's scratch
constexpr int kBatchNumLists = 5;        // range items of 512 and of 256 threads, all items of 128, azimuth items of 256, 512

// How the kernel runs lines of one length.
struct BatchGeom {
    const char *schedule;   // name of the compiled schedule of the same geometry; nullptr: length not supported
    int threads;            // of a worker
    int lines;              // that a worker holds at once
    int set;                // lines of a range item that are stored together
    bool parks;             // such a set needs the scratch
};
// whole_block: range items of 2048, 4096 and 8192 samples on all 512 threads.
BatchGeom batch_geometry(int n, bool whole_block = false);

// One launch: the items of list i are items[begin[i]] ... items[begin[i + 1]
// - 1].  done[n_strips] and next[kBatchNumLists] must be zero (the caller
// clears them before every launch); status is set to 5 when a bounded wait
// runs out, and then nobody takes items any more.  scratch: batch_grid() *
// kBatchScratch samples, or nullptr where no range item is longer than the
// lines its worker holds.
struct BatchLists {
    const BItem *items;
    int32_t begin[kBatchNumLists + 1];
    const BStrip *strips;
    int *done, *next, *status;
    long long wait_cycles;
    float2 *scratch;
};
// Blocks of the kernel resident on the whole current device (0 on error).
int batch_grid();
cudaError_t launch_batch_persistent(const BatchLists &lists, cudaStream_t st);
cudaError_t prepare_batch_persistent();

}  // namespace sar
