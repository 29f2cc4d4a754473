// A ragged batch in one persistent launch.
//
// Every strip of the batch is two sets of line items: range items (k
// consecutive azimuth rows of the raw echo, compressed along range and
// written straight into the corner-turned image) and azimuth items (k
// consecutive range bins of the image, compressed along azimuth in place).
// One block of 512 threads per SM stays resident.  It is one, two or four
// workers, by the length of the lines: 512 threads for 16384 samples, 256 for
// 8192, 128 up to 4096 (several lines at a time below 4096), each on its share
// of the block's shared memory (the padded buffer of one 16384-sample line).
// A worker takes items from a list through an atomic counter and waits for no
// other worker, so that the lines of an SM are out of phase with one another
// and one loads while another computes, as in the one-length kernels with
// four blocks per SM.  Bound by latency (one block, sixteen warps per SM:
// issue 38 %, L1 55 %).  16 strips of 1024 ... 16384 x 337 ... 4054 samples
// (148 M): 2.71 ms, against 3.07 with items of the whole block throughout and
// every exchange and table access through generic pointers; 1024 x 256 strips
// 150 us per 2^24 samples against 283, 4096 x 256 177 against 255, 16384 x 256
// 234 against 327.
//
// Corner turn: a range item is at least four consecutive azimuth rows.  Where
// a worker holds fewer lines at once, it compresses them one after the other
// and parks all but the last, in natural order, in its own scratch (384 KiB
// per block, 58 MB over the GPU: it stays in L2).  Then it stores each range
// bin's samples of all the rows as one run of at least 32 bytes of the image
// row: the separate transpose and its 16 bytes per sample of HBM traffic
// disappear, without clusters and without a barrier among the workers.
//
// A batch of few range lines of 2048 samples or more has them in items of the
// whole block instead (all the lines it holds at once, none parked): fewer
// steps one after the other (batch.cu).
//
// Phases: the lists are walked one after the other, range items of workers of
// 512, 256 and 128 threads, then azimuth items of 128, 256 and 512; only
// between two of them does the whole block meet.
//
// Dependencies: an azimuth item of strip s reads whole image rows, which
// every range item of s writes into.  Range items count their finished lines
// in done[s] (all stores of the worker, its barrier, a device-scope fence,
// then the atomic add); an azimuth item's first thread waits, with an
// acquire load, until done[s] reaches the strip's n_az, and the threads read
// the rows through L2 only (ld.global.cg).  A block comes to the azimuth items
// only once every range item has been taken by a resident block, so an item
// only ever waits for items that are being computed, and the wait ends.  It is
// bounded all the same: after `wait_cycles` SM clocks the thread sets *status
// to 5 (timeout), and nobody takes items any more once *status is set.  No
// block waits for another one to start.
#include "batch_persistent.h"
#include "line_engine.cuh"
#include "streamed.cuh"

namespace sar {

namespace {

// the line engines of the batch kernel: E = 32 (E = 16 at n = 256) samples
// per thread, the default geometry of every length
using B256 = Sched<256, 16, 16, 16>;
using B512 = Sched<512, 32, 16, 32>;
using B1024 = Sched<1024, 32, 32, 32>;
using B2048 = Sched<2048, 32, 16, 8, 16>;
using B4096 = Sched<4096, 32, 16, 16, 16>;
using B8192 = Sched<8192, 32, 16, 32, 16>;
using B16384 = Sched<16384, 32, 16, 32, 32>;

// A worker: WT threads holding K lines at once, and the stride of their
// shared-memory buffers, one line's padded exchange layout plus a shift of
// 16/k bank pairs (1 for k >= 16), so that the transposed store's reads of k
// lines at one range bin (k lanes of a half-warp) hit distinct bank pairs.  A
// uniform shift of a line's buffer leaves the passes' own access patterns
// conflict-free.
template <class SC, int WT_ = (SC::T > 128 ? SC::T : 128)>
struct BGeo {
    static constexpr int WT = WT_;
    static constexpr int K = WT / SC::T;
    static_assert(K * SC::T == WT && kBatchThreads % WT == 0, "lines fill a worker, workers the block");
    static constexpr int SHIFT = K >= 16 ? 1 : 16 / K;
    static constexpr int BS = SC::SMEM_ELEMS + (K > 1 ? SHIFT : 0);
    static constexpr int W = K < kLongLines ? kLongLines : K;   // lines of one set of a range item
    static constexpr int PARKED = (W - K) * SC::N;              // samples of a set in the scratch
    static_assert(PARKED * (kBatchThreads / WT) <= kBatchScratch, "the workers' scratch fits the block's");
};
constexpr int kSmemElems = 4 * BGeo<B2048>::K * BGeo<B2048>::BS;   // per block (the largest need); a worker has its share
template <class G>
constexpr bool worker_fits() {
    return G::K * G::BS * (kBatchThreads / G::WT) <= kSmemElems;
}
static_assert(worker_fits<BGeo<B256>>() && worker_fits<BGeo<B512>>() && worker_fits<BGeo<B1024>>() &&
                  worker_fits<BGeo<B2048>>() && worker_fits<BGeo<B4096>>() && worker_fits<BGeo<B8192>>() &&
                  worker_fits<BGeo<B16384>>() && worker_fits<BGeo<B2048, 512>>() && worker_fits<BGeo<B4096, 512>>() &&
                  worker_fits<BGeo<B8192, 512>>(),
              "a worker's lines fit its share of the shared memory");

// The item that a worker is at, and its strip, in shared memory: read where
// they are needed.  Held in registers, or in local memory behind the calls,
// they cost the engines spills.
struct BWork {
    BItem it;
    BStrip st;
};
constexpr int kWorkElems = (int)(sizeof(BWork) + 7) / 8;   // of float2
constexpr int kSmem = (kSmemElems + 4 * kWorkElems) * (int)sizeof(float2);

// The block's shared memory: the workers' line buffers, then their BWork.  The
// item routines, which are calls, find it by this name and not through a
// pointer argument, and say which pointers are global ones: behind a generic
// pointer every exchange and table access is a generic load, which waits like
// a global one (16 strips of 256 lines of 4096: 193 us against 231, 3 of 4096 x
// 4096 715 against 858).
extern __shared__ __align__(16) float2 batch_smem[];
__device__ __forceinline__ BWork& work_of(int w) {
    return reinterpret_cast<BWork*>(batch_smem + kSmemElems)[w];
}
template <class T>
__device__ __forceinline__ T* global_ptr(T* p) {
    __builtin_assume(__isGlobal(p));
    return p;
}

// Barriers.  The lines of a block synchronise on ids 1 ... 8: up to two lines
// of 64 threads or more per worker, which may be at another length than its
// neighbours, so worker w of four has ids 1 + 2 w and 2 + 2 w.  Workers: id 0
// for the whole block, 5 and 6 for halves (whose lines have 1 and 2 and the
// staggered starts 9 ... 15), 9 ... 12 for quarters.
template <int WT>
__device__ __forceinline__ void worker_sync(int w) {
    if constexpr (WT == kBatchThreads)
        __syncthreads();
    else
        asm volatile("bar.sync %0, %1;" ::"r"((WT == 256 ? 5 : 9) + w), "r"(WT) : "memory");
}
// the engine's line index (its barrier id less 1) of line `lib` of the block
template <class SC>
__device__ __forceinline__ int line_barrier(int lib) {
    return SC::T == 128 ? 2 * lib : lib;
}
// lines per block as the engines count them (1: the line is the whole block)
template <class SC>
__host__ __device__ constexpr int block_lines() { return kBatchThreads / SC::T; }

// Inverse pass 1 of group-streamed line `lib`: shared memory -> conjugate
// twiddles -> inverse DFT; emit(lo, x) receives natural-order samples
// lo + r*S1.
template <class SC, int LPB, class Emit>
__device__ __forceinline__ void b_inverse_pass1(const float2* sm, const float2* tw, int t, int lib, Emit&& emit) {
    constexpr int R1 = SC::R1, G1 = SC::E / R1;
#pragma unroll 1
    for (int s = 0; s < G1; ++s) {
        float2 x[R1];
        streamed_final_group<SC, LPB>(sm, tw, t, lib, s, x);
        emit(t + SC::T * s, x);
    }
}

// Range item: lines line0 .. line0 + nlines - 1 (azimuth rows) of the strip,
// compressed along range and stored transposed into the image, in sets of W
// lines, each set in rounds of the K lines that the worker holds.  Stored by
// themselves the 1 or 2 lines would write 8 or 16 bytes of every 32-byte
// sector (8192 range samples: 230 us for 2^24 samples, 16384: 250, where the
// line passes alone take 78 and 103).  scratch == nullptr (no memory for it)
// or a batch of few lines: items of at most K lines, one round.
// The item routines are calls: inlined into one kernel the fourteen of them
// spill 3.5 KiB a thread under the block's 128 registers, though each alone
// spills nothing up to 4096 samples.  A call saves about 40 registers, so an
// item is a few rounds.
template <class SC, class G = BGeo<SC>>
__device__ __noinline__ void range_item(float2* scratch) {
    constexpr int R1 = SC::R1, S1 = SC::S1, LPB = block_lines<SC>();
    const int tid = threadIdx.x % G::WT, lib = tid / SC::T, t = tid % SC::T;
    const int bar = line_barrier<SC>(threadIdx.x / SC::T);
    const int w = threadIdx.x / G::WT;
    const BWork& wk = work_of(w);
    float2* smem = batch_smem + w * (kSmemElems / (kBatchThreads / G::WT));
    float2* sm = smem + lib * G::BS;
    scratch = global_ptr(scratch);
    const float2 *filt = global_ptr(wk.st.filt_r), *tw = global_ptr(wk.st.tw_r);
    const float2* raw = global_ptr(wk.st.raw) + (int64_t)wk.it.line0 * SC::N;
    for (int base = 0; base < wk.it.nlines; base += G::K) {   // one round: lines base ... base + K - 1
        const int set = base - base % G::W, end = min(set + G::W, wk.it.nlines), l = base + lib;
        const bool last = base + G::K >= end;                 // round of the set
        if (l < end) {
            streamed_until_last<SC, LPB, true>(raw + (int64_t)l * SC::N, sm, filt, tw, t, bar);
            if (last) {
                // natural-order results back into the slots they were read from
                b_inverse_pass1<SC, LPB>(sm, tw, t, bar, [&](int lo, const float2 (&x)[R1]) {
#pragma unroll
                    for (int r = 0; r < R1; ++r) sm[smem_pos(lo + r * S1, SC::PADSH)] = x[r];
                });
            } else {
                float2* park = scratch + (int64_t)(l - set) * SC::N;
                b_inverse_pass1<SC, LPB>(sm, tw, t, bar, [&](int lo, const float2 (&x)[R1]) {
#pragma unroll
                    for (int r = 0; r < R1; ++r) __stcg(park + lo + r * S1, x[r]);
                });
            }
        }
        if (!last) continue;
        worker_sync<G::WT>(w);
        // range bin n of the set's lines -> image[n][line0 + set ...]: a
        // thread takes one line q of the set, parked or in shared memory, and
        // every (WT / W)-th bin, UN loads in flight
        constexpr int UN = 8, STEP = G::WT / G::W;
        static_assert(SC::N % (STEP * UN) == 0, "whole batches of bins");
        const int q = tid % G::W, n0 = tid / G::W, parked = base - set;
        const int64_t n_az = wk.st.n_az;
        float2* dst = global_ptr(wk.st.image) + n0 * n_az + wk.it.line0 + set + q;
        const float2* pq = scratch + (int64_t)q * SC::N;
        const float2* sq = smem + (q - parked) * G::BS;
        if (set + q < end) {
#pragma unroll 1
            for (int n = n0; n < SC::N; n += STEP * UN) {
                float2 v[UN];
                if (G::PARKED > 0 && q < parked) {
#pragma unroll
                    for (int j = 0; j < UN; ++j) v[j] = __ldcg(pq + n + STEP * j);
                } else {
#pragma unroll
                    for (int j = 0; j < UN; ++j) v[j] = sq[smem_pos(n + STEP * j, SC::PADSH)];
                }
#pragma unroll
                for (int j = 0; j < UN; ++j) __stcs(dst + (n - n0 + STEP * j) * n_az, v[j]);
            }
        }
        worker_sync<G::WT>(w);   // the next set overwrites the buffers and the scratch
    }
}

// Azimuth item: range bins line0 .. line0 + nlines - 1 of the image,
// compressed along azimuth in place (transform length l_az, the n_az stored
// samples zero-padded).  Each of the worker's line groups takes every K-th
// line and waits for no other group.  8192 and 16384 samples run without the
// staggered starts, which delay the loads behind the calls' spills: 6000 lines
// of 1024 range samples 116.9 us against 129.9, 9000 x 4096 782 against 864.
template <class SC>
__device__ __noinline__ void az_item() {
    using G = BGeo<SC>;
    constexpr int R1 = SC::R1, S1 = SC::S1, LPB = block_lines<SC>();
    const int tid = threadIdx.x % G::WT, lib = tid / SC::T, t = tid % SC::T;
    const int bar = line_barrier<SC>(threadIdx.x / SC::T);
    const int w = threadIdx.x / G::WT;
    const BWork& wk = work_of(w);
    float2* sm = batch_smem + w * (kSmemElems / (kBatchThreads / G::WT)) + lib * G::BS;
    const float2 *filt = global_ptr(wk.st.filt_a), *tw = global_ptr(wk.st.tw_a);
    const int64_t n_az = wk.st.n_az;
    float2* image = global_ptr(wk.st.image) + (int64_t)wk.it.line0 * n_az;
    for (int l = lib; l < wk.it.nlines; l += G::K) {
        float2* row = image + l * n_az;
        // the inverse pass 1 below reads and the next line's pass 1 writes a
        // thread's own slots only: no barrier between two lines of a group
        streamed_until_last<SC, LPB, true, true, true>(row, sm, filt, tw, t, bar, (int)n_az);
        b_inverse_pass1<SC, LPB>(sm, tw, t, bar, [&](int lo, const float2 (&x)[R1]) {
#pragma unroll
            for (int r = 0; r < R1; ++r) {
                const int i = lo + r * S1;
                if (i < (int)n_az) __stcs(row + i, x[r]);
            }
        });
    }
}

// Bounded wait of one thread for *ctr >= expect (acquire); false when the
// bound ran out or another block recorded a failure.
__device__ __forceinline__ bool wait_count(const int* ctr, int expect, const int* status, long long wait_cycles) {
    const long long t0 = clock64();
    for (;;) {
        int v;
        asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
        if (v >= expect) return true;
        if (*(volatile const int*)status != 0) return false;
        if (clock64() - t0 > wait_cycles) return false;
        __nanosleep(200);
    }
}

// Asks L2 for the image rows of an azimuth item (whole 16-byte units inside
// them: the instruction needs an aligned address and size).  For lines of 8192
// and 16384, one or two per SM with nothing else to hide their loads: 12000 x
// 4096, larger than L2, 954 us against 995, 6000 x 8192 1003 against 1029.
// Range items and short azimuth lines gain nothing or lose.
__device__ __forceinline__ void prefetch_rows(const BItem& it, const BStrip& st) {
    const uintptr_t p = (uintptr_t)(st.image + (int64_t)it.line0 * st.n_az);
    const uintptr_t e = (p + (uintptr_t)it.nlines * st.n_az * 8) & ~(uintptr_t)15;
    for (uintptr_t q = (p + 15) & ~(uintptr_t)15; q < e; q += 65536) {
        const uint32_t n = (uint32_t)((e - q) < 65536 ? (e - q) : 65536);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(q), "r"(n) : "memory");
    }
}

// One thread takes the next item of a list (*next counts them) into wk and,
// for an azimuth item, waits for its strip's range lines.  it.strip is -1
// where the list is empty or a wait ran out.  ahead > 0 (azimuth lists): the
// rows of the item that many further, about the worker's next, are asked for.
__device__ __forceinline__ void take_item(BWork& wk, const BItem* items, int n_items, const BStrip* strips,
                                          const int* done, int* next, int* status, long long wait_cycles, int ahead) {
    // three trips to L2: what does not depend on one another is in flight together
    const int i = atomicAdd(next, 1), failed = *(volatile int*)status;
    wk.it.strip = -1;
    if (i >= n_items || failed) return;
    const BItem it = items[i];
    if (ahead > 0 && i < n_items - ahead) {
        const BItem later = items[i + ahead];
        prefetch_rows(later, strips[later.strip]);
    }
    int seen = 0;
    if (it.kind == 1)
        asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(seen) : "l"(done + it.strip) : "memory");
    wk.st = strips[it.strip];
    if (it.kind == 1 && seen < wk.st.expect &&
        !wait_count(done + it.strip, wk.st.expect, status, wait_cycles)) {
        atomicMax(status, 5);
        return;
    }
    wk.it = it;
}

// One list, walked by workers of WT threads until it is empty.
template <int WT, bool PREFETCH = false>
__device__ __forceinline__ void walk_list(const BatchLists& a, int list, float2* scratch) {
    const int w = threadIdx.x / WT;
    constexpr int SHARE = kBatchThreads / WT;
    BWork& wk = work_of(w);
    if (scratch) scratch += w * (kBatchScratch / SHARE);
    const BItem* items = a.items + a.begin[list];
    const int n_items = a.begin[list + 1] - a.begin[list];
    if (n_items == 0) return;
    for (;;) {
        if (threadIdx.x % WT == 0)
            take_item(wk, items, n_items, a.strips, a.done, a.next + list, a.status, a.wait_cycles,
                      PREFETCH ? (int)gridDim.x * SHARE : 0);
        worker_sync<WT>(w);
        if (wk.it.strip < 0) break;
        if (wk.it.kind == 0) {
            if constexpr (WT == 512) {
                switch (wk.st.n_range) {
                    case 2048: range_item<B2048, BGeo<B2048, 512>>(scratch); break;
                    case 4096: range_item<B4096, BGeo<B4096, 512>>(scratch); break;
                    case 8192: range_item<B8192, BGeo<B8192, 512>>(scratch); break;
                    default: range_item<B16384>(scratch); break;
                }
            }
            if constexpr (WT == 256) range_item<B8192>(scratch);
            if constexpr (WT == 128) {
                switch (wk.st.n_range) {
                    case 256: range_item<B256>(scratch); break;
                    case 512: range_item<B512>(scratch); break;
                    case 1024: range_item<B1024>(scratch); break;
                    case 2048: range_item<B2048>(scratch); break;
                    default: range_item<B4096>(scratch); break;
                }
            }
            // every store of the item was issued before its last barrier
            if (threadIdx.x % WT == 0) {
                __threadfence();
                atomicAdd(a.done + wk.it.strip, wk.it.nlines);
            }
        } else {
            if constexpr (WT == 512) az_item<Unstaggered<B16384>>();
            if constexpr (WT == 256) az_item<Unstaggered<B8192>>();
            if constexpr (WT == 128) {
                switch (wk.st.l_az) {
                    case 256: az_item<B256>(); break;
                    case 512: az_item<B512>(); break;
                    case 1024: az_item<B1024>(); break;
                    case 2048: az_item<B2048>(); break;
                    default: az_item<B4096>(); break;
                }
            }
        }
        worker_sync<WT>(w);   // the next item overwrites wk and the shared memory, maybe in another length's layout
    }
    __syncthreads();   // the next list's workers share these workers' memory
}

__global__ void __launch_bounds__(kBatchThreads, 1) batch_persistent_kernel(const __grid_constant__ BatchLists a) {
    float2* scratch = a.scratch ? a.scratch + (int64_t)blockIdx.x * kBatchScratch : nullptr;
    walk_list<512>(a, 0, scratch);
    walk_list<256>(a, 1, scratch);
    walk_list<128>(a, 2, scratch);   // range items, then azimuth items
    walk_list<256, true>(a, 3, scratch);
    walk_list<512, true>(a, 4, scratch);
}

}  // namespace

template <class G>
constexpr BatchGeom geom_of(const char *schedule) {
    return BatchGeom{schedule, G::WT, G::K, G::W, G::PARKED > 0};
}

// The schedules named are those whose geometry the engines have: twiddle
// tables and filter order are built from them.
BatchGeom batch_geometry(int n, bool whole_block) {
    switch (n) {
        case 256: return geom_of<BGeo<B256>>("n256_e16_r16x16_l8");
        case 512: return geom_of<BGeo<B512>>("n512_e32_r16x32_l8");
        case 1024: return geom_of<BGeo<B1024>>("n1024_e32_r32x32_l4");
        case 2048:
            return whole_block ? geom_of<BGeo<B2048, 512>>("n2048_e32_r16x8x16_sr2")
                               : geom_of<BGeo<B2048>>("n2048_e32_r16x8x16_sr2");
        case 4096:
            return whole_block ? geom_of<BGeo<B4096, 512>>("n4096_e32_r16x16x16_sr1")
                               : geom_of<BGeo<B4096>>("n4096_e32_r16x16x16_sr1");
        case 8192:
            return whole_block ? geom_of<BGeo<B8192, 512>>("n8192_e32_r16x32x16_sr1")
                               : geom_of<BGeo<B8192>>("n8192_e32_r16x32x16_sr1");
        case 16384: return geom_of<BGeo<B16384>>("n16384_e32_r16x32x32_sr1");
        default: return BatchGeom{nullptr, 0, 0, 0, false};
    }
}

cudaError_t prepare_batch_persistent() {
    return cudaFuncSetAttribute(batch_persistent_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
}

int batch_grid() {
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (!cached[dev]) {
        int per_sm = 0, sms = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_persistent_kernel, kBatchThreads, kSmem) !=
                cudaSuccess ||
            per_sm < 1) {
            cudaGetLastError();
            return 0;
        }
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cached[dev] = per_sm * sms;
    }
    return cached[dev];
}

cudaError_t launch_batch_persistent(const BatchLists &lists, cudaStream_t st) {
    const int grid = batch_grid();
    if (grid <= 0) return cudaErrorInvalidConfiguration;
    batch_persistent_kernel<<<(unsigned)grid, kBatchThreads, kSmem, st>>>(lists);
    return cudaGetLastError();
}

}  // namespace sar
