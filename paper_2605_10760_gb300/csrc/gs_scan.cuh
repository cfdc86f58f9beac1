// gs_scan.cuh -- decoupled look-back scan, partition claims and claim classes, shared by the binning
// kernels.
#pragma once

#include "gs_kernels.cuh"

namespace gs {

constexpr unsigned long long kFlagAgg64 = 1ull << 62, kFlagInc64 = 2ull << 62, kVal64 = (1ull << 62) - 1;

// ------------------------------------------------------------------------------------------
// inclusive scan with decoupled look-back
// ------------------------------------------------------------------------------------------
template <int THREADS>
struct ScanShared {
    unsigned long long wsum[THREADS / 32];
    unsigned long long prefix;
};

// Global exclusive prefix of this thread's first count in partition `part`, given tsum, the sum of
// the thread's counts (threads in order).  Block scan of the per-thread sums; warp 0 publishes the
// partition total, looks back over the predecessors (a warp reads 32 at a time, the nearest
// inclusive word ends it; bounded spins) and publishes the inclusive prefix; the last partition
// writes K and checks the capacity (TOTAL).  sh.prefix holds the partition's prefix on return.
template <int THREADS, bool TOTAL = true>
__device__ unsigned long long scan_partition(const BinArgs &a, ScanShared<THREADS> &sh, long long part,
                                             long long nparts, unsigned long long tsum) {
    static_assert(THREADS / 32 <= 32, "warp 0 scans the warp sums");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long incl = tsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sh.wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        unsigned long long w = lane < THREADS / 32 ? sh.wsum[lane] : 0ull;
        unsigned long long wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < THREADS / 32) sh.wsum[lane] = wi - w;   // exclusive warp offsets
        const unsigned long long total = __shfl_sync(0xffffffffu, wi, THREADS / 32 - 1);
        const bool silent = (part == a.fault_scan_part);
        unsigned long long prefix = 0;
        if (part == 0) {
            if (lane == 0 && !silent) st_relaxed_u64(a.scan_state, kFlagInc64 | total);
        } else {
            if (lane == 0 && !silent) st_relaxed_u64(a.scan_state + part, kFlagAgg64 | total);
            // warp look-back: lane i reads predecessor j - i; the nearest inclusive word ends it
            long long j = part - 1;
            unsigned long long spins = 0;
            bool timed_out = false;
            for (;;) {
                const long long jj = j - lane;
                const unsigned long long w2 = jj >= 0 ? ld_relaxed_u64(a.scan_state + jj) : kFlagInc64;
                const unsigned long long fl = w2 & ~kVal64;
                const unsigned ready = __ballot_sync(0xffffffffu, fl != 0);
                const unsigned inc = __ballot_sync(0xffffffffu, fl == kFlagInc64);
                const int first = inc ? __ffs(inc) - 1 : 32;               // nearest inclusive lane
                const unsigned need = first >= 31 ? 0xffffffffu : ((2u << first) - 1u);
                if ((ready & need) == need) {
                    unsigned long long v = (lane <= first) ? (w2 & kVal64) : 0ull;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    prefix += v;
                    if (inc) break;
                    j -= 32;
                    continue;
                }
                if (++spins > a.spin_limit) { timed_out = true; break; }
                __nanosleep(100);
            }
            if (lane == 0) {
                if (timed_out) record_error(a.st, GS_ERR_TIMEOUT, 1);
                if (!silent) st_relaxed_u64(a.scan_state + part, kFlagInc64 | ((prefix + total) & kVal64));
            }
        }
        if (lane == 0) {
            sh.prefix = prefix;
            if (TOTAL && part == nparts - 1) {
                const unsigned long long K = prefix + total;
                a.st->num_keys = K;
                if (K > (unsigned long long)a.cap) {
                    a.st->required_keys = K;
                    record_error(a.st, GS_ERR_CAPACITY, 2);
                }
            }
        }
    }
    __syncthreads();
    return sh.prefix + sh.wsum[warp] + (incl - tsum);
}

__device__ __forceinline__ uint32_t sat32(unsigned long long x) { return x > 0xffffffffull ? 0xffffffffu : (uint32_t)x; }

// Next partition of a scan or onesweep CTA (thread 0), in claim order.  A CTA whose grid covers
// every partition claims once; otherwise every CTA ends with one claim past the partitions.  The
// launch's last claim returns the counter to zero for the next launch, so the counters need no
// clearing between launches (gs_workspace_init leaves them zero).
__device__ __forceinline__ uint32_t claim_part(uint32_t *ctr, long long nparts) {
    const uint32_t c = atomicAdd(ctr, 1u);
    const long long last = nparts <= (long long)gridDim.x ? (long long)gridDim.x - 1 : nparts + gridDim.x - 1;
    if ((long long)c == last) *ctr = 0u;
    return c;
}

// The persistent compositing kernels claim (view, tile) items from a counter.  Claimed in tile
// order, a long list taken near the end keeps its CTA running after the others have finished;
// claimed longest first, the last items are the short ones.  So every item is appended, once its
// list length is known, to the list of its claim class (half-octave length classes, class 0 the
// longest), and the kernels claim class by class.  The position inside a class is arbitrary: the
// order moves no result, only when each tile is composited.
__device__ __forceinline__ int claim_class(uint32_t n) {
    const int e = 31 - __clz(n | 1u);
    if (e > 15) return 0;
    const int half = e >= 1 ? (int)((n >> (e - 1)) & 1u) : 0;
    return kClaimClasses - 1 - (2 * e + half);
}


}  // namespace gs
