// gs_sort.cu -- radix binning: pairs sorted by depth, then their keys by tile; and the scan alone.
//
// A tile's list is its entries in (depth, pair index) order.  The visible pairs are far fewer than
// the keys (one key per touched tile), so the depth digits are sorted on the pairs and only the tile
// digits on the keys, with a stable LSD onesweep radix sort both times.  All launches are
// stream-ordered, without host synchronisation; the numbers of pairs and keys are read from device
// memory:
//   1. k_scan_chunks<true> (gs_bin.cu): key and visible-pair offsets of every 256-pair chunk;
//   2. k_compact     a warp per chunk: tiles_touched becomes its inclusive sums; every visible pair
//                    writes (depth bits, position) and its rectangle in pair order, clears its
//                    backward accumulator and counts its depth digits;
//   3. k_onesweep    four passes over the depth digits of the pairs;
//   4. k_emit_sorted scan of the key counts in depth order with decoupled look-back; as soon as a
//                    partition of pairs has its prefix, the CTA emits its (tile, pair) keys, a
//                    thread per key, and counts the tile digits;
//   5. k_onesweep    ceil(tile bits / 8) passes over the tile digits of the keys (at most 8 bits each,
//                    split evenly);
//   6. k_records     [start, end) of every global tile, the sorted keys and values and every entry's
//                    record copied into list order (so a tile's list is one contiguous block for TMA);
//   7. k_claims      every tile under the claim class of its list length.
// Both sorts are stable and the pairs start in ascending pair index, so entries of equal depth keep
// that order.  Depth is positive (z > near > 0): its float bits order like its value.
// Against one sort of all keys by (tile, depth) (8 + 4 bytes, 4 depth passes over the keys), a
// 64-view floor of 71 M visible pairs and 194 M keys moves a third of the bytes: 13.1 ms (2.2 compaction,
// 5.3 the seven passes, 1.9 emission, 3.5 records) where that sort took 24.7.
#include <algorithm>

#include "gs_scan.cuh"

namespace gs {

constexpr uint32_t kFlagAgg = 1u << 30, kFlagInc = 2u << 30, kVal = (1u << 30) - 1;

// The IPT counts of this thread (consecutive pairs from base).
template <int IPT>
__device__ __forceinline__ void scan_load(const BinArgs &a, long long base, uint32_t (&x)[IPT]) {
    if (base + IPT <= a.P) {
        const uint4 *src = reinterpret_cast<const uint4 *>(a.touched + base);
#pragma unroll
        for (int q = 0; q < IPT / 4; ++q) {
            uint4 u = src[q];
            x[4 * q] = u.x; x[4 * q + 1] = u.y; x[4 * q + 2] = u.z; x[4 * q + 3] = u.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < IPT; ++k) x[k] = (base + k < a.P) ? a.touched[base + k] : 0u;
    }
}

// Inclusive sums y of this thread's counts back into tiles_touched.
template <int IPT>
__device__ __forceinline__ void scan_store(const BinArgs &a, long long base, const uint32_t (&y)[IPT]) {
    if (base + IPT <= a.P) {
        uint4 *dst = reinterpret_cast<uint4 *>(a.touched + base);
#pragma unroll
        for (int q = 0; q < IPT / 4; ++q) dst[q] = make_uint4(y[4 * q], y[4 * q + 1], y[4 * q + 2], y[4 * q + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < IPT; ++k)
            if (base + k < a.P) a.touched[base + k] = y[k];
    }
}

// Scan alone: counts -> inclusive sums in place (pruning and the bounded-wait test).
__global__ void __launch_bounds__(kScanThreads) k_scan(BinArgs a) {
    __shared__ uint32_t s_part;
    __shared__ ScanShared<kScanThreads> sh;
    const long long nparts = (a.P + kScanTile - 1) / kScanTile;
    for (;;) {
        if (threadIdx.x == 0) s_part = claim_part(&a.st->ctr[kCtrScan], nparts);
        __syncthreads();
        const long long part = s_part;
        if (part >= nparts) break;
        const long long base = part * kScanTile + (long long)threadIdx.x * kScanIPT;
        uint32_t x[kScanIPT];
        scan_load<kScanIPT>(a, base, x);
        unsigned long long tsum = 0;
#pragma unroll
        for (int k = 0; k < kScanIPT; ++k) tsum += x[k];
        unsigned long long run = scan_partition<kScanThreads>(a, sh, part, nparts, tsum);
        uint32_t y[kScanIPT];
#pragma unroll
        for (int k = 0; k < kScanIPT; ++k) {
            run += x[k];
            y[k] = sat32(run);
        }
        scan_store<kScanIPT>(a, base, y);
        __syncthreads();
        if (nparts <= (long long)gridDim.x) break;   // every partition was taken by a first claim
    }
}

// ------------------------------------------------------------------------------------------
// 2. visible pairs in pair order
// ------------------------------------------------------------------------------------------
// Persistent CTAs of eight warps, a warp per chunk of 256 pairs in eight rounds of 32 consecutive
// pairs.  A chunk without keys only stores its offset.  The digit histograms of all four depth
// passes are counted per CTA (the upper two digits of a chunk are nearly constant: equal digits of a
// warp are added once).
constexpr int kCpThreads = 256;
__global__ void __launch_bounds__(kCpThreads) k_compact(BinArgs a) {
    __shared__ uint32_t s_hist[4][256];
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < 4 * 256; i += kCpThreads) (&s_hist[0][0])[i] = 0u;
    __syncthreads();
    const unsigned lt = lanemask_lt();
    constexpr int kRounds = kChunk / 32;
    for (long long c = (long long)blockIdx.x * (kCpThreads / 32) + (threadIdx.x >> 5); c < a.chunks;
         c += (long long)gridDim.x * (kCpThreads / 32)) {
        const uint4 b = a.blk[c];
        const int v = blk_view(b.y);
        const ViewEntry ve = a.views[v];
        const long long local = (c - ve.chunk_off) * kChunk, fbase = ve.pair_off + local;
        const int np = (int)min((long long)kChunk, ve.count - local);
        unsigned long long keys = b.w;
        if (blk_visible(b.y) == 0u) {
#pragma unroll
            for (int r = 0; r < kRounds; ++r)
                if (r * 32 + lane < np) a.touched[fbase + r * 32 + lane] = (uint32_t)keys;
            continue;
        }
        uint32_t x[kRounds], sl[kRounds];
#pragma unroll
        for (int r = 0; r < kRounds; ++r) x[r] = r * 32 + lane < np ? a.touched[fbase + r * 32 + lane] : 0u;
#pragma unroll
        for (int r = 0; r < kRounds; ++r) sl[r] = x[r] ? a.slot[fbase + r * 32 + lane] : kNoSlot;
        unsigned long long at = b.z;                    // position among all visible pairs
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            uint32_t incl = x[r];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const long long f = fbase + r * 32 + lane;
            if (r * 32 + lane < np) a.touched[f] = sat32(keys + incl);
            keys += __shfl_sync(0xffffffffu, incl, 31);
            const unsigned vis = __ballot_sync(0xffffffffu, x[r] != 0u);
            const unsigned long long pos = at + (unsigned)__popc(vis & lt);
            at += (unsigned)__popc(vis);
            uint32_t z = 0u;
            bool ok = x[r] != 0u;
            if (ok && (unsigned long long)sl[r] >= (unsigned long long)a.vcap) {   // only after an earlier recorded failure
                record_error(a.st, GS_ERR_DEVICE_FAULT, 7);
                ok = false;
            }
            ok = ok && pos < (unsigned long long)a.cap;    // K exceeds the capacity too (one key or more per pair)
            if (ok) {
                const size_t s3 = 3 * (size_t)sl[r];
                const float4 r0 = a.proj[s3], r1 = a.proj[s3 + 1];
                int x0, x1, y0, y1;
                spec_rect(r0.x, r0.y, r1.w, a.itw, a.ith, (float)a.Tx, (float)a.Ty, x0, x1, y0, y1);
                if ((uint32_t)((x1 - x0) * (y1 - y0)) != x[r]) record_error(a.st, GS_ERR_DEVICE_FAULT, 3);
                z = __float_as_uint(r1.z);
                a.pkey[0][pos] = z;
                a.pval[0][pos] = (uint32_t)pos;
                a.info[pos] = make_uint4((uint32_t)((unsigned long long)v * a.Tx * a.Ty + (unsigned long long)(y0 * a.Tx + x0)),
                                         (uint32_t)max(x1 - x0, 1), x[r], (uint32_t)f);
                const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
                a.g2d[s3] = z4;
                a.g2d[s3 + 1] = z4;
                a.g2d[s3 + 2] = z4;
            }
            const unsigned in = __ballot_sync(0xffffffffu, ok);
            if (ok) {
                atomicAdd(&s_hist[0][z & 255u], 1u);
                atomicAdd(&s_hist[1][(z >> 8) & 255u], 1u);
#pragma unroll
                for (int p = 2; p < 4; ++p) {
                    const uint32_t dg = (z >> (8 * p)) & 255u;
                    const unsigned peers = __match_any_sync(in, dg);
                    if ((peers & lt) == 0u) atomicAdd(&s_hist[p][dg], (uint32_t)__popc(peers));
                }
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 4 * 256; i += kCpThreads) {
        const uint32_t n = (&s_hist[0][0])[i];
        if (n) atomicAdd(a.hist + i, n);
    }
}

// ------------------------------------------------------------------------------------------
// 4. keys in depth order
// ------------------------------------------------------------------------------------------
// A partition of 1024 pairs per CTA of 256 threads: (1) each pair's rectangle, gathered by position;
// (2) the scan of the key counts; (3) a thread per key: consecutive threads write consecutive keys,
// each finding its pair by a binary search over the partition's inclusive sums.
constexpr int kEsThreads = 256, kEsIPT = kEmitPart / kEsThreads;
__global__ void __launch_bounds__(kEsThreads) k_emit_sorted(BinArgs a) {
    __shared__ uint32_t s_inc[kEmitPart], s_g0[kEmitPart], s_wr[kEmitPart], s_f[kEmitPart];
    __shared__ uint32_t s_hist[kMaxTilePasses][256];
    __shared__ uint32_t s_part;
    __shared__ ScanShared<kEsThreads> sh;
    const int tid = threadIdx.x;
    for (int i = tid; i < kMaxTilePasses * 256; i += kEsThreads) (&s_hist[0][0])[i] = 0u;
    const unsigned long long cap = (unsigned long long)a.cap;
    const long long M = (long long)min(a.st->bin_pairs, cap), nparts = (M + kEmitPart - 1) / kEmitPart;
    for (;;) {
        if (tid == 0) s_part = claim_part(&a.st->ctr[kCtrEmitSorted], nparts);
        __syncthreads();
        const long long part = s_part;
        if (part >= nparts) break;
        const long long pbase = part * kEmitPart;
        uint32_t pv[kEsIPT];
#pragma unroll
        for (int j = 0; j < kEsIPT; ++j) {
            const int li = j * kEsThreads + tid;
            pv[j] = pbase + li < M ? a.pval[0][pbase + li] : 0xffffffffu;
        }
#pragma unroll
        for (int j = 0; j < kEsIPT; ++j) {
            const int li = j * kEsThreads + tid;
            const uint4 it = (long long)pv[j] < M ? a.info[pv[j]] : make_uint4(0u, 1u, 0u, 0u);
            s_inc[li] = it.z;
            s_g0[li] = it.x;
            s_wr[li] = it.y;
            s_f[li] = it.w;
        }
        __syncthreads();
        uint32_t x[kEsIPT];
        unsigned long long tsum = 0;
#pragma unroll
        for (int k = 0; k < kEsIPT; ++k) {
            x[k] = s_inc[tid * kEsIPT + k];
            tsum += x[k];
        }
        unsigned long long run = scan_partition<kEsThreads, false>(a, sh, part, nparts, tsum);
        const unsigned long long pstart = sh.prefix;
#pragma unroll
        for (int k = 0; k < kEsIPT; ++k) {
            run += x[k];
            s_inc[tid * kEsIPT + k] = sat32(run - pstart);   // sums of this partition
        }
        __syncthreads();
        const unsigned long long room = pstart < cap ? cap - pstart : 0ull;
        const uint32_t n = (uint32_t)min((unsigned long long)s_inc[kEmitPart - 1], room);
        for (uint32_t m = tid; m < n; m += kEsThreads) {
            uint32_t li = 0;              // the pair: smallest li with inc[li] > m
#pragma unroll
            for (int step = kEmitPart / 2; step > 0; step >>= 1)
                if (s_inc[li + step - 1] <= m) li += step;
            const uint32_t r = m - (li ? s_inc[li - 1] : 0u), w = s_wr[li], row = r / w;
            const uint32_t g = s_g0[li] + row * (uint32_t)a.Tx + (r - row * w);
            a.tkey[0][pstart + m] = g;
            a.tval[0][pstart + m] = s_f[li];
            for (int p = 0; p < a.tile_passes; ++p) atomicAdd(&s_hist[p][(g >> (a.tile_bits * p)) & ((1u << a.tile_bits) - 1u)], 1u);
        }
        __syncthreads();
        if (nparts <= (long long)gridDim.x) break;
    }
    __syncthreads();
    for (int i = tid; i < a.tile_passes * 256; i += kEsThreads) {
        const uint32_t c = (&s_hist[0][0])[i];
        if (c) atomicAdd(a.hist + 4 * 256 + i, c);
    }
}

// ------------------------------------------------------------------------------------------
// 3., 5. onesweep pass
// ------------------------------------------------------------------------------------------
struct SweepArgs {
    const uint32_t *kin, *vin;
    uint32_t *kout, *vout;
    const uint32_t *hist;        // [256] digit counts of this pass over all keys
    const unsigned long long *count;   // number of keys (those beyond cap are not there)
    uint32_t *state;             // [parts][256]
    uint32_t *ctr;
    DevStatus *st;
    long long cap;
    int shift;
    uint32_t mask;               // digit = (key >> shift) & mask, at most 255
    unsigned long long spin_limit;
};

constexpr int kSweepWarps = kSortThreads / 32;
template <int IPT>
constexpr size_t sweep_dyn_smem() { return (size_t)kSortThreads * IPT * 2 * sizeof(uint32_t); }

// Predecessors whose digit words one look-back round loads together.  A partition's keys, values
// and ranks already sit in shared memory when it looks back, so the window costs registers only
// while it is consumed; a window this wide lets a partition of a small sort (tens of partitions,
// all running at once) add up every predecessor's published count in one or two rounds.
constexpr int kLookback = 32;

template <int IPT>
__global__ void __launch_bounds__(kSortThreads) k_onesweep(SweepArgs a) {
    constexpr int kSortIPT = IPT;
    constexpr int kSortTile = kSortThreads * IPT;
    extern __shared__ __align__(16) unsigned char sw_smem[];
    uint32_t *s_keys = reinterpret_cast<uint32_t *>(sw_smem);
    uint32_t *s_vals = s_keys + kSortTile;
    __shared__ uint32_t s_wcnt[kSweepWarps][256];
    __shared__ uint32_t s_tstart[256];
    __shared__ uint32_t s_gbase[256];
    __shared__ uint32_t s_wsum[kSweepWarps];
    __shared__ uint32_t s_part;
    __shared__ int s_bad;
    __shared__ uint32_t s_goff[256];      // exclusive global start of each digit in this pass
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the first partition is claimed while the pass histogram is read and scanned
    if (threadIdx.x == 0) {
        s_part = atomicAdd(a.ctr, 1u);
        s_bad = 0;
    }
#pragma unroll
    for (int w = 0; w < kSweepWarps; ++w) s_wcnt[w][threadIdx.x] = 0;
    {
        // exclusive scan of the pass's 256 digit counts, once per CTA
        const uint32_t c = a.hist[threadIdx.x];
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_wsum[warp] = incl;
        __syncthreads();
        uint32_t off = 0;
        for (int w = 0; w < warp; ++w) off += s_wsum[w];
        s_goff[threadIdx.x] = off + incl - c;
        __syncthreads();
    }
    const unsigned long long Kll = min(*a.count, (unsigned long long)a.cap);
    const uint32_t K = (uint32_t)Kll;
    const uint32_t nparts = (K + kSortTile - 1) / kSortTile;
    const unsigned lt_mask = lanemask_lt();
    {   // the first claim, made before nparts was known, may be the launch's last one (claim_part)
        const long long last =
            (long long)nparts <= (long long)gridDim.x ? (long long)gridDim.x - 1 : (long long)nparts + gridDim.x - 1;
        if (threadIdx.x == 0 && (long long)s_part == last) *a.ctr = 0u;
    }
    for (;;) {
        const uint32_t part = s_part;
        if (part >= nparts) break;
        const uint32_t base = part * kSortTile;
        const uint32_t tile_n = min((uint32_t)kSortTile, K - base);
        const int d = threadIdx.x;            // thread d owns digit d from the digit totals on
        uint32_t total = 0, tstart = 0;
        {
            uint32_t k[kSortIPT];
            uint32_t val[kSortIPT];
            uint32_t rk[kSortIPT];
#pragma unroll
            for (int r = 0; r < kSortIPT; ++r) {
                const uint32_t li = warp * (kSortIPT * 32) + r * 32 + lane;
                const bool valid = li < tile_n;
                k[r] = valid ? a.kin[base + li] : 0u;
                val[r] = valid ? a.vin[base + li] : 0u;
            }
            // stable rank inside the warp: match_any groups equal digits, per-warp digit counters
#pragma unroll
            for (int r = 0; r < kSortIPT; ++r) {
                const uint32_t li = warp * (kSortIPT * 32) + r * 32 + lane;
                const uint32_t dg = li < tile_n ? (k[r] >> a.shift) & a.mask : 256u;
                const unsigned peers = __match_any_sync(0xffffffffu, dg);
                const uint32_t c = dg < 256u ? s_wcnt[warp][dg] : 0u;
                __syncwarp();
                if (dg < 256u && lane == __ffs(peers) - 1) s_wcnt[warp][dg] = c + __popc(peers);
                __syncwarp();
                rk[r] = c + __popc(peers & lt_mask);
            }
            __syncthreads();
#pragma unroll
            for (int w = 0; w < kSweepWarps; ++w) {
                const uint32_t c = s_wcnt[w][d];
                s_wcnt[w][d] = total;
                total += c;
            }
            // publish this partition's digit count before anything else, for the successors
            if ((uint32_t)d <= a.mask) st_relaxed_u32(a.state + (size_t)part * 256 + d, (part == 0 ? kFlagInc : kFlagAgg) | total);
            // exclusive scan of the digit totals inside the partition
            uint32_t incl = total;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) s_wsum[warp] = incl;
            __syncthreads();
            uint32_t woff = 0;
            for (int w = 0; w < warp; ++w) woff += s_wsum[w];
            tstart = woff + incl - total;
            s_tstart[d] = tstart;
            __syncthreads();
            // local scatter: the partition in digit order in shared memory (needs no global offset)
#pragma unroll
            for (int r = 0; r < kSortIPT; ++r) {
                const uint32_t li = warp * (kSortIPT * 32) + r * 32 + lane;
                if (li < tile_n) {
                    const uint32_t dd = (k[r] >> a.shift) & a.mask;
                    const uint32_t lp = s_tstart[dd] + s_wcnt[warp][dd] + rk[r];
                    s_keys[lp] = k[r];
                    s_vals[lp] = val[r];
                }
            }
        }
        // look back over the predecessors' counts of digit d: a window of kLookback words loaded
        // together, consumed nearest first until an inclusive word (done) or a not-yet-published
        // one (wait, then reload from there); every wait is bounded
        uint32_t excl = 0;
        if (part > 0 && (uint32_t)d <= a.mask) {
            int j = (int)part - 1;
            unsigned long long spins = 0;
            bool timed_out = false;
            for (;;) {
                uint32_t w[kLookback];
#pragma unroll
                for (int q = 0; q < kLookback; ++q)
                    w[q] = (j - q >= 0) ? ld_relaxed_u32(a.state + (size_t)(j - q) * 256 + d) : kFlagInc;
                bool found = false, stop = false;
                int adv = 0;
#pragma unroll
                for (int q = 0; q < kLookback; ++q) {
                    if (!stop) {
                        const uint32_t fl = w[q] & ~kVal;
                        if (fl == 0u) {
                            stop = true;
                        } else {
                            excl += w[q] & kVal;
                            ++adv;
                            if (fl == kFlagInc) found = stop = true;
                        }
                    }
                }
                if (found) break;
                j -= adv;
                if (stop) {
                    if (++spins > a.spin_limit) { timed_out = true; break; }
                    __nanosleep(64);
                }
            }
            st_relaxed_u32(a.state + (size_t)part * 256 + d, kFlagInc | ((excl + total) & kVal));
            if (timed_out) {
                s_bad = 1;
                record_error(a.st, GS_ERR_TIMEOUT, 4);
            }
        }
        s_gbase[d] = s_goff[d] + excl - tstart;
        __syncthreads();
        if (!s_bad) {
            for (uint32_t i = threadIdx.x; i < tile_n; i += kSortThreads) {
                const uint32_t key = s_keys[i];
                const uint32_t dd = (key >> a.shift) & a.mask;
                const uint32_t gp = s_gbase[dd] + i;
                if (gp < K) {
                    a.kout[gp] = key;
                    a.vout[gp] = s_vals[i];
                }
            }
        }
        // a grid that covers every partition claimed them all with its first claims: leave without
        // another claim round trip
        if (nparts <= gridDim.x) break;
        __syncthreads();
        // next partition; the per-warp digit counters start from zero again
        if (threadIdx.x == 0) {
            s_part = claim_part(a.ctr, (long long)nparts);
            s_bad = 0;
        }
#pragma unroll
        for (int w = 0; w < kSweepWarps; ++w) s_wcnt[w][threadIdx.x] = 0;
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------------------
// 6. tile ranges and records in list order
// ------------------------------------------------------------------------------------------
// A warp per 32 keys: a lane per key finds the range borders, the pair's slot and the value, then the
// 96 16-byte parts of the 32 records are copied by consecutive lanes (a record's three parts by three
// neighbouring lanes, so every store instruction writes 512 contiguous bytes).  The lists are streamed past the
// L2 (64 B a key written once): it is the records of the view in hand, gathered about three times each, that
// should stay there.  The step of 64 views of 4 M
// Gaussians (194 M keys) goes from 61.3 to 59.3 ms with it; lists that fit the L2 neither gain nor lose.
constexpr int kRecThreads = 256;
__global__ void __launch_bounds__(kRecThreads) k_records(BinArgs a) {
    const unsigned long long K = min(a.st->num_keys, (unsigned long long)a.cap);
    const int lane = threadIdx.x & 31;
    uint64_t *kout = a.keys[a.passes & 1];
    uint32_t *vout = a.vals[a.passes & 1];
    const uint32_t *tk = a.tkey[a.tile_passes & 1], *tv = a.tval[a.tile_passes & 1];
    const unsigned long long stride = (unsigned long long)gridDim.x * kRecThreads;
    for (unsigned long long i0 = (unsigned long long)blockIdx.x * kRecThreads + (threadIdx.x & ~31u); i0 < K; i0 += stride) {
        const unsigned long long i = i0 + lane;
        const uint32_t g = i < K ? tk[i] : 0xffffffffu;
        const uint32_t f = i < K ? tv[i] : 0u;
        uint32_t prev = __shfl_up_sync(0xffffffffu, g, 1), next = __shfl_down_sync(0xffffffffu, g, 1);
        if (lane == 0) prev = i0 > 0 ? tk[i0 - 1] : 0xffffffffu;
        if (lane == 31) next = i + 1 < K ? tk[i + 1] : 0xffffffffu;
        uint32_t sl = kNoSlot;
        if (i < K) {
            if ((long long)g >= a.G || (long long)f >= a.P) {   // only after an earlier recorded failure
                record_error(a.st, GS_ERR_DEVICE_FAULT, 5);
            } else {
                if (g != prev) a.ranges[2 * (size_t)g] = (uint32_t)i;
                if (g != next) a.ranges[2 * (size_t)g + 1] = (uint32_t)(i + 1);
                __stcs(vout + i, f);
                sl = a.slot[f];
                if (sl >= (unsigned long long)a.vcap) {         // only after an earlier recorded failure
                    record_error(a.st, GS_ERR_DEVICE_FAULT, 8);
                    sl = kNoSlot;
                }
            }
        }
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const int q = t * 32 + lane, e = q / 3, part = q - 3 * e;
            const uint32_t se = __shfl_sync(0xffffffffu, sl, e), ge = __shfl_sync(0xffffffffu, g, e);
            if (se != kNoSlot) {
                float4 r = a.proj[3 * (size_t)se + part];
                if (part == 1) {
                    __stcs(reinterpret_cast<unsigned long long *>(kout) + i0 + e, ((unsigned long long)ge << 32) | __float_as_uint(r.z));
                    r.w = __uint_as_float(se);   // the radius (used only by the emission) gives way to the slot
                }
                __stcs(a.srec + 3 * i0 + q, r);
            }
        }
    }
}

// ------------------------------------------------------------------------------------------
// host driver
// ------------------------------------------------------------------------------------------
static int occupancy(const void *fn, int threads, size_t dyn) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, threads, dyn) != cudaSuccess || b < 1) b = 1;
    return b;
}

int run_scan_only(const BinArgs &a, cudaStream_t s) {
    if (cudaMemsetAsync(&a.st->ctr[kCtrScan], 0, sizeof(uint32_t), s) != cudaSuccess) return GS_ERR_CUDA;
    const long long parts = (a.P + kScanTile - 1) / kScanTile;
    if (parts > 0) {
        if (cudaMemsetAsync(a.scan_state, 0, sizeof(unsigned long long) * parts, s) != cudaSuccess) return GS_ERR_CUDA;
        static PerDevice per;
        const int occ = per.get(current_device(), [] { return occupancy((const void *)k_scan, kScanThreads, 0); });
        long long grid = std::min<long long>(parts, (long long)device_sm_count() * occ);
        k_scan<<<(unsigned)grid, kScanThreads, 0, s>>>(a);
        count_launches(1);
    } else {
        // no pairs: K = 0
        if (cudaMemsetAsync(&a.st->num_keys, 0, sizeof(unsigned long long), s) != cudaSuccess) return GS_ERR_CUDA;
    }
    return check_launch();
}

static int sweep(const BinArgs &a, SweepArgs sa, int pass, cudaStream_t s) {
    static PerDevice attr, per;
    const int dev = current_device();
    if (!attr.get(dev, [] {
            return cudaFuncSetAttribute((const void *)k_onesweep<kSortIPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)sweep_dyn_smem<kSortIPT>()) == cudaSuccess;
        }))
        return GS_ERR_CUDA;
    const int occ = per.get(dev, [] { return occupancy((const void *)k_onesweep<kSortIPT>, kSortThreads, sweep_dyn_smem<kSortIPT>()); });
    const long long grid = std::max<long long>(1, std::min<long long>(a.sort_parts, (long long)device_sm_count() * occ));
    sa.hist = a.hist + 256 * pass;
    sa.state = a.sort_state + (size_t)256 * a.sort_parts * pass;
    sa.ctr = &a.st->ctr[kCtrSort0 + pass];
    sa.st = a.st;
    sa.cap = a.cap;
    sa.spin_limit = a.spin_limit;
    k_onesweep<kSortIPT><<<(unsigned)grid, kSortThreads, sweep_dyn_smem<kSortIPT>(), s>>>(sa);
    count_launches(1);
    return GS_OK;
}

int run_onesweep(const BinArgs &a, cudaStream_t s) {
    // look-back words of the scans and of every pass, digit histograms and tile ranges (the claim counters
    // return to zero at the end of every launch and k_scan_chunks clears the claim-class counts)
    if (cudaMemsetAsync(a.clear_begin, 0, a.clear_bytes, s) != cudaSuccess) return GS_ERR_CUDA;
    const long long sms = device_sm_count();
    launch_scan_chunks(a, true, s);
    static PerDevice per_c, per_e;
    const int dev = current_device();
    const int occ_c = per_c.get(dev, [] { return occupancy((const void *)k_compact, kCpThreads, 0); });
    k_compact<<<(unsigned)std::max<long long>(1, std::min<long long>((a.chunks + 7) / 8, sms * occ_c)), kCpThreads, 0, s>>>(a);
    count_launches(1);
    SweepArgs sa;
    sa.count = &a.st->bin_pairs;
    sa.mask = 255u;
    for (int p = 0; p < 4; ++p) {
        sa.kin = a.pkey[p & 1];
        sa.vin = a.pval[p & 1];
        sa.kout = a.pkey[(p + 1) & 1];
        sa.vout = a.pval[(p + 1) & 1];
        sa.shift = 8 * p;
        const int rc = sweep(a, sa, p, s);
        if (rc) return rc;
    }
    BinArgs e = a;
    e.scan_state = a.emit_scan_state;
    const int occ_e = per_e.get(dev, [] { return occupancy((const void *)k_emit_sorted, kEsThreads, 0); });
    const long long parts = std::max<long long>(1, (std::min(a.cap, a.P) + kEmitPart - 1) / kEmitPart);
    k_emit_sorted<<<(unsigned)std::min<long long>(parts, sms * occ_e), kEsThreads, 0, s>>>(e);
    count_launches(1);
    sa.count = &a.st->num_keys;
    sa.mask = (1u << a.tile_bits) - 1u;
    for (int p = 0; p < a.tile_passes; ++p) {
        sa.kin = a.tkey[p & 1];
        sa.vin = a.tval[p & 1];
        sa.kout = a.tkey[(p + 1) & 1];
        sa.vout = a.tval[(p + 1) & 1];
        sa.shift = a.tile_bits * p;
        const int rc = sweep(a, sa, 4 + p, s);
        if (rc) return rc;
    }
    k_records<<<(unsigned)(sms * 8), kRecThreads, 0, s>>>(a);
    count_launches(1);
    launch_claims(a, s);
    return check_launch();
}

}  // namespace gs
