// gs_bin.cu -- tile-first binning: every key dropped into its tile's slice, then every slice sorted.
//
// A tile's list is its entries ordered by (depth bits, pair index).  Instead of sorting all K keys
// by (tile, depth) digit by digit, the keys are counted per tile, scattered into per-tile slices in
// arbitrary order and each slice is sorted on chip by the 64-bit word (depth bits << 32 | pair
// index); the pair index makes the words of a tile distinct, so the result is exactly the stable
// global order.  Five launches, each stream-ordered, K read from device memory:
//   1. k_scan_chunks  the projection left every 256-pair chunk's key count in its block record; their
//                     exclusive prefix sums give each chunk its key offset (and K);
//   2. k_emit_tiles   one CTA per chunk: the pairs' tile rectangles, the chunk's inclusive key sums,
//                     then a thread per key takes the key's rank inside its tile by one atomic on
//                     the tile's counter and writes (tile, rank, depth bits, pair index);
//   3. k_tile_scan    prefix sums of the G tile counts: the tile ranges and the claim classes;
//   4. k_scatter      each key's word to the slice start plus its rank;
//   5. k_tile_sort    every slice sorted, the keys, values and records written in list order.
// Memory per key: 16 B written and read once (the records' own buffer, free until step 5), 8 B
// written and read once, and the 60 B of outputs, against 24 B per key and radix pass of a global sort.
// Small problems are bound by the chain of dependent loads of five launches (a 500k-Gaussian view, 256k
// keys: 4.4, 9.3, 6.9, 5.1 and 16.5 us), large ones by the sort's instructions.
#include <algorithm>

#include "gs_scan.cuh"

namespace gs {

// ------------------------------------------------------------------------------------------
// 1. key offset of every chunk
// ------------------------------------------------------------------------------------------
constexpr int kCsThreads = 1024, kCsIPT = 4;
static_assert(kCsThreads * kCsIPT == kScanTile, "the layout sizes the look-back words by kScanTile");

// blk[c].z = keys of chunk c -> blk[c].w = keys of the chunks before it (saturated at 2^32 - 1, far
// above any capacity).  PAIRS: blk[c].z then becomes the visible pairs before it.  Otherwise a chunk with more than
// a.emit_keys keys also lists its further portions of that many keys as extra work items of k_emit_tiles (those that
// start below the capacity).
template <bool PAIRS>
__global__ void __launch_bounds__(kCsThreads) k_scan_chunks(BinArgs a) {
    __shared__ uint32_t s_part;
    __shared__ ScanShared<kCsThreads> sh;
    const long long nparts = (a.chunks + kScanTile - 1) / kScanTile;
    // the claim classes of this binning start empty (k_tile_scan fills them; the compositing launches
    // of the previous binning, which read them, are complete)
    if (blockIdx.x == 0 && threadIdx.x < kClaimClasses) a.st->claim_cnt[threadIdx.x] = 0u;
    for (;;) {
        if (threadIdx.x == 0) s_part = nparts == 1 ? 0u : claim_part(&a.st->ctr[kCtrScan], nparts);
        __syncthreads();
        const long long part = s_part;
        if (part >= nparts) break;
        const long long base = part * kScanTile + (long long)threadIdx.x * kCsIPT;
        uint32_t x[kCsIPT], nv[kCsIPT];
        unsigned long long tsum = 0, vsum = 0;
#pragma unroll
        for (int k = 0; k < kCsIPT; ++k) {
            const uint4 b = base + k < a.chunks ? a.blk[base + k] : make_uint4(0u, 0u, 0u, 0u);
            x[k] = b.z;
            nv[k] = blk_visible(b.y);
            tsum += x[k];
            vsum += nv[k];
        }
        unsigned long long run = scan_partition<kCsThreads>(a, sh, part, nparts, tsum);
        if constexpr (PAIRS) {
            __syncthreads();              // sh.prefix has been read
            BinArgs av = a;
            av.scan_state = a.vis_scan_state;
            unsigned long long vrun = scan_partition<kCsThreads, false>(av, sh, part, nparts, vsum);
            if (part == nparts - 1 && threadIdx.x == kCsThreads - 1) a.st->bin_pairs = vrun + vsum;
#pragma unroll
            for (int k = 0; k < kCsIPT; ++k) {
                if (base + k < a.chunks) a.blk[base + k].z = sat32(vrun);
                vrun += nv[k];
            }
        }
#pragma unroll
        for (int k = 0; k < kCsIPT; ++k) {
            if (base + k >= a.chunks) break;
            a.blk[base + k].w = sat32(run);
            if (!PAIRS && x[k] > a.emit_keys && run < (unsigned long long)a.cap) {
                const uint32_t below = (uint32_t)min((unsigned long long)x[k], (unsigned long long)a.cap - run);
                const uint32_t extra = (below - 1u) / a.emit_keys;   // portions 1 .. extra
                const uint32_t at = extra ? atomicAdd(&a.st->ctr[kCtrEmitExtra], extra) : 0u;
                for (uint32_t j = 0; j < extra; ++j)
                    if (at + j < a.extra_cap) a.extra[at + j] = make_uint2((uint32_t)(base + k), j + 1u);
            }
            run += x[k];
        }
        __syncthreads();
        if (nparts <= (long long)gridDim.x) break;
    }
}

// ------------------------------------------------------------------------------------------
// 2. keys of a chunk, each with its rank inside its tile
// ------------------------------------------------------------------------------------------
// One CTA of 128 threads per chunk: 256 pairs (two per thread in the scan), their keys a thread
// each.  The rank is the old value of the tile's counter, so the keys of a tile are ranked in the
// order their atomics arrive; the sort of step 5 makes the list's order independent of it.  Four
// keys per thread are in flight together (binary search over the chunk's inclusive sums, atomic,
// 16-byte store).  CTAs beyond the chunks take the extra portions of heavy chunks.
//
// A view whose Gaussians pile up in few tiles has them all at the same counters, and one address takes an atomic every
// 1.5 ns.  There the keys of a batch are counted per tile in shared memory (a table of hashed tiles; a key that finds
// another tile in its place goes to the counter itself) and every tile in the table takes one atomic.  An item does
// so where an eighth of its first keys have the tile of the key 16 lanes on, or where some tile is known to hold more
// than kEtHot keys: always, it costs latency that short problems cannot hide (a 500 k room's binning 67 -> 70 us).
// (32 registers, so that it does not lower the resident CTAs: 32 views 518 us at 40 registers, 511 at 32, as without.)
// Views of at most kPile Gaussians do without (25 us at the worst).  Binning of a 640 x 480 view, us, one atomic a
// key / counted first: 400 k Gaussians in 4 tiles 323 / 145, 2 M 1307 / 412; 2 M in 36 tiles 771 / 526.
constexpr int kEtThreads = 128, kEtBatch = 4;
constexpr int kEtTableBits = 9, kEtTable = 1 << kEtTableBits;
constexpr int kEtShared = kEtThreads / 8;
constexpr uint32_t kEtHot = 4096;
constexpr long long kPile = 16384;
constexpr uint32_t kNoTile = 0xffffffffu;
static_assert(kChunk == 2 * kEtThreads, "two pairs per thread");

template <bool PILES>
__global__ void __launch_bounds__(kEtThreads, 16) k_emit_tiles(BinArgs a) {
    __shared__ uint32_t s_inc[kChunk];    // keys of the chunk's pairs up to and including each
    __shared__ uint32_t s_g0[kChunk];     // global tile of the rectangle's top-left corner
    __shared__ uint32_t s_wr[kChunk];     // rectangle width
    __shared__ uint32_t s_z[kChunk];      // depth bits
    __shared__ uint32_t s_wsum[kEtThreads / 32];
    __shared__ uint32_t s_tile[PILES ? kEtTable : 1], s_cnt[PILES ? kEtTable : 1];   // tiles of a batch and its keys in them
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long nextra =
        (long long)blockIdx.x < a.chunks ? 0 : (long long)min(a.st->ctr[kCtrEmitExtra], a.extra_cap);
    for (long long q = (long long)blockIdx.x - a.chunks; q < 0 || q < nextra; q += gridDim.x - a.chunks) {
        const uint2 it = q < 0 ? make_uint2(blockIdx.x, 0u) : a.extra[q];
        const uint4 b = a.blk[it.x];
        const bool hot = PILES && ld_relaxed_u32(a.coop + kCoopHot) != 0u;
        const int v = blk_view(b.y);
        const ViewEntry ve = a.views[v];
        const long long local = ((long long)it.x - ve.chunk_off) * kChunk;
        const long long fbase = ve.pair_off + local;
        const unsigned long long vc = (unsigned long long)a.vcap;
        const uint32_t n0 = b.x < vc ? (uint32_t)min((unsigned long long)blk_candidates(b.y), vc - b.x) : 0u;
        s_inc[tid] = s_inc[tid + kEtThreads] = 0u;
        __syncthreads();
        for (uint32_t u = tid; u < n0; u += kEtThreads) {
            const size_t sl = (size_t)b.x + u;
            const uint32_t li = a.slane[sl];
            if (li & kSlotHole) continue;
            const float4 r0 = a.proj[3 * sl], r1 = a.proj[3 * sl + 1];
            int x0, x1, y0, y1;
            spec_rect(r0.x, r0.y, r1.w, a.itw, a.ith, (float)a.Tx, (float)a.Ty, x0, x1, y0, y1);
            const uint32_t i = li & 0xffu;
            s_inc[i] = (uint32_t)((x1 - x0) * (y1 - y0));
            s_g0[i] = (uint32_t)((unsigned long long)v * a.Tx * a.Ty + (unsigned long long)(y0 * a.Tx + x0));
            s_wr[i] = (uint32_t)max(x1 - x0, 1);
            s_z[i] = __float_as_uint(r1.z);
            if (it.y == 0u) {             // the backward accumulator of the slot
                const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
                a.g2d[3 * sl] = z4;
                a.g2d[3 * sl + 1] = z4;
                a.g2d[3 * sl + 2] = z4;
            }
        }
        __syncthreads();
        // inclusive sums over the chunk's pairs, two consecutive pairs per thread
        const uint32_t c0 = s_inc[2 * tid], c1 = s_inc[2 * tid + 1];
        uint32_t incl = c0 + c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_wsum[warp] = incl;
        __syncthreads();
        uint32_t off = 0, total = 0;
#pragma unroll
        for (int w = 0; w < kEtThreads / 32; ++w) {
            if (w < warp) off += s_wsum[w];
            total += s_wsum[w];
        }
        s_inc[2 * tid] = off + incl - c1;
        s_inc[2 * tid + 1] = off + incl;
        __syncthreads();
        if (it.y == 0u) {
            if (total != b.z && tid == 0) record_error(a.st, GS_ERR_DEVICE_FAULT, 3);
            if (a.touched) {              // counts -> inclusive sums over all pairs
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int li = tid + h * kEtThreads;
                    if (local + li < ve.count && gs_guard(a.st, fbase + li < a.P, 13))
                        a.touched[fbase + li] = sat32((unsigned long long)b.w + s_inc[li]);
                }
            }
        }
        // this item's keys [lo, hi) of the chunk, those below the capacity
        const unsigned long long room = (unsigned long long)b.w < (unsigned long long)a.cap ? (unsigned long long)a.cap - b.w : 0ull;
        const uint32_t lim = (uint32_t)min((unsigned long long)min(total, b.z), room);
        const uint32_t lo = it.y * a.emit_keys;
        const uint32_t hi = lim - min(lim, lo) > a.emit_keys ? lo + a.emit_keys : lim;
        bool few = false;                 // keys are counted per tile in shared memory first
        for (uint32_t mb = lo; mb < hi; mb += kEtThreads * kEtBatch) {
            const uint32_t m0 = mb + tid;
            uint32_t g[kEtBatch], p[kEtBatch], rank[kEtBatch];
#pragma unroll
            for (int k = 0; k < kEtBatch; ++k) {
                const uint32_t m = m0 + k * kEtThreads;
                // the pair: smallest li with inc[li] > m (pairs without keys repeat their predecessor's sum)
                uint32_t li = 0;
                g[k] = kNoTile;
                if (m < hi) {
#pragma unroll
                    for (int step = kChunk / 2; step > 0; step >>= 1)
                        if (s_inc[li + step - 1] <= m) li += step;
                    const uint32_t r = m - (li ? s_inc[li - 1] : 0u), w = s_wr[li], row = r / w;
                    g[k] = s_g0[li] + row * (uint32_t)a.Tx + (r - row * w);
                    if (!gs_guard(a.st, (long long)g[k] < a.G, 14)) g[k] = kNoTile;
                }
                p[k] = li;
            }
            if (PILES && mb == lo) {
                const uint32_t near = __shfl_xor_sync(0xffffffffu, g[0], 16);
                // (counted, so that every thread decides alike although each has read the note by itself)
                few = __syncthreads_count(hot || (g[0] != kNoTile && near == g[0])) >= kEtShared;
            }
            if (!PILES || !few) {
#pragma unroll
                for (int k = 0; k < kEtBatch; ++k)
                    if (g[k] != kNoTile) rank[k] = atomicAdd(a.tile_cnt + g[k], 1u);
#pragma unroll
                for (int k = 0; k < kEtBatch; ++k)
                    if (PILES && g[k] != kNoTile && rank[k] == kEtHot) st_relaxed_u32(a.coop + kCoopHot, 1u);
            } else {
                int at[kEtBatch];
                for (int i = tid; i < kEtTable; i += kEtThreads) {
                    s_tile[i] = kNoTile;
                    s_cnt[i] = 0u;
                }
                __syncthreads();
#pragma unroll
                for (int k = 0; k < kEtBatch; ++k) {
                    at[k] = -1;
                    if (g[k] == kNoTile) continue;
                    const int h = (int)((g[k] * 0x9e3779b1u) >> (32 - kEtTableBits));
                    uint32_t t = *(volatile uint32_t *)(s_tile + h);
                    if (t == kNoTile) t = atomicCAS(s_tile + h, kNoTile, g[k]);
                    if (t == kNoTile || t == g[k]) {
                        at[k] = h;
                        rank[k] = atomicAdd(s_cnt + h, 1u);
                    } else {              // another tile's place
                        rank[k] = atomicAdd(a.tile_cnt + g[k], 1u);
                    }
                }
                __syncthreads();
                for (int i = tid; i < kEtTable; i += kEtThreads) {
                    if (s_tile[i] == kNoTile) continue;
                    const uint32_t n = s_cnt[i], from = atomicAdd(a.tile_cnt + s_tile[i], n);
                    if (from <= kEtHot && from + n > kEtHot) st_relaxed_u32(a.coop + kCoopHot, 1u);
                    s_cnt[i] = from;
                }
                __syncthreads();
#pragma unroll
                for (int k = 0; k < kEtBatch; ++k)
                    if (at[k] >= 0) rank[k] += s_cnt[at[k]];
                __syncthreads();          // before the next batch's table
            }
#pragma unroll
            for (int k = 0; k < kEtBatch; ++k) {
                const uint32_t m = m0 + k * kEtThreads;
                if (m < hi) a.items[(size_t)b.w + m] = make_uint4(g[k], rank[k], s_z[p[k]], (uint32_t)(fbase + p[k]));
            }
        }
        if (q < 0) break;
        __syncthreads();                  // the shared tables are rebuilt for the next item
    }
}

// ------------------------------------------------------------------------------------------
// 3. tile ranges and claim classes
// ------------------------------------------------------------------------------------------
// Every item of a partition is filed under its claim class with one global atomic per class and
// partition (the position inside the partition's run from a shared counter).
__device__ __forceinline__ uint32_t class_position(uint32_t *s_cls, int c, bool in) {
    // (few classes are met by many tiles: one shared atomic per warp and class)
    const unsigned peers = __match_any_sync(0xffffffffu, in ? c : -1);
    const int lead = __ffs(peers) - 1;
    uint32_t at = 0;
    if (in && (int)(threadIdx.x & 31) == lead) at = atomicAdd(&s_cls[c], (uint32_t)__popc(peers));
    return __shfl_sync(0xffffffffu, at, lead) + (uint32_t)__popc(peers & lanemask_lt());
}

__global__ void __launch_bounds__(kCsThreads) k_tile_scan(BinArgs a) {
    __shared__ uint32_t s_part;
    __shared__ ScanShared<kCsThreads> sh;
    __shared__ uint32_t s_cls[kClaimClasses], s_base[kClaimClasses];
    const long long nparts = (a.G + kScanTile - 1) / kScanTile;
    if (blockIdx.x == 0 && threadIdx.x == 0) {   // the compositing launches on this binning count anew
        a.st->fwd_pairs = 0ull;
        a.st->bwd_pairs = 0ull;
    }
    for (;;) {
        if (threadIdx.x == 0) s_part = nparts == 1 ? 0u : claim_part(&a.st->ctr[kCtrTileScan], nparts);
        if (threadIdx.x < kClaimClasses) s_cls[threadIdx.x] = 0u;
        __syncthreads();
        const long long part = s_part;
        if (part >= nparts) break;
        const long long base = part * kScanTile + (long long)threadIdx.x * kCsIPT;
        uint32_t x[kCsIPT], pos[kCsIPT];
        unsigned long long tsum = 0;
#pragma unroll
        for (int k = 0; k < kCsIPT; ++k) {
            x[k] = base + k < a.G ? a.tile_cnt[base + k] : 0u;
            tsum += x[k];
            pos[k] = class_position(s_cls, claim_class(x[k]), base + k < a.G);
        }
        unsigned long long run = scan_partition<kCsThreads, false>(a, sh, part, nparts, tsum);
        if (threadIdx.x < kClaimClasses) {
            const uint32_t c = s_cls[threadIdx.x];
            s_base[threadIdx.x] = c ? atomicAdd(&a.st->claim_cnt[threadIdx.x], c) : 0u;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kCsIPT; ++k) {
            const long long g = base + k;
            if (g >= a.G) break;
            // an empty tile reads [0, 0)
            a.ranges[2 * g] = x[k] ? sat32(run) : 0u;
            a.ranges[2 * g + 1] = x[k] ? sat32(run + x[k]) : 0u;
            run += x[k];
            const int c = claim_class(x[k]);
            const unsigned long long at = (unsigned long long)s_base[c] + pos[k];
            if (at < (unsigned long long)a.G) a.clist[(size_t)c * a.G + at] = (uint32_t)g;
            else record_error(a.st, GS_ERR_DEVICE_FAULT, 12);
        }
        __syncthreads();
        if (nparts <= (long long)gridDim.x) break;
    }
}

// The claim classes alone, from the ranges (after the radix binning).
__global__ void __launch_bounds__(kCsThreads) k_claims(BinArgs a) {
    __shared__ uint32_t s_cls[kClaimClasses], s_base[kClaimClasses];
    if (blockIdx.x == 0 && threadIdx.x == 0) {   // the compositing launches on this binning count anew
        a.st->fwd_pairs = 0ull;
        a.st->bwd_pairs = 0ull;
    }
    if (threadIdx.x < kClaimClasses) s_cls[threadIdx.x] = 0u;
    __syncthreads();
    const long long g = (long long)blockIdx.x * kCsThreads + threadIdx.x;
    int c = 0;
    if (g < a.G) {
        const uint2 r = reinterpret_cast<const uint2 *>(a.ranges)[g];
        c = claim_class(r.y - r.x);
    }
    const uint32_t pos = class_position(s_cls, c, g < a.G);
    __syncthreads();
    if (threadIdx.x < kClaimClasses) {
        const uint32_t n = s_cls[threadIdx.x];
        s_base[threadIdx.x] = n ? atomicAdd(&a.st->claim_cnt[threadIdx.x], n) : 0u;
    }
    __syncthreads();
    if (g < a.G) {
        const unsigned long long at = (unsigned long long)s_base[c] + pos;
        if (at < (unsigned long long)a.G) a.clist[(size_t)c * a.G + at] = (uint32_t)g;
        else record_error(a.st, GS_ERR_DEVICE_FAULT, 12);
    }
}

// ------------------------------------------------------------------------------------------
// 4. words into their slices
// ------------------------------------------------------------------------------------------
constexpr int kScThreads = 256, kScBatch = 4;
__global__ void __launch_bounds__(kScThreads) k_scatter(BinArgs a) {
    const unsigned long long K = min(a.st->num_keys, (unsigned long long)a.cap);
    if (blockIdx.x == 0 && threadIdx.x == 0) a.st->ctr[kCtrEmitExtra] = 0u;   // k_emit_tiles is complete
    const unsigned long long stride = (unsigned long long)gridDim.x * kScThreads;
    for (unsigned long long i0 = (unsigned long long)blockIdx.x * kScThreads + threadIdx.x; i0 < K; i0 += stride * kScBatch) {
        uint4 it[kScBatch];
        uint32_t start[kScBatch];
#pragma unroll
        for (int k = 0; k < kScBatch; ++k)
            if (i0 + k * stride < K) it[k] = a.items[i0 + k * stride];
#pragma unroll
        for (int k = 0; k < kScBatch; ++k) {
            start[k] = 0xffffffffu;
            if (i0 + k * stride < K && (long long)it[k].x < a.G) start[k] = a.ranges[2 * (size_t)it[k].x];
        }
#pragma unroll
        for (int k = 0; k < kScBatch; ++k) {
            if (i0 + k * stride >= K) continue;
            const unsigned long long dst = (unsigned long long)start[k] + it[k].y;
            if (dst < K) a.words[dst] = ((unsigned long long)it[k].z << 32) | it[k].w;
            else record_error(a.st, GS_ERR_DEVICE_FAULT, 5);   // only after an earlier recorded failure
        }
    }
}

// ------------------------------------------------------------------------------------------
// 5. sort of every slice
// ------------------------------------------------------------------------------------------
// Lists of up to 256 words are sorted by one warp in registers (bitonic, 1 to 8 words per lane), longer
// ones by a CTA: every warp sorts 256 words the same way, the sorted chunks are merged pairwise in shared
// memory, each thread finding its outputs' position in the two runs by a binary search along its
// diagonal (merge path), and lists beyond one shared-memory run are sorted run by run and the runs
// merged block by block between the tile's slices of the two key buffers.  The register sort works on
// 32-bit words (24 bits of depth relative to the list's range, 8 bits of position; one min and one max
// per exchange instead of six instructions) and sorts the 64-bit words themselves only when two
// entries that the 24 bits cannot tell apart came out in the wrong order.
constexpr int kTlKPT = 8;                            // words per thread of a full shared-memory run
constexpr int kWarpSort = 256;                       // lists of at most so many words are sorted by one warp
constexpr int kLongClass = 15;                       // claim classes 0 .. 15 hold the lists of 256 entries and more
typedef unsigned long long word_t;

__device__ __forceinline__ int pd(int i) { return i + (i >> 3); }   // one spare word in nine: strided runs without bank conflicts

// Words that come from run A (na words from a0) among the first d of A merged with run B (nb words
// from b0), both ascending, by AT(i) = word i.
template <class At>
__device__ __forceinline__ int merge_split(At at, int a0, int na, int b0, int nb, int d) {
    int lo = max(0, d - nb), hi = min(d, na);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (at(a0 + mid) < at(b0 + d - 1 - mid)) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The same for runs of na and nb words at r, by a warp: 32 probes a step, so that runs in global memory cost a few
// loads in a chain instead of one per bit of their length.
__device__ __forceinline__ int warp_split(const word_t *r, int na, int nb, int d, int lane) {
    int lo = max(0, d - nb), hi = min(d, na);
    while (lo < hi) {                     // (lo and hi are the same in every lane)
        const int step = (hi - lo + 31) >> 5, mid = lo + (lane + 1) * step - 1;
        const int below = __popc(__ballot_sync(0xffffffffu, mid < hi && r[mid] < r[na + d - 1 - mid]));
        const int from = lo + below * step;
        hi = min(hi, from + step - 1);
        lo = from;
    }
    return lo;
}

// KPT outputs of the merge of A and B in shared memory from diagonal d on (past the end: ~0)
template <int KPT>
__device__ __forceinline__ void merge_regs(const word_t *s, int a0, int na, int b0, int nb, int d, word_t (&out)[KPT]) {
    int ia = merge_split([&](int i) { return s[pd(i)]; }, a0, na, b0, nb, d);
    int ib = d - ia;
    word_t wa = ia < na ? s[pd(a0 + ia)] : ~0ull, wb = ib < nb ? s[pd(b0 + ib)] : ~0ull;
#pragma unroll
    for (int r = 0; r < KPT; ++r) {
        const bool ta = wa <= wb;
        out[r] = ta ? wa : wb;
        if (ta) ++ia;
        else ++ib;
        const bool in = ta ? ia < na : ib < nb;
        const word_t nx = in ? s[pd(ta ? a0 + ia : b0 + ib)] : ~0ull;
        if (ta) wa = nx;
        else wb = nx;
    }
}

// Bitonic network over 32 E elements, element lane * E + r in x[r]; ascending.  The phases that cross lanes
// are loops, not unrolled: straight-line code for all of them costs more in instruction fetches than it
// saves when a CTA sorts one list.  A lane of a descending block holds complemented elements during
// its phase, so every exchange inside a lane is one min and one max.
template <int E, class T>
__device__ __forceinline__ void bitonic_warp(T (&x)[E], int lane) {
    T flip = 0;
#pragma unroll
    for (int k = 2; k < E; k <<= 1)       // blocks inside a lane
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int r = 0; r < E; ++r)
                if ((r & j) == 0) {
                    const T lo = min(x[r], x[r | j]), hi = max(x[r], x[r | j]);
                    x[r] = (r & k) == 0 ? lo : hi;
                    x[r | j] = (r & k) == 0 ? hi : lo;
                }
#pragma unroll 1
    for (int m = E > 1 ? 1 : 2; m <= 32; m <<= 1) {   // blocks of m lanes, descending where lane & m
        const T f = (lane & m) ? ~(T)0 : (T)0;        // (lane < 32: the last block is ascending)
#pragma unroll
        for (int r = 0; r < E; ++r) x[r] ^= flip ^ f;
        flip = f;
#pragma unroll 1
        for (int l = m >> 1; l > 0; l >>= 1) {
            const bool lower = (lane & l) == 0;
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const T y = __shfl_xor_sync(0xffffffffu, x[r], l);
                x[r] = lower ? min(x[r], y) : max(x[r], y);
            }
        }
#pragma unroll
        for (int j = E >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int r = 0; r < E; ++r)
                if ((r & j) == 0) {
                    const T lo = min(x[r], x[r | j]);
                    x[r | j] = max(x[r], x[r | j]);
                    x[r] = lo;
                }
    }
}

// n <= 32 E words from src, ascending over (lane, r): lane's words are x[0 .. E) at lane E + r (~0 past n)
template <int E>
__device__ __forceinline__ void sort_warp(word_t (&x)[E], const word_t *src, int n, int lane) {
    static_assert(32 * E <= 256, "8 bits of position");
    uint32_t z[E], zmin = 0xffffffffu, zmax = 0u;
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const int e = r * 32 + lane;
        z[r] = e < n ? reinterpret_cast<const uint32_t *>(src)[2 * e + 1] : 0u;   // depth bits
        zmin = e < n ? min(zmin, z[r]) : zmin;
        zmax = max(zmax, z[r]);
    }
    zmin = __reduce_min_sync(0xffffffffu, zmin);
    zmax = __reduce_max_sync(0xffffffffu, zmax);
    const int shift = max(0, 8 - __clz(zmax - zmin));
#pragma unroll
    for (int r = 0; r < E; ++r) {   // (a real word is below 2^32 - 1: with a position of 255 there is no padding)
        const int e = r * 32 + lane;
        z[r] = e < n ? ((z[r] - zmin) >> shift) << 8 | (uint32_t)e : 0xffffffffu;
    }
    bitonic_warp<E>(z, lane);
#pragma unroll
    for (int r = 0; r < E; ++r) x[r] = lane * E + r < n ? src[z[r] & 255u] : ~0ull;
    bool bad = false;
    const word_t next = __shfl_down_sync(0xffffffffu, x[0], 1);
#pragma unroll
    for (int r = 0; r < E; ++r) bad |= x[r] > (r + 1 < E ? x[r + 1 < E ? r + 1 : r] : (lane < 31 ? next : ~0ull));
    if (__any_sync(0xffffffffu, bad)) bitonic_warp<E>(x, lane);
}

// one merge level over the n words of s (padded positions; n a multiple of KPT), runs of w words; whole CTA
template <int THREADS, int KPT>
__device__ __forceinline__ void merge_level(word_t *s, int n, int w) {
    const int at = threadIdx.x * KPT;
    const bool act = at < n;
    word_t x[KPT];
    if (act) {
        const int base = at / (2 * w) * (2 * w);
        const int na = min(w, n - base), nb = min(w, n - base - na);
        merge_regs<KPT>(s, base, na, base + na, nb, at - base, x);
    }
    __syncthreads();
    if (act) {
#pragma unroll
        for (int r = 0; r < KPT; ++r) s[pd(at + r)] = x[r];
    }
    __syncthreads();
}

// n <= 8 THREADS words from src into s (padded positions, ~0 up to a multiple of 256), ascending; whole CTA
template <int THREADS>
__device__ __forceinline__ void sort_smem(word_t *s, const word_t *src, int n) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c0 = warp * 256;
    if (c0 < n) {
        word_t x[8];
        sort_warp<8>(x, src + c0, min(256, n - c0), lane);
#pragma unroll
        for (int r = 0; r < 8; ++r) s[pd(c0 + lane * 8 + r)] = x[r];
    }
    __syncthreads();
    const int np = (n + 255) & ~255;
    for (int w = 256; w < np; w <<= 1) {
        if (np <= 4 * THREADS) merge_level<THREADS, 4>(s, np, w);
        else merge_level<THREADS, 8>(s, np, w);
    }
}

// key and value of list position pos of tile g; the entry's slot (kNoSlot after an earlier failure)
__device__ __forceinline__ uint32_t emit_entry(const BinArgs &a, uint64_t *kout, uint32_t *vout, long long g, long long pos,
                                               word_t w) {
    const uint32_t f = (uint32_t)w;
    kout[pos] = ((unsigned long long)g << 32) | (w >> 32);
    vout[pos] = f;
    uint32_t sl = (long long)f < a.P ? a.slot[f] : kNoSlot;
    if (sl >= (unsigned long long)a.vcap) {
        record_error(a.st, GS_ERR_DEVICE_FAULT, 6);
        sl = kNoSlot;
    }
    return sl;
}

// The records of list positions s0 .. s0 + n - 1 by THREADS threads: a thread keeps one of the three
// float4s of a record and steps THREADS / 3 records on, so that neighbouring threads write
// neighbouring 16 bytes; slot(e) is entry e's slot.  The radius field (used only by the emission)
// carries the slot.
template <int THREADS, class Slot>
__device__ __forceinline__ void copy_records(const BinArgs &a, long long s0, int n, int t, Slot slot) {
    constexpr int kStep = THREADS / 3;
    if (t >= 3 * kStep) return;
    const int part = t % 3;
    const float4 *src = a.proj + part;
    float4 *dst = a.srec + 3 * (size_t)s0 + t;
#pragma unroll 4
    for (int e = t / 3; e < n; e += kStep, dst += 3 * kStep) {
        const uint32_t sl = slot(e);
        if (sl == kNoSlot) continue;
        float4 r = src[3 * (size_t)sl];
        if (part == 1) r.w = __uint_as_float(sl);
        *dst = r;
    }
}

template <int E>
__device__ __forceinline__ void warp_list(const BinArgs &a, uint64_t *kout, uint32_t *vout, long long g, long long s0, int n,
                                          uint32_t *slots, int lane) {
    word_t x[E];
    sort_warp<E>(x, a.words + s0, n, lane);
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const int e = lane * E + r;
        if (e < n) slots[e] = emit_entry(a, kout, vout, g, s0 + e, x[r]);
    }
    __syncwarp();
    copy_records<32>(a, s0, n, lane, [&](int e) { return slots[e]; });
    __syncwarp();
}

// The short list of tile g, one warp.
__device__ __forceinline__ void sort_short(const BinArgs &a, long long g, uint32_t *slots, int lane) {
    if (g >= a.G) return;
    uint64_t *kout = a.keys[a.passes & 1];
    uint32_t *vout = a.vals[a.passes & 1];
    const unsigned long long K = min(a.st->num_keys, (unsigned long long)a.cap);
    const uint2 r = reinterpret_cast<const uint2 *>(a.ranges)[g];
    if (r.y < r.x || (unsigned long long)r.y > K) {   // only after an earlier recorded failure
        if (lane == 0) record_error(a.st, GS_ERR_DEVICE_FAULT, 9);
        return;
    }
    const int n = (int)(r.y - r.x);
    if (n == 0 || n > kWarpSort) return;
    if (n <= 32) warp_list<1>(a, kout, vout, g, r.x, n, slots, lane);
    else if (n <= 64) warp_list<2>(a, kout, vout, g, r.x, n, slots, lane);
    else if (n <= 128) warp_list<4>(a, kout, vout, g, r.x, n, slots, lane);
    else warp_list<8>(a, kout, vout, g, r.x, n, slots, lane);
}

// Output block b (kRun words) of one merge level of a list of n words: runs of w words of `in` merged pairwise into
// `out`; whole CTA.  Two warps find where the block's first and last outputs split the two runs.
template <int THREADS>
__device__ __forceinline__ void merge_block(word_t *s, int *split, const word_t *in, word_t *out, int n, int b, long long w) {
    constexpr int kRun = kTlKPT * THREADS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = (int)((long long)b * kRun / (2 * w) * (2 * w));
    const int na = (int)min(w, (long long)n - base), nb = (int)min(w, (long long)n - base - na);
    const int d0 = b * kRun - base, d1 = min(d0 + kRun, na + nb);
    if (warp < 2) {
        const int at = warp_split(in + base, na, nb, warp ? d1 : d0, lane);
        if (lane == 0) split[warp] = at;
    }
    __syncthreads();
    const int a0 = split[0], ca = split[1] - a0, cb = d1 - d0 - ca;
    const word_t *ra = in + base + a0, *rb = in + base + na + (d0 - a0);
    for (int e = tid; e < ca + cb; e += THREADS) s[pd(e)] = e < ca ? ra[e] : rb[e - ca];
    __syncthreads();
    word_t x[kTlKPT];
    const bool act = tid * kTlKPT < ca + cb;
    if (act) merge_regs<kTlKPT>(s, 0, ca, ca, cb, tid * kTlKPT, x);
    __syncthreads();
    if (act) {
#pragma unroll
        for (int r = 0; r < kTlKPT; ++r) s[pd(tid * kTlKPT + r)] = x[r];
    }
    __syncthreads();
    for (int e = tid; e < ca + cb; e += THREADS) out[b * kRun + e] = s[pd(e)];
    __syncthreads();
}

// Keys, values and records of `len` sorted words from position r0 of tile g's list at s0; whole CTA.  (`in` may be the
// key buffer itself: an entry's key is written by the thread that read its word.)
template <int THREADS>
__device__ __forceinline__ void finish_run(const BinArgs &a, word_t *s, const word_t *in, long long g, long long s0, int r0, int len) {
    uint32_t *slots = reinterpret_cast<uint32_t *>(s);
    uint64_t *kout = a.keys[a.passes & 1];
    uint32_t *vout = a.vals[a.passes & 1];
    for (int e = threadIdx.x; e < len; e += THREADS) slots[e] = emit_entry(a, kout, vout, g, s0 + r0 + e, in[r0 + e]);
    __syncthreads();
    copy_records<THREADS>(a, s0 + r0, len, threadIdx.x, [&](int e) { return slots[e]; });
    __syncthreads();
}

// Lists of more than kCoopMin words and of more than a 192nd of all keys are sorted by all long-list CTAs together: a
// tile may hold every Gaussian of a view, and a list of 131 k words takes one CTA 3.1 ms.  The work is split into items of one run or output block each:
// stage 0 sorts the runs in place, each further stage is one merge level, the last one writes keys, values and
// records.  CTAs claim items by a ticket, all lists' items of a stage before the next stage's, and an item waits
// until every item of its list's earlier stages is counted in the list's done word.  All those have smaller
// tickets, whose holders are running CTAs that wait for smaller ones only, so no wait depends on a CTA that has yet
// to start (and each is bounded).  The share of the keys keeps a view of many long lists at one list per CTA, without
// waits, and bounds the number of shared lists by kCoopLists.
//   Binning of a 640 x 480 view, us, one CTA per list / lists shared: 60 k Gaussians in 4 tiles 465 / 111, 400 k
// 3268 / 324, 2 M 22976 / 1306 (the emission takes 190 and 960 of it); 400 k in 36 tiles 538 / 185; 2 M in 144 tiles
// 1062 / 698.  (kCoopMin 16384: 400 k in 36 tiles 425.)  No list is shared in a 500 k room (67 and 67 us) or in 32
// views of submaps (503 and 508).
constexpr int kCoopLists = 192;
constexpr uint32_t kCoopMin = 4096;

struct CoopLists {
    uint32_t start[kCoopLists], n[kCoopLists], g[kCoopLists];
    uint32_t upto[kCoopLists];           // items of the stage in this and the lists before
    uint32_t warp_cnt[32];
    uint32_t ticket;
    int count, levels, ok;
};
static_assert(kCoopHot == 1 + kCoopLists, "ticket and done words");

__device__ __forceinline__ int merge_levels(uint32_t runs) { return runs > 1u ? 32 - __clz(runs - 1u) : 0; }

// The shared lists in claim order (the same in every CTA): of the first `cand` claims those of more than `above` words.
template <int THREADS>
__device__ __forceinline__ void coop_collect(const BinArgs &a, CoopLists &c, const uint32_t *coff, long long cand, uint32_t above,
                                             unsigned long long K) {
    constexpr int kRun = kTlKPT * THREADS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) c.count = c.levels = 0;
    __syncthreads();
    for (long long i0 = 0; i0 < cand; i0 += THREADS) {
        const long long i = i0 + threadIdx.x;
        const long long g = i < cand ? claim_at(coff, a.clist, a.G, i) : a.G;
        const uint2 r = g < a.G ? reinterpret_cast<const uint2 *>(a.ranges)[g] : make_uint2(0u, 0u);
        const bool in = r.y > r.x && (unsigned long long)r.y <= K && r.y - r.x > above;
        const unsigned vote = __ballot_sync(0xffffffffu, in);
        if (lane == 0) c.warp_cnt[warp] = (uint32_t)__popc(vote);
        __syncthreads();
        uint32_t at = (uint32_t)c.count + (uint32_t)__popc(vote & lanemask_lt()), all = 0;
#pragma unroll 1
        for (int w = 0; w < THREADS / 32; ++w) {
            if (w < warp) at += c.warp_cnt[w];
            all += c.warp_cnt[w];
        }
        if (in && at < (uint32_t)kCoopLists) {
            c.start[at] = r.x;
            c.n[at] = r.y - r.x;
            c.g[at] = (uint32_t)g;
            atomicMax(&c.levels, merge_levels((r.y - r.x + kRun - 1u) / kRun));
        }
        __syncthreads();
        if (threadIdx.x == 0) c.count = min(c.count + (int)all, kCoopLists);
        __syncthreads();
    }
}

// upto[] of a stage and its number of items; whole CTA
template <int THREADS>
__device__ __forceinline__ uint32_t coop_stage(CoopLists &c, int stage) {
    constexpr uint32_t kRun = kTlKPT * THREADS;
    const int lane = threadIdx.x & 31;
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t before = 0;
        for (int i0 = 0; i0 < c.count; i0 += 32) {
            const int i = i0 + lane;
            const uint32_t runs = i < c.count ? (c.n[i] + kRun - 1u) / kRun : 0u;
            uint32_t x = stage == 0 || stage > c.levels || merge_levels(runs) >= stage ? runs : 0u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (i < c.count) c.upto[i] = before + x;
            before += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    __syncthreads();
    return c.upto[c.count - 1];
}

// Waits until `want` items of a list are done (thread 0; bounded).  The barrier after it makes what their CTAs wrote
// visible to the whole CTA.
__device__ __forceinline__ bool coop_wait(const BinArgs &a, const uint32_t *done, uint32_t want) {
    for (unsigned long long spins = 0; ld_relaxed_u32(done) < want; ++spins) {
        if (spins > a.spin_limit) {
            record_error(a.st, GS_ERR_TIMEOUT, 13);
            return false;
        }
        __nanosleep(64);
    }
    __threadfence();
    return true;
}

// false after a wait that ran out
template <int THREADS>
__device__ __forceinline__ bool coop_sort(const BinArgs &a, CoopLists &c, word_t *s, int *split) {
    constexpr int kRun = kTlKPT * THREADS;
    const int tid = threadIdx.x, last = c.levels + 1;
    uint64_t *kout = a.keys[a.passes & 1];
    if (tid == 0) c.ticket = atomicAdd(a.coop, 1u);
    uint32_t before = 0, items = coop_stage<THREADS>(c, 0);   // (its barriers publish the ticket)
    int stage = 0;
    for (;;) {
        const uint32_t t = c.ticket;
        while (stage <= last && t - before >= items) {
            before += items;
            if (++stage <= last) items = coop_stage<THREADS>(c, stage);
        }
        if (stage > last) return true;
        const uint32_t at = t - before;
        int lo = 0, hi = c.count - 1;     // the list: smallest i with upto[i] > at
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (c.upto[mid] > at) hi = mid;
            else lo = mid + 1;
        }
        const int i = lo, b = (int)(at - (i ? c.upto[i - 1] : 0u)), n = (int)c.n[i], r0 = b * kRun;
        const uint32_t runs = (c.n[i] + kRun - 1u) / kRun;
        const int levels = merge_levels(runs);
        uint32_t next = 0;
        if (tid == 0) {
            next = atomicAdd(a.coop, 1u);    // on its way while the item is worked on
            c.ok = stage == 0 || coop_wait(a, a.coop + 1 + i, runs * (uint32_t)min(stage, levels + 1));
        }
        __syncthreads();
        if (!c.ok) return false;
        word_t *buf[2] = {a.words + c.start[i], reinterpret_cast<word_t *>(kout) + c.start[i]};
        if (stage == 0) {
            const int len = min(kRun, n - r0);
            sort_smem<THREADS>(s, buf[0] + r0, len);
            for (int e = tid; e < len; e += THREADS) buf[0][r0 + e] = s[pd(e)];
        } else if (stage < last) {
            merge_block<THREADS>(s, split, buf[(stage - 1) & 1], buf[stage & 1], n, b, (long long)kRun << (stage - 1));
        } else {
            finish_run<THREADS>(a, s, buf[levels & 1], c.g[i], c.start[i], r0, min(kRun, n - r0));
        }
        __syncthreads();
        if (tid == 0) {
            __threadfence();                 // the item's words before its count
            atomicAdd(a.coop + 1 + i, 1u);
            c.ticket = next;
        }
        __syncthreads();
    }
}

// The first a.long_blocks CTAs take the longer lists (the longest of them together, then a CTA each, longest first):
// runs of 8 words per thread sorted in shared memory, the runs of a longer list merged pairwise, a run of outputs
// at a time, between the tile's slices of the two key buffers.  The other CTAs sort the short lists beside them, a
// tile per warp.
template <int kTlThreads>
constexpr size_t kTileSortSmem = sizeof(word_t) * (kTlKPT * kTlThreads + kTlThreads);

template <int kTlThreads>
__global__ void __launch_bounds__(kTlThreads, 1024 / kTlThreads) k_tile_sort(BinArgs a) {
    constexpr int kRun = kTlKPT * kTlThreads, kWarps = kTlThreads / 32;
    extern __shared__ __align__(16) unsigned char ts_smem[];
    word_t *s = reinterpret_cast<word_t *>(ts_smem);
    static_assert(kWarps * kWarpSort * sizeof(uint32_t) <= kTileSortSmem<kTlThreads>, "a warp's slots");
    if ((long long)blockIdx.x >= a.long_blocks) {
        const int warp = threadIdx.x >> 5;
        sort_short(a, ((long long)blockIdx.x - a.long_blocks) * kWarps + warp, reinterpret_cast<uint32_t *>(s) + warp * kWarpSort,
                   threadIdx.x & 31);
        return;
    }
    __shared__ uint32_t coff[kClaimClasses + 1];
    __shared__ int s_split[2];
    __shared__ CoopLists s_coop;
    const int tid = threadIdx.x;
    uint64_t *kout = a.keys[a.passes & 1];
    uint32_t *vout = a.vals[a.passes & 1];
    claim_offsets(a.st, coff);
    __syncthreads();
    const long long nlong = min((long long)coff[kLongClass + 1], a.G);
    const unsigned long long K = min(a.st->num_keys, (unsigned long long)a.cap);
    const uint32_t above = (uint32_t)max((unsigned long long)kCoopMin, K / kCoopLists + 1ull);
    const long long cand = min((long long)coff[claim_class(above) + 1], a.G);
    if (cand > 0) {
        coop_collect<kTlThreads>(a, s_coop, coff, cand, above, K);
        if (s_coop.count > 0 && !coop_sort<kTlThreads>(a, s_coop, s, s_split)) return;
    }
    for (long long i = blockIdx.x; i < nlong; i += a.long_blocks) {
        const long long g = claim_at(coff, a.clist, a.G, i);
        const uint2 rng = g < a.G ? reinterpret_cast<const uint2 *>(a.ranges)[g] : make_uint2(1u, 0u);
        if (rng.y < rng.x || (unsigned long long)rng.y > K) {   // only after an earlier recorded failure
            if (tid == 0) record_error(a.st, GS_ERR_DEVICE_FAULT, 9);
            continue;
        }
        const long long s0 = rng.x;
        const int n = (int)(rng.y - rng.x);
        if (n <= kWarpSort) continue;     // exactly 256 words: a short list
        if (rng.y - rng.x > above) continue;   // sorted above
        // (the words lie in the key buffer that is not the output)
        word_t *in = a.words + s0, *out = reinterpret_cast<word_t *>(kout) + s0;
        if (n <= kRun) {
            sort_smem<kTlThreads>(s, in, n);
            for (int e = tid; e < n; e += kTlThreads) s[pd(e)] = emit_entry(a, kout, vout, g, s0 + e, s[pd(e)]);
            __syncthreads();
            copy_records<kTlThreads>(a, s0, n, tid, [&](int e) { return (uint32_t)s[pd(e)]; });
            __syncthreads();
            continue;
        }
        // sorted runs, in place
        for (int r0 = 0; r0 < n; r0 += kRun) {
            const int len = min(kRun, n - r0);
            sort_smem<kTlThreads>(s, in + r0, len);
            for (int e = tid; e < len; e += kTlThreads) in[r0 + e] = s[pd(e)];
            __syncthreads();
        }
        const int nblk = (n + kRun - 1) / kRun;
        for (long long w = kRun; w < n; w <<= 1) {
            for (int b = 0; b < nblk; ++b) merge_block<kTlThreads>(s, s_split, in, out, n, b, w);
            word_t *x = in;
            in = out;
            out = x;
        }
        for (int r0 = 0; r0 < n; r0 += kRun) finish_run<kTlThreads>(a, s, in, g, s0, r0, min(kRun, n - r0));
    }
}

// ------------------------------------------------------------------------------------------
// host driver
// ------------------------------------------------------------------------------------------
static int occupancy(const void *fn, int threads) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, threads, 0) != cudaSuccess || b < 1) b = 1;
    return b;
}

// (a.chunks > 0)
void launch_scan_chunks(const BinArgs &a, bool pairs, cudaStream_t s) {
    const long long parts = (a.chunks + kScanTile - 1) / kScanTile;
    static PerDevice per;
    const int occ = per.get(current_device(), [] {
        return std::min(occupancy((const void *)k_scan_chunks<true>, kCsThreads),
                        occupancy((const void *)k_scan_chunks<false>, kCsThreads));
    });
    const unsigned grid = (unsigned)std::min<long long>(parts, (long long)device_sm_count() * occ);
    if (pairs) k_scan_chunks<true><<<grid, kCsThreads, 0, s>>>(a);
    else k_scan_chunks<false><<<grid, kCsThreads, 0, s>>>(a);
    count_launches(1);
}

void launch_claims(const BinArgs &a, cudaStream_t s) {
    k_claims<<<(unsigned)((a.G + kCsThreads - 1) / kCsThreads), kCsThreads, 0, s>>>(a);
    count_launches(1);
}

template <int THREADS>
static int launch_tile_sort(BinArgs a, cudaStream_t s) {
    static PerDevice attr;
    if (!attr.get(current_device(), [] {
            return cudaFuncSetAttribute((const void *)k_tile_sort<THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)kTileSortSmem<THREADS>) == cudaSuccess;
        }))
        return GS_ERR_CUDA;
    constexpr int kWarps = THREADS / 32;
    // a view's Gaussians bound its lists; CTAs beyond the lists are there to share them (a 10 k cloud over 300
    // tiles, where nothing is shared: 41.5 us for the binning, 44 us with them)
    a.long_blocks = a.max_count > kWarpSort ? (long long)device_sm_count() * (1024 / THREADS) : 0;
    if (a.max_count <= kPile) a.long_blocks = std::min(a.long_blocks, a.G);
    k_tile_sort<THREADS><<<(unsigned)(a.long_blocks + (a.G + kWarps - 1) / kWarps), THREADS, kTileSortSmem<THREADS>, s>>>(a);
    return GS_OK;
}

static int run_tile_first(BinArgs a, cudaStream_t s) {
    const long long sms = device_sm_count();
    // tile counts and the look-back words of both scans
    if (cudaMemsetAsync(a.bucket_clear_begin, 0, a.bucket_clear_bytes, s) != cudaSuccess) return GS_ERR_CUDA;
    // keys per work item of the emission: few chunks (fewer than eight per SM) are split finely so that
    // every SM has keys to emit, many only to bound the work of a CTA whose pairs cover many tiles
    a.emit_keys = a.chunks < 8 * sms ? kEmitKeysMin : 4096u;
    if (a.chunks > 0) {
        launch_scan_chunks(a, false, s);
        const unsigned grid = (unsigned)(a.chunks + 4 * sms);
        if (a.max_count > kPile) k_emit_tiles<true><<<grid, kEtThreads, 0, s>>>(a);
        else k_emit_tiles<false><<<grid, kEtThreads, 0, s>>>(a);
        count_launches(1);
    } else if (cudaMemsetAsync(&a.st->num_keys, 0, sizeof(unsigned long long), s) != cudaSuccess ||
               cudaMemsetAsync(a.st->claim_cnt, 0, sizeof(uint32_t) * kClaimClasses, s) != cudaSuccess) {
        return GS_ERR_CUDA;   // no pairs: K = 0, and the claim classes start empty
    }
    BinArgs t = a;
    t.scan_state = a.tile_scan_state;
    static PerDevice per_t, per_s;
    const int dev = current_device();
    const int occ_t = per_t.get(dev, [] { return occupancy((const void *)k_tile_scan, kCsThreads); });
    const long long gparts = (a.G + kScanTile - 1) / kScanTile;
    k_tile_scan<<<(unsigned)std::min<long long>(gparts, sms * occ_t), kCsThreads, 0, s>>>(t);
    const int occ_s = per_s.get(dev, [] { return occupancy((const void *)k_scatter, kScThreads); });
    k_scatter<<<(unsigned)std::max<long long>(1, std::min<long long>((a.cap + kScThreads - 1) / kScThreads, sms * occ_s)),
                kScThreads, 0, s>>>(a);
    // fewer tiles than SMs: a CTA of 1024 threads per list, whose runs hold 8192 words, else 256 threads
    const int rc = a.G <= sms ? launch_tile_sort<1024>(a, s) : launch_tile_sort<256>(a, s);
    if (rc) return rc;
    count_launches(3);
    return check_launch();
}

// Which binning.  The tile-first one sorts every list by one warp or CTA and moves 48 B per key besides
// the outputs; the radix one sorts the pairs' depths in four launches whose latency small problems
// cannot hide and moves 16 B per key and tile pass.  Measured (us, tile-first / radix / one radix sort of
// all keys by tile and depth, which the two replaced): 500k-Gaussian room, 1 view of 3225 tiles (256k keys)
// 39 / 142 / 88; 10k cloud, 300 tiles (64k keys) 37 / 95 / 122; 4 views of a 500k room (2.5M keys)
// 198 / 268 / 287; 8 agents' rooms, 32 views (7.3M keys, 62 pairs per tile) 479 / 559 / 883; 4 views of a 1M
// room (4.9M keys, 310 pairs per tile) 376 / 373 / 529; 8 views of it (10.9M keys) 846 / 733 / 1096; 4 views
// of a 2M floor (8.0M keys, 620 pairs per tile) 1138 / 608 / 885.  So: up to 4M pairs, or as long as the lists
// are short, on average: how the pairs fall into tiles is not known here, and a view may have them all in a few (the
// sort then shares the long lists among its CTAs).  Beyond 16384 pairs per tile always the radix binning.
constexpr long long kTileFirstPairs = 4000000, kShortListPairs = 128, kMaxPairsPerTile = 16384;

int run_bin_sort(const BinArgs &a, cudaStream_t s) {
    const bool tile_first = a.P <= kMaxPairsPerTile * a.G && (a.P <= kTileFirstPairs || a.P <= kShortListPairs * a.G);
    if (a.sort_mode == GS_SORT_TILE_BUCKET || a.chunks == 0 || tile_first) return run_tile_first(a, s);
    return run_onesweep(a, s);
}

}  // namespace gs
