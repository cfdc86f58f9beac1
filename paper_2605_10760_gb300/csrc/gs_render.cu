// gs_render.cu -- per-tile compositing (forward) and its adjoint (backward).
//
// One CTA = one tile of TW x TH pixels, two vertically adjacent pixels per thread; a warp covers an
// 8 x 8 block of the tile and each quarter of it (eight lanes) a cell of 4 x 4 pixels.  Both kernels are
// persistent: a grid of (#SM x resident CTAs) claims (view, tile) work items from a device counter, so
// one launch covers every tile of every view of every scene, whatever the per-tile list lengths.
//
// Staging: a tile's list is a contiguous block of records (gs_bin_sort writes them in list order),
// so each batch of TW*TH records is one TMA bulk copy (cp.async.bulk) issued by one thread into one
// of two shared-memory buffers and completed on that buffer's mbarrier; the next batch is copied
// while the current one is processed.  All mbarrier waits are bounded (error + drain + return).
//
// Forward: each thread walks the staged records front to back for its two pixels taking the FP32
// decisions of the decision chain (sigma < 0 skip, alpha < alpha_min skip, stop before blending
// when T (1 - alpha) < t_min).  The CTA leaves the list once every pixel has stopped.  Each record
// carries a cut-off sigma_cut = ln(o / alpha_min) + 1e-3: for sigma > sigma_cut the exponential is
// not evaluated because alpha < alpha_min is certain (the decision-chain exp is within 2 ulp of
// e^x), so every decision is exactly the one the full test takes.
//
// Backward: from final_T and last_idx of each pixel the CTA walks the list back to front,
// recovering T_j = T_{j+1} / (1 - alpha_j) and one running scalar Q (the upstream-weighted colour
// and depth accumulated behind each entry, with the background and alpha-output terms), so no
// per-pixel list is stored.  Each thread sums the 10 per-Gaussian gradient components of its two
// pixels, then each quarter warp reduces them with a transposed butterfly (10 shuffles for four
// entries at once) and its lanes issue one atomic add per component.
//
// Both kernels are bound by instruction issue.  A small footprint covers a third of the 8 x 8 blocks it
// touches but most of its 4 x 4 cells, so the quarters of a warp walk their own entries: per batch each
// thread marks the cells that an entry may reach (cell_mask), a ballot per cell of the warp gives each
// quarter the bit list of its next 32 entries, and a step takes every quarter's next one.  Control flow
// is uniform per warp: a pixel that skips an entry blends alpha 0.  Measured on 8 agents x 4 views (7.3M
// list entries) against one 8 x 8 block and one entry per warp and step: forward 1515 -> 1297 us,
// backward 2322 -> 2110 us (12 % fewer instructions each); deeper forms of the same idea were slower
// (per-quarter lists over the whole batch save another tenth of the steps but cost more instructions).
//
// A thread's two pixels are the two components of packed FP32x2 arithmetic (one instruction for both
// pixels, each component rounded exactly as the scalar operation, so the decision chain is unchanged
// bit for bit); the decisions themselves are scalar compares and selects.  The forward can also
// evaluate the L1 terms of the mapping loss and their gradient in its per-pixel epilogue
// (gs_render_fwd_l1).
#include <type_traits>

#include "gs_kernels.cuh"

namespace gs {

constexpr int kPPT = 2;   // pixels per thread
constexpr int kWX = 8;    // warp block: kWX columns x (32 / kWX) * kPPT rows
constexpr int kWY = 32 / kWX * kPPT;
constexpr int kCell = 4;  // a quarter warp's pixels: kCell x kCell

// Pixel of a thread inside its tile: warp w takes block (w mod (TW / kWX), w div (TW / kWX)), and each
// quarter of the warp (eight lanes) one cell of 4 x 4 pixels of the block.
template <int TW>
__device__ __forceinline__ void thread_pixel(int tid, int &lx, int &ly) {
    const int w = tid >> 5, lane = tid & 31, q = lane >> 3;
    lx = (w % (TW / kWX)) * kWX + (q & 1) * kCell + (lane & 3);
    ly = (w / (TW / kWX)) * kWY + (q >> 1) * kCell + ((lane >> 2) & 1) * kPPT;
}

// sigma(d) = 1/2 (A dx^2 + C dy^2) + B dx dy in the decision chain's operation order (spec_sigma),
// used for the box minimum below so that its rounding error has the same bound
__device__ __forceinline__ float sigma_rn(float A, float B, float C, float dx, float dy) {
    const float q = fp::fma(fp::mul(A, dx), dx, fp::mul(fp::mul(C, dy), dy));
    return fp::fma(fp::mul(B, dx), dy, fp::mul(0.5f, q));
}

// True when the decision chain's sigma exceeds `cut` at every pixel centre of the box
// [xa, xb] x [ya, yb] (pixel centres; the mean (mx, my) and the conic (A, B, C) as recorded), so
// that every pixel of the box skips the entry.
//
// The box minimum of the convex quadratic sigma is 0 when the mean is inside the box, else it is
// attained on an edge at the 1-D minimiser clamped to that edge; s is that minimum evaluated in
// FP32.  Error bound, with u = 2^-24 and M = 1/2 (A Dx^2 + C Dy^2) + |B| Dx Dy (Dx, Dy the largest
// |offset| of the box from the mean along each axis, so M bounds the sum of the magnitudes of the
// three terms of sigma anywhere in the box):
//  * the decision chain at a pixel rounds dx and dy once (at most 2u M on sigma), forms the
//    non-negative A dx^2 + C dy^2 with three roundings (3u M) and adds B dx dy with one fused
//    rounding (u M): it is within 6u M of the exact sigma of that pixel;
//  * s rounds each candidate's edge offset once and evaluates sigma with the same sequence
//    (6u M); its minimiser, computed with an approximate reciprocal, is off by a relative
//    O(u), which raises sigma only by O(u^2) M (sigma is quadratic about the minimiser);
// so s - 12u M (up to O(u^2) M) is below the chain's sigma at every pixel of the box.  The box
// is skipped when s > cut + 0.01 + 1e-3 |cut| + 32u M: the 32u term covers the 12u bound with
// room for the rounding of M itself, and for thin footprints (conic entries of 1e4 and more,
// where B dx dy cancels most of the other two terms) it is what keeps the skip exact.  Non-finite
// or non-positive-definite input never skips.
__device__ __forceinline__ bool box_skips(float A, float B, float C, float mx, float my, float xa, float xb,
                                          float ya, float yb, float cut) {
    if (!(A > 0.f && C > 0.f && A < 1e30f && C < 1e30f && fabsf(B) < 1e30f && fabsf(mx) < 1e30f &&
          fabsf(my) < 1e30f && fabsf(cut) < 1e30f))
        return false;
    const float dxa = xa - mx, dxb = xb - mx, dya = ya - my, dyb = yb - my;
    if (dxa <= 0.f && dxb >= 0.f && dya <= 0.f && dyb >= 0.f) return false;
    const float iA = __fdividef(1.f, A), iC = __fdividef(1.f, C);
    float best = 3.0e38f;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float dx = e ? dxb : dxa;
        const float dy = fminf(fmaxf(-B * dx * iC, dya), dyb);
        best = fminf(best, sigma_rn(A, B, C, dx, dy));
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float dy = e ? dyb : dya;
        const float dx = fminf(fmaxf(-B * dy * iA, dxa), dxb);
        best = fminf(best, sigma_rn(A, B, C, dx, dy));
    }
    const float Dx = fmaxf(fabsf(dxa), fabsf(dxb)), Dy = fmaxf(fabsf(dya), fabsf(dyb));
    const float M = 0.5f * (A * Dx * Dx + C * Dy * Dy) + fabsf(B) * Dx * Dy;
    const float thr = cut + 0.01f + 1e-3f * fabsf(cut) + 0x1p-19f * M;
    return best > thr;   // false for a NaN or infinite threshold
}

__device__ __forceinline__ float sqrt_approx(float x) {   // (relative error about 2^-23)
    float y;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Bit r (TW / 4) + c set <=> the cell of 4 x 4 pixels in row r and column c of the tile may blend the
// entry.  A cleared bit means the decision chain's sigma exceeds the cut at every pixel of the cell, so
// that a quarter warp may skip the entry without evaluating it.
//
// Where sigma stays below a level the pixels form an ellipse, whose part in a band of pixel rows covers one
// interval of x: in offsets from the mean, the right end (-B dy + sqrt(2 A level - det dy^2)) / A at the
// dy of the ellipse's rightmost point, clamped to the band; the left end likewise.  Four rows of cells are
// four bands, and each interval gives its row's columns at once.  The level is the cut raised by
// box_skips' margin 0.01 + 1e-3 |cut| + 32u M with M taken over the whole tile, which bounds the rounding
// of the chain's sigma at any pixel; the ends are widened by 0.05 + 1e-3 of their distance from the mean,
// far above their own rounding while det keeps three digits (det > 1e-3 A C; det's error is below 2u A C).
// More elongated footprints take box_skips per block of four cells.  Non-finite or non-positive-definite
// input never skips; a negative cut (alpha < alpha_min even at the mean) always does.
template <int TW, int TH>
__device__ __forceinline__ uint32_t cell_mask(const float4 &r0, const float4 &r1, float cut, int tile_x0, int tile_y0) {
    constexpr int NC = TW / kCell, NR = TH / kCell;
    static_assert(NC * NR <= 32 && NC <= 8, "a bit per cell");
    constexpr uint32_t kAll = NC * NR == 32 ? 0xffffffffu : (1u << (NC * NR)) - 1u;
    const float A = r0.z, B = r0.w, C = r1.x, mx = r0.x, my = r0.y;
    if (cut < 0.f) return 0u;
    if (!(A > 0.f && C > 0.f && A < 1e30f && C < 1e30f && fabsf(B) < 1e30f && fabsf(mx) < 1e30f && fabsf(my) < 1e30f &&
          cut < 1e30f))
        return kAll;
    const float xo = (float)tile_x0 - mx, yo = (float)tile_y0 - my;      // tile corner, from the mean
    const float det = A * C - B * B;
    if (!(det > 1e-3f * A * C)) {
        uint32_t m = 0;
#pragma unroll 1
        for (int w = 0; w < NC * NR / 4; ++w) {
            const int bx = w % (TW / kWX), by = w / (TW / kWX);
            const float xa = (float)(tile_x0 + bx * kWX) + 0.5f, ya = (float)(tile_y0 + by * kWY) + 0.5f;
            if (!box_skips(A, B, C, mx, my, xa, xa + (float)(kWX - 1), ya, ya + (float)(kWY - 1), cut))
                m |= ((3u << (2 * bx)) * (1u | (1u << NC))) << (2 * by * NC);
        }
        return m;
    }
    const float Dx = fmaxf(fabsf(xo), fabsf(xo + (float)TW)), Dy = fmaxf(fabsf(yo), fabsf(yo + (float)TH));
    const float M = 0.5f * (A * Dx * Dx + C * Dy * Dy) + fabsf(B) * Dx * Dy;
    const float lev2 = 2.0f * (cut + 0.01f + 1e-3f * cut + 0x1p-19f * M);
    const float irt = rsqrtf(det), iA = __fdividef(1.0f, A);
    const float ym = sqrt_approx(lev2 * A) * irt;                             // the ellipse's extent in y
    const float dyr = -B * sqrt_approx(__fdividef(lev2, C)) * irt;            // row of its rightmost point
    const float yr = ym * 1.001f + 0.05f;
    if (!(yr < 1e30f)) return kAll;
    uint32_t m = 0;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const float ya = yo + ((float)(r * kCell) + 0.5f), yb = ya + (float)(kCell - 1);
        if (ya > yr || yb < -yr) continue;
        const float tr = fminf(fmaxf(dyr, ya), yb), tl = fminf(fmaxf(-dyr, ya), yb);
        float xr = (sqrt_approx(fmaxf(lev2 * A - det * tr * tr, 0.f)) - B * tr) * iA;
        float xl = (-sqrt_approx(fmaxf(lev2 * A - det * tl * tl, 0.f)) - B * tl) * iA;
        xr += 0.05f + 1e-3f * fabsf(xr);
        xl -= 0.05f + 1e-3f * fabsf(xl);
        // columns c with xo + 4 c + 0.5 <= xr and xo + 4 c + 3.5 >= xl
        const int c1 = (int)fminf(fmaxf(floorf((xr - xo - 0.5f) * 0.25f), -1.f), (float)(NC - 1));
        const int c0 = (int)fminf(fmaxf(ceilf((xl - xo - 3.5f) * 0.25f), 0.f), (float)NC);
        m |= (((1u << (c1 + 1)) - 1u) & ~((1u << c0) - 1u)) << (r * NC);   // (none where c1 < c0)
    }
    return m;
}

// Bit of the first cell of warp w's block; the quarters' cells are at + 0, + 1, + NC, + NC + 1.
template <int TW>
__device__ __forceinline__ uint32_t first_cell(int w) {
    return (uint32_t)((w / (TW / kWX)) * 2 * (TW / kCell) + (w % (TW / kWX)) * 2);
}
// The entries (of 32, cell mask m each) that this lane's quarter visits.
template <int TW>
__device__ __forceinline__ uint32_t quarter_bits(uint32_t m, uint32_t cell0, int lane) {
    m >>= cell0;
    const uint32_t b0 = __ballot_sync(0xffffffffu, m & 1u), b1 = __ballot_sync(0xffffffffu, m & 2u);
    const uint32_t b2 = __ballot_sync(0xffffffffu, m & (1u << (TW / kCell))), b3 = __ballot_sync(0xffffffffu, m & (2u << (TW / kCell)));
    return lane & 16 ? (lane & 8 ? b3 : b2) : (lane & 8 ? b1 : b0);
}

constexpr unsigned long long kTmaWaitLimit = 1ull << 22;   // polls of a batch's mbarrier before giving up

// Next work item of a persistent compositing CTA (thread 0), -1 when all are taken.  Every CTA
// makes exactly one claim past the last item; the CTA that draws the last of those (every other
// claim of the launch is made by then) returns the counter to zero for the next launch.  Class
// lists inconsistent with G (only after an earlier binning failure) record a device fault; the
// claim then falls back to the counter's own value.
__device__ __forceinline__ long long claim_item(DevStatus *st, uint32_t *ctr, const uint32_t *coff,
                                                const uint32_t *clist, long long G) {
    const long long c = (long long)atomicAdd(ctr, 1u);
    const long long total = min((long long)coff[kClaimClasses], G);
    if (c >= total) {
        if (c == total + (long long)gridDim.x - 1) *ctr = 0u;
        return -1;
    }
    const long long g = claim_at(coff, clist, G, c);
    if (g >= G) {
        record_error(st, GS_ERR_DEVICE_FAULT, 10);
        return c;
    }
    return g;
}

// A CTA leaving early (after a failed wait, an error already recorded) claims until it draws a
// value past the items, skipping the items it draws, so that every CTA still makes exactly one
// claim past them and the launch's last claim returns the counter to zero.
__device__ __forceinline__ void claim_exit(uint32_t *ctr, const uint32_t *coff, long long G) {
    if (threadIdx.x == 0) {
        const long long total = min((long long)coff[kClaimClasses], G);
        long long c;
        do {
            c = (long long)atomicAdd(ctr, 1u);
        } while (c < total);
        if (c == total + (long long)gridDim.x - 1) *ctr = 0u;
    }
}

// Shared memory of one render CTA: two batches of records (double buffer filled by TMA), the
// per-entry cell masks of each batch, one mbarrier per buffer.
// NB records per staged batch: 64, 128 or 256, at most one per pixel of the tile (two buffers of
// 256 records take 24 KB)
template <int NB>
struct __align__(128) RenderSmem {
    float4 rec[2][3 * NB];
    uint32_t mask[NB];                  // cell_mask of each entry of the batch being walked
    uint64_t bar[2];
    long long item;
    int maxlast;
    uint32_t coff[kClaimClasses + 1];   // claim-class offsets (claim_offsets)
};

// Waits for both buffers' outstanding copies (bounded) after a failed wait, so that the CTA never
// leaves with a copy still targeting its shared memory unless that copy is itself stuck.
template <int NB>
__device__ __forceinline__ void drain_after_timeout(RenderSmem<NB> &sm, const uint32_t (&parity)[2],
                                                    const bool (&pending)[2], DevStatus *st) {
    if (threadIdx.x == 0) {
        record_error(st, GS_ERR_TIMEOUT, 8);
        for (int bb = 0; bb < 2; ++bb)
            if (pending[bb]) mbar_wait_bounded(&sm.bar[bb], parity[bb], kTmaWaitLimit);
    }
    __syncthreads();
}

// Resident CTAs per SM (32 warps of 64 registers when whole batches are staged, else 40 of 48): with short
// lists the chain of claim, range, copy and masks of the next tile is hidden by more warps, with long
// ones the walk itself runs faster with more registers.
template <int TW, int TH, int NB>
constexpr bool kWide = NB >= 256 || NB >= TW * TH;
template <int TW, int TH, int NB>
constexpr int kResident = (kWide<TW, TH, NB> ? 2048 : 2560) / (TW * TH);

// The walks blend a pixel that skips an entry with weight 0 instead of branching around it, which leaves its sums as
// they are only while the entry's colour and depth and the pixel's upstream gradient are tame: 0 x NaN is NaN, and a
// lane whose quarter has no entry left reads another entry of the batch.  The projection gives other entries an
// infinite cut-off, and their batches (and, in the backward, those of a tile with other gradients) take the SLOW
// walk, in which a pixel's sums meet only the entries that it blends.  The backward of short lists looks at gradients and
// sums once a batch: a flag kept through the walk cost it 1 % (32 views, 7.3M list entries: 2119 for 2093 us).  That of
// long lists keeps the flag, and a tile stays with the SLOW walk once an entry has asked for it (8 views, 10.7M: 2247 us
// with a look per batch, 2236 with a look after each SLOW walk, 2212 so, 2203 without any of this).
__device__ __forceinline__ float2 select2(bool x, bool y, float2 a, float2 b) {
    return make_float2(x ? a.x : b.x, y ? a.y : b.y);
}

// Cell masks of a staged batch; true where this thread saw an entry for the SLOW walk: a cut-off beyond
// spec_exp_neg's range.
template <int TW, int TH, int NB>
__device__ __forceinline__ bool stage_masks(const float4 *rec, uint32_t *mask, int cnt, int x0, int y0) {
    bool slow = false;
    for (int e = threadIdx.x; e < cnt; e += TW * TH / kPPT) {
        const float4 r0 = rec[3 * e], r1 = rec[3 * e + 1];
        const float cut = rec[3 * e + 2].w;
        mask[e] = cell_mask<TW, TH>(r0, r1, cut, x0, y0);
        slow |= !(cut < kFastCut);
    }
    return slow;
}

template <int TW, int TH, int NB>
__global__ void __launch_bounds__(TW *TH / kPPT, kResident<TW, TH, NB>) k_render_fwd(FwdArgs a) {
    static_assert(NB <= TW * TH, "at most one staged record per pixel of the tile");
    constexpr int NT = TW * TH / kPPT;            // threads
    __shared__ RenderSmem<NB> sm;
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t cell0 = first_cell<TW>(tid >> 5);
    const long long tpv = (long long)a.Tx * a.Ty;
    const long long HW = (long long)a.W * a.H;
    int lx, ly;
    thread_pixel<TW>(tid, lx, ly);
    if (tid == 0) {
        mbar_init(&sm.bar[0], 1);
        mbar_init(&sm.bar[1], 1);
        fence_proxy_async_smem();
    }
    claim_offsets(a.st, sm.coff);
    __syncthreads();
    uint32_t parity[2] = {0u, 0u};
    unsigned long long pairs = 0;
    // per-thread sums of |rendered - target| (L1 epilogue): a tile's terms in FP32, added to a pair of floats so
    // that the total does not depend on how many tiles a thread has seen
    float2 l1_rgb = make_float2(0.f, 0.f), l1_d = make_float2(0.f, 0.f);
    for (;;) {
        if (tid == 0) sm.item = claim_item(a.st, &a.st->fwd_items, sm.coff, a.clist, a.G);
        __syncthreads();
        const long long g = sm.item;
        if (g < 0) break;
        const int v = (int)(g / tpv);
        const int tl = (int)(g - (long long)v * tpv);
        const int ty = tl / a.Tx, tx = tl - ty * a.Tx;
        const int x = tx * TW + lx, y0 = ty * TH + ly;
        const uint32_t start = a.ranges[2 * g], end = a.ranges[2 * g + 1];
        // the tile's list must lie inside the records (its batches are copied by TMA)
        const int n = gs_guard(a.st, end >= start && (long long)end <= a.cap, 10) ? (int)(end - start) : 0;
        // per-pixel state of the thread's two pixels, packed (component p = pixel p)
        static_assert(kPPT == 2, "two pixels per thread, one per packed component");
        bool done[kPPT];
        int last[kPPT];
        float2 T = fp2::splat(1.0f), C0 = fp2::splat(0.f), C1 = fp2::splat(0.f), C2 = fp2::splat(0.f),
               D = fp2::splat(0.f);
        const float px = (float)x + 0.5f;
        float2 py = make_float2((float)y0 + 0.5f, (float)(y0 + 1) + 0.5f);
        const float kNaN = __int_as_float(0x7fffffff);   // row of a pixel that is done: its sigma is NaN
#pragma unroll
        for (int p = 0; p < kPPT; ++p) {
            done[p] = !(x < a.W && y0 + p < a.H);
            last[p] = 0;
            pairs += done[p] ? 0ull : (unsigned long long)n;   // entries visited by the pixel: all, until it stops
        }
        if (done[0]) py.x = kNaN;
        if (done[1]) py.y = kNaN;
        // every pixel of the lane's quarter / of the warp is done
        uint32_t bdone = __ballot_sync(0xffffffffu, done[0] && done[1]);
        bool qdone = ((bdone >> (lane & 24)) & 255u) == 255u;
        // one batch's entries, front to back; SLOW: see stage_masks
        auto walk = [&](auto is_slow, const float4 *rec, const uint32_t *msk, int b, int cnt) {
            constexpr bool SLOW = decltype(is_slow)::value;
            for (int k0 = 0; k0 < cnt; k0 += 32) {
                const int kk = k0 + lane;
                uint32_t bits = quarter_bits<TW>(kk < cnt ? msk[kk] : 0u, cell0, lane);
                if (qdone) bits = 0u;
                // the quarters walk their own entries side by side, as many steps as the longest of them has
                for (int left = __reduce_max_sync(0xffffffffu, __popc(bits)); left > 0; --left) {
                    const bool has = bits != 0u;
                    const int k = has ? k0 + __ffs(bits) - 1 : k0;
                    bits &= bits - 1u;
                    const float4 r0 = rec[3 * k], r1 = rec[3 * k + 1], r2 = rec[3 * k + 2];
                    const float cut = r2.w;
                    const float dx = fp::sub(px, r0.x);
                    const float2 sg = spec_sigma2(r0.z, r0.w, r1.x, dx, fp2::add(py, fp2::splat(-r0.y)));
                    bool ev0, ev1;
                    float2 e;
                    if (SLOW) {
                        ev0 = has && !done[0] && !(sg.x < 0.0f) && !(sg.x > cut);
                        ev1 = has && !done[1] && !(sg.y < 0.0f) && !(sg.y > cut);
                        e = spec_expf2(fp2::neg(sg));
                    } else {
                        // 0 <= sigma <= cut as one unsigned compare of the bits: negative and NaN are larger
                        // (cut >= 0: cell_mask drops the other entries)
                        const uint32_t lim = has ? __float_as_uint(cut) + 1u : 0u;
                        ev0 = __float_as_uint(sg.x) < lim;
                        ev1 = __float_as_uint(sg.y) < lim;
                        e = spec_exp_neg(sg);
                    }
                    const float2 ar = fp2::mul(fp2::splat(r1.y), e);
                    float2 al = make_float2(fminf(a.amax, ar.x), fminf(a.amax, ar.y));
                    // both pixels of every lane without branches: a pixel that skips the entry blends alpha 0,
                    // which leaves its transmittance (T x 1) and its sums as they are
                    bool bl0 = ev0 && !(al.x < a.amin), bl1 = ev1 && !(al.y < a.amin);
                    al = make_float2(bl0 ? al.x : 0.f, bl1 ? al.y : 0.f);
                    float2 Tn = fp2::mul(T, fp2::add(fp2::splat(1.0f), fp2::neg(al)));
                    float2 w = fp2::mul(al, T);
                    if (__any_sync(0xffffffffu, Tn.x < a.tmin || Tn.y < a.tmin)) {
                        // a pixel stops before blending (T >= t_min until then)
                        if (Tn.x < a.tmin) {
                            bl0 = false;
                            done[0] = true;
                            pairs -= (unsigned long long)(n - (b + k + 1));
                            py.x = kNaN;
                            Tn.x = T.x;
                            w.x = 0.f;
                        }
                        if (Tn.y < a.tmin) {
                            bl1 = false;
                            done[1] = true;
                            pairs -= (unsigned long long)(n - (b + k + 1));
                            py.y = kNaN;
                            Tn.y = T.y;
                            w.y = 0.f;
                        }
                        bdone = __ballot_sync(0xffffffffu, done[0] && done[1]);
                        qdone = ((bdone >> (lane & 24)) & 255u) == 255u;
                        if (qdone) bits = 0u;
                        if (bdone == 0xffffffffu) left = 1;   // every pixel of the warp
                    }
                    float2 c0 = fp2::splat(r2.x), c1 = fp2::splat(r2.y), c2 = fp2::splat(r2.z), z = fp2::splat(r1.z);
                    if (SLOW) {
                        const float2 zero = fp2::splat(0.f);
                        c0 = select2(bl0, bl1, c0, zero);
                        c1 = select2(bl0, bl1, c1, zero);
                        c2 = select2(bl0, bl1, c2, zero);
                        z = select2(bl0, bl1, z, zero);
                    }
                    C0 = fp2::fma(c0, w, C0);
                    C1 = fp2::fma(c1, w, C1);
                    C2 = fp2::fma(c2, w, C2);
                    D = fp2::fma(z, w, D);
                    T = Tn;
                    last[0] = bl0 ? b + k + 1 : last[0];
                    last[1] = bl1 ? b + k + 1 : last[1];
                }
                if (bdone == 0xffffffffu) break;
            }
        };
        const int nb = (n + NB - 1) / NB;
        auto issue = [&](int bi, int bb) {     // thread 0: batch bi of this tile into buffer bb
            const int b = bi * NB;
            fence_proxy_async_smem();
            tma_load_1d(&sm.rec[bb][0], a.srec + 3 * (size_t)(start + b), (uint32_t)min(NB, n - b) * 48u,
                        &sm.bar[bb]);
        };
        if (tid == 0 && nb > 0) issue(0, 0);
        int buf = 0;
        for (int bi = 0; bi < nb; ++bi) {
            const int b = bi * NB, cnt = min(NB, n - b);
            if (tid == 0 && bi + 1 < nb) issue(bi + 1, buf ^ 1);
            const bool ok = mbar_wait_bounded(&sm.bar[buf], parity[buf], kTmaWaitLimit);
            if (__syncthreads_or(!ok)) {
                const bool pending[2] = {buf == 0 || bi + 1 < nb, buf == 1 || bi + 1 < nb};
                drain_after_timeout(sm, parity, pending, a.st);
                claim_exit(&a.st->fwd_items, sm.coff, a.G);
                return;
            }
            parity[buf] ^= 1u;
            const float4 *rec = sm.rec[buf];
            const bool slow = __syncthreads_or(stage_masks<TW, TH, NB>(rec, sm.mask, cnt, tx * TW, ty * TH));
            if (bdone != 0xffffffffu) {
                if (slow) walk(std::true_type(), rec, sm.mask, b, cnt);
                else walk(std::false_type(), rec, sm.mask, b, cnt);
            }
            const bool all_done = __syncthreads_and(bdone == 0xffffffffu);   // also: buffer reads finished
            if (all_done) {
                if (bi + 1 < nb) {   // the prefetched batch must land before its buffer is reused
                    const bool ok2 = mbar_wait_bounded(&sm.bar[buf ^ 1], parity[buf ^ 1], kTmaWaitLimit);
                    if (__syncthreads_or(!ok2)) {
                        const bool pending[2] = {buf == 1, buf == 0};
                        drain_after_timeout(sm, parity, pending, a.st);
                        claim_exit(&a.st->fwd_items, sm.coff, a.G);
                        return;
                    }
                    parity[buf ^ 1] ^= 1u;
                }
                break;
            }
            buf ^= 1;
        }
        float t_rgb = 0.f, t_d = 0.f;
#pragma unroll
        for (int p = 0; p < kPPT; ++p) {
            if (x < a.W && y0 + p < a.H) {
                const long long pix = (long long)(y0 + p) * a.W + x;
                const float Tp = p ? T.y : T.x, Dp = p ? D.y : D.x;
                const float c[3] = {(p ? C0.y : C0.x) + Tp * a.bg0, (p ? C1.y : C1.x) + Tp * a.bg1,
                                    (p ? C2.y : C2.x) + Tp * a.bg2};
                if (a.rgb) {
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) a.rgb[(3 * (long long)v + ch) * HW + pix] = c[ch];
                }
                if (a.depth) a.depth[(long long)v * HW + pix] = Dp;
                if (a.alpha) a.alpha[(long long)v * HW + pix] = 1.0f - Tp;
                a.finalT[(long long)v * HW + pix] = Tp;
                a.last[(long long)v * HW + pix] = last[p];
                if (a.rgb_t) {   // L1 terms and their gradient, as gs_loss_l1 computes them
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) {
                        const long long idx = (3 * (long long)v + ch) * HW + pix;
                        const float d = c[ch] - a.rgb_t[idx];
                        t_rgb += fabsf(d);
                        a.d_rgb[idx] = (d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f)) * a.sc_rgb;
                    }
                    if (a.depth_t) {
                        const long long idx = (long long)v * HW + pix;
                        const float d = Dp - a.depth_t[idx];
                        t_d += fabsf(d);
                        a.d_depth[idx] = (d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f)) * a.sc_d;
                    }
                }
            }
        }
        if (a.rgb_t) {
            add_to_pair(l1_rgb, t_rgb);
            add_to_pair(l1_d, t_d);
        }
        __syncthreads();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
    if ((tid & 31) == 0 && pairs) atomicAdd(&a.st->fwd_pairs, pairs);
    if (a.rgb_t) {   // one double atomic per warp for the loss
        double l = pair_value(l1_rgb) * a.sc_rgb + pair_value(l1_d) * a.sc_d;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if ((tid & 31) == 0 && l != 0.0) atomicAdd(a.loss, l);
    }
}

// Transposed butterfly over the eight lanes of a quarter warp: v[0 .. 9] are the lane's terms of the 10
// gradient components; afterwards v[0] is the quarter's sum of component b0 + 3 b1 + 5 b2 (b_k = bit k of
// the lane) and v[2] that of component 2 + 5 b2.  10 shuffles.
__device__ __forceinline__ void quarter_transpose_reduce(float (&v)[10], int lane) {
    {
        const bool up = lane & 4;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const float send = up ? v[i] : v[i + 5], keep = up ? v[i + 5] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
        }
    }
    {
        const bool up = lane & 2;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float send = up ? v[i] : v[i + 3], keep = up ? v[i + 3] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
        }
        v[2] += __shfl_xor_sync(0xffffffffu, v[2], 2);
    }
    {
        const bool up = lane & 1;
        const float send = up ? v[0] : v[1], keep = up ? v[1] : v[0];
        v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
        v[2] += __shfl_xor_sync(0xffffffffu, v[2], 1);
    }
}

// the gradient components, in the order of the grad2d record
enum : int { kGMx, kGMy, kGA, kGB, kGC, kGO, kGZ, kGR, kGG, kGBl };

template <int TW, int TH, int NB>
__global__ void __launch_bounds__(TW *TH / kPPT, kResident<TW, TH, NB>) k_render_bwd(BwdArgs a) {
    static_assert(NB <= TW * TH, "at most one staged record per pixel of the tile");
    constexpr int NT = TW * TH / kPPT;
    __shared__ RenderSmem<NB> sm;
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t cell0 = first_cell<TW>(tid >> 5);
    const int comp0 = (lane & 1) + 3 * ((lane >> 1) & 1) + 5 * ((lane >> 2) & 1);   // components this lane adds to grad2d
    const int comp2 = 2 + 5 * ((lane >> 2) & 1);                                    // (comp2: lanes 0 and 4 of a quarter)
    const long long tpv = (long long)a.Tx * a.Ty;
    const long long HW = (long long)a.W * a.H;
    int lx, ly;
    thread_pixel<TW>(tid, lx, ly);
    if (tid == 0) {
        mbar_init(&sm.bar[0], 1);
        mbar_init(&sm.bar[1], 1);
        fence_proxy_async_smem();
    }
    claim_offsets(a.st, sm.coff);
    __syncthreads();
    uint32_t parity[2] = {0u, 0u};
    unsigned long long pairs = 0;
    for (;;) {
        if (tid == 0) {
            sm.item = claim_item(a.st, &a.st->bwd_items, sm.coff, a.clist, a.G);
            sm.maxlast = 0;
        }
        __syncthreads();
        const long long g = sm.item;
        if (g < 0) break;
        const int v = (int)(g / tpv);
        const int tl = (int)(g - (long long)v * tpv);
        const int ty = tl / a.Tx, tx = tl - ty * a.Tx;
        const int x = tx * TW + lx, y0 = ty * TH + ly;
        const uint32_t start = a.ranges[2 * g], end = a.ranges[2 * g + 1];
        const int n = gs_guard(a.st, end >= start && (long long)end <= a.cap, 11) ? (int)(end - start) : 0;
        const float px = (float)x + 0.5f;
        // per-pixel state of the thread's two pixels, packed (component p = pixel p)
        static_assert(kPPT == 2, "two pixels per thread, one per packed component");
        int lst[kPPT];
        float tT[kPPT], tQ[kPPT], tC0[kPPT], tC1[kPPT], tC2[kPPT], tD[kPPT];
        int tmax = 0;
#pragma unroll
        for (int p = 0; p < kPPT; ++p) {
            lst[p] = 0;
            tT[p] = 1.0f;
            tC0[p] = tC1[p] = tC2[p] = tD[p] = 0.f;
            float gA = 0.f;
            if (x < a.W && y0 + p < a.H) {
                const long long pix = (long long)(y0 + p) * a.W + x;
                lst[p] = min(max(a.last[(long long)v * HW + pix], 0), n);   // never past the list
                tT[p] = a.finalT[(long long)v * HW + pix];
                if (a.d_rgb) {
                    tC0[p] = a.d_rgb[(3 * (long long)v + 0) * HW + pix];
                    tC1[p] = a.d_rgb[(3 * (long long)v + 1) * HW + pix];
                    tC2[p] = a.d_rgb[(3 * (long long)v + 2) * HW + pix];
                }
                if (a.d_depth) tD[p] = a.d_depth[(long long)v * HW + pix];
                if (a.d_alpha) gA = a.d_alpha[(long long)v * HW + pix];
            }
            // rgb = sum c alpha T + T_final bg, alpha_out = 1 - T_final
            tQ[p] = tT[p] * (tC0[p] * a.bg0 + tC1[p] * a.bg1 + tC2[p] * a.bg2 - gA);
            pairs += (unsigned long long)lst[p];
            tmax = max(tmax, lst[p]);
        }
        // Q = sum over blended entries behind the current one of (gC . c + gD z) alpha T, plus the
        // background and alpha-output terms: dL/dalpha_j = T_j (gC . c_j + gD z_j) - Q / (1 - alpha_j)
        float2 T = make_float2(tT[0], tT[1]), Q = make_float2(tQ[0], tQ[1]);
        const float2 gC0 = make_float2(tC0[0], tC0[1]), gC1 = make_float2(tC1[0], tC1[1]),
                     gC2 = make_float2(tC2[0], tC2[1]), gD = make_float2(tD[0], tD[1]);
        const float2 py = make_float2((float)y0 + 0.5f, (float)(y0 + 1) + 0.5f);
        const int wmax = __reduce_max_sync(0xffffffffu, tmax);
        if (lane == 0) atomicMax(&sm.maxlast, wmax);
        // (kWide) an upstream gradient of this thread is not tame; from the first batch on, of the tile, or an entry
        // so far asked for the SLOW walk (which may have spoilt a sum)
        bool slow = kWide<TW, TH, NB> && !(tame(tC0[0], tC1[0], tC2[0], tD[0]) && tame(tC0[1], tC1[1], tC2[1], tD[1]) &&
                                           tame(tQ[0], tQ[1], 0.f, 0.f));
        // the quarter's largest last index
        int qmax = tmax;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) qmax = max(qmax, __shfl_xor_sync(0xffffffffu, qmax, o));
        // one batch's entries (positions lo on), back to front; SLOW: see stage_masks
        auto walk = [&](auto is_slow, const float4 *rec, const uint32_t *msk, int lo, int kend) {
            constexpr bool SLOW = decltype(is_slow)::value;
            for (int k0 = ((kend - 1) >> 5) << 5; k0 >= 0 && kend > 0; k0 -= 32) {
                const int kk = k0 + lane;
                uint32_t bits = quarter_bits<TW>(kk < kend ? msk[kk] : 0u, cell0, lane);
                // entries at or beyond the quarter's largest last index contribute nothing to it
                const int over = qmax - lo - k0;
                if (over < 32) bits &= over > 0 ? (1u << over) - 1u : 0u;
                // the quarters walk their own entries side by side, as many steps as the longest of them has
                for (int left = __reduce_max_sync(0xffffffffu, __popc(bits)); left > 0; --left) {
                    const bool has = bits != 0u;
                    const int kb = has ? 31 - __clz(bits) : 0, k = k0 + kb;
                    bits &= ~(1u << kb);
                    const int pos = lo + k;
                    const float4 r0 = rec[3 * k], r1 = rec[3 * k + 1], r2 = rec[3 * k + 2];
                    const float cut = r2.w;
                    const float dx = fp::sub(px, r0.x);
                    const float2 dy = fp2::add(py, fp2::splat(-r0.y));
                    const float2 sg = spec_sigma2(r0.z, r0.w, r1.x, dx, dy);
                    bool ev0, ev1;
                    float2 e;
                    if (SLOW) {
                        ev0 = has && pos < lst[0] && !(sg.x < 0.0f) && !(sg.x > cut);
                        ev1 = has && pos < lst[1] && !(sg.y < 0.0f) && !(sg.y > cut);
                        e = spec_expf2(fp2::neg(sg));
                    } else {
                        // 0 <= sigma <= cut as one unsigned compare of the bits: negative and NaN are larger
                        // (cut >= 0: cell_mask drops the other entries)
                        const uint32_t lim = has ? __float_as_uint(cut) + 1u : 0u;
                        ev0 = pos < lst[0] && __float_as_uint(sg.x) < lim;
                        ev1 = pos < lst[1] && __float_as_uint(sg.y) < lim;
                        e = spec_exp_neg(sg);
                    }
                    const float2 araw = fp2::mul(fp2::splat(r1.y), e);
                    float2 al = make_float2(fminf(a.amax, araw.x), fminf(a.amax, araw.y));
                    // both pixels of every lane without branches; a pixel that does not blend the entry takes
                    // alpha 0 and contributes zero
                    const bool bl0 = ev0 && !(al.x < a.amin), bl1 = ev1 && !(al.y < a.amin);
                    const uint32_t contrib = __ballot_sync(0xffffffffu, bl0 || bl1);
                    if (contrib == 0u) continue;
                    al = make_float2(bl0 ? al.x : 0.f, bl1 ? al.y : 0.f);
                    const float2 oma = fp2::add(fp2::splat(1.0f), fp2::neg(al));
                    const float2 ioma = make_float2(__fdividef(1.0f, oma.x), __fdividef(1.0f, oma.y));
                    const float2 Tj = fp2::mul(T, ioma);
                    const float2 w = fp2::mul(al, Tj);
                    const float2 Pj = fp2::fma(gD, fp2::splat(r1.z),
                                               fp2::fma(gC2, fp2::splat(r2.z),
                                                        fp2::fma(gC1, fp2::splat(r2.y), fp2::mul(gC0, fp2::splat(r2.x)))));
                    float2 dLda = fp2::fma(Tj, Pj, fp2::neg(fp2::mul(Q, ioma)));
                    if (SLOW) {
                        dLda = select2(bl0, bl1, dLda, fp2::splat(0.f));
                        Q = select2(bl0, bl1, fp2::fma(Pj, w, Q), Q);
                    } else {
                        Q = fp2::fma(Pj, w, Q);
                    }
                    T = make_float2(bl0 ? Tj.x : T.x, bl1 ? Tj.y : T.y);
                    float gv[10];
                    float2 cR = fp2::mul(gC0, w), cG = fp2::mul(gC1, w), cB = fp2::mul(gC2, w), cZ = fp2::mul(gD, w);
                    if (SLOW) {
                        const float2 zero = fp2::splat(0.f);
                        cR = select2(bl0, bl1, cR, zero);
                        cG = select2(bl0, bl1, cG, zero);
                        cB = select2(bl0, bl1, cB, zero);
                        cZ = select2(bl0, bl1, cZ, zero);
                    }
                    gv[kGR] = cR.x + cR.y;
                    gv[kGG] = cG.x + cG.y;
                    gv[kGBl] = cB.x + cB.y;
                    gv[kGZ] = cZ.x + cZ.y;
                    // dL/dsigma per pixel (a capped alpha has no gradient with respect to opacity and sigma); the
                    // conic and mean gradients are sums over the two pixels of dL/dsigma times 1/2 dx^2, dx dy,
                    // 1/2 dy^2 and -(A dx + B dy), -(B dx + C dy): dx is the pair's, so only s0 = sum dL/dsigma,
                    // s1 = sum dL/dsigma dy and s2 = sum dL/dsigma dy^2 need both pixels
                    const bool un0 = araw.x <= a.amax, un1 = araw.y <= a.amax;
                    float2 dLds = fp2::mul(dLda, make_float2(un0 ? -al.x : 0.f, un1 ? -al.y : 0.f));
                    if (SLOW) dLds = select2(un0, un1, dLds, fp2::splat(0.f));
                    const float2 t1 = fp2::mul(dLds, dy);
                    const float2 t2 = fp2::mul(t1, dy);
                    const float s0 = dLds.x + dLds.y, s1 = t1.x + t1.y, s2 = t2.x + t2.y;
                    const float s0dx = s0 * dx;
                    gv[kGA] = 0.5f * s0dx * dx;
                    gv[kGB] = s1 * dx;
                    gv[kGC] = 0.5f * s2;
                    gv[kGMx] = -(r0.z * s0dx + r0.w * s1);
                    gv[kGMy] = -(r0.w * s0dx + r1.x * s1);
                    // dL/do = sum of dL/dalpha e = -(sum of dL/dsigma) / o, divided once after the reduction (o is
                    // at least alpha_min for a blended entry); with alpha_min = 0 (SLOW) an opacity of 0 blends
                    // too, and the sum itself is taken
                    gv[kGO] = s0;
                    if (SLOW) {
                        const float2 oe = fp2::mul(dLda, e);
                        gv[kGO] = (bl0 && un0 ? oe.x : 0.f) + (bl1 && un1 ? oe.y : 0.f);
                    }
                    quarter_transpose_reduce(gv, lane);
                    bool add = ((contrib >> (lane & 24)) & 255u) != 0u;
                    if constexpr (kWide<TW, TH, NB>) {
                        // a footprint that covers the block is every quarter's next entry at once: one sum for the
                        // warp, so that the many additions to a large footprint's gradient (and their rounding)
                        // are a quarter.  With short lists of small footprints the test alone costs 7 %.
                        const int klead = __shfl_sync(0xffffffffu, k, 0);
                        if (__all_sync(0xffffffffu, has && k == klead)) {
#pragma unroll
                            for (int o = 8; o <= 16; o <<= 1) {
                                gv[0] += __shfl_xor_sync(0xffffffffu, gv[0], o);
                                gv[2] += __shfl_xor_sync(0xffffffffu, gv[2], o);
                            }
                            add = lane < 8;
                        }
                    }
                    if (!SLOW && comp0 == kGO) gv[0] = __fdividef(gv[0], -r1.y);
                    const uint32_t sl = __float_as_uint(r1.w);   // the record's slot in g2d
                    if (add && gs_guard(a.st, (long long)sl < a.P, 12)) {
                        float *dst = a.g2d + 12 * (size_t)sl;
                        atomicAdd(dst + comp0, gv[0]);
                        if ((lane & 3) == 0) atomicAdd(dst + comp2, gv[2]);
                    }
                }
            }
        };
        __syncthreads();
        const int maxl = sm.maxlast;
        const int nb = (maxl + NB - 1) / NB;   // batches, back to front: [max(0, maxl-(bi+1)NB), maxl-bi NB)
        auto issue = [&](int bi, int bb) {
            const int hi = maxl - bi * NB, lo = max(0, hi - NB);
            fence_proxy_async_smem();
            tma_load_1d(&sm.rec[bb][0], a.srec + 3 * (size_t)(start + lo), (uint32_t)(hi - lo) * 48u, &sm.bar[bb]);
        };
        if (tid == 0 && nb > 0) issue(0, 0);
        int buf = 0;
        for (int bi = 0; bi < nb; ++bi) {
            const int hi = maxl - bi * NB, lo = max(0, hi - NB), cnt = hi - lo;
            if (tid == 0 && bi + 1 < nb) issue(bi + 1, buf ^ 1);
            const bool ok = mbar_wait_bounded(&sm.bar[buf], parity[buf], kTmaWaitLimit);
            if (__syncthreads_or(!ok)) {
                const bool pending[2] = {buf == 0 || bi + 1 < nb, buf == 1 || bi + 1 < nb};
                drain_after_timeout(sm, parity, pending, a.st);
                claim_exit(&a.st->bwd_items, sm.coff, a.G);
                return;
            }
            parity[buf] ^= 1u;
            const float4 *rec = sm.rec[buf];
            if constexpr (!kWide<TW, TH, NB>)
                slow = !(tame(gC0.x, gC1.x, gC2.x, gD.x) && tame(gC0.y, gC1.y, gC2.y, gD.y) && tame(Q.x, Q.y, 0.f, 0.f));
            slow = __syncthreads_or(stage_masks<TW, TH, NB>(rec, sm.mask, cnt, tx * TW, ty * TH) | slow);
            // entries at or beyond the warp's largest last_idx contribute nothing to this warp
            const int kend = min(hi, wmax) - lo;
            if (slow) walk(std::true_type(), rec, sm.mask, lo, kend);
            else walk(std::false_type(), rec, sm.mask, lo, kend);
            __syncthreads();                          // buffer reads finished before its refill
            buf ^= 1;
        }
        __syncthreads();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
    if (lane == 0 && pairs) atomicAdd(&a.st->bwd_pairs, pairs);
}

template <class F>
static int persistent_grid(F fn, int threads) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, threads, 0) != cudaSuccess || b < 1) b = 1;
    return b * device_sm_count();
}

template <int TW, int TH, int NB>
static int fwd_t(const FwdArgs &a, cudaStream_t s) {
    constexpr int NT = TW * TH / kPPT;
    static PerDevice per;
    const int grid = per.get(current_device(), [] { return persistent_grid(k_render_fwd<TW, TH, NB>, NT); });
    if (a.rgb_t && cudaMemsetAsync(a.loss, 0, sizeof(double), s) != cudaSuccess) return GS_ERR_CUDA;
    const long long g = std::min<long long>(grid, std::max<long long>(1, a.G));
    k_render_fwd<TW, TH, NB><<<(unsigned)g, NT, 0, s>>>(a);
    count_launches(1);
    return check_launch();
}

template <int TW, int TH, int NB>
static int bwd_t(const BwdArgs &a, cudaStream_t s) {
    constexpr int NT = TW * TH / kPPT;
    static PerDevice per;
    const int grid = per.get(current_device(), [] { return persistent_grid(k_render_bwd<TW, TH, NB>, NT); });
    const long long g = std::min<long long>(grid, std::max<long long>(1, a.G));
    k_render_bwd<TW, TH, NB><<<(unsigned)g, NT, 0, s>>>(a);
    count_launches(1);
    return check_launch();
}

// (tile, records per batch) pairs with a compiled kernel; the API layer validates the values
int launch_render_fwd(int tw, int th, int nb, const FwdArgs &a, cudaStream_t s) {
    if (tw == 16 && th == 16)
        return nb == 64 ? fwd_t<16, 16, 64>(a, s) : nb == 128 ? fwd_t<16, 16, 128>(a, s) : fwd_t<16, 16, 256>(a, s);
    if (tw == 16 && th == 8) return nb == 64 ? fwd_t<16, 8, 64>(a, s) : fwd_t<16, 8, 128>(a, s);
    if (tw == 32 && th == 16)
        return nb == 64 ? fwd_t<32, 16, 64>(a, s) : nb == 128 ? fwd_t<32, 16, 128>(a, s) : fwd_t<32, 16, 256>(a, s);
    return GS_ERR_INVALID_ARG;
}

int launch_render_bwd(int tw, int th, int nb, const BwdArgs &a, cudaStream_t s) {
    if (tw == 16 && th == 16)
        return nb == 64 ? bwd_t<16, 16, 64>(a, s) : nb == 128 ? bwd_t<16, 16, 128>(a, s) : bwd_t<16, 16, 256>(a, s);
    if (tw == 16 && th == 8) return nb == 64 ? bwd_t<16, 8, 64>(a, s) : bwd_t<16, 8, 128>(a, s);
    if (tw == 32 && th == 16)
        return nb == 64 ? bwd_t<32, 16, 64>(a, s) : nb == 128 ? bwd_t<32, 16, 128>(a, s) : bwd_t<32, 16, 256>(a, s);
    return GS_ERR_INVALID_ARG;
}

}  // namespace gs
