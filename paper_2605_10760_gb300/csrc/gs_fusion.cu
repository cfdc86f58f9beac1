// gs_fusion.cu -- occupancy-aware fusion of aligned submaps (Sec. III-C, Eqs. 19-22).
//
//  * k_sim3: the Sim(3) correction C = (s, R, t) acting on Gaussians (Eq. 19): mu' = s R mu + t,
//    rotation q' = q_R (x) q, log-scales + ln s; opacity and colour copied.
//  * Voxel sets: open-addressing hash sets of 64-bit keys (voxel index kappa(x) = floor(x / v) per
//    axis, 21 bits per axis with offset 2^20); insertion by compare-and-swap, membership by probing
//    to the first empty slot.  Blocks of 4 x 2 x 2 voxels hash to lines of 16 slots, so neighbouring
//    voxels meet in one line (VoxProbe).  Probing is bounded by the capacity; a full table records
//    GS_ERR_CAPACITY in the set's status word instead of looping.
//  * k_add_boxes (Eq. 20): every voxel of [kappa(mu - k s), kappa(mu + k s)]; a warp spreads the
//    voxels of its 32 boxes over its lanes.
//  * k_add_rays (Eq. 21): one thread per (keyframe, strided pixel), a warp per 8 x 4 of them, walks the voxels crossed by the
//    segment from the camera centre to the back-projected depth point, t in [0, 1), with a 3-D
//    digital differential analyser (ties between axes go to the lowest axis).
//  * k_keep (Eq. 22): keep a borrowed Gaussian iff kappa(mu) is in neither set.
// Every voxel decision uses the same FP32 operation sequence as the fusion oracle (explicit
// round-to-nearest intrinsics, never contracted), so the voxel sets agree bit for bit.
#include <algorithm>
#include <cmath>

#include "gs_kernels.cuh"

namespace gs {

constexpr unsigned long long kEmptyKey = ~0ull;
constexpr int kKeyBits = 21;
constexpr long long kKeyOff = 1LL << 20;
// words of a set's 256-byte header beside the status (bytes 8 .. 15 are gs_voxset_status's)
constexpr int kStoredOffset = 16;      // keys stored, as far as reported
constexpr int kLongestOffset = 24;     // the largest number of pauses (VoxProbe) that a stored key has made
constexpr uint32_t kPatience = 32;     // slots between two pauses of a key
constexpr int kMaxRaySteps = 1 << 16;  // voxels after the first of one ray before it is flagged
constexpr int kMaxBoxExtent = 64;      // voxels per axis of one Gaussian's box before it is flagged

struct VoxSet {
    int32_t *status;                   // first error
    unsigned long long *keys;          // [capacity]
    uint32_t blocks;                   // lines of slots - 1
    uint32_t pos;                      // slots of a line - 1 (15, or capacity - 1 of a smaller set)
    int shift;                         // log2 of the slots of a line
};

static VoxSet voxset_of_host(void *mem, long long capacity) {
    VoxSet s;
    s.status = reinterpret_cast<int32_t *>(mem);
    s.keys = reinterpret_cast<unsigned long long *>(static_cast<char *>(mem) + 256);
    s.shift = 0;
    while (s.shift < 4 && (2LL << s.shift) <= capacity) ++s.shift;
    s.pos = (1u << s.shift) - 1u;
    s.blocks = (uint32_t)((capacity >> s.shift) - 1);
    return s;
}

// a voxel index as it enters a key: clamped to [-2^20, 2^20), offset to [0, 2^21)
__device__ __forceinline__ uint32_t key_coord(int i) {
    return (uint32_t)(min(max(i, (int)-kKeyOff), (int)kKeyOff - 1) + (int)kKeyOff);
}
__device__ __forceinline__ unsigned long long vox_key(int ix, int iy, int iz) {
    return ((unsigned long long)key_coord(ix) << (2 * kKeyBits)) | ((unsigned long long)key_coord(iy) << kKeyBits) |
           key_coord(iz);
}

// Where the key of a voxel may stand.  The 16 voxels of a 4 x 2 x 2 block share a line (128 bytes; 2 x 2 x 1 of
// them a sector), whose number is a hash of the block: a ray of 70 voxels touches about 30 lines and its
// neighbours in the warp the same ones, where a hash of the voxel itself touches 70 sectors of its own.  The
// place within the line is the voxel's place in its block, XORed with hash bits (so that flat sets, which use
// half of every block's voxels, still use all slots alike).  The sequence visits that place in other lines, a
// hashed odd number of lines apart (the lines are a power of two), then the next place in every line, so that
// every slot is visited once in `capacity` probes: the slots of one place behave like a double-hashed table of
// random keys.  (Carved space fills whole blocks, so a line's neighbours are no better than any other line, and
// steps of one line would form long runs: at 89 % of the slots in use 41 probes to find a key absent, hashed
// steps 9.  7 views into a set filled to 73 % and 89 %: 3.25 ms with steps of one line, 0.69 ms.)
struct VoxProbe {
    unsigned long long key;
    uint32_t mix, block, pos;

    __device__ __forceinline__ VoxProbe(const VoxSet &s, unsigned long long k) : key(k) {
        const uint32_t lo = (uint32_t)k, hi = (uint32_t)(k >> 32);   // y's low 11 bits and z; x and y's high 10 bits
        // the block (two bits of x, one of y and z masked off) through odd multipliers, then a multiplication
        // whose halves are folded onto each other, and the high part of another one (the multipliers are primes
        // of xxHash32)
        const uint32_t h = (lo & ~0x00200001u) * 0x9e3779b1u + (hi & ~0x00000c00u) * 0x85ebca77u;
        const unsigned long long m = (unsigned long long)h * 0xc2b2ae3du;
        mix = (uint32_t)m ^ (uint32_t)(m >> 32);
        block = home(s);
        pos = first(s);
    }
    __device__ __forceinline__ uint32_t first(const VoxSet &s) const {
        const uint32_t lo = (uint32_t)key, hi = (uint32_t)(key >> 32);
        const uint32_t place = ((hi >> 10) & 3u) | ((lo >> 19) & 4u) | ((lo << 3) & 8u);
        return (place ^ mix) & s.pos;
    }
    __device__ __forceinline__ uint32_t home(const VoxSet &s) const { return __umulhi(mix * 0x27d4eb2fu, s.blocks + 1u); }
    __device__ __forceinline__ size_t slot(const VoxSet &s) const { return ((size_t)block << s.shift) | pos; }
    // On to the next line; true at a pause: after every kPatience slots (the step is odd, so the low bits of the line's
    // number come round) and where the lines have come round, at home.
    __device__ __forceinline__ bool advance(const VoxSet &s) {
        block = (block + ((mix >> 5) | 1u)) & s.blocks;
        return ((block ^ home(s)) & (kPatience - 1u)) == 0u;
    }
    // At a pause: on to the next place if this is home; false once all have been visited.
    __device__ __forceinline__ bool turn(const VoxSet &s) {
        if (block != home(s)) return true;
        pos = (pos + 1u) & s.pos;
        return pos != first(s);
    }
};

template <class T>
__device__ __forceinline__ volatile T *voxset_word(const VoxSet &s, int offset) {
    return reinterpret_cast<volatile T *>(reinterpret_cast<char *>(s.status) + offset);
}

// Reports the keys that this CTA has stored since its last report (`taken`).
__device__ __forceinline__ void voxset_report(const VoxSet &s, uint32_t *taken) {
    const uint32_t n = atomicExch(taken, 0u);
    if (n) atomicAdd((unsigned long long *)voxset_word<unsigned long long>(s, kStoredOffset), (unsigned long long)n);
}

// A key that pauses reports its CTA's keys and asks whether the set is full (every CTA reports the rest when it ends, so
// that is known soon after the last slot was taken).  A full set changes no more: with an error recorded the key may
// leave it, and otherwise only needs to know whether it is in there, for which it looks no further than any stored
// key has come.  Without the two words it would walk the whole set, or a sixteenth of it after an error.  2^17 slots
// offered 10 times as many keys 0.19 ms, 2^22 slots 4 times 2.1 ms, 2^25 slots 1.5 times 18 ms (0.05, 0.7 and 2.5 ms
// into a set that holds them).  The count is kept by the CTA, not the thread: a lane that waits for a neighbour's key
// could not report its own.  It costs the rays 4 % (8 views of 600 x 340, 488 -> 507 us timed alone).
__device__ __forceinline__ void voxset_insert(const VoxSet &s, unsigned long long key, uint32_t *taken) {
    VoxProbe p(s, key);
    uint32_t pauses = 0;
    for (;;) {
        unsigned long long *slot = s.keys + p.slot(s);
        const unsigned long long cur = *slot;
        if (cur == p.key) return;
        if (cur == kEmptyKey) {
            const unsigned long long prev = atomicCAS(slot, kEmptyKey, p.key);
            if (prev == kEmptyKey) {
                if (pauses) {
                    atomicMax((uint32_t *)voxset_word<uint32_t>(s, kLongestOffset), pauses);
                    __threadfence();           // before the count that may fill the set
                }
                atomicAdd(taken, 1u);
            }
            if (prev == kEmptyKey || prev == p.key) return;
        }
        if (p.advance(s)) {
            ++pauses;
            voxset_report(s, taken);
            if (*voxset_word<unsigned long long>(s, kStoredOffset) >= ((unsigned long long)s.blocks + 1ull) << s.shift) {
                __threadfence();
                if (*voxset_word<int32_t>(s, 0) != 0) return;
                if (pauses > *voxset_word<uint32_t>(s, kLongestOffset)) break;
            }
            if (!p.turn(s)) break;
        }
    }
    atomicCAS(s.status, 0, GS_ERR_CAPACITY);
}

// `cur` is what the caller found in the first slot.  Up to the first empty slot, or as far as any stored key has come:
// an overfull set has no empty slot, and a key that is not in it would be compared with all the others.  (1 M Gaussians
// outside a set of 2^22 slots: 0.04 ms half full, 0.13 ms at 94 %, 2.6 ms overfull.)
__device__ __forceinline__ bool voxset_contains(const VoxSet &s, VoxProbe p, unsigned long long cur) {
    uint32_t pauses = 0;
    for (;;) {
        if (cur == p.key) return true;
        if (cur == kEmptyKey) return false;
        if (p.advance(s) && (++pauses > *voxset_word<uint32_t>(s, kLongestOffset) || !p.turn(s))) return false;
        cur = s.keys[p.slot(s)];
    }
}

__device__ __forceinline__ long long vox_index(float x, float v) { return (long long)floorf(fp::div(x, v)); }
// the same for a key alone: beyond +-2^30 every index enters keys as the same limit
__device__ __forceinline__ int vox_clamp(long long i) { return (int)min(max(i, -(1LL << 30)), 1LL << 30); }

// ------------------------------------------------------------------------------------------
__global__ void k_voxset_clear(unsigned long long *keys, long long capacity, int32_t *status) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < capacity;
         i += (long long)gridDim.x * blockDim.x)
        keys[i] = kEmptyKey;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *status = 0;
        *reinterpret_cast<unsigned long long *>(reinterpret_cast<char *>(status) + kStoredOffset) = 0ull;
        *reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(status) + kLongestOffset) = 0u;
    }
}

// One Gaussian per lane for the box, then the warp's voxels one per lane in turn, those of a box along z first:
// boxes of one warp differ in size (one to hundreds of voxels), and a lane that walked its own would wait for a
// probe of memory per voxel.  2 M Gaussians, a set of 2^25: 151 us, bound by instruction issue (75 %); 545 us with
// a box per lane and voxels hashed one by one.
__global__ void __launch_bounds__(256) k_add_boxes(VoxSet s, long long n, const float *means, const float *log_scales,
                                                   float k, float v) {
    __shared__ uint32_t s_taken;
    if (threadIdx.x == 0) s_taken = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < n; i0 += stride) {
        const long long i = i0 + lane;
        int lo[3] = {0, 0, 0}, ext[3] = {0, 0, 0};
        bool big = false;
        if (i < n) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float mu = means[3 * i + a];
                const float ks = fp::mul(k, spec_expf(log_scales[3 * i + a]));
                const long long l = vox_index(fp::sub(mu, ks), v), h = vox_index(fp::add(mu, ks), v);
                lo[a] = vox_clamp(l);
                const unsigned long long span = (unsigned long long)h - (unsigned long long)l;
                big |= h >= l && span >= kMaxBoxExtent;
                ext[a] = h >= l ? (int)min(span, kMaxBoxExtent - 1ull) + 1 : 0;
            }
        }
        if (big) atomicCAS(s.status, 0, GS_ERR_INVALID_ARG);   // a box wider than kMaxBoxExtent voxels
        const int count = big ? 0 : ext[0] * ext[1] * ext[2];
        int end = count;                                       // inclusive prefix sum over the lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += up;
        }
        const int total = __shfl_sync(0xffffffffu, end, 31);
        const int begin = end - count, dims = ext[1] << 8 | ext[2];
        for (int base = 0; base < total; base += 32) {
            const int item = base + lane;
            int owner = 0;                                     // number of lanes whose voxels end at or before `item`
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, end, owner + o - 1) <= item) owner += o;
            const int d = __shfl_sync(0xffffffffu, dims, owner), at = item - __shfl_sync(0xffffffffu, begin, owner);
            const int x0 = __shfl_sync(0xffffffffu, lo[0], owner), y0 = __shfl_sync(0xffffffffu, lo[1], owner);
            const int z0 = __shfl_sync(0xffffffffu, lo[2], owner);
            if (item < total) {
                // at < 2^18 and extents <= 64: (at + 1/2) / extent is at least 1/128 away from an integer,
                // and the approximate division (2 ulp) puts it within 2^-9 of where it belongs
                const int ny = d >> 8, nz = d & 255;
                const int row = (int)__fdividef((float)at + 0.5f, (float)nz), z = at - row * nz;
                const int x = (int)__fdividef((float)row + 0.5f, (float)ny), y = row - x * ny;
                voxset_insert(s, vox_key(x0 + x, y0 + y, z0 + z), &s_taken);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) voxset_report(s, &s_taken);
}

struct RayArgs {
    VoxSet s;
    const gs_camera *cams;
    const float *depth;       // [V,H,W] camera depth (z) per pixel; <= 0 or non-finite: no ray
    int V, W, H, stride, sw, sh;   // sw x sh rays a view
    int pw, ph;               // patches of 8 x 4 rays across and down, one per warp
    float v;
};

// Bound by the instructions of a step (about 40: the analyser, the hash, the probe), not by memory: the rays of a
// patch walk together through the lines near the camera.  8 views of 600 x 340 rays, some 70 voxels each, a set of
// 2^25: 442 us (419 us with probe steps of one line, see VoxProbe; 48 warps an SM 477 us); before those hashed steps
// 467 us with a warp's rays along a row; 827 us with voxels hashed one by one and 64-bit indices.  Settling a voxel
// only after the next one's load was issued: 650 us (more instructions, and more slots found empty that another
// warp had just filled).
__global__ void __launch_bounds__(256, 8) k_add_rays(RayArgs a) {
    __shared__ uint32_t s_taken;
    if (threadIdx.x == 0) s_taken = 0u;
    __syncthreads();
    const long long total = (long long)a.V * a.pw * a.ph * 32;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < total; r += (long long)gridDim.x * blockDim.x) {
        const int lane = threadIdx.x & 31;
        const long long patch = r >> 5, k = patch / ((long long)a.pw * a.ph);
        const int at = (int)(patch - k * a.pw * a.ph), sy = at / a.pw * 4 + (lane >> 3), sx = at % a.pw * 8 + (lane & 7);
        if (sy >= a.sh || sx >= a.sw) continue;
        const int y = sy * a.stride, x = sx * a.stride;
        const float d = a.depth[((long long)k * a.H + y) * a.W + x];
        if (!(d > 0.f) || !isfinite(d)) continue;
        const gs_camera cam = a.cams[k];
        const float *R = cam.R, *t = cam.t;
        float c[3], p[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) c[q] = -fp::fma(R[q], t[0], fp::fma(R[3 + q], t[1], fp::mul(R[6 + q], t[2])));
        const float xn = fp::div(fp::sub(fp::add((float)x, 0.5f), cam.cx), cam.fx);
        const float yn = fp::div(fp::sub(fp::add((float)y, 0.5f), cam.cy), cam.fy);
        const float pc0 = fp::sub(fp::mul(xn, d), t[0]), pc1 = fp::sub(fp::mul(yn, d), t[1]), pc2 = fp::sub(d, t[2]);
#pragma unroll
        for (int q = 0; q < 3; ++q) p[q] = fp::fma(R[q], pc0, fp::fma(R[3 + q], pc1, fp::mul(R[6 + q], pc2)));
        // digital differential analyser over [c, p)
        int cur[3], step[3];
        float tmax[3], tdel[3];
        const float inf = __int_as_float(0x7f800000);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const long long at = vox_index(c[q], a.v);
            cur[q] = vox_clamp(at);
            const float dq = fp::sub(p[q], c[q]);
            if (dq > 0.f) {
                step[q] = 1;
                tmax[q] = fp::div(fp::sub(fp::mul((float)(at + 1), a.v), c[q]), dq);
                tdel[q] = fp::div(a.v, dq);
            } else if (dq < 0.f) {
                step[q] = -1;
                tmax[q] = fp::div(fp::sub(fp::mul((float)at, a.v), c[q]), dq);
                tdel[q] = fp::div(-a.v, dq);
            } else {
                step[q] = 0;
                tmax[q] = inf;
                tdel[q] = inf;
            }
        }
        unsigned long long key = vox_key(cur[0], cur[1], cur[2]);
        voxset_insert(a.s, key, &s_taken);
        int n = 0;
        // A ray that starts far enough inside the range of keys never meets its limits: its key moves by the
        // step's own bits.
        constexpr int kInside = (int)kKeyOff - (kMaxRaySteps + 1);
        if (max(max(abs(cur[0]), abs(cur[1])), abs(cur[2])) <= kInside) {
            const unsigned long long kx = (unsigned long long)(long long)step[0] << (2 * kKeyBits);
            const unsigned long long ky = (unsigned long long)(long long)step[1] << kKeyBits;
            const unsigned long long kz = (unsigned long long)(long long)step[2];
            for (; n < kMaxRaySteps; ++n) {
                const bool b1 = tmax[1] < tmax[0];
                const float t01 = b1 ? tmax[1] : tmax[0];
                const bool q2 = tmax[2] < t01;
                if (!((q2 ? tmax[2] : t01) < 1.0f)) break;
                const float n0 = fp::add(tmax[0], tdel[0]), n1 = fp::add(tmax[1], tdel[1]), n2 = fp::add(tmax[2], tdel[2]);
                key += q2 ? kz : b1 ? ky : kx;
                tmax[0] = !q2 && !b1 ? n0 : tmax[0];
                tmax[1] = !q2 && b1 ? n1 : tmax[1];
                tmax[2] = q2 ? n2 : tmax[2];
                voxset_insert(a.s, key, &s_taken);
            }
        } else {
            for (; n < kMaxRaySteps; ++n) {
                int q = 0;
                if (tmax[1] < tmax[0]) q = 1;
                if (tmax[2] < (q ? tmax[1] : tmax[0])) q = 2;
                if (!((q == 2 ? tmax[2] : q == 1 ? tmax[1] : tmax[0]) < 1.0f)) break;
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    if (d == q) {
                        cur[d] += step[d];
                        tmax[d] = fp::add(tmax[d], tdel[d]);
                    }
                voxset_insert(a.s, vox_key(cur[0], cur[1], cur[2]), &s_taken);
            }
        }
        if (n == kMaxRaySteps) atomicCAS(a.s.status, 0, GS_ERR_INVALID_ARG);   // ray longer than allowed
    }
    __syncthreads();
    if (threadIdx.x == 0) voxset_report(a.s, &s_taken);
}

__global__ void k_keep(long long n, const float *means, VoxSet occ, VoxSet fre, bool has_free, float v,
                       uint8_t *keep) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int x = vox_clamp(vox_index(means[3 * i], v)), y = vox_clamp(vox_index(means[3 * i + 1], v)),
                  z = vox_clamp(vox_index(means[3 * i + 2], v));
        const unsigned long long key = vox_key(x, y, z);
        const VoxProbe po(occ, key), pf(fre, key);
        const unsigned long long co = occ.keys[po.slot(occ)];   // both sets are asked before either answers
        const unsigned long long cf = has_free ? fre.keys[pf.slot(fre)] : kEmptyKey;
        const bool drop = voxset_contains(occ, po, co) || voxset_contains(fre, pf, cf);
        keep[i] = drop ? 0 : 1;
    }
}

__global__ void k_sim3(long long n, gs_gaussians in, gs_gaussian_arrays out, float s, float R00, float R01, float R02,
                       float R10, float R11, float R12, float R20, float R21, float R22, float t0, float t1, float t2,
                       float qw, float qx, float qy, float qz, float ln_s) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float m0 = in.means[3 * i], m1 = in.means[3 * i + 1], m2 = in.means[3 * i + 2];
        out.means[3 * i] = s * (R00 * m0 + R01 * m1 + R02 * m2) + t0;
        out.means[3 * i + 1] = s * (R10 * m0 + R11 * m1 + R12 * m2) + t1;
        out.means[3 * i + 2] = s * (R20 * m0 + R21 * m1 + R22 * m2) + t2;
#pragma unroll
        for (int a = 0; a < 3; ++a) out.log_scales[3 * i + a] = in.log_scales[3 * i + a] + ln_s;
        const float bw = in.quats[4 * i], bx = in.quats[4 * i + 1], by = in.quats[4 * i + 2], bz = in.quats[4 * i + 3];
        out.quats[4 * i] = qw * bw - qx * bx - qy * by - qz * bz;
        out.quats[4 * i + 1] = qw * bx + qx * bw + qy * bz - qz * by;
        out.quats[4 * i + 2] = qw * by - qx * bz + qy * bw + qz * bx;
        out.quats[4 * i + 3] = qw * bz + qx * by - qy * bx + qz * bw;
        out.opacities[i] = in.opacities[i];
#pragma unroll
        for (int a = 0; a < 3; ++a) out.colors[3 * i + a] = in.colors[3 * i + a];
    }
}

static int grid_for(long long n) {
    return (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, (long long)device_sm_count() * 16));
}

int launch_voxset_clear(void *mem, long long capacity, cudaStream_t s) {
    k_voxset_clear<<<grid_for(capacity), 256, 0, s>>>(
        reinterpret_cast<unsigned long long *>(static_cast<char *>(mem) + 256), capacity, reinterpret_cast<int32_t *>(mem));
    count_launches(1);
    return check_launch();
}

int launch_voxset_add_boxes(void *mem, long long capacity, long long n, const float *means, const float *log_scales,
                            float k, float v, cudaStream_t s) {
    if (n > 0) {
        k_add_boxes<<<grid_for(n), 256, 0, s>>>(voxset_of_host(mem, capacity), n, means, log_scales, k, v);
        count_launches(1);
    }
    return check_launch();
}

int launch_voxset_add_rays(void *mem, long long capacity, int V, int W, int H, const gs_camera *cams,
                           const float *depth, int stride, float v, cudaStream_t s) {
    RayArgs a;
    a.s = voxset_of_host(mem, capacity);
    a.cams = cams;
    a.depth = depth;
    a.V = V; a.W = W; a.H = H; a.stride = stride;
    a.sw = (W + stride - 1) / stride;
    a.sh = (H + stride - 1) / stride;
    a.v = v;
    a.pw = (a.sw + 7) / 8;
    a.ph = (a.sh + 3) / 4;
    const long long total = (long long)V * a.pw * a.ph * 32;
    k_add_rays<<<grid_for(total), 256, 0, s>>>(a);
    count_launches(1);
    return check_launch();
}

int launch_voxset_keep(long long n, const float *means, void *occ, long long occ_cap, void *fre, long long free_cap,
                       float v, uint8_t *keep, cudaStream_t s) {
    if (n > 0) {
        const VoxSet o = voxset_of_host(occ, occ_cap);
        const VoxSet f = fre ? voxset_of_host(fre, free_cap) : o;
        k_keep<<<grid_for(n), 256, 0, s>>>(n, means, o, f, fre != nullptr, v, keep);
        count_launches(1);
    }
    return check_launch();
}

int launch_sim3(long long n, const gs_gaussians &in, const float q[4], const float t[3], float sc,
                const gs_gaussian_arrays &out, cudaStream_t s) {
    // rotation matrix of the unit quaternion (normalised here, in double on the host)
    const double nq = sqrt((double)q[0] * q[0] + (double)q[1] * q[1] + (double)q[2] * q[2] + (double)q[3] * q[3]);
    const double w = q[0] / nq, x = q[1] / nq, y = q[2] / nq, z = q[3] / nq;
    const float R[9] = {(float)(1 - 2 * (y * y + z * z)), (float)(2 * (x * y - w * z)), (float)(2 * (x * z + w * y)),
                        (float)(2 * (x * y + w * z)), (float)(1 - 2 * (x * x + z * z)), (float)(2 * (y * z - w * x)),
                        (float)(2 * (x * z - w * y)), (float)(2 * (y * z + w * x)), (float)(1 - 2 * (x * x + y * y))};
    if (n > 0) {
        k_sim3<<<grid_for(n), 256, 0, s>>>(n, in, out, sc, R[0], R[1], R[2], R[3], R[4], R[5], R[6], R[7], R[8], t[0],
                                           t[1], t[2], (float)w, (float)x, (float)y, (float)z, (float)log((double)sc));
        count_launches(1);
    }
    return check_launch();
}

}  // namespace gs
