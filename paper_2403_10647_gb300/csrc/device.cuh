// Device-side definitions shared by the grid-construction kernels.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace gg {

// Error bits raised by kernels into Ctl::err and turned into GRID_* codes on
// the host.  No kernel traps: a failed check records a bit and skips the
// offending access.
constexpr unsigned ERR_BADINDEX = 1u;   // triangle references a vertex outside [0, nverts)
constexpr unsigned ERR_NONFINITE = 2u;  // NaN / Inf vertex coordinate
constexpr unsigned ERR_OVERFLOW = 4u;   // a prefix sum passed INT32_MAX
constexpr unsigned ERR_TIMEOUT = 8u;    // a bounded look-back wait gave up
constexpr unsigned ERR_RANGE = 16u;     // a key outside [0, ncells) or out of order reached range
                                        // extraction, or a sort scatter fell outside the output
constexpr unsigned ERR_TILE_REDO = 64u;        // not an error: count/scan could not record every pair
                                               // tile's first object; the host runs tile_search
constexpr unsigned ERR_BTILE_REDO = 128u;      // not an error: the same for the brick entries' tiles
constexpr unsigned ERR_LOCAL_FALLBACK = 32u;   // not an error: a group of buckets too large for the
                                               // per-bucket counting sort; the host places the build
                                               // by radix passes over every key bit instead

// Spin limit of every look-back wait (each iteration sleeps ~0.1-1 us).
constexpr unsigned SPIN_LIMIT = 1u << 20;

constexpr int MAX_PASSES = 4;
constexpr int MAX_RADIX = 1 << 11;

// Per-build control block, zero before the first kernel: a context has two, and
// a single-mesh build's bounds kernel zeroes the one for the next build; where no
// build did, a memset does.  A count that is run again (the host's grid
// metadata in place of the device's) starts from err, tickets[0], npairs and count_done
// zeroed anew; it writes nrefs over.
struct Ctl {
    unsigned lo_inv[3];         // atomicMax of ~ordered(min coordinate) per axis
    unsigned hi_ord[3];         // atomicMax of ordered(max coordinate) per axis
    unsigned err;               // ERR_* bits
    unsigned bounds_done;       // blocks of the bounds kernel that finished (the last one plans)
    unsigned long long nrefs;   // NO, written by the last count/scan tile (with the brick entries in the
                                // bits from BRICK_SUM_BITS on when it counted them)
    unsigned tickets[8];        // tile tickets: [0] count/scan, [5] cell scan (its look-back's tiles, or the
                                // blocks of its first pass that finished), [7] culling emit; counts: [1] cells
                                // of many objects, [2] the hybrid placement's bucket groups or a culled brick
                                // build's words of entries, [3] the brick items, [4] their chunk slots, [6] the
                                // empty bricks
    unsigned long long nkept;   // pairs that culling kept: by the culling emit's last tile, or added up by the
                                // brick count
    unsigned long long npairs;  // a count with brick entries: NO added up on its own, exact
    unsigned count_done, place_done;   // blocks of count/scan, and of the placement's last kernel, that
                                       // finished (publish_ctl)
    // grid metadata M computed on the device from the bounds above (plan_kernel),
    // for count/scan to read without a host round trip; the host checks it
    // against its own plan from the same bounds
    float plan_lo[3];
    float plan_scale[3];
    int plan_res[3];
    unsigned plan_pad;
};
static_assert(sizeof(Ctl) == 136, "Ctl layout");

// One object's box in grid coordinates and its pair offset (grid_objrec).
struct __align__(16) ObjRec {
    uint16_t lo[3];
    uint16_t hi[3];
    uint32_t start;
};
static_assert(sizeof(ObjRec) == 16, "ObjRec layout");

// Order-preserving map float -> uint32 (larger float, larger key).
__host__ __device__ __forceinline__ unsigned float_to_ordered(float f)
{
#ifdef __CUDA_ARCH__
    unsigned b = __float_as_uint(f);
#else
    unsigned b;
    __builtin_memcpy(&b, &f, 4);
#endif
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__host__ __device__ __forceinline__ float ordered_to_float(unsigned k)
{
    unsigned b = (k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k;
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float f;
    __builtin_memcpy(&f, &b, 4);
    return f;
#endif
}

// ---- bricks ----
//
// A brick is a box of 2^lx x 2^ly x 2^lz cells, at most 512.  A brick build
// sorts one entry per (brick, object whose box meets it) instead of one pair
// per cell; an entry carries the object's box inside the brick as two local
// cell indices of 9 bits each.
constexpr int BRICK_CELLS_LOG = 9;
constexpr int BRICK_CELLS = 1 << BRICK_CELLS_LOG;
constexpr int BRICK_INFO_BITS = 2 * BRICK_CELLS_LOG;
// Count and scan of pairs and brick entries at once: one 62-bit sum holds the
// pairs in its low BRICK_SUM_BITS bits and the entries above them (never more
// than the pairs).  Whether the pairs overflowed shows in their own exact sum.
constexpr int BRICK_SUM_BITS = 31;
constexpr unsigned BRICK_SUM_MASK = (1u << BRICK_SUM_BITS) - 1u;

__host__ __device__ __forceinline__ unsigned ceil_log2(unsigned v)
{
    unsigned b = 0;
    while ((1u << b) < v) ++b;
    return b;
}

// Brick shape of a grid, lx | ly << 4 | lz << 8: 8 cells along each axis, fewer
// where the grid is thinner than that (in x at least 4, as the fill takes four
// neighbours in x at a time); a thin grid's bricks are 16 cells
// wide in x while the brick stays within 512 cells and its cell columns, rows
// and layers within 32 (one bit each in a warp's 32 x 32 bit transpose).
__host__ __device__ __forceinline__ unsigned brick_shape(int rx, int ry, int rz)
{
    unsigned cx = ceil_log2((unsigned)rx), cy = ceil_log2((unsigned)ry), cz = ceil_log2((unsigned)rz);
    unsigned lx = cx < 2u ? 2u : cx < 3u ? cx : 3u, ly = cy < 3u ? cy : 3u, lz = cz < 3u ? cz : 3u;
    if (cx > 3u && lx + ly + lz < (unsigned)BRICK_CELLS_LOG) lx = 4u;
    return lx | (ly << 4) | (lz << 8);
}

// How a brick build's entries are packed into 32-bit keys and values: the
// brick id in the key's low kb bits, the object in the value's low ob bits, the
// box's BRICK_INFO_BITS in the bits above them (key first).
struct BrickGen {
    unsigned shape;      // single mesh: brick_shape, bricks per axis x and y
    unsigned nbx, nby;
    int kb, ob;
};

__host__ __device__ __forceinline__ int brick_key_info_bits(int kb)
{
    return 32 - kb < BRICK_INFO_BITS ? 32 - kb : BRICK_INFO_BITS;
}

__host__ __device__ __forceinline__ bool brick_packs(int kb, int ob)
{
    return ob + BRICK_INFO_BITS - brick_key_info_bits(kb) <= 32 && ob < 32 && kb < 32;
}

#ifdef __CUDACC__

__device__ __forceinline__ unsigned ld_relaxed_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed_u32(unsigned *p, unsigned v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Four consecutive 32-bit words, each read with relaxed gpu-scope semantics
// (16-byte aligned address).
__device__ __forceinline__ uint4 ld_relaxed_v4(const unsigned *p)
{
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed_u64(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Grid coordinate of world value p on one axis: floor((p - lo) * scale) with
// both operations rounded to FP32 separately (the intrinsics are never
// contracted into an FMA), clamped to [0, res - 1]; NaN maps to 0.
__device__ __forceinline__ int cell_coord(float p, float lo, float scale, int res)
{
    float u = __fmul_rn(__fsub_rn(p, lo), scale);
    if (!(u >= 1.0f)) return 0;                 // u < 1 (incl. negative) or NaN
    if (u >= (float)res) return res - 1;        // floor(u) > res - 1
    return __float2int_rz(u);                   // u in [1, res): truncation == floor
}

// ---- block and grid primitives ----

template <typename T>
__device__ __forceinline__ T warp_incl_sum(T v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

__device__ __forceinline__ unsigned warp_incl_max(unsigned v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = max(v, u);
    }
    return v;
}

// First statement of every kernel that launch_after (kernels.h) starts: waits
// for everything before it on the stream to have finished.  The kernels do not
// let their successors start early (griddepcontrol.launch_dependents): waiting
// blocks in the way of running ones cost more than that hides (100,000
// triangles: 109 us without dependent launch, 115 with early starts, 99 so).
__device__ __forceinline__ void after_stream() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// For the kernel ahead of a host wait on a small build: the last block to
// finish (*done counts them) writes the control block to its pinned host
// mirror, in place of a copy of its own on the stream (about 4 us of a 115 us
// build).  Every thread of every block calls it, last thing.
__device__ __forceinline__ void publish_ctl(const Ctl *ctl, Ctl *host, unsigned *done)
{
    if (!host) return;
    __shared__ unsigned s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(done, 1u) + 1u == gridDim.x;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const unsigned *from = reinterpret_cast<const unsigned *>(ctl);
    volatile unsigned *to = reinterpret_cast<volatile unsigned *>(host);
    for (unsigned i = threadIdx.x; i < sizeof(Ctl) / sizeof(unsigned); i += blockDim.x) to[i] = __ldcg(from + i);
    __threadfence_system();
}

// Exclusive block-wide sum of one value per thread; s_tmp holds BLOCK/32
// entries.  Returns the exclusive prefix, writes the block total to *total.
template <int BLOCK, typename T>
__device__ __forceinline__ T block_excl_sum(T v, T *s_tmp, T *total)
{
    constexpr int W = BLOCK / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    T inc = warp_incl_sum(v);
    if (lane == 31) s_tmp[w] = inc;
    __syncthreads();
    if (w == 0) {
        T x = lane < W ? s_tmp[lane] : T(0);
        x = warp_incl_sum(x);
        if (lane < W) s_tmp[lane] = x;
    }
    __syncthreads();
    T wex = w ? s_tmp[w - 1] : T(0);
    *total = s_tmp[W - 1];
    __syncthreads();
    return wex + inc - v;
}

constexpr unsigned long long LB64_AGG = 1ull << 62;
constexpr unsigned long long LB64_PREFIX = 2ull << 62;
constexpr unsigned long long LB64_VALUE = (1ull << 62) - 1ull;

// Decoupled look-back of tile t over 64-bit status words (flag | value), run
// by one whole warp: publishes t's aggregate, reads 32 predecessors per round
// trip (lane q reads tile k - q), adds every aggregate up to the nearest
// inclusive prefix, then publishes t's own inclusive prefix.  A word not yet
// published ahead of that prefix means polling the window again, at most
// SPIN_LIMIT times (then ERR_TIMEOUT and the partial sum).  Returns the
// exclusive prefix in every lane.
__device__ __forceinline__ unsigned long long warp_lookback64(unsigned long long *st, unsigned t,
                                                              unsigned long long total, Ctl *ctl)
{
    const int lane = threadIdx.x & 31;
    unsigned long long excl = 0;
    if (t == 0) {
        if (lane == 0) st_relaxed_u64(&st[0], LB64_PREFIX | total);
        return 0ull;
    }
    if (lane == 0) st_relaxed_u64(&st[t], LB64_AGG | total);
    long long k = (long long)t - 1;
    unsigned spins = 0;
    while (true) {
        const long long idx = k - lane;
        const unsigned long long v = idx >= 0 ? ld_relaxed_u64(&st[idx]) : LB64_PREFIX;
        const unsigned pre = __ballot_sync(0xffffffffu, (v & LB64_PREFIX) != 0ull);
        const unsigned zero = __ballot_sync(0xffffffffu, v == 0ull);
        const int p = pre ? __ffs(pre) - 1 : 32;                // nearest prefix in the window
        const unsigned upto = p < 31 ? (2u << p) - 1u : 0xffffffffu;
        if (zero & upto) {                                       // a nearer tile has not published
            if (++spins > SPIN_LIMIT) {
                if (lane == 0) atomicOr(&ctl->err, ERR_TIMEOUT);
                break;
            }
            if (spins > 8) __nanosleep(64);
            continue;
        }
        unsigned long long part = lane <= p ? (v & LB64_VALUE) : 0ull;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
        excl += part;
        if (p < 32) break;
        k -= 32;
    }
    if (lane == 0) st_relaxed_u64(&st[t], LB64_PREFIX | ((excl + total) & LB64_VALUE));
    return excl;
}

#endif  // __CUDACC__

}  // namespace gg
