// Brick builds (sm_103a): RadixSort, RunLengthEncode, NonEmptyCells and
// ExclusiveSum of Algorithm 1 over bricks of cells instead of single cells.
//
// A triangle's pairs fill a box of cells, so the sort need not carry them one
// by one.  The grid is cut into bricks (8 x 8 x 8 cells); the sorted entries are
// (brick, object) with the object's box inside the brick packed into the spare
// key and value bits (BrickGen): 1.2 to 1.6 entries per triangle on the
// scenes of scenes/, against 3 to 140 pairs.  The stable radix passes leave
// every brick's entries in ascending object order, and the pairs first appear
// in device memory as the final refs.
//
//   split   work items: a brick's entries, at most BRICK_CHUNK each.
//   count   objects per cell.
//   scan    exclusive sums of the counts: G (localized per mesh in a batch).
//   fill    refs: every cell's objects in ascending order at G[cell].
//
// count and fill find the objects of a cell by bit masks.  32 entries at a
// time, a warp turns the boxes into 32 rows of feature bits (columns x, rows
// y, layers z that the box covers) and transposes them, so that lane f holds
// which of the 32 entries cover feature f; the entries covering cell (x, y, z)
// are then X[x] & Y[y] & Z[z].  No atomics, no per-pair search, and ascending
// bits are ascending objects.
//
// Measured, whole builds, sorted pairs then bricks: 10M-triangle building (2.4
// pairs per cell, 2.0e8 pairs) 4.00 -> 1.72 ms; soup of 1M triangles (8.3e7 pairs)
// 1.68 -> 0.33; soup of 7.3M (1.0e9 pairs) 22.7 -> 1.95; 64 soups (1.6e9 pairs)
// 35.5 -> 3.6.  The pair path moved 12.8, 5.5, 70 and 91 GB for them, the
// bricks 4.0, 0.6, 6.1 and 9.5.
#include <atomic>
#include <cstdint>

#include "cull.cuh"
#include "device.cuh"
#include "kernels.h"

namespace gg {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr unsigned NO_SLOT = 0xFFFFFFFFu;
constexpr int GROUPS = BRICK_CELLS / 32;   // groups of 32 cells, in cell order

// Decoded BrickItem::dims.
struct Dims {
    unsigned nx, ny, nz;   // cells inside the grid per axis
    unsigned lx, ly, lz;
};

__device__ __forceinline__ Dims decode(unsigned d)
{
    return Dims{(d & 31u) + 1u, ((d >> 5) & 31u) + 1u, ((d >> 10) & 31u) + 1u, (d >> 15) & 7u, (d >> 18) & 7u,
                (d >> 21) & 7u};
}

__device__ __forceinline__ BrickItem load_item(const BrickItem *p)
{
    const uint4 a = __ldg(reinterpret_cast<const uint4 *>(p)), b = __ldg(reinterpret_cast<const uint4 *>(p) + 1);
    return BrickItem{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
}

// Bits a .. b (inclusive) set.
__device__ __forceinline__ unsigned bit_run(unsigned a, unsigned b) { return (2u << b) - (1u << a); }

// Feature bits of an entry's box: columns at bit 0, rows at 2^lx, layers at
// 2^lx + 2^ly.
__device__ __forceinline__ unsigned feature_row(unsigned info, const Dims &d)
{
    const unsigned l0 = info & (BRICK_CELLS - 1u), l1 = (info >> BRICK_CELLS_LOG) & (BRICK_CELLS - 1u);
    const unsigned mx = (1u << d.lx) - 1u, my = (1u << d.ly) - 1u, mz = (1u << d.lz) - 1u;
    const unsigned lxy = d.lx + d.ly;
    const unsigned X = bit_run(l0 & mx, l1 & mx);
    const unsigned Y = bit_run((l0 >> d.lx) & my, (l1 >> d.lx) & my);
    const unsigned Z = bit_run((l0 >> lxy) & mz, (l1 >> lxy) & mz);
    return X | (Y << (1u << d.lx)) | (Z << ((1u << d.lx) + (1u << d.ly)));
}

// 32 x 32 bit transpose across the warp: bit j of lane i moves to bit i of
// lane j.
__device__ __forceinline__ unsigned transpose32(unsigned x)
{
    const unsigned lane = threadIdx.x & 31u;
    unsigned m = 0x0000FFFFu;
#pragma unroll
    for (unsigned j = 16u; j; j >>= 1, m ^= m << j) {
        const unsigned y = __shfl_xor_sync(FULL, x, j);
        x = (lane & j) ? (x & ~m) | ((y & ~m) >> j) : (x & m) | ((y & m) << j);
    }
    return x;
}

// Entry e + k of an item (n entries left from e) in lane 31 - k, so that in a
// transposed mask counting leading zeros walks the entries in ascending order.
struct Entry {
    unsigned key, val;
    bool ok;
};

__device__ __forceinline__ Entry load_entry(const BrickArgs &a, unsigned e, unsigned n)
{
    const unsigned k = 31u - (threadIdx.x & 31u);
    Entry r{0u, 0u, k < n};
    if (r.ok) {
        r.key = __ldg(a.keys + e + k);
        r.val = __ldg(a.vals + e + k);
    }
    return r;
}

// The packed box, and the object.
__device__ __forceinline__ unsigned entry_info(const BrickArgs &a, const Entry &r)
{
    return (r.key >> a.kb) | ((r.val >> a.ob) << brick_key_info_bits(a.kb));
}

__device__ __forceinline__ unsigned entry_obj(const BrickArgs &a, const Entry &r) { return r.val & ((1u << a.ob) - 1u); }

// Mesh of a brick (the last m with brick_base[m] <= b; every mesh has bricks).
__device__ __forceinline__ int mesh_of_brick(const MeshTab &mt, unsigned b)
{
    int lo = 0, hi = mt.nm - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&mt.md[mid].brick_base) <= b)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// First entry of brick b (b <= nbricks): the number of keys of bricks below b.
__device__ __forceinline__ unsigned brick_start(const BrickArgs &a, unsigned b)
{
    if (b >= a.nbricks) return a.count;
    const unsigned mask = (1u << a.kb) - 1u;
    unsigned lo = 0, hi = a.count;
    while (lo < hi) {
        const unsigned mid = lo + ((hi - lo) >> 1);
        if ((__ldg(a.keys + mid) & mask) < b)
            lo = mid + 1u;
        else
            hi = mid;
    }
    return lo;
}

}  // namespace

// ---------------------------------------------------------------------------
// split: bricks -> work items
// ---------------------------------------------------------------------------

// One thread per brick: its first entry by binary search.  The block then writes
// its bricks' items (and, for culled builds, their words) one after another, a
// thread per item, so that a brick of thousands of chunks takes no longer than
// as many bricks: with each thread writing its own brick's, a brick of 4M entries
// took 145 us (774 culled), now under 20 (76).  Empty bricks go to the other end of the
// list: only the count visits them, to write their zeros.  Bound by the
// searches' dependent loads (21 us for 163,000 bricks).
constexpr unsigned SPLIT_BLOCK = 256;

__global__ void __launch_bounds__(SPLIT_BLOCK) brick_split_kernel(BrickArgs a)
{
    after_stream();
    __shared__ unsigned s_start[SPLIT_BLOCK + 1];
    __shared__ unsigned s_tmp[SPLIT_BLOCK / 32];
    __shared__ unsigned s_base, s_ebase, s_wbase;
    __shared__ BrickItem s_item[SPLIT_BLOCK];       // the brick, its entries as one item; slot: the first chunk's
    __shared__ unsigned s_iex[SPLIT_BLOCK], s_wex[SPLIT_BLOCK];   // items and words of the bricks before
    const unsigned tid = threadIdx.x, b0 = blockIdx.x * SPLIT_BLOCK, b = b0 + tid;
    if (b <= a.nbricks) s_start[tid] = brick_start(a, b);
    if (tid == SPLIT_BLOCK - 1u && b + 1u <= a.nbricks) s_start[SPLIT_BLOCK] = brick_start(a, b + 1u);
    __syncthreads();
    const bool ok = b < a.nbricks;
    BrickItem it{};
    unsigned k = 0u;
    if (ok) {
        it.first = s_start[tid];
        it.count = s_start[tid + 1] - it.first;
        k = (it.count + BRICK_CHUNK - 1u) / BRICK_CHUNK;
        unsigned shape = a.shape, nbx = a.nbx, nby = a.nby, lb = b;
        int r[3] = {a.res[0], a.res[1], a.res[2]};
        unsigned long long c0 = 0ull;
        if (a.mt.md) {
            const int q = mesh_of_brick(a.mt, b);
            const MeshDesc &md = a.mt.md[q];
            shape = md.shape;
            nbx = md.nbx;
            nby = md.nby;
            lb = b - md.brick_base;
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) r[ax] = md.res[ax];
            c0 = (unsigned long long)__ldg(a.cells_off + q);
            it.base = __ldg(a.pair_base + q);
        }
        const unsigned lx = shape & 15u, ly = (shape >> 4) & 15u, lz = (shape >> 8) & 15u;
        const unsigned bz = lb / (nbx * nby), rem = lb - bz * nbx * nby, by = rem / nbx, bx = rem - by * nbx;
        const unsigned x0 = bx << lx, y0 = by << ly, z0 = bz << lz;
        it.rx = (unsigned)r[0];
        it.rxy = (unsigned)r[0] * (unsigned)r[1];
        it.cell0 = (unsigned)(c0 + x0 + (unsigned long long)it.rx * (y0 + (unsigned long long)r[1] * z0));
        const unsigned ex = min(1u << lx, (unsigned)r[0] - x0) - 1u, ey = min(1u << ly, (unsigned)r[1] - y0) - 1u,
                       ez = min(1u << lz, (unsigned)r[2] - z0) - 1u;
        it.dims = ex | (ey << 5) | (ez << 10) | (lx << 15) | (ly << 18) | (lz << 21);
        it.slot = k > 1u ? atomicAdd(&a.ctl->tickets[4], k) : NO_SLOT;
    }
    const bool empty = ok && k == 0u;
    unsigned total, etotal, wtotal = 0u;
    const unsigned iex = block_excl_sum<SPLIT_BLOCK>(k, s_tmp, &total);
    const unsigned eex = block_excl_sum<SPLIT_BLOCK>(empty ? 1u : 0u, s_tmp, &etotal);
    if (a.masks) s_wex[tid] = block_excl_sum<SPLIT_BLOCK>((it.count + 31u) / 32u, s_tmp, &wtotal);
    s_item[tid] = it;
    s_iex[tid] = iex;
    if (tid == 0u) {
        s_wbase = wtotal ? atomicAdd(&a.ctl->tickets[2], wtotal) : 0u;
        s_base = total ? atomicAdd(&a.ctl->tickets[3], total) : 0u;
        s_ebase = etotal ? atomicAdd(&a.ctl->tickets[6], etotal) : 0u;
    }
    __syncthreads();
    bool bad = false;   // never: the host sizes the lists for every split of `count` entries
    if (empty) {
        const unsigned p = s_ebase + eex;
        if (p < a.max_items)
            a.items[a.max_items - 1u - p] = it;
        else
            bad = true;
    }
    // the last brick of the block with before[q] <= i: the one that holds item (or word) i
    auto brick_of = [](const unsigned *before, unsigned i) {
        unsigned lo = 0u;
#pragma unroll
        for (unsigned step = SPLIT_BLOCK / 2u; step; step >>= 1)
            if (before[lo + step] <= i) lo += step;
        return lo;
    };
    for (unsigned i = tid; i < total; i += SPLIT_BLOCK) {
        const unsigned q = brick_of(s_iex, i), j = i - s_iex[q], p = s_base + i;
        BrickItem o = s_item[q];
        const unsigned m = o.count, chunks = (m + BRICK_CHUNK - 1u) / BRICK_CHUNK, slot0 = o.slot;
        o.first += j * BRICK_CHUNK;
        o.count = min((unsigned)BRICK_CHUNK, m - j * BRICK_CHUNK);
        if (chunks > 1u) {
            o.slot = slot0 + j;
            if (o.slot >= a.max_slots) {
                bad = true;
                continue;
            }
            a.slot_meta[o.slot] = make_uint2(slot0, chunks);
            a.arrive[o.slot] = 0u;
        }
        if (p >= a.max_items) {
            bad = true;
            continue;
        }
        a.items[p] = o;
        if (a.masks) {
            const unsigned w0 = s_wbase + s_wex[q] + j * (BRICK_CHUNK / 32), words = (o.count + 31u) / 32u;
            const bool fits = w0 + words <= a.max_words;
            a.mask0[p] = fits ? w0 : 0u;
            if (fits)
                for (unsigned w = 0; w < words; ++w) a.word_item[w0 + w] = p;
            bad |= !fits;
        }
    }
    if (bad) atomicOr(&a.ctl->err, ERR_RANGE);
}

// ---------------------------------------------------------------------------
// count: objects per cell
// ---------------------------------------------------------------------------

constexpr int COUNT_WARPS = 4;

// Adds an item's entries to cnt: lane l of group g counts cell 32 g + l.  The
// next word's entries are loaded while one is counted.
__device__ __forceinline__ void count_words(const BrickArgs &a, const BrickItem &it, const Dims &d,
                                            unsigned (&cnt)[GROUPS])
{
    const unsigned lane = threadIdx.x & 31u;
    const unsigned fy = 1u << d.lx, fz = fy + (1u << d.ly);
    const bool cube = d.lx == 3u && d.ly == 3u && d.lz == 3u;
    const int ngroups = max(1, 1 << (d.lx + d.ly + d.lz) >> 5);
    Entry next = load_entry(a, it.first, it.count);
    for (unsigned e = 0; e < it.count; e += 32u) {
        const Entry cur = next;
        const unsigned en = e + 32u;
        next = load_entry(a, it.first + en, en < it.count ? it.count - en : 0u);
        const unsigned f = transpose32(cur.ok ? feature_row(entry_info(a, cur), d) : 0u);
        if (cube) {   // cell 32 g + l is (l % 8, 4 (g % 2) + l / 8, g / 2)
            const unsigned mx = __shfl_sync(FULL, f, lane & 7u);
            const unsigned m0 = mx & __shfl_sync(FULL, f, 8u + (lane >> 3));
            const unsigned m1 = mx & __shfl_sync(FULL, f, 12u + (lane >> 3));
#pragma unroll
            for (int z = 0; z < 8; ++z) {
                const unsigned mz = __shfl_sync(FULL, f, 16 + z);
                cnt[2 * z] += __popc(m0 & mz);
                cnt[2 * z + 1] += __popc(m1 & mz);
            }
        } else {
#pragma unroll
            for (int g = 0; g < GROUPS; ++g) {
                if (g < ngroups) {
                    const unsigned c = 32u * g + lane;
                    const unsigned mx = __shfl_sync(FULL, f, c & ((1u << d.lx) - 1u));
                    const unsigned my = __shfl_sync(FULL, f, fy + ((c >> d.lx) & ((1u << d.ly) - 1u)));
                    const unsigned mz = __shfl_sync(FULL, f, (fz + (c >> (d.lx + d.ly))) & 31u);
                    cnt[g] += __popc(mx & my & mz);
                }
            }
        }
    }
}

// Cells of BRICK_BIG objects and more: a table of open addresses, at most half
// full (each such cell holds 65,535 pairs).  As a list searched from its front it
// made the scans of 512 cells of 65,000 objects take 147 us, now under 20.
__device__ __forceinline__ unsigned big_place(int bits, unsigned cell)
{
    return (cell * 0x9E3779B1u) >> (32 - bits);   // Fibonacci hashing (Knuth)
}

__device__ __noinline__ bool note_big(uint2 *big, int bits, unsigned cell, unsigned count)
{
    const unsigned mask = (1u << bits) - 1u;
    unsigned h = big_place(bits, cell);
    for (unsigned k = 0; k <= mask; ++k, h = (h + 1u) & mask) {
        if (atomicCAS(&big[h].x, 0u, cell + 1u) == 0u) {
            big[h].y = count;
            return true;
        }
    }
    return false;
}

__device__ __noinline__ unsigned big_count(const uint2 *big, int bits, unsigned cell)
{
    const unsigned mask = (1u << bits) - 1u;
    unsigned h = big_place(bits, cell);
    for (unsigned k = 0; k <= mask; ++k, h = (h + 1u) & mask) {
        const uint2 e = big[h];
        if (e.x == cell + 1u) return e.y;
        if (e.x == 0u) break;
    }
    return 0u;
}

// Rows of a brick in k > 1 chunks: its chunks' counts at slots [s, s + k) and, when
// k > MERGE_CHUNKS, the sums of merge_group(k) chunks each at group_row.
constexpr unsigned MERGE_CHUNKS = 32;

// The smallest power of two whose square is at least k, 16 at the least.
__host__ __device__ __forceinline__ unsigned merge_group(unsigned k)
{
    unsigned g = 16u;
    while (g < 65536u && g * g < k) g <<= 1;
    return g;
}

// First of a brick's group rows, behind the max_slots chunk rows: more than
// MERGE_CHUNKS chunks make at most k / 8 groups, so the rows of two bricks
// (their slots follow one another) stay apart.
__device__ __forceinline__ unsigned group_row(const BrickArgs &a, unsigned slot0) { return a.max_slots + (slot0 + 7u) / 8u; }

// Turns n rows of counts into offsets (each the sum of the rows before) and
// adds them up in cnt (one warp; lane l of group g has cell 32 g + l).
__device__ __forceinline__ void scan_rows(unsigned *rows, unsigned n, unsigned (&cnt)[GROUPS])
{
    const unsigned lane = threadIdx.x & 31u;
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) cnt[g] = 0u;
    for (unsigned j = 0; j < n; ++j) {
        unsigned *row = rows + (size_t)j * BRICK_CELLS + lane, v[GROUPS];
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) v[g] = __ldcg(row + 32 * g);
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) {
            row[32 * g] = cnt[g];
            cnt[g] += v[g];
        }
    }
}

// One more of n arrivals at *count: is it the last?  What the warps that
// arrived before wrote is visible to the last.
__device__ __forceinline__ bool last_to_arrive(unsigned *count, unsigned n)
{
    __threadfence();
    __syncwarp();
    unsigned last = 0u;
    if ((threadIdx.x & 31u) == 0u) last = atomicAdd(count, 1u) + 1u == n;
    last = __shfl_sync(FULL, last, 0);
    if (last) __threadfence();
    return last;
}

// Writes an item's counts (lane l of group g has cell 32 g + l; one warp).  A
// brick in one item writes its cells' counts; a chunk writes its own to its
// slot, and the last chunk of the brick to arrive turns the slots into offsets
// inside each cell and writes the sums.  A slot costs that warp a round trip to
// L2 (0.24 us), so a brick of more than MERGE_CHUNKS chunks is added up in two
// levels: the last chunk of each group to arrive does the group's slots, the
// last group the groups' sums.
__device__ __forceinline__ void finish_counts(const BrickArgs &a, const BrickItem &it, const Dims &d,
                                              unsigned (&cnt)[GROUPS])
{
    const unsigned lane = threadIdx.x & 31u;
    if (it.slot != NO_SLOT) {
        unsigned *sl = a.slots + (size_t)it.slot * BRICK_CELLS;
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) sl[32 * g + lane] = cnt[g];
        const uint2 meta = a.slot_meta[it.slot];   // the brick's first slot, its chunks
        bool top = meta.y <= MERGE_CHUNKS;
        const unsigned per = top ? meta.y : merge_group(meta.y), q = (it.slot - meta.x) / per;
        unsigned row0 = meta.x + q * per, n = min(per, meta.y - q * per), *arrive = a.arrive + row0;
        for (;;) {
            if (!last_to_arrive(arrive, n)) return;
            scan_rows(a.slots + (size_t)row0 * BRICK_CELLS, n, cnt);
            if (top) break;
            top = true;
            row0 = group_row(a, meta.x);
            n = (meta.y + per - 1u) / per;
            arrive = a.arrive + meta.x + 1u;   // no group starts at a brick's second slot
            unsigned *sum = a.slots + (size_t)(row0 + q) * BRICK_CELLS + lane;
#pragma unroll
            for (int g = 0; g < GROUPS; ++g) sum[32 * g] = cnt[g];
        }
    }
    unsigned most = 0u;
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) most = max(most, cnt[g]);
    const bool big = most >= BRICK_BIG;
    if (d.nx == 8u && d.ny == 8u && d.nz == 8u && !big) {   // a whole cube: steps of 4 rows and of a layer
        unsigned short *p = a.counts + (it.cell0 + (lane & 7u) + it.rx * (lane >> 3));
#pragma unroll
        for (int g = 0; g < GROUPS; ++g)
            p[(size_t)(g & 1) * (4u * it.rx) + (size_t)(g >> 1) * it.rxy] = (unsigned short)cnt[g];
        return;
    }
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) {
        const unsigned c = 32u * g + lane;
        const unsigned x = c & ((1u << d.lx) - 1u), y = (c >> d.lx) & ((1u << d.ly) - 1u), z = c >> (d.lx + d.ly);
        if (x < d.nx && y < d.ny && z < d.nz) {
            const unsigned cell = it.cell0 + x + it.rx * y + it.rxy * z;
            a.counts[cell] = (unsigned short)min(cnt[g], BRICK_BIG);
            if (cnt[g] >= BRICK_BIG) {
                atomicAdd(&a.ctl->tickets[1], 1u);
                if (!note_big(a.big, a.big_bits, cell, cnt[g]))
                    atomicOr(&a.ctl->err, ERR_RANGE);   // never: half of the table stays free
            }
        }
    }
}

// A warp per item.  CULLED: the kept masks of its words instead of the boxes,
// and their sum in ctl->nkept.
//
// Bound by the latency of an item's loads (its record, its entries, an object's
// spilled box bits) with 8 blocks of 4 warps per SM, then by issue: 193 us at
// 163,000 bricks (80M cells, 1.6e7 entries), 96 us at 59,000 bricks of crowded
// cells.  More resident blocks spill (9, 10, 12 per SM: 189, 201, 206 us and 107,
// 100, 120); 6 and 7 hide less (207, 205).
template <bool CULLED>
__global__ void __launch_bounds__(32 * COUNT_WARPS, 8) brick_count_kernel(BrickArgs a)
{
    after_stream();
    const unsigned lane = threadIdx.x & 31u;
    const unsigned nitems = min(ld_relaxed_u32(&a.ctl->tickets[3]), a.max_items);
    const unsigned nempty = min(ld_relaxed_u32(&a.ctl->tickets[6]), a.max_items);
    for (unsigned i = blockIdx.x * COUNT_WARPS + (threadIdx.x >> 5); i < nitems + nempty; i += gridDim.x * COUNT_WARPS) {
        const BrickItem it = load_item(a.items + (i < nitems ? i : a.max_items - 1u - (i - nitems)));
        const Dims d = decode(it.dims);
        unsigned cnt[GROUPS];
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) cnt[g] = 0u;
        if (CULLED) {
            if (it.count) {
                const unsigned *in = a.masks + (size_t)__ldg(a.mask0 + i) * BRICK_CELLS + lane;
                for (unsigned e = 0; e < it.count; e += 32u, in += BRICK_CELLS) {
#pragma unroll
                    for (int g = 0; g < GROUPS; ++g) cnt[g] += __popc(__ldg(in + 32 * g));
                }
                unsigned sum = 0u;
#pragma unroll
                for (int g = 0; g < GROUPS; ++g) sum += cnt[g];
                sum = __reduce_add_sync(FULL, sum);
                if (lane == 0u && sum) atomicAdd(&a.ctl->nkept, (unsigned long long)sum);
            }
        } else {
            count_words(a, it, d, cnt);
        }
        finish_counts(a, it, d, cnt);
    }
}

// ---------------------------------------------------------------------------
// cull: the entries that each cell keeps, and their counts (culled builds)
// ---------------------------------------------------------------------------

// The test of cull.cuh decides every pair exactly as the pair path does; what
// changes is which pairs reach it, and that full warps run it.  A word of 32
// entries per warp: a lane sets up its entry's triangle and looks through the
// box inside the brick when that has at most CULL_OWN cells; the warp looks
// through a larger one, two rows of the brick per lane.  A cell that holds a
// vertex is kept at once; one whose centre lies further from the triangle's
// plane than any cell that the normal's axis could keep is dropped after one
// multiply-add (most cells of a large triangle's box); the others are listed,
// and the test runs over the list, a pair per lane.
//
// That bound, T: the test drops a cell when the three projections p_k = n . w_k
// all lie beyond R = S (1/2 + max|w| 2^-16 + 2^-10) on one side, S = |n_x| + |n_y| +
// |n_z|.  The cell is dropped here when its plane value v, p_0 but for rounding,
// lies beyond T: so T has to exceed R by what the three can differ from v.  Let
// the FP32 edges have components up to L, and |w| be up to W over the
// brick; S <= 4 L^2 (a 3 x 3 determinant of entries up to 1 is at most 4).
//  - n . (q_k - q_0) is not zero: each component of the FP32 cross product is off by
//    4 u L^2 (u = 2^-24) and each edge by u L, which makes 16 u L^3 for k = 1 and 28 u
//    L^3 for k = 2 (the three rounded edges do not add up to zero).
//  - The test's rounding of a projection (w, three products, two sums): 4 u S W.
//  - The rounding of v (q - c0, three fused steps to the brick's first cell, three
//    to this one): 7 u S W.
// Together 28 u L^3 + 11 u S W <= 28 u L^3 + 44 u L^2 W.  T = S (1/2 + W 2^-16 + 2^-10)
// (1 + 2^-10) + 2^-18 L^2 (L + W) exceeds R by more than 64 u L^3 + 64 u L^2 W.
//
// Bound by issue (73% of cycles).  Tests and compaction pair by pair, ahead of a
// sort of the pairs, then this kernel: 1150 -> 297 us on the soup of 1M triangles,
// 764 -> 706 on a building of 2M.  A block per item instead of a warp per word:
// 408 and 2038; rows of large boxes one lane each: 820 and 5018.
constexpr int CULL_WARPS = 4;
constexpr unsigned CULL_OWN = 16;
constexpr unsigned CULL_LIST = 512;   // pairs listed for the test
static_assert(CULL_LIST >= BRICK_CELLS && CULL_LIST >= 32 * CULL_OWN, "one step lists no more than fits");
constexpr int CULL_TRI = 25;   // words per triangle in shared memory (24 and a pad)

__global__ void __launch_bounds__(32 * CULL_WARPS, 7) brick_cull_kernel(BrickArgs a)
{
    after_stream();
    __shared__ unsigned s_keep[CULL_WARPS][BRICK_CELLS];   // per cell: the word's kept entries; zero between words
    __shared__ float s_tri[CULL_WARPS][32 * CULL_TRI];
    __shared__ unsigned short s_list[CULL_WARPS][CULL_LIST];   // (entry's lane, cell) of pairs to test
    const unsigned lane = threadIdx.x & 31u, w = threadIdx.x >> 5, below = lanemask_lt();
    const unsigned nwords = min(ld_relaxed_u32(&a.ctl->tickets[2]), a.max_words);
    const float lo[3] = {a.lo[0], a.lo[1], a.lo[2]}, scale[3] = {a.scale[0], a.scale[1], a.scale[2]};
    const float resf[3] = {(float)a.res[0], (float)a.res[1], (float)a.res[2]};
    const unsigned zero3[3] = {0u, 0u, 0u};
    const unsigned last3[3] = {(unsigned)a.res[0] - 1u, (unsigned)a.res[1] - 1u, (unsigned)a.res[2] - 1u};
    unsigned *keep = s_keep[w];
    float *tris = s_tri[w];
    unsigned short *list = s_list[w];
    for (unsigned c = lane; c < BRICK_CELLS; c += 32u) keep[c] = 0u;
    __syncwarp();
    for (unsigned word = blockIdx.x * CULL_WARPS + w; word < nwords; word += gridDim.x * CULL_WARPS) {
        const unsigned item = __ldg(a.word_item + word);
        const BrickItem it = load_item(a.items + item);
        const unsigned q = word - __ldg(a.mask0 + item);
        if (32u * q >= it.count) continue;   // never with consistent lists
        const Dims d = decode(it.dims);
        const unsigned lxy = d.lx + d.ly, mskx = (1u << d.lx) - 1u, msky = (1u << d.ly) - 1u;
        const unsigned bz = it.cell0 / it.rxy, by = (it.cell0 - bz * it.rxy) / it.rx, bx = it.cell0 - bz * it.rxy - by * it.rx;
        const unsigned org[3] = {bx, by, bz};   // the brick's first cell
        const Entry en = load_entry(a, it.first + 32u * q, it.count - 32u * q);
        const unsigned info = entry_info(a, en);
        const unsigned l0 = info & (BRICK_CELLS - 1u), l1 = (info >> BRICK_CELLS_LOG) & (BRICK_CELLS - 1u);
        const unsigned nx = (l1 & mskx) - (l0 & mskx) + 1u, ny = ((l1 >> d.lx) & msky) - ((l0 >> d.lx) & msky) + 1u;
        const unsigned vol = en.ok ? nx * ny * ((l1 >> lxy) - (l0 >> lxy) + 1u) : 0u;
        GridTri t;
        unsigned live = 0u;
        float A = 0.0f, T = 0.0f;   // the plane's value at the centre of the brick's first cell, the bound
        if (en.ok) {
            grid_tri(a.verts, a.nverts, a.tris, entry_obj(a, en), lo, scale, resf, t, a.ctl);
            live = live_axes(t);
            float W = 0.0f, L = 0.0f;
            const unsigned ext[3] = {mskx, msky, (1u << d.lz) - 1u};
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                const float c0 = (float)org[ax] + 0.5f, c1 = c0 + (float)ext[ax];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    W = fmaxf(W, fmaxf(fabsf(t.q[3 * k + ax] - c0), fabsf(t.q[3 * k + ax] - c1)));
                    L = fmaxf(L, fabsf(t.e[3 * k + ax]));
                }
                A = fmaf(t.n[ax], t.q[ax] - c0, A);
            }
            const float S = fabsf(t.n[0]) + fabsf(t.n[1]) + fabsf(t.n[2]);
            T = fmaf(S, (0.5f + 9.765625e-04f + W * 1.52587890625e-05f) * 1.0009765625f,
                     3.814697265625e-06f * (L * L) * (L + W));
            if (!(live & 1u)) T = __int_as_float(0x7f800000);   // the test skips the normal: no bound from it
        }
        if (en.ok) {
            float *o = tris + lane * CULL_TRI;
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                o[k] = t.q[k];
                o[9 + k] = t.e[k];
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) o[18 + k] = t.n[k];
            o[21] = A;
            o[22] = T;
            o[23] = __uint_as_float(live);
        }
        unsigned listed = 0u;
        auto append = [&](bool cand, unsigned c, unsigned e) {   // the lanes with cand list (e, c)
            const unsigned m = __ballot_sync(FULL, cand);
            if (cand) list[listed + __popc(m & below)] = (unsigned short)((e << BRICK_CELLS_LOG) | c);
            listed += __popc(m);
        };
        auto test = [&]() {
            __syncwarp();
            for (unsigned k = lane; k < listed; k += 32u) {
                const unsigned v = list[k], c = v & (BRICK_CELLS - 1u), e = v >> BRICK_CELLS_LOG;
                const float *o = tris + e * CULL_TRI;
                GridTri g;
#pragma unroll
                for (int j = 0; j < 9; ++j) {
                    g.q[j] = o[j];
                    g.e[j] = o[9 + j];
                }
#pragma unroll
                for (int j = 0; j < 3; ++j) g.n[j] = o[18 + j];
                if (!tri_cell_separated(g, __float_as_uint(o[23]), bx + (c & mskx), by + ((c >> d.lx) & msky),
                                        bz + (c >> lxy)))
                    atomicOr(&keep[c], 1u << e);
            }
            listed = 0u;
            __syncwarp();
        };
        {
            // boxes of few cells: the lane's own, cell by cell in box order
            const bool own = vol <= CULL_OWN;
            unsigned long long vc[3] = {0ull, 0ull, 0ull};
            if (own && en.ok) {
#pragma unroll
                for (int k = 0; k < 3; ++k) vc[k] = vertex_cell(t, k, zero3, last3);
            }
            unsigned c = l0, x = nx, y = ny;
            const unsigned steps = __reduce_max_sync(FULL, own ? vol : 0u);
            for (unsigned k = 0; k < steps; ++k) {
                bool cand = own && k < vol;
                if (cand) {
                    const unsigned cx = c & mskx, cy = (c >> d.lx) & msky, cz = c >> lxy;
                    const unsigned long long rc = (unsigned long long)(bx + cx) |
                                                  ((unsigned long long)(by + cy) << 16) |
                                                  ((unsigned long long)(bz + cz) << 32);
                    if (rc == vc[0] || rc == vc[1] || rc == vc[2]) {
                        atomicOr(&keep[c], 1u << lane);
                        cand = false;
                    } else {
                        const float v =
                            fmaf(-t.n[0], (float)cx, fmaf(-t.n[1], (float)cy, fmaf(-t.n[2], (float)cz, A)));
                        cand = !(fabsf(v) > T);
                    }
                }
                append(cand, c, lane);
                ++c;
                if (--x == 0u) {
                    x = nx;
                    c += (1u << d.lx) - nx;
                    if (--y == 0u) {
                        y = ny;
                        c += (1u << lxy) - (ny << d.lx);
                    }
                }
            }
        }
        __syncwarp();
        for (unsigned large = __ballot_sync(FULL, vol > CULL_OWN); large; large &= large - 1u) {
            const unsigned from = (unsigned)__ffs(large) - 1u;
            const unsigned b0 = __shfl_sync(FULL, l0, from), bnx = __shfl_sync(FULL, nx, from),
                           bny = __shfl_sync(FULL, ny, from), bv = __shfl_sync(FULL, vol, from);
            const float *o = tris + from * CULL_TRI;
            const float n0 = o[18], n1 = o[19], n2 = o[20], pA = o[21], pT = o[22];
            const unsigned rx = 65535u / bnx + 1u, ry = 65535u / bny + 1u;   // exact quotients below 512
            if (listed + bv > CULL_LIST) test();
            for (unsigned k0 = 0; k0 < bv; k0 += 32u) {
                const unsigned k = k0 + lane, u = (k * rx) >> 16, z = (u * ry) >> 16;
                const unsigned c = b0 + (k - u * bnx) + ((u - z * bny) << d.lx) + (z << lxy);
                const unsigned cx = c & mskx, cy = (c >> d.lx) & msky, cz = c >> lxy;
                const float v = fmaf(-n0, (float)cx, fmaf(-n1, (float)cy, fmaf(-n2, (float)cz, pA)));
                append(k < bv && !(fabsf(v) > pT), c & (BRICK_CELLS - 1u), from);
            }
        }
        if (listed) test();
        __syncwarp();
        unsigned *out = a.masks + (size_t)word * BRICK_CELLS;
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) {
            out[32 * g + lane] = keep[32 * g + lane];
            keep[32 * g + lane] = 0u;
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// scan: counts -> G
// ---------------------------------------------------------------------------

// Exclusive sums of the counts into the cells array.  A warp takes 256 J
// consecutive cells in J coalesced 16-byte loads per lane.  In a batch each
// mesh's slice ends in one word more than its cells (counted 0, so it gets the
// mesh's total) and the sums are less the mesh's first pair; a single mesh is
// a batch of one.
//
// Up to SCAN_ONE_PASS cells: one pass, look-back between tiles.  Beyond, the
// look-back's chain would set the time (32 tiles per round trip): a first
// pass adds up each tile, its last block scans the sums, a second pass reads
// the counts again, half of them from L2 (80M cells: 165 us against 192 for
// the look-back, in the forms of that time).
//
// Both passes wait on their loads: what helps is bytes in flight and few, long
// blocks.  With SCAN_J_BIG loads per lane 80M cells take 123 us (J = 4: 149, 12:
// 119, 16: 117) and 25M 49 us (J = 4: 56, 12: 52, 16: 53); 4M cells fill
// the chip better with SCAN_J (16 us against 18), 8M take 22 us either way.
constexpr int SCAN_BLOCK = 256;
constexpr int SCAN_WARPS = SCAN_BLOCK / 32;
constexpr long long SCAN_ONE_PASS = 1ll << 20, SCAN_BIG = 1ll << 23;
constexpr int SCAN_J = 4, SCAN_J_BIG = 8;   // loads per lane of the two passes

template <int J>
__host__ __device__ constexpr long long scan_tile() { return (long long)SCAN_BLOCK * 8 * J; }

struct Counts8 {
    unsigned v[8];
};

// Mesh holding word p of the cells array (the last m with cells_off[m] <= p).
__device__ __forceinline__ int mesh_of_word(const BrickArgs &a, long long p)
{
    int lo = 0, hi = a.mt.nm - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(a.cells_off + mid) <= p)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// The 16-bit counts of words p .. p + 7 (p a multiple of 8) as they lie in
// memory, zero beyond the last word.
__device__ __forceinline__ uint4 load_raw(const BrickArgs &a, long long p)
{
    if (p + 8 <= a.ncells_out) return __ldcg(reinterpret_cast<const uint4 *>(a.counts + p));
    unsigned w[4] = {0u, 0u, 0u, 0u};
    for (int k = 0; k < 8; ++k)
        if (p + k < a.ncells_out) w[k >> 1] |= (unsigned)__ldcg(a.counts + p + k) << (16 * (k & 1));
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Is one of eight counts in 16 bits BRICK_BIG?
__device__ __forceinline__ bool has_big(const uint4 &q)
{
    return ((__vcmpeq2(q.x, 0xFFFFFFFFu) | __vcmpeq2(q.y, 0xFFFFFFFFu)) |
            (__vcmpeq2(q.z, 0xFFFFFFFFu) | __vcmpeq2(q.w, 0xFFFFFFFFu))) != 0u;
}

// The eight counts: zero at the end of a mesh's slice, the table's value for a
// cell of BRICK_BIG objects or more.  *m: a mesh at or before word p's on
// entry (batched), word p's on return.
__device__ __forceinline__ Counts8 unpack(const BrickArgs &a, const uint4 &q, long long p, int *m)
{
    Counts8 c;
    const long long n = a.ncells_out;
    const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        c.v[2 * k] = w[k] & 0xFFFFu;
        c.v[2 * k + 1] = w[k] >> 16;
    }
    if (a.mt.md) {
        if (p < n) {
            int s = *m;
            long long end = __ldg(a.cells_off + s + 1);
            while (end <= p) end = __ldg(a.cells_off + ++s + 1);
            *m = s;
            if (end <= p + 8) {   // a slice ends among the eight words
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (p + k < n) {
                        while (end <= p + k) end = __ldg(a.cells_off + ++s + 1);
                        if (p + k + 1 == end) c.v[k] = 0u;
                    }
                }
            }
        }
    } else if (p + 8 >= n) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (p + k + 1 >= n) c.v[k] = 0u;
    }
    if (has_big(q)) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (c.v[k] == BRICK_BIG) c.v[k] = big_count(a.big, a.big_bits, (unsigned)(p + k));
    }
    return c;
}

__device__ __forceinline__ unsigned sum8(const Counts8 &c)
{
    return ((c.v[0] + c.v[1]) + (c.v[2] + c.v[3])) + ((c.v[4] + c.v[5]) + (c.v[6] + c.v[7]));
}

// Eight words at a multiple of 32 bytes (the cells arrays start on 256), whole sectors
// at a time: as two 16-byte stores the scan took 172 against 151 us at 80M cells.
__device__ __forceinline__ void store8(unsigned *p, const unsigned (&o)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(o[0]), "r"(o[1]), "r"(o[2]),
                 "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
                 : "memory");
}

// G of words p .. p + 7 from the sum x before them.
__device__ __forceinline__ void store_offsets(const BrickArgs &a, long long p, const Counts8 &c, unsigned x, int m)
{
    unsigned o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        o[k] = x;
        x += c.v[k];
    }
    if (a.mt.md && p < a.ncells_out) {
        long long end = __ldg(a.cells_off + m + 1);
        unsigned base = __ldg(a.pair_base + m);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (p + k < a.ncells_out) {
                while (end <= p + k) {
                    end = __ldg(a.cells_off + ++m + 1);
                    base = __ldg(a.pair_base + m);
                }
                o[k] -= base;
            }
        }
    }
    if (p + 8 <= a.ncells_out) {
        store8(a.G + p, o);
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (p + k < a.ncells_out) a.G[p + k] = o[k];
    }
}

// A warp's words [p, p + 256 J): `inner` when they lie inside one mesh's slice,
// short of its last word, and none of their cells is in the table of big ones.
// Their counts are then the halves of the loaded words (raw), and `base` is the
// mesh's first pair.
struct WarpWords {
    int m;   // mesh of word p
    unsigned base;
    bool inner;
};

template <int J>
__device__ __forceinline__ WarpWords warp_words(const BrickArgs &a, long long p, const uint4 (&raw)[J])
{
    WarpWords s{0, 0u, false};
    long long end = a.ncells_out;
    const unsigned nbig = ld_relaxed_u32(&a.ctl->tickets[1]);
    if (a.mt.md && p < end) {
        s.m = mesh_of_word(a, p);
        end = __ldg(a.cells_off + s.m + 1);
        s.base = __ldg(a.pair_base + s.m);
    }
    s.inner = p + 256 * J < end;
    if (nbig && s.inner) {
        bool big = false;
#pragma unroll
        for (int j = 0; j < J; ++j) big |= has_big(raw[j]);
        s.inner = !__any_sync(FULL, big);
    }
    return s;
}

// The loads of load_raw where eight words are there.
template <int J>
__device__ __forceinline__ void load_words(const BrickArgs &a, long long p, uint4 (&raw)[J])
{
#pragma unroll
    for (int j = 0; j < J; ++j)
        raw[j] = p + 256 * j + 8 <= a.ncells_out ? __ldcg(reinterpret_cast<const uint4 *>(a.counts + p + 256 * j))
                                                 : make_uint4(0u, 0u, 0u, 0u);
}

__device__ __forceinline__ unsigned sum_halves(const uint4 &q)
{
    return __dp2a_lo(q.w, 0x0101u, __dp2a_lo(q.z, 0x0101u, __dp2a_lo(q.y, 0x0101u, __dp2a_lo(q.x, 0x0101u, 0u))));
}

// First pass: the sum of every tile; the last block to finish turns the sums
// into offsets.
template <int J>
__global__ void __launch_bounds__(SCAN_BLOCK, J > SCAN_J ? 4 : 6) cell_sums_kernel(const __grid_constant__ BrickArgs a, unsigned ntiles)
{
    after_stream();
    __shared__ unsigned s_warp[SCAN_WARPS];
    __shared__ unsigned s_last;
    unsigned *sums = reinterpret_cast<unsigned *>(a.status);
    const unsigned tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
    const long long pw = (long long)blockIdx.x * scan_tile<J>() + (long long)w * (256 * J), p0 = pw + 8 * lane;
    uint4 raw[J];
    load_words(a, p0, raw);
    const WarpWords ww = warp_words<J>(a, pw, raw);
    unsigned sum = 0u;
    if (ww.inner) {
#pragma unroll
        for (int j = 0; j < J; ++j) sum += sum_halves(raw[j]);
    } else {
        int m = ww.m;
#pragma unroll 1
        for (int j = 0; j < J; ++j) sum += sum8(unpack(a, load_raw(a, p0 + 256 * j), p0 + 256 * j, &m));
    }
    sum = __reduce_add_sync(FULL, sum);
    if (lane == 0u) s_warp[w] = sum;
    __syncthreads();
    if (tid == 0u) {
        unsigned t = 0u;
#pragma unroll
        for (int k = 0; k < SCAN_WARPS; ++k) t += s_warp[k];
        sums[blockIdx.x] = t;
        __threadfence();
        s_last = atomicAdd(&a.ctl->tickets[5], 1u) + 1u == gridDim.x;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    unsigned carry = 0u;
    for (unsigned c0 = 0; c0 < ntiles; c0 += 4u * SCAN_BLOCK) {
        const unsigned i = c0 + 4u * tid;
        unsigned v[4];
#pragma unroll
        for (unsigned k = 0; k < 4u; ++k) v[k] = i + k < ntiles ? __ldcg(sums + i + k) : 0u;
        unsigned total;
        unsigned x = carry + block_excl_sum<SCAN_BLOCK>(v[0] + v[1] + v[2] + v[3], s_warp, &total);
#pragma unroll
        for (unsigned k = 0; k < 4u; ++k) {
            if (i + k < ntiles) sums[i + k] = x;
            x += v[k];
        }
        carry += total;
    }
}

// The scan of one tile, from the first pass's offset or (LOOKBACK) from the
// tiles before it.
template <int J, bool LOOKBACK>
__global__ void __launch_bounds__(SCAN_BLOCK, J > SCAN_J ? 4 : 5) cell_scan_kernel(const __grid_constant__ BrickArgs a)
{
    after_stream();
    __shared__ unsigned s_tile;
    __shared__ unsigned s_warp[SCAN_WARPS];
    __shared__ unsigned s_excl;
    const unsigned tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
    unsigned tile = blockIdx.x;
    if (LOOKBACK) {   // tiles in ticket order, so every tile a look-back waits for has started
        if (tid == 0u) s_tile = atomicAdd(&a.ctl->tickets[5], 1u);
        __syncthreads();
        tile = s_tile;
    }
    const long long pw = (long long)tile * scan_tile<J>() + (long long)w * (256 * J), p0 = pw + 8 * lane;
    uint4 raw[J];
    load_words(a, p0, raw);
    const WarpWords ww = warp_words<J>(a, pw, raw);
    unsigned off[J];   // words of the warp before this lane's load j
    unsigned run = 0u;
    if (ww.inner) {
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const unsigned sum = sum_halves(raw[j]), inc = warp_incl_sum(sum);
            off[j] = run + inc - sum;
            run += __shfl_sync(FULL, inc, 31);
        }
    } else {
        int m = ww.m;
#pragma unroll 1
        for (int j = 0; j < J; ++j)
            run += __reduce_add_sync(FULL, sum8(unpack(a, load_raw(a, p0 + 256 * j), p0 + 256 * j, &m)));
    }
    if (lane == 31u) s_warp[w] = run;
    __syncthreads();
    if (w == 0u) {
        const unsigned x = lane < (unsigned)SCAN_WARPS ? s_warp[lane] : 0u;
        const unsigned inc = warp_incl_sum(x);
        if (lane < (unsigned)SCAN_WARPS) s_warp[lane] = inc - x;
        if (LOOKBACK) {
            const unsigned total = __shfl_sync(FULL, inc, SCAN_WARPS - 1);
            const unsigned long long excl = warp_lookback64(a.status, tile, total, a.ctl);
            if (lane == 0u) s_excl = (unsigned)excl;
        } else if (lane == 0u) {
            s_excl = __ldg(reinterpret_cast<const unsigned *>(a.status) + tile);
        }
    }
    __syncthreads();
    unsigned base = s_excl + s_warp[w];
    if (ww.inner) {
        base -= ww.base;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const unsigned c[4] = {raw[j].x, raw[j].y, raw[j].z, raw[j].w};
            unsigned o[8];
            o[0] = base + off[j];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                o[2 * k + 1] = o[2 * k] + (c[k] & 0xFFFFu);
                if (k < 3) o[2 * k + 2] = o[2 * k + 1] + (c[k] >> 16);
            }
            store8(a.G + p0 + 256 * j, o);
        }
        return;
    }
    int m = ww.m;
#pragma unroll 1
    for (int j = 0; j < J; ++j) {
        const Counts8 c = unpack(a, load_raw(a, p0 + 256 * j), p0 + 256 * j, &m);
        const unsigned sum = sum8(c), inc = warp_incl_sum(sum);
        store_offsets(a, p0 + 256 * j, c, base + inc - sum, m);
        base += __shfl_sync(FULL, inc, 31);
    }
}

// ---------------------------------------------------------------------------
// fill: refs
// ---------------------------------------------------------------------------

constexpr unsigned MASK_PITCH = 36;   // words a row of 32 masks: rows of different words in different banks
constexpr int FILL_WARPS = 4;         // a warp per 128 cells of the brick
static_assert(BRICK_CHUNK <= 1024, "10 bits of entry in a tag");
static_assert(BRICK_CELLS == FILL_WARPS * 128, "four cells per lane");

// The masks of a lane's four cells in word q: from the word's feature masks in
// shared memory, or (culled builds) from the kept masks in device memory.
struct BoxMasks {
    const unsigned *mx, *my, *mz;
    __device__ __forceinline__ uint4 operator()(unsigned q) const
    {
        const uint4 X = *reinterpret_cast<const uint4 *>(mx + MASK_PITCH * q);
        const unsigned yz = my[MASK_PITCH * q] & mz[MASK_PITCH * q];
        return make_uint4(X.x & yz, X.y & yz, X.z & yz, X.w & yz);
    }
};

struct KeptMasks {
    const unsigned *m;
    __device__ __forceinline__ uint4 operator()(unsigned q) const
    {
        return __ldg(reinterpret_cast<const uint4 *>(m + (size_t)BRICK_CELLS * q));
    }
};

// Stages the entries of words [q0, q1) that cover the lane's four cells, as
// 16-bit tags: each cell's from its own position p on.  The four cells' lists
// grow together, so finding an entry's bit is paid once for the cells it
// covers.  A tag is `owner` over the entry; PER_CELL adds the cell of the four.
template <bool PER_CELL, typename Masks>
__device__ __forceinline__ void stage_entries(unsigned short *stage, const Masks &masks, unsigned q0, unsigned q1,
                                              unsigned owner, unsigned (&p)[4])
{
    for (unsigned q = q0; q < q1; ++q) {
        const uint4 M = masks(q);
        const unsigned m[4] = {M.x, M.y, M.z, M.w};
        unsigned u = m[0] | m[1] | m[2] | m[3];
        const unsigned tag = owner | (q << 5);
        while (u) {
            const unsigned b = __clz(u), t = 0x80000000u >> b;
            u &= ~t;
            const unsigned v = tag | b;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (m[i] & t) {
                    stage[p[i]] = (unsigned short)(PER_CELL ? v | (unsigned)(i << 10) : v);
                    ++p[i];
                }
            }
        }
    }
}

// The same, staging the entries' objects.
template <typename Masks>
__device__ __forceinline__ void stage_objects(unsigned *stage, const unsigned *s_obj, const Masks &masks, unsigned q0,
                                              unsigned q1, unsigned (&p)[4])
{
    for (unsigned q = q0; q < q1; ++q) {
        const uint4 M = masks(q);
        const unsigned m[4] = {M.x, M.y, M.z, M.w};
        unsigned u = m[0] | m[1] | m[2] | m[3];
        while (u) {
            const unsigned b = __clz(u), t = 0x80000000u >> b;
            u &= ~t;
            const unsigned v = s_obj[32u * q + b];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (m[i] & t) {
                    stage[p[i]] = v;
                    ++p[i];
                }
            }
        }
    }
}

// A block per item, a warp per 128 cells, four neighbours in x per lane.  Of
// every four rows each warp takes another one, skewed from layer to layer: a
// surface that follows a plane of the brick keeps all warps busy.  The
// pairs are staged in shared memory in output order, as (cells,
// entry) in 16 bits, and copied out as objects with consecutive lanes on
// consecutive refs (the cells of a row of the brick are neighbours in refs
// too).  128 cells go at once when their pairs fit the stage, else 32 cells at
// a time, four lanes per four cells with a quarter of the entries each, and
// where 32 cells do not fit either, in windows of entries.
//
// DENSE: where 128 cells do not fit the stage (and no four cells overflow it on
// their own) the objects themselves are staged, for 8, 4, 2 or 1 lanes' cells
// at a time, the other lanes sharing their entries; four cells' refs are one
// run then, copied by whole warps without a tag, a lookup of its place and
// one of its object per ref.  Shared memory bounds the fill there (91% of its
// rate with tags): 1.47 -> 1.26 ms on the soup of 7.3M triangles, 1.0e9 refs.
//
// Bound by issue (78% of cycles) and shared memory (47 to 59% of its wavefronts);
// device memory is at a quarter of its rate.  Masks alone, no pairs written: 0.25
// of 0.64 ms at the 10M building.  One cell per lane 1.09, four 0.73 (one bit
// search serves four lists), two refs per lane in flight and one range check per
// cell 0.67, objects staged 0.66, the wider grid 0.64.  Measured and dropped: 16
// warps per block, lanes walking words independently (0.92 against 0.73), a lane
// per entry with popcount ranks (1.41), the next item's record loaded early.
template <unsigned STAGE, int MIN_BLOCKS, bool CULLED, bool DENSE>
__global__ void __launch_bounds__(32 * FILL_WARPS, MIN_BLOCKS) brick_fill_kernel(BrickArgs a)
{
    after_stream();
    static_assert(STAGE >= 1024, "one word of 32 cells fits");
    constexpr unsigned W = FILL_WARPS;
    __shared__ __align__(16) unsigned s_mask[CULLED ? 4 : BRICK_CHUNK / 32 * MASK_PITCH];   // [word][feature]
    __shared__ unsigned s_obj[BRICK_CHUNK];
    __shared__ __align__(16) unsigned short s_stage[W][STAGE];
    __shared__ unsigned s_delta[W][32];                      // per cell: its refs' place less its staged place
    const unsigned lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    const unsigned nitems = min(ld_relaxed_u32(&a.ctl->tickets[3]), a.max_items);
    unsigned short *stage = s_stage[w];
    unsigned *sdelta = s_delta[w];
    bool bad = false;
    for (unsigned i = blockIdx.x; i < nitems; i += gridDim.x) {
        const BrickItem it = load_item(a.items + i);
        const Dims d = decode(it.dims);
        const unsigned nw = (it.count + 31u) >> 5;
        Entry next = load_entry(a, it.first + 32u * w, 32u * w < it.count ? it.count - 32u * w : 0u);
        // the lane's four cells: where each one's refs start and, of a brick in
        // one item, how many it has; loaded ahead of the masks
        const unsigned rr = 4u * (lane >> (d.lx - 2u)), row = rr + ((w + 2u * (rr >> d.ly)) & 3u);
        const unsigned x = 4u * (lane & ((1u << (d.lx - 2u)) - 1u)), y = row & ((1u << d.ly) - 1u), z = row >> d.ly;
        const unsigned c0 = (row << d.lx) + x;
        unsigned dst[4], num[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) dst[k] = num[k] = 0u;
        if (y < d.ny && z < d.nz) {
            const unsigned *gp = a.G + it.cell0 + x + it.rx * y + it.rxy * z;
            unsigned g[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) g[k] = x + k <= d.nx ? __ldg(gp + k) : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (x + k < d.nx) {
                    dst[k] = it.base + g[k];
                    num[k] = g[k + 1] - g[k];
                    bad |= num[k] > a.nrefs || dst[k] > a.nrefs - num[k];
                    // the cell's other chunks come first; this one's share is counted below
                    if (it.slot != NO_SLOT) dst[k] += __ldg(a.slots + (size_t)it.slot * BRICK_CELLS + c0 + k);
                }
            }
        }
        if (it.slot != NO_SLOT) {   // those of a brick in many chunks: the groups before this one's
            const uint2 meta = a.slot_meta[it.slot];
            if (meta.y > MERGE_CHUNKS && y < d.ny && z < d.nz) {
                const unsigned row = group_row(a, meta.x) + (it.slot - meta.x) / merge_group(meta.y);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (x + k < d.nx) dst[k] += __ldg(a.slots + (size_t)row * BRICK_CELLS + c0 + k);
            }
        }
        __syncthreads();   // the previous item's masks and objects are read
        for (unsigned q = w; q < nw; q += W) {
            const Entry cur = next;
            const unsigned en = 32u * (q + W);
            next = load_entry(a, it.first + en, en < it.count ? it.count - en : 0u);
            if (!CULLED) s_mask[MASK_PITCH * q + lane] = transpose32(cur.ok ? feature_row(entry_info(a, cur), d) : 0u);
            s_obj[32u * q + 31u - lane] = entry_obj(a, cur);
        }
        __syncthreads();
        const unsigned fy = 1u << d.lx, fz = fy + (1u << d.ly);
        // the masks of four cells that start at local cell cc = (xx, yy, zz)
        const unsigned *kept = CULLED ? a.masks + (size_t)__ldg(a.mask0 + i) * BRICK_CELLS : nullptr;
        auto masks = [&](unsigned xx, unsigned yy, unsigned zz, unsigned cc) {
            if constexpr (CULLED) {
                return KeptMasks{kept + cc};
            } else {
                (void)cc;
                return BoxMasks{s_mask + xx, s_mask + fy + yy, s_mask + ((fz + zz) & 31u)};
            }
        };
        // a cells array that points outside refs (never with consistent lists): nothing is written
        if (__any_sync(FULL, bad)) continue;
        const unsigned lsum = num[0] + num[1] + num[2] + num[3];
        const unsigned inc = warp_incl_sum(lsum);
        const unsigned total = __shfl_sync(FULL, inc, 31);
        if (total == 0u) continue;
        if (total <= STAGE && it.slot == NO_SLOT) {
            unsigned p[4] = {inc - lsum, 0u, 0u, 0u};
#pragma unroll
            for (int k = 1; k < 4; ++k) p[k] = p[k - 1] + num[k - 1];
            const unsigned delta = dst[0] - p[0];   // the lane's cells follow one another in refs as in the stage
            if (lsum)
                stage_entries<false>(stage, masks(x, y, z, c0), 0u, nw, lane << 10, p);
            __syncwarp();
            for (unsigned p0 = 0; p0 < total; p0 += 64u) {   // two refs per lane in flight
                const unsigned q0 = p0 + lane, q1 = q0 + 32u;
                const unsigned v0 = q0 < total ? stage[q0] : 0u, v1 = q1 < total ? stage[q1] : 0u;
                const unsigned r0 = q0 + __shfl_sync(FULL, delta, v0 >> 10), r1 = q1 + __shfl_sync(FULL, delta, v1 >> 10);
                const unsigned o0 = s_obj[v0 & 1023u], o1 = s_obj[v1 & 1023u];
                if (q0 < total) __stcs(a.refs + r0, o0);
                if (q1 < total) __stcs(a.refs + r1, o1);
            }
            __syncwarp();
            continue;
        }
        if (DENSE && it.slot == NO_SLOT && !__any_sync(FULL, lsum > STAGE / 2u)) {
            unsigned *ostage = reinterpret_cast<unsigned *>(stage);
            for (unsigned l0 = 0; l0 < 32u;) {   // the cells of lanes l0 .. l0 + nl - 1
                const unsigned before = l0 ? __shfl_sync(FULL, inc, l0 - 1u) : 0u;
                unsigned nl = l0 + 8u <= 32u ? 8u : l0 + 4u <= 32u ? 4u : l0 + 2u <= 32u ? 2u : 1u;
                while (__shfl_sync(FULL, inc, l0 + nl - 1u) - before > STAGE / 2u) nl >>= 1;
                const unsigned q = lane & (nl - 1u), from = l0 + q, subs = 32u / nl, sub = lane / nl;
                const unsigned len = __shfl_sync(FULL, lsum, from), at = __shfl_sync(FULL, inc, from) - len - before;
                const unsigned to = __shfl_sync(FULL, dst[0], from);
                const auto four = masks(__shfl_sync(FULL, x, from), __shfl_sync(FULL, y, from), __shfl_sync(FULL, z, from),
                                        __shfl_sync(FULL, c0, from));
                const unsigned n0 = __shfl_sync(FULL, num[0], from), n1 = __shfl_sync(FULL, num[1], from),
                               n2 = __shfl_sync(FULL, num[2], from);
                const unsigned qa = nw * sub / subs, qb = nw * (sub + 1u) / subs;
                unsigned k[4] = {0u, 0u, 0u, 0u}, p[4] = {at, at + n0, at + n0 + n1, at + n0 + n1 + n2};
                if (len) {
                    for (unsigned qq = qa; qq < qb; ++qq) {
                        const uint4 M = four(qq);
                        k[0] += __popc(M.x);
                        k[1] += __popc(M.y);
                        k[2] += __popc(M.z);
                        k[3] += __popc(M.w);
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {   // behind the entries of the lanes that share the cells before this one
                    unsigned v = k[j];
                    for (unsigned o = nl; o < 32u; o <<= 1) {
                        const unsigned t = __shfl_up_sync(FULL, v, o);
                        if (lane >= o) v += t;
                    }
                    p[j] += v - k[j];
                }
                if (len) stage_objects(ostage, s_obj, four, qa, qb, p);
                __syncwarp();
                for (unsigned i4 = 0; i4 < nl; ++i4) {
                    const unsigned n = __shfl_sync(FULL, len, i4), src = __shfl_sync(FULL, at, i4);
                    unsigned *out = a.refs + __shfl_sync(FULL, to, i4);
                    for (unsigned r = lane; r < n; r += 32u) __stcs(out + r, ostage[src + r]);
                }
                __syncwarp();
                l0 += nl;
            }
            continue;
        }
        const unsigned quad = lane & 7u, sub = lane >> 3;
        for (unsigned g = 0; g < 4u; ++g) {
            // cells 32 g .. 32 g + 31 of the warp's: those of lanes 8 g .. 8 g + 7
            const unsigned from = 8u * g + quad;
            unsigned to[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) to[k] = __shfl_sync(FULL, dst[k], from);
            const bool live = __shfl_sync(FULL, lsum, from) != 0u;   // a cell beyond a small brick has no features
            if (!__any_sync(FULL, live)) continue;
            const unsigned qx = __shfl_sync(FULL, x, from), qy = __shfl_sync(FULL, y, from),
                           qz = __shfl_sync(FULL, z, from);
            const auto four = masks(qx, qy, qz, __shfl_sync(FULL, c0, from));
            unsigned win = nw;
            for (unsigned q0 = 0; q0 < nw;) {
                unsigned nq = min(win, nw - q0), qa, qb, k[4], pre[4], sum[4], base, cnt;
                for (;;) {
                    qa = q0 + nq * sub / 4u;
                    qb = q0 + nq * (sub + 1u) / 4u;
                    k[0] = k[1] = k[2] = k[3] = 0u;
                    if (live) {
                        for (unsigned q = qa; q < qb; ++q) {
                            const uint4 M = four(q);
                            k[0] += __popc(M.x);
                            k[1] += __popc(M.y);
                            k[2] += __popc(M.z);
                            k[3] += __popc(M.w);
                        }
                    }
                    // each cell's entries of the lower quarters, its sum, and the cells before
                    unsigned all = 0u;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        unsigned v = k[j];
                        const unsigned v1 = __shfl_up_sync(FULL, v, 8);
                        if (sub >= 1u) v += v1;
                        const unsigned v2 = __shfl_up_sync(FULL, v, 16);
                        if (sub >= 2u) v += v2;
                        pre[j] = v - k[j];
                        sum[j] = __shfl_sync(FULL, v, 24u + quad);
                        all += sum[j];
                    }
                    unsigned v = all;
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) {
                        const unsigned t = __shfl_up_sync(FULL, v, o, 8);
                        if (quad >= (unsigned)o) v += t;
                    }
                    base = v - all;
                    cnt = __shfl_sync(FULL, v, 7);
                    if (cnt <= STAGE) break;
                    win = nq = nq / 2u;   // one word always fits
                }
                unsigned p[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    p[j] = base + pre[j];
                    if (sub == 0u) sdelta[4u * quad + j] = to[j] - base;
                    base += sum[j];
                    to[j] += sum[j];
                }
                if (live) stage_entries<true>(stage, four, qa, qb, quad << 12, p);
                __syncwarp();
                unsigned p0 = lane;
                for (; p0 + 32u < cnt; p0 += 64u) {   // two refs per lane in flight
                    const unsigned v0 = stage[p0], v1 = stage[p0 + 32u];
                    const unsigned r0 = p0 + sdelta[v0 >> 10], r1 = p0 + 32u + sdelta[v1 >> 10];
                    const unsigned o0 = s_obj[v0 & 1023u], o1 = s_obj[v1 & 1023u];
                    __stcs(a.refs + r0, o0);
                    __stcs(a.refs + r1, o1);
                }
                if (p0 < cnt) {
                    const unsigned v = stage[p0];
                    __stcs(a.refs + (p0 + sdelta[v >> 10]), s_obj[v & 1023u]);
                }
                __syncwarp();
                q0 += nq;
            }
        }
    }
    if (bad) atomicOr(&a.ctl->err, ERR_RANGE);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

// A brick in k > 1 chunks holds more than (k - 1) BRICK_CHUNK entries, at least
// k BRICK_CHUNK / 2.
unsigned brick_max_slots(unsigned count) { return 2u * (count / BRICK_CHUNK) + 2u; }

// Group rows behind the slots (group_row).
unsigned brick_max_groups(unsigned count) { return brick_max_slots(count) / 8u + 2u; }

unsigned brick_max_items(unsigned nbricks, unsigned count)
{
    const unsigned long long n = (unsigned long long)nbricks + brick_max_slots(count);
    return n > 0xFFFFFFFFull ? 0xFFFFFFFFu : (unsigned)n;
}

// A table of twice as many places as there can be cells of BRICK_BIG objects.
int brick_big_bits(unsigned nrefs)
{
    int bits = 1;
    while ((1u << bits) < 2u * (nrefs / BRICK_BIG + 1u)) ++bits;
    return bits;
}

unsigned long long cell_scan_tiles(long long ncells_out)
{
    const long long t = ncells_out > SCAN_BIG        ? scan_tile<SCAN_J_BIG>()
                        : ncells_out > SCAN_ONE_PASS ? scan_tile<SCAN_J>()
                                                     : scan_tile<1>();
    return (unsigned long long)((ncells_out + t - 1) / t);
}

cudaError_t launch_brick_split(const BrickArgs &a, cudaStream_t s)
{
    launch_after(brick_split_kernel, (a.nbricks + 255u) / 256u, 256, 0, s, a);
    return cudaGetLastError();
}

cudaError_t launch_brick_count(const BrickArgs &a, int nsm, cudaStream_t s)
{
    const unsigned blocks = (a.max_items + COUNT_WARPS - 1u) / COUNT_WARPS, cap = (unsigned)nsm * 64u;
    const unsigned grid = blocks < cap ? blocks : cap;
    if (a.masks)
        launch_after(brick_count_kernel<true>, grid, 32 * COUNT_WARPS, 0, s, a);
    else
        launch_after(brick_count_kernel<false>, grid, 32 * COUNT_WARPS, 0, s, a);
    return cudaGetLastError();
}

int cell_scan_launches(long long ncells_out) { return ncells_out > SCAN_ONE_PASS ? 2 : 1; }

cudaError_t launch_cell_scan(const BrickArgs &a, cudaStream_t s)
{
    const unsigned tiles = (unsigned)cell_scan_tiles(a.ncells_out);
    if (a.ncells_out > SCAN_BIG) {
        launch_after(cell_sums_kernel<SCAN_J_BIG>, tiles, SCAN_BLOCK, 0, s, a, tiles);
        launch_after(cell_scan_kernel<SCAN_J_BIG, false>, tiles, SCAN_BLOCK, 0, s, a);
    } else if (a.ncells_out > SCAN_ONE_PASS) {
        launch_after(cell_sums_kernel<SCAN_J>, tiles, SCAN_BLOCK, 0, s, a, tiles);
        launch_after(cell_scan_kernel<SCAN_J, false>, tiles, SCAN_BLOCK, 0, s, a);
    } else {
        launch_after(cell_scan_kernel<1, true>, tiles, SCAN_BLOCK, 0, s, a);
    }
    return cudaGetLastError();
}

// In crowded cells the larger stage wins, in the others the more resident blocks.
// Larger against smaller, us, at so many pairs per cell: buildings 2.5: 186 / 147,
// 4.5: 101 / 99, 6.3: 91 / 97; soups of 4M triangles 4.0: 242 / 199, 6.8: 305 / 283, 7.9:
// 206 / 251, 13.6: 268 / 349, 128: 559 / 604; of 400,000 4.0: 31 / 29, 6.8: 38 / 46; soups of
// uneven triangles 19.5: 134 / 203.
constexpr double DENSE_PAIRS_PER_CELL = 6.0;

cudaError_t launch_brick_fill(const BrickArgs &a, int nsm, cudaStream_t s)
{
    // many more blocks than fit, so that bricks of many entries even out: 638 us at the 10M building, 656 with 64
    // per SM, 667 with a block per item
    const unsigned cap = (unsigned)nsm * 256u, grid = a.max_items < cap ? a.max_items : cap;
    if (a.masks)
        launch_after(brick_fill_kernel<1024, 10, true, false>, grid, 32 * FILL_WARPS, 0, s, a);
    else if ((double)a.nrefs > DENSE_PAIRS_PER_CELL * (double)a.ncells_out)
        launch_after(brick_fill_kernel<3072, 6, false, true>, grid, 32 * FILL_WARPS, 0, s, a);
    else
        launch_after(brick_fill_kernel<1024, 10, false, true>, grid, 32 * FILL_WARPS, 0, s, a);
    return cudaGetLastError();
}

unsigned brick_max_words(unsigned nbricks, unsigned count)
{
    // every item rounds its last word up
    const unsigned long long n = (unsigned long long)count / 32u + brick_max_items(nbricks < count ? nbricks : count, count);
    return n > 0xFFFFFFFEull ? 0xFFFFFFFEu : (unsigned)n;
}

cudaError_t launch_brick_cull(const BrickArgs &a, int nsm, cudaStream_t s)
{
    const unsigned blocks = (a.max_words + CULL_WARPS - 1u) / CULL_WARPS, cap = (unsigned)nsm * 64u;
    launch_after(brick_cull_kernel, blocks < cap ? blocks : cap, 32 * CULL_WARPS, 0, s, a);
    return cudaGetLastError();
}

}  // namespace gg
