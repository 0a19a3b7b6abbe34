// CSF builder, splitter sort: the sort and the per-level compression of large tensors (csf_build.cu holds the radix sort that
// takes the others, and everything around the two).
//
// The nonzeros go through memory three times instead of once per 8 or 9 key bits:
//   1. a sample of the keys, ranked all against all, gives splitters that cut the key space into buckets of about equal
//      counts, whatever the distribution (split_sample, split_rank);
//   2. every tile packs its coordinates, deals them to the buckets and appends each run to its bucket, which is a list of
//      fixed chunks that are handed out as it grows (split_tile, first level);
//   3. per bucket a sample gives splitters for parts of about kPartMean nonzeros (split_sample2), and every chunk deals its
//      nonzeros to the parts, each of which has room for kPartRoom (split_tile, second level);
//   4. a block sorts a part in shared memory, writes values and leaf coordinates to their final places and lists the nodes that
//      open at the level above the leaves (part_sort); a scan numbers the nodes (part_scan), and once the host has sized the
//      arrays the lists are turned into the upper levels (part_nodes).
// None of the moves has to keep the order of equal keys (a coordinate that occurs twice is an error, and two equal keys meet in
// one part), so places are handed out by counters: no ballots per key bit, no chain from tile to tile.
// A part that outgrows its room, or a bucket that outgrows its list, sets `gave_up`; the host then takes the radix sort.
#include <algorithm>

#include "csf_build.cuh"

namespace cb {
namespace {

// Measured on 77 M nonzeros of Zipf slices (43-bit keys, fp32) unless it says otherwise, us for the kernel named.
// A tile of 2048 (4096: split_buckets 1573 against 1094).
constexpr int kThreads = 256, kItems = 8, kTile = kThreads * kItems;
// Blocks of split_tile resident per SM: three of 80 registers for the first level, which keeps coordinates (four: 907 against 822, two: 894
// against 821; fp64 uniform, two: 814 against 757; order 4, which spills a few registers at three, 30 M, two against three: fp32 316 / 305,
// fp64 361 / 361), four of 64 for the second (three: 733 against 680).
constexpr int tile_blocks(bool first) { return first ? 3 : 4; }
constexpr int kWide = 512;                         // threads of the blocks that sort up to kPartRoom numbers, kItems each
constexpr int kChunk = 4096;                       // elements of a bucket's chunk, at least a tile: a run spans two at most
// Parts of 1365 on average: with kOverParts samples a part, one in seventy is larger than the 2048 of an ordinary block, and one in
// 10^10 outgrows its room of three times the average.
constexpr int kPartRoom = kWide * kItems, kPartMean = 1365;
constexpr int kSampleThreads = 1024;               // of the block that sorts a bucket's sample
// Two levels of ways about alike: 256 buckets of up to 512 parts (both levels together 1645; 512 of 256: 1720; 128 of 512: 1665).
constexpr int kMaxBuckets = 256, kMaxParts = 512;
constexpr int kCells = 1 << 10;                    // of the classification: stretches of equal length of the key space or of a bucket
constexpr int kOverBuckets = 16, kOverParts = 24;  // samples per bucket and per part
constexpr int kPad = 4;                            // numbers behind the room of the keys: even, what follows is read 16 bytes at a time
constexpr int kTogether = 4;                       // elements of a thread that look through their bins side by side
constexpr int kSlack = 3;                          // elements of a bin compared without a loop
template <int NT> constexpr int kBins = NT < 512 ? 2048 : 4 * NT;      // of a sort of NT threads
constexpr int kSpinLimit = 1 << 21;
constexpr int kCursorGap = 16;                     // words between the buckets' cursors, which every tile adds to: a line of the cache for two
constexpr int kPartBits = 9;                       // part_owner: bucket << kPartBits | part of the bucket
static_assert(kMaxParts <= 1 << kPartBits && kMaxParts <= kWide && kMaxBuckets <= kWide && kTile <= kChunk, "one thread per part");

struct PartInfo {
    uint64_t first, last;                          // keys: the part's ends
    uint32_t count, start;                         // nonzeros, position of the first one
    uint32_t opened[kMaxOrder - 1];                // nodes that open in the part, its first element counted at every level
    uint32_t cont;                                 // bit l: at level l the first element goes on with a node of an earlier part
};

struct PartJob {                                   // a part as part_sort takes it
    uint64_t lo, range;                            // its keys lie in [lo, lo + range]
    uint32_t start, count;
};

struct Tables {
    uint32_t *result;                              // totals [0..3), parts [3], status [16], gave up [17]
    uint32_t *arrived, *next_chunk, *large, *ready, *cursor, *part_count, *chunk_of;     // cleared
    uint64_t *samples, *bucket_split, *part_split;
    uint32_t *bucket_cells, *part_cells;
    uint32_t *part_base, *bucket_parts, *part_owner, *part_nodes, *bucket_nodes;
    PartJob *jobs;
    uint32_t *large_parts;                         // parts for the second launch of part_sort
    uint2 *chunk_owner;
    PartInfo *infos;
    uint64_t key_max;
    int64_t n;
    int buckets, bucket_shift, chunk_rows;
    uint32_t max_chunks;
    __device__ __forceinline__ int32_t *status() const { return reinterpret_cast<int32_t *>(result + 16); }
    __device__ __forceinline__ uint32_t *gave_up() const { return result + 17; }
};

template <int ORDER>
__device__ __forceinline__ uint64_t pack_key(const PackArgs &a, const uint32_t *x, bool &bad) {
    uint64_t key = 0;
#pragma unroll
    for (int l = 0; l < ORDER; ++l) {
        uint32_t c = x[l];
        if (c >= (uint32_t)a.dim[l]) { bad = true; c = 0; }              // extents are below 2^31: a negative number is beyond them too
        key |= l + 1 < ORDER ? (uint64_t)c << a.shift[l] : (uint64_t)c;
    }
    return key;
}

// One position of [0, n) out of the t-th of `of` equal stretches, anywhere inside it: the input may be sorted or periodic.
__device__ __forceinline__ int64_t sample_at(uint32_t t, uint32_t of, int64_t n) {
    const int64_t lo = n * t / of, hi = n * (t + 1) / of;
    uint32_t h = t * 2654435761u + 0x9e3779b9u;
    h ^= h >> 16; h *= 0x85ebca6bu; h ^= h >> 13; h *= 0xc2b2ae35u; h ^= h >> 16;
    return hi > lo ? lo + (int64_t)(h % (uint32_t)(hi - lo)) : lo;
}

template <int ORDER>
__global__ void __launch_bounds__(kThreads) split_sample(PackArgs a, Tables t, uint32_t samples) {
    const uint32_t x = blockIdx.x * kThreads + threadIdx.x;
    bool bad = false;
    start_next_kernel();
    if (x >= samples) return;
    const int64_t e = sample_at(x, samples, t.n);
    uint32_t c[ORDER];
#pragma unroll
    for (int l = 0; l < ORDER; ++l) c[l] = (uint32_t)__ldg(a.c[l] + e);
    t.samples[x] = pack_key<ORDER>(a, c, bad);
}

// For every key the number of splitters not above it.  The key's cell gives the splitters before the cell (low half, as a byte
// offset) and how many lie in it (high half).  The powers of two no larger than that are tried from the largest down, for all
// keys of a thread side by side.
__device__ __forceinline__ void classify(const uint64_t (&key)[kItems], uint32_t (&way)[kItems], uint64_t lo, int shift, const uint64_t *split,
                                         const uint32_t *cells) {
    auto splitter = [&](uint32_t offset) { return *reinterpret_cast<const uint64_t *>(reinterpret_cast<const unsigned char *>(split) + offset); };
    uint32_t most = 0;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        way[i] = cells[(uint32_t)((key[i] - lo) >> shift)];
        most = max(most, way[i]);
    }
    most = __reduce_max_sync(0xffffffffu, most) >> 16;
    for (uint32_t h = most ? 1u << (31 - __clz(most)) : 0u; h; h >>= 1) {
        const uint32_t least = h << 16, step = 8 * h - (h << 16), mid = 8 * (h - 1);
        uint64_t s[kItems];                                             // lanes without so many read the first: no branches, one bank
#pragma unroll
        for (int i = 0; i < kItems; ++i) s[i] = splitter(way[i] >= least ? (way[i] & 0xffffu) + mid : 0u);
#pragma unroll
        for (int i = 0; i < kItems; ++i) way[i] += way[i] >= least && s[i] <= key[i] ? step : 0u;
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i) way[i] = (way[i] & 0xffffu) >> 3;
}

// right shift that leaves `bits` bits of every number up to `range`
__device__ __forceinline__ int cell_shift(uint64_t range, int bits) { return max(0, 64 - __clzll((long long)range) - bits); }

// cells[c] = splitters in the cells before c, times 8 | splitters in c << 16
__device__ __forceinline__ void fill_cells(uint32_t *cells, const uint64_t *split, int splits, uint64_t lo, int shift) {
    for (int c = threadIdx.x; c < kCells; c += blockDim.x) {
        int at[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int a = 0, b = splits;
            while (a < b) {
                const int mid = (a + b) >> 1;
                if ((int)((split[mid] - lo) >> shift) < c + h) a = mid + 1; else b = mid;
            }
            at[h] = a;
        }
        cells[c] = 8u * (uint32_t)at[0] | (uint32_t)(at[1] - at[0]) << 16;
    }
}

// Rank of every sample among all, eight lanes per sample (4096 samples: 128 blocks, 15 us);
// every kOverBuckets-th becomes a splitter.  The last block to finish fills the cells.
__global__ void __launch_bounds__(kThreads) split_rank(Tables t, uint32_t samples) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *all = reinterpret_cast<uint64_t *>(smem);
    after_last_kernel();
    start_next_kernel();
    for (uint32_t x = threadIdx.x; x < samples; x += kThreads) all[x] = t.samples[x];
    __syncthreads();
    const uint32_t me = blockIdx.x * (kThreads / 8) + threadIdx.x / 8, sub = threadIdx.x % 8;
    const uint64_t key = all[me];                                       // samples is a multiple of 32
    uint32_t rank = 0;
    uint32_t x = sub;                                                   // equal keys by their numbers
#pragma unroll 8
    for (; x < me; x += 8) rank += all[x] <= key;
#pragma unroll 8
    for (; x < samples; x += 8) rank += all[x] < key;
#pragma unroll
    for (int off = 4; off; off >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, off);
    if (sub == 0 && rank > 0 && rank % kOverBuckets == 0) t.bucket_split[rank / kOverBuckets - 1] = key;
    if (!last_block(t.arrived)) return;
    const int splits = t.buckets - 1;
    for (int y = threadIdx.x; y < splits; y += kThreads) all[y] = __ldcg(t.bucket_split + y);
    __syncthreads();
    fill_cells(t.bucket_cells, all, splits, 0ull, t.bucket_shift);
}

__device__ __forceinline__ uint64_t bucket_low(const Tables &t, int b) { return b > 0 ? t.bucket_split[b - 1] : 0ull; }
__device__ __forceinline__ uint64_t bucket_top(const Tables &t, int b) { return b + 1 < t.buckets ? t.bucket_split[b] - 1 : t.key_max; }

// The chunk behind place q of bucket b's list, plus one; 0 where there is no room.  Published for the tiles that append to it.
__device__ __forceinline__ uint32_t take_chunk(const Tables &t, uint32_t b, uint32_t q, int withhold) {
    if (q >= (uint32_t)t.chunk_rows) return 0;
    const uint32_t ch = atomicAdd(t.next_chunk, 1u);
    if (ch >= t.max_chunks) return 0;                                   // cannot happen: every bucket has one chunk that is not full
    t.chunk_owner[ch] = make_uint2(b, q);
    if (!withhold) *reinterpret_cast<volatile uint32_t *>(t.chunk_of + (size_t)b * t.chunk_rows + q) = ch + 1;
    return ch + 1;
}

// Deals tiles to their buckets (ORDER > 0: packs the coordinates first) or a chunk of a bucket to the bucket's parts (ORDER 0),
// appending each run to its target.  A block goes over several tiles, with the tables loaded once; the loads of the next tile are
// under way while the present one is written out.
// What bounds it: the shared-memory pipe (52 and 40 wavefronts per 32 nonzeros in the two levels: cells and splitters, counters, the
// reorder; it is 72 and 79 % busy) and, between the phases of a tile, too few loads under way.  77 M: 821 us and 691 us for the two
// levels, 2.6 and 2.7 TB/s (uniform: 662 and 687); a radix pass over the same data takes 560.
template <typename V, int ORDER>
__global__ void __launch_bounds__(kThreads, tile_blocks(ORDER > 0)) split_tile(PackArgs a, Tables t, const uint64_t *kin,
                                                                 const V *vin, uint64_t *kout, V *vout,
                                                                 int spin_limit, int withhold) {
    constexpr bool kFirst = ORDER > 0;
    constexpr int kWays = kFirst ? kMaxBuckets : kMaxParts, kPer = kWays / kThreads;
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *keybuf = reinterpret_cast<uint64_t *>(smem);
    V *valbuf = reinterpret_cast<V *>(smem + kTile * sizeof(uint64_t));
    uint16_t *waybuf = reinterpret_cast<uint16_t *>(smem + kTile * (sizeof(uint64_t) + sizeof(V)));
    __shared__ uint64_t split[kWays];
    __shared__ uint32_t cells[kCells];
    __shared__ uint32_t place[kWays], to1[kFirst ? kWays : 1];
    __shared__ uint2 to0[kWays];                                        // target, end of the part of the run that goes there
    __shared__ int s_bad;

    const int tid = threadIdx.x;
    uint32_t b = 0;
    uint64_t lo = 0;
    int shift = t.bucket_shift;
    int64_t base = (int64_t)blockIdx.x * kTile, end = t.n, stride = (int64_t)gridDim.x * kTile;
    if (!kFirst) {
        after_last_kernel();
        start_next_kernel();
        if (tid == 0) s_bad = *reinterpret_cast<volatile uint32_t *>(t.gave_up()) != 0;
        __syncthreads();
        if (s_bad || blockIdx.x >= *t.next_chunk) return;
        const uint2 owner = t.chunk_owner[blockIdx.x];
        b = owner.x;
        base = (int64_t)blockIdx.x * kChunk;
        end = base + min((uint32_t)kChunk, t.cursor[b * kCursorGap] - owner.y * kChunk);
        stride = kTile;
        lo = bucket_low(t, (int)b);
        shift = cell_shift(bucket_top(t, (int)b) - lo, 10);
    }
    // All loads of a tile are under way before the first is used; beyond the end they repeat the last element.
    int32_t c[kFirst ? ORDER : 1][kItems];
    uint64_t key[kItems];
    V val[kItems];
    auto load = [&](int64_t from) {
        const int last = (int)min((int64_t)kTile, end - from) - 1;
        auto at = [&](auto offset) {                                    // offset(i): of this thread's i-th element
            if (kFirst) {
#pragma unroll
                for (int l = 0; l < ORDER; ++l) {
                    const int32_t *p = a.c[l] + from;
#pragma unroll
                    for (int i = 0; i < kItems; ++i) c[l][i] = __ldg(p + offset(i));
                }
            } else {
                const uint64_t *p = kin + from;
#pragma unroll
                for (int i = 0; i < kItems; ++i) key[i] = p[offset(i)];
            }
            const V *p = vin + from;
#pragma unroll
            for (int i = 0; i < kItems; ++i) val[i] = p[offset(i)];
        };
        if (last == kTile - 1) at([&](int i) { return i * kThreads + tid; });
        else at([&](int i) { return min(i * kThreads + tid, last); });
    };
    if (base >= end) return;
    load(base);                                                         // (first level: the caller's arrays, no earlier kernel's)
    if (kFirst) {
        after_last_kernel();
        start_next_kernel();
    }
    const int splits = kFirst ? t.buckets - 1 : (int)t.bucket_parts[b] - 1;
    const uint64_t *from_split = kFirst ? t.bucket_split : t.part_split + (size_t)b * kMaxParts;
    const uint32_t *from_cells = kFirst ? t.bucket_cells : t.part_cells + (size_t)b * kCells;
    for (int x = tid; x < splits; x += kThreads) split[x] = from_split[x];
    for (int x = tid; x < kCells; x += kThreads) cells[x] = from_cells[x];

    for (; base < end; base += stride) {
        const int nvalid = (int)min((int64_t)kTile, end - base);
        if (kFirst) {
            bool bad = false;
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                uint32_t x[ORDER ? ORDER : 1];
#pragma unroll
                for (int l = 0; l < ORDER; ++l) x[l] = (uint32_t)c[l][i];
                key[i] = pack_key<ORDER>(a, x, bad);
            }
            if (bad) report(t.status(), CONST_ERR_COORD_RANGE);
        }
        for (int x = tid; x < kWays; x += kThreads) place[x] = 0;
        if (tid == 0) s_bad = 0;
        __syncthreads();

        uint32_t way[kItems];
        classify(key, way, lo, shift, split, cells);
        // way[i] becomes (way << 16) | place in the run; lanes that all go the same way (sorted input) are counted with one addition
        const uint32_t w0 = __shfl_sync(0xffffffffu, way[0], 0);
        if (nvalid == kTile && __all_sync(0xffffffffu, way[0] == w0)) {
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const uint32_t same = __match_any_sync(0xffffffffu, way[i]);
                const int head = __ffs(same) - 1, lane = tid & 31;
                uint32_t r = 0;
                if (lane == head) r = atomicAdd(&place[way[i]], (uint32_t)__popc(same));
                way[i] = (way[i] << 16) | (__shfl_sync(0xffffffffu, r, head) + __popc(same & ((1u << lane) - 1u)));
            }
        } else {
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                uint32_t r = 0;
                if (i * kThreads + tid < nvalid) r = atomicAdd(&place[way[i]], 1u);
                way[i] = (way[i] << 16) | r;
            }
        }
        __syncthreads();
        uint32_t count[kPer], at[kPer], excl[kPer], chunk0[kPer], chunk1[kPer];
        {
            uint32_t sum = 0, total;
#pragma unroll
            for (int q = 0; q < kPer; ++q) { count[q] = place[tid * kPer + q]; sum += count[q]; }
            uint32_t run = block_scan(sum, total);
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                const uint32_t w = tid * kPer + q;
                excl[q] = run;
                place[w] = run;
                run += count[q];
                at[q] = 0;
                chunk0[q] = chunk1[q] = 0;
                if (count[q]) at[q] = atomicAdd(kFirst ? t.cursor + w * kCursorGap : t.part_count + t.part_base[b] + w, count[q]);
            }
        }
        bool failed = false;
        if (kFirst) {                                                   // the chunks that this tile's runs open, before anything waits
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                if (!count[q]) continue;
                const uint32_t w = tid * kPer + q, row = at[q] / kChunk, off = at[q] % kChunk;
                if (off == 0) { chunk0[q] = take_chunk(t, w, row, withhold); failed = failed || !chunk0[q]; }
                if (off + count[q] > kChunk) { chunk1[q] = take_chunk(t, w, row + 1, withhold); failed = failed || !chunk1[q]; }
                if (off != 0 && row < (uint32_t)t.chunk_rows)
                    chunk0[q] = *reinterpret_cast<volatile uint32_t *>(t.chunk_of + (size_t)w * t.chunk_rows + row);
            }
            __syncwarp();
        }
        __syncthreads();                                                // `place` is complete
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            if (i * kThreads + tid < nvalid) {
                const uint32_t w = way[i] >> 16, p = place[w] + (way[i] & 0xffffu);
                keybuf[p] = key[i];
                valbuf[p] = val[i];
                waybuf[p] = (uint16_t)w;
            }
        }
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const uint32_t w = tid * kPer + q;
            if (!count[q]) continue;
            if (kFirst) {
                const uint32_t row = at[q] / kChunk, off = at[q] % kChunk;
                if (off != 0) {                                         // opened by another tile, which waits for nothing in between
                    if (row < (uint32_t)t.chunk_rows) {
                        volatile uint32_t *slot = t.chunk_of + (size_t)w * t.chunk_rows + row;
                        for (int spins = 0; !chunk0[q] && spins < spin_limit; ++spins) {
                            __nanosleep(100);
                            chunk0[q] = *slot;
                        }
                        if (!chunk0[q]) report(t.status(), CONST_ERR_TIMEOUT);
                    }
                    failed = failed || !chunk0[q];
                }
                const uint32_t stop = excl[q] + (kChunk - off);
                to0[w] = make_uint2((chunk0[q] - 1) * kChunk + off - excl[q], stop);   // modulo 2^32; adding a position in the tile gives the place
                to1[w] = (chunk1[q] - 1) * kChunk - stop;
            } else {
                failed = failed || at[q] + count[q] > kPartRoom;
                to0[w].x = (t.part_base[b] + w) * kPartRoom + at[q] - excl[q];
            }
        }
        if (failed) {
            atomicExch(t.gave_up(), 1u);
            s_bad = 1;
        }
        if (base + stride < end) load(base + stride);
        __syncthreads();
        if (s_bad) return;
#pragma unroll
        for (int m = 0; m < kItems; ++m) {
            const uint32_t p = tid + m * kThreads;
            if (p < (uint32_t)nvalid) {
                const uint32_t w = waybuf[p];
                uint32_t o;
                if (kFirst) {
                    const uint2 to = to0[w];
                    o = to.x;
                    if (p >= to.y) o = to1[w];
                } else {
                    o = to0[w].x;
                }
                o += p;
                kout[o] = keybuf[p];
                vout[o] = valbuf[p];
            }
        }
        __syncthreads();
    }
}

// Bin of a number in [lo, lo + range], and how far it lies inside the bin (in 2^-32 of its length).
template <int NT>
struct Bins {
    int shift;
    uint32_t scale;
    uint64_t lo;
    __device__ __forceinline__ Bins(uint64_t low, uint64_t range) : lo(low) {
        shift = cell_shift(range, 32);
        const uint64_t wide = (range >> shift) + 1;
        // rounded down by more than the divisions can be off: the largest number stays below the last bin's end
        scale = wide <= kBins<NT> ? 0u : (uint32_t)((float)kBins<NT> * 4294965000.0f / (float)wide);
    }
    __device__ __forceinline__ uint32_t bin(uint32_t d, uint32_t &inside) const {
        if (!scale) { inside = 0; return min(d, (uint32_t)kBins<NT> - 1); }
        const uint64_t x = (uint64_t)d * scale;
        inside = (uint32_t)x;
        return min((uint32_t)(x >> 32), (uint32_t)kBins<NT> - 1);
    }
    __device__ __forceinline__ uint32_t of(uint32_t x, uint32_t &inside) const { return bin(x - (uint32_t)lo, inside); }     // ranges below 2^32
    __device__ __forceinline__ uint32_t of(uint64_t x, uint32_t &inside) const { return bin((uint32_t)((x - lo) >> shift), inside); }
};

// Turns the counts of the bins into the first places of the bins: as they are into `bins` (where SELF), and in 16 bits into
// `start`.  Returns the sum of the squares of the counts.
template <int NT, bool SELF>
__device__ __forceinline__ uint32_t scan_bins(uint32_t *counts, uint16_t *start, int m) {
    __shared__ uint32_t s_squares;
    constexpr int PER = kBins<NT> / NT;
    static_assert(PER % 4 == 0, "whole words of four per thread");
    const int tid = threadIdx.x;
    uint32_t word[PER], sum = 0, squares = 0, total;
#pragma unroll
    for (int x = 0; x < PER / 4; ++x) *reinterpret_cast<uint4 *>(word + 4 * x) = reinterpret_cast<uint4 *>(counts)[tid * (PER / 4) + x];
#pragma unroll
    for (int x = 0; x < PER; ++x) { sum += word[x]; squares += word[x] * word[x]; }
    if (tid == 0) s_squares = 0;
    squares = __reduce_add_sync(0xffffffffu, squares);
    uint32_t run = block_scan<NT>(sum, total);                           // (its barriers stand behind the clearing)
    if ((tid & 31) == 0) atomicAdd(&s_squares, squares);
#pragma unroll
    for (int x = 0; x < PER; ++x) { const uint32_t c = word[x]; word[x] = run; run += c; }
#pragma unroll
    for (int x = 0; x < PER / 4; ++x) {
        if (SELF) reinterpret_cast<uint4 *>(counts)[tid * (PER / 4) + x] = *reinterpret_cast<uint4 *>(word + 4 * x);
        reinterpret_cast<uint2 *>(start)[tid * (PER / 4) + x] =
            make_uint2(word[4 * x] | word[4 * x + 1] << 16, word[4 * x + 2] | word[4 * x + 3] << 16);
    }
    if (tid == 0) {
        if (SELF) counts[kBins<NT>] = m;
        start[kBins<NT>] = (uint16_t)m;
    }
    __syncthreads();
    return s_squares;
}

// Whether `other` comes in front of `x`, `earlier` settling it between equal ones.  32-bit numbers stay below 2^32 - 1 (part_sort), 64-bit
// ones may be any.
__device__ __forceinline__ bool in_front(uint32_t other, uint32_t x, bool earlier) { return other < x + earlier; }
__device__ __forceinline__ bool in_front(uint64_t other, uint64_t x, bool earlier) { return earlier ? other <= x : other < x; }

// Sorts m <= kItems x NT numbers of type K: thread x holds dist[i] for element i * NT + x.
// They are dealt to bins of equal ranges -- where that leaves many in few bins, to new ones whose borders follow the counts of
// the old -- and every one then finds its place among those of its bin (a warp works on neighbouring places, so its lanes meet
// bins of like size); `put(place, number, was)` hears of it, `was` being where `stash(was, i)` was told to keep what goes with
// dist[i].  Where even the new bins are crowded (some 96 to compare with on average) a bitonic network takes over.
// buf has room for kPad more than m, bins for kBins + 4, start for kBins + 8.
template <int NT, class K, class Stash, class Put>
__device__ __forceinline__ void sort_block(K *buf, uint16_t *order, uint32_t *bins, uint16_t *start, int m, const Bins<NT> &bins_of,
                                           K (&dist)[kItems], Stash stash, Put put) {
    constexpr int kHalve = NT > kThreads ? 1 : 0;                        // places per new bin, as a shift
    static_assert((kItems * NT >> kHalve) <= kBins<NT>, "a new bin for every place");
    const int tid = threadIdx.x;
    uint32_t rank[kItems];                                               // bin | place in the bin << 16
    auto clear = [&](uint32_t *counts) {
#pragma unroll
        for (int x = 0; x < kBins<NT> / NT / 4; ++x) reinterpret_cast<uint4 *>(counts)[tid + x * NT] = make_uint4(0, 0, 0, 0);
        __syncthreads();
    };
    bool renewed = false;
    auto bin_of = [&](K x) {
        uint32_t inside;
        const uint32_t bin = bins_of.of(x, inside);
        if (!renewed) return bin;
        const uint32_t from = bins[bin];
        return (from + __umulhi(inside, bins[bin + 1] - from)) >> kHalve;
    };
    auto count = [&](uint32_t *counts) {
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            rank[i] = bin_of(dist[i]);
            if (i * NT + tid < m) rank[i] |= atomicAdd(&counts[rank[i]], 1u) << 16;
        }
        __syncthreads();
    };
    clear(bins);
    count(bins);
    uint32_t squares = scan_bins<NT, true>(bins, start, m);
    if (squares > 6u * (uint32_t)m && bins_of.scale) {
        renewed = true;
        uint32_t *counts = reinterpret_cast<uint32_t *>(buf);            // nothing is there yet
        clear(counts);
        count(counts);
        squares = scan_bins<NT, false>(counts, start, m);
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        if (i * NT + tid < m) {
            const uint32_t p = start[rank[i] & 0xffffu] + (rank[i] >> 16);
            buf[p] = dist[i];
            stash(p, i);
        }
    }
    const bool crowded = squares > 96u * (uint32_t)m;
    __syncthreads();
    if (!crowded) {
#pragma unroll
        for (int i0 = 0; i0 < kItems; i0 += kTogether) {
            if (i0 * NT >= m) break;
            // behind m lie numbers of no meaning: they give a bin all the same, and are not put anywhere
            uint32_t from[kTogether], to[kTogether];
#pragma unroll
            for (int z = 0; z < kTogether; ++z) dist[i0 + z] = buf[(i0 + z) * NT + tid];
#pragma unroll
            for (int z = 0; z < kTogether; ++z) {
                const uint32_t bin = bin_of(dist[i0 + z]);
                rank[i0 + z] = from[z] = start[bin];
                to[z] = start[bin + 1];
            }
#pragma unroll
            for (uint32_t x = 0; x < kSlack; ++x) {                     // equal keys keep their order
                K other[kTogether];
#pragma unroll
                for (int z = 0; z < kTogether; ++z) other[z] = buf[from[z] + x];
#pragma unroll
                for (int z = 0; z < kTogether; ++z) {
                    const uint32_t q = from[z] + x;
                    rank[i0 + z] += (q < to[z]) & in_front(other[z], dist[i0 + z], q < (uint32_t)((i0 + z) * NT + tid));
                }
            }
#pragma unroll
            for (int z = 0; z < kTogether; ++z) {
                const uint32_t p = (i0 + z) * NT + tid;
                if (p >= (uint32_t)m) continue;
                for (uint32_t q = from[z] + kSlack; q < to[z]; ++q) rank[i0 + z] += in_front(buf[q], dist[i0 + z], q < p);
                put(rank[i0 + z], dist[i0 + z], p);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kItems; ++i)
            if (i * NT + tid < m) buf[rank[i]] = dist[i];
        __syncthreads();
        return;
    }
    if (order)
        for (int x = tid; x < m; x += NT) order[x] = (uint16_t)x;
    __syncthreads();
    int bits = 1;
    while ((1 << bits) < m) ++bits;
    const int half = 1 << (bits - 1);
    auto exchange = [&](int x, int y) {                                  // x < y; what lies beyond m counts as larger than all
        if (y >= m) return;
        const K dx = buf[x], dy = buf[y];
        if (dx > dy) {
            buf[x] = dy;
            buf[y] = dx;
            if (order) {
                const uint16_t o = order[x];
                order[x] = order[y];
                order[y] = o;
            }
        }
    };
    // A warp compares a run of neighbours: while what is merged is no longer than the run, warps need not wait for one another.
    constexpr int kWarps = NT / 32;
    const int each = max(half / kWarps, 32), first = (tid >> 5) * each + (tid & 31), end = min(((tid >> 5) + 1) * each, half);
    for (int size = 1; size <= bits; ++size) {
        const bool far = (1 << size) > 2 * each;
        if (far) __syncthreads();
        for (int x = first; x < end; x += 32) {
            const int from = x >> (size - 1) << size, j = x & ((1 << (size - 1)) - 1);
            exchange(from + j, from + (1 << size) - 1 - j);
        }
        for (int stride = size - 2; stride >= 0; --stride) {
            if (2 << (stride + 1) > 2 * each) __syncthreads();           // the step before went beyond the runs
            else __syncwarp();
            for (int x = first; x < end; x += 32) {
                const int from = (x >> stride << (stride + 1)) | (x & ((1 << stride) - 1));
                exchange(from, from + (1 << stride));
            }
        }
        __syncwarp();
    }
    __syncthreads();
    for (int x = tid; x < m; x += NT) put(x, buf[x], order ? order[x] : 0);
    __syncthreads();
}

__device__ __forceinline__ uint32_t parts_of(uint32_t size) { return min((size + kPartMean - 1) / kPartMean, (uint32_t)kMaxParts); }

// One block per bucket: where it starts, how many parts it gets, and their splitters from a sorted sample of it.
__global__ void __launch_bounds__(kSampleThreads, 1) split_sample2(Tables t, const uint64_t *keys) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *keybuf = reinterpret_cast<uint64_t *>(smem);
    uint32_t *bins = reinterpret_cast<uint32_t *>(smem + (kSampleThreads * kItems + kPad) * sizeof(uint64_t));
    __shared__ uint64_t split[kMaxParts];
    after_last_kernel();
    start_next_kernel();
    if (*t.gave_up()) return;
    const int tid = threadIdx.x, b = blockIdx.x;
    uint32_t parts_before = 0, first_part;
    for (int x = tid; x < b; x += kSampleThreads) parts_before += parts_of(t.cursor[x * kCursorGap]);
    block_scan<kSampleThreads>(parts_before, first_part);
    const uint32_t size = t.cursor[b * kCursorGap], parts = parts_of(size);
    if (tid == 0) {
        t.part_base[b] = first_part;
        t.bucket_parts[b] = parts;
        if (b == t.buckets - 1) t.result[3] = first_part + parts;
    }
    if (tid < (int)parts) t.part_owner[first_part + tid] = (uint32_t)b << kPartBits | (uint32_t)tid;
    if (parts == 0) return;
    const uint64_t lo = bucket_low(t, b), range = bucket_top(t, b) - lo;
    if (parts > 1) {
        const uint32_t m = min((uint32_t)(kSampleThreads * kItems), parts * kOverParts);
        uint64_t dist[kItems];
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const uint32_t x = i * kSampleThreads + tid;
            dist[i] = lo;
            if (x < m) {
                const uint32_t v = (uint32_t)sample_at(x, m, size);
                const uint32_t ch = t.chunk_of[(size_t)b * t.chunk_rows + v / kChunk];
                if (ch) dist[i] = keys[(size_t)(ch - 1) * kChunk + v % kChunk];
                else report(t.status(), CONST_ERR_TIMEOUT);             // not published (const_debug_set), and no tile had to wait for it
            }
        }
        sort_block<kSampleThreads>(keybuf, (uint16_t *)nullptr, bins, reinterpret_cast<uint16_t *>(bins + kBins<kSampleThreads> + 4), (int)m,
                                   Bins<kSampleThreads>(lo, range), dist, [](uint32_t, int) {}, [](uint32_t, uint64_t, uint32_t) {});
        if (tid < (int)parts - 1) {
            split[tid] = keybuf[(uint32_t)(tid + 1) * m / parts];
            t.part_split[(size_t)b * kMaxParts + tid] = split[tid];
        }
    }
    __syncthreads();
    fill_cells(t.part_cells + (size_t)b * kCells, split, (int)parts - 1, lo, cell_shift(range, 10));
}

// Where every part begins and what its keys lie between: one block per bucket, one thread per part.
__global__ void __launch_bounds__(kWide) part_jobs(Tables t) {
    after_last_kernel();
    start_next_kernel();
    if (*t.gave_up()) return;
    const int tid = threadIdx.x, b = blockIdx.x;
    uint32_t before = 0, start, total;
    for (int x = tid; x < b; x += kWide) before += t.cursor[x * kCursorGap];
    block_scan<kWide>(before, start);
    const int parts = (int)t.bucket_parts[b];
    const uint32_t g = t.part_base[b] + tid, m = tid < parts ? t.part_count[g] : 0;
    start += block_scan<kWide>(m, total);
    if (tid >= parts) return;
    const uint64_t *split = t.part_split + (size_t)b * kMaxParts;
    const uint64_t lo = tid > 0 ? split[tid - 1] : bucket_low(t, b);
    const uint64_t top = tid + 1 < parts ? split[tid] - 1 : bucket_top(t, b);
    t.jobs[g] = PartJob{lo, top - lo, start, m};
    if (m == 0) t.infos[g].count = 0;
    if (m > kTile) t.large_parts[atomicAdd(t.large, 1u)] = g;
}

// Sorts a part, writes its values and leaf coordinates and lists the nodes above the leaves.  The numbers sorted are what the keys
// have beyond `base`, the root coordinate of the part's lowest key: 32 bits wherever those suffice.
template <typename K, int NT, typename V, int ORDER>
__device__ __forceinline__ void sort_part(unsigned char *smem, const Tables &t, const LevelShifts &ls, uint32_t leaf_mask, uint32_t g, const PartJob &job,
                                          uint64_t base, const uint64_t (&key)[kItems], const V (&val)[kItems], V *vals_out,
                                          int32_t *leaf_crd, uint64_t *list_keys, uint32_t *list_pos) {
    constexpr int D = ORDER - 2;                                        // the level above the leaves
    constexpr int kRoom = kItems * NT, kWarps = NT / 32;
    __shared__ uint32_t opened[kWarps][D + 1];
    V *valbuf = reinterpret_cast<V *>(smem);
    K *buf = reinterpret_cast<K *>(smem + kRoom * sizeof(V));
    uint32_t *bins = reinterpret_cast<uint32_t *>(smem + kRoom * sizeof(V) + (kRoom + kPad) * sizeof(uint64_t));
    uint16_t *order = reinterpret_cast<uint16_t *>(bins);                // of the bitonic network, which needs the bins no more
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, m = (int)job.count;
    const uint32_t start = job.start;
    K x[kItems];
#pragma unroll
    for (int i = 0; i < kItems; ++i) x[i] = (K)(key[i] - base);
    sort_block<NT>(buf, order, bins, reinterpret_cast<uint16_t *>(bins + kBins<NT> + 4), m, Bins<NT>(job.lo - base, job.range), x,
                   [&](uint32_t p, int i) { valbuf[p] = val[i]; },
                   [&](uint32_t f, K y, uint32_t p) {
                       vals_out[start + f] = valbuf[p];
                       leaf_crd[start + f] = (int32_t)((uint32_t)y & leaf_mask);
                   });

    // every warp goes over a run of neighbours
    const int run = (m + NT - 1) / NT * 32, from = warp * run;
    uint32_t heads[kItems], mine[D + 1] = {};
    bool dup = false;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        heads[i] = 0;
        if (i * 32 < run) {
            const int p = from + i * 32 + lane;
            K diff = 0;
            bool open = false;
            if (p < m) {
                open = p == 0;
                if (p > 0) {
                    diff = buf[p] ^ buf[p - 1];
                    dup = dup || diff == 0;
                }
            }
#pragma unroll
            for (int l = 0; l <= D; ++l) {
                const unsigned all = __ballot_sync(0xffffffffu, open || (diff >> ls.shift[l]) != 0);
                mine[l] += __popc(all);
                if (l == D) heads[i] = all;
            }
        }
    }
    if (dup) report(t.status(), CONST_ERR_DUPLICATE_COORD);
    if (lane == 0)
#pragma unroll
        for (int l = 0; l <= D; ++l) opened[warp][l] = mine[l];
    __syncthreads();
    uint32_t at = start;
#pragma unroll
    for (int w = 0; w < kWarps - 1; ++w) at += w < warp ? opened[w][D] : 0;
    const uint64_t base_node = base >> ls.shift[D];
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        if (i * 32 < run) {
            const int p = from + i * 32 + lane;
            if ((heads[i] >> lane) & 1u) {
                const uint32_t o = at + __popc(heads[i] & ((1u << lane) - 1u));
                list_keys[o] = base_node + (buf[p] >> ls.shift[D]);
                list_pos[o] = start + p;
            }
            at += __popc(heads[i]);
        }
    }
    if (tid <= D) {
        uint32_t sum = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) sum += opened[w][tid];
        t.infos[g].opened[tid] = sum;
    }
    if (tid == 0) {
        PartInfo &info = t.infos[g];
        info.first = base + buf[0];
        info.last = base + buf[m - 1];
        info.count = m;
        info.start = start;
    }
}

// NT = kThreads: a block takes one part of at most kTile nonzeros.  NT = kWide: few blocks go over the list of the larger ones; that
// launch comes first and lets the other one start beside it, which therefore may not wait for its end to read what part_jobs and the
// kernels before left: the wide launch, having waited for part_jobs, releases the number of parts, and a block that acquires it sees all
// that the releasing thread could see.  A block that does not find it waits like any other, and so does the last one, so
// that the narrow launch ends after the wide one (builds, us, this against all blocks waiting: 77 M 2600 / 2626, 5 M 241 / 251, 1 M of Zipf
// slices 124 / 137).  What bounds it: instruction issue (250 thread instructions per
// nonzero), 66 % busy at 30 warps per SM.  77 M: 835 us beside 47 of the wide launch (uniform: 857);
// 5 M uniform: 70.
template <typename V, int ORDER, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) part_sort(Tables t, LevelShifts ls, int leaf_bits, const uint64_t *keys,
                                                          const V *vals, V *vals_out, int32_t *leaf_crd,
                                                          uint64_t *list_keys, uint32_t *list_pos, int withhold) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool kLarge = NT == kWide;
    auto parts = [&]() { return *t.gave_up() ? 0u : t.result[3]; };
    uint32_t todo;
    if (kLarge) {
        after_last_kernel();
        todo = *t.gave_up() ? 0u : *t.large;
        if (blockIdx.x == 0 && threadIdx.x == 0 && !withhold)
            asm volatile("st.release.gpu.global.u32 [%0], %1;" :: "l"(t.ready), "r"(parts() + 1) : "memory");
        start_next_kernel();
    } else {
        start_next_kernel();
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(todo) : "l"(t.ready) : "memory");
        if (todo == 0 || blockIdx.x == gridDim.x - 1) {
            after_last_kernel();
            todo = parts() + 1;
        }
        --todo;
    }
    const uint32_t leaf_mask = (uint32_t)((1ull << leaf_bits) - 1ull);
    for (uint32_t turn = blockIdx.x; turn < todo; turn += gridDim.x) {
        const uint32_t g = kLarge ? t.large_parts[turn] : turn;
        const PartJob job = t.jobs[g];
        if (job.count == 0 || job.count > kItems * NT) continue;
        const uint64_t *kp = keys + (size_t)g * kPartRoom;
        const V *vp = vals + (size_t)g * kPartRoom;
        uint64_t key[kItems];
        V val[kItems];
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const int x = i * NT + threadIdx.x;
            key[i] = job.lo;
            val[i] = 0;
            if (x < (int)job.count) { key[i] = kp[x]; val[i] = vp[x]; }
        }
        const uint64_t base = job.lo >> ls.shift[0] << ls.shift[0];
        if (job.lo - base + job.range < 0xffffffffull && ls.shift[0] < 32)
            sort_part<uint32_t, NT, V, ORDER>(smem, t, ls, leaf_mask, g, job, base, key, val, vals_out, leaf_crd, list_keys, list_pos);
        else
            sort_part<uint64_t, NT, V, ORDER>(smem, t, ls, leaf_mask, g, job, base, key, val, vals_out, leaf_crd, list_keys, list_pos);
        if (kLarge) __syncthreads();
    }
}

// Numbers the nodes: one block per bucket, one thread per part; the last block adds up the buckets.
template <int ORDER>
__global__ void __launch_bounds__(kWide) part_scan(Tables t, LevelShifts ls) {
    constexpr int L = ORDER - 1;
    after_last_kernel();
    if (*t.gave_up()) return;
    const int tid = threadIdx.x, b = blockIdx.x;
    const uint32_t parts = t.bucket_parts[b], g = t.part_base[b] + tid;
    const bool in = tid < (int)parts;
    uint32_t count[L] = {};
    if (in && t.infos[g].count > 0) {
        PartInfo &info = t.infos[g];
        uint32_t cont = 0, q = g;
        while (q > 0 && t.infos[q - 1].count == 0) --q;                 // parts without nonzeros have no ends
        const uint64_t prev = q > 0 ? t.infos[q - 1].last : 0ull;
#pragma unroll
        for (int l = 0; l < L; ++l) {
            const bool same = q > 0 && (prev >> ls.shift[l]) == (info.first >> ls.shift[l]);
            cont |= (uint32_t)same << l;
            count[l] = info.opened[l] - same;
        }
        info.cont = cont;
    }
#pragma unroll
    for (int l = 0; l < L; ++l) {
        uint32_t total;
        const uint32_t before = block_scan<kWide>(count[l], total);
        if (in) t.part_nodes[(size_t)g * (kMaxOrder - 1) + l] = before;
        if (tid == 0) t.bucket_nodes[b * (kMaxOrder - 1) + l] = total;
    }
    if (!last_block(t.arrived + 1)) return;
#pragma unroll
    for (int l = 0; l < L; ++l) {
        uint32_t total;
        const uint32_t in_bucket = tid < t.buckets ? __ldcg(t.bucket_nodes + tid * (kMaxOrder - 1) + l) : 0;
        const uint32_t at = block_scan<kWide>(in_bucket, total);
        if (tid < t.buckets) t.bucket_nodes[tid * (kMaxOrder - 1) + l] = at;
        if (tid == 0) t.result[l] = total;
    }
}

// The upper levels out of the lists of nodes: crd and pos of all levels above the leaves, slice_ptr, and behind the last nonzero
// the ends of the pos arrays.
constexpr int kNodeThreads = 128;
template <int ORDER>
__global__ void __launch_bounds__(kNodeThreads) part_nodes(const PartInfo *__restrict__ infos, const uint32_t *__restrict__ part_base,
                                                          const uint32_t *__restrict__ bucket_base, const uint32_t *__restrict__ part_owner,
                                                          const uint64_t *__restrict__ list_keys, const uint32_t *__restrict__ list_pos,
                                                          uint32_t n, LevelShifts ls, CsfArrays out, int32_t *__restrict__ slice_ptr) {
    constexpr int L = ORDER - 1, D = L - 1;
    __shared__ uint32_t warps[2][kNodeThreads / 32][L];
    const uint32_t g = blockIdx.x;
    const PartInfo info = infos[g];
    if (info.count == 0) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t run[L];
#pragma unroll
    for (int l = 0; l < L; ++l)
        run[l] = bucket_base[(part_owner[g] >> kPartBits) * (kMaxOrder - 1) + l] + part_base[(size_t)g * (kMaxOrder - 1) + l];
    const uint32_t nodes = info.opened[D];
    const bool last_part = info.start + info.count == n;
    for (uint32_t f0 = 0, turn = 0; f0 < nodes; f0 += kNodeThreads, turn ^= 1u) {
        const uint32_t f = f0 + tid;
        uint64_t key = 0, diff = 0;
        uint32_t pos = 0;
        if (f < nodes) {
            key = list_keys[info.start + f];
            pos = list_pos[info.start + f];
            diff = f > 0 ? key ^ list_keys[info.start + f - 1] : 0;
        }
        unsigned open[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            const bool opens = f < nodes && (f == 0 ? !((info.cont >> l) & 1u) : (diff >> (ls.shift[l] - ls.shift[D])) != 0);
            open[l] = __ballot_sync(0xffffffffu, opens);
            if (lane == 0) warps[turn][warp][l] = __popc(open[l]);
        }
        __syncthreads();
        uint32_t at[L];
#pragma unroll
        for (int l = 0; l < L; ++l) {
            at[l] = run[l] + __popc(open[l] & ((1u << lane) - 1u));
#pragma unroll
            for (int w = 0; w < kNodeThreads / 32; ++w) {
                if (w < warp) at[l] += warps[turn][w][l];
                run[l] += warps[turn][w][l];
            }
        }
        if (f < nodes) {
#pragma unroll
            for (int l = 0; l < L; ++l) {
                if ((open[l] >> lane) & 1u) {
                    out.crd[l][at[l]] = (int32_t)((key >> (ls.shift[l] - ls.shift[D])) & ((1ull << out.bits[l]) - 1ull));
                    out.pos[l + 1][at[l]] = l < D ? (int32_t)at[l < D ? l + 1 : l] : (int32_t)pos;
                    if (l == 0) slice_ptr[at[0]] = (int32_t)pos;
                }
            }
            if (last_part && f + 1 == nodes) {
#pragma unroll
                for (int l = 0; l < L; ++l) at[l] += (open[l] >> lane) & 1u;
                out.pos[0][0] = 0;
                out.pos[0][1] = (int32_t)at[0];
#pragma unroll
                for (int l = 0; l < L; ++l) out.pos[l + 1][at[l]] = l < D ? (int32_t)at[l < D ? l + 1 : l] : (int32_t)n;
                slice_ptr[at[0]] = (int32_t)n;
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------
// host
// ------------------------------------------------------------------------------------------------
// The splitter sort has nine launches and two samplings where the radix sort has two and one per pass: it takes tensors of
// at least 200 000 nonzeros whose count, times the passes beyond two, is 700 000 or more.  Both sides around the line (build, us,
// radix / splitters; uniform, Zipf-sized slices): five passes, keys of 44 bits, 150 K 102 / 93, 103 / 95, 200 K 112 / 94, 114 / 96, 260 K
// 114 / 95, 116 / 101; of 41 bits, 150 K 97 / 94, 96 / 92, 200 K 101 / 94, 101 / 93; four passes, 150 K 84 / 86, 82 / 94, 200 K 85 / 89,
// 86 / 91, 260 K 90 / 92, 91 / 93, 300 K 98 / 90, 98 / 93, 500 K 98 / 93, 98 / 97; three, uniform, 500 K 99 / 93, 700 K 105 / 101.  The
// line lies where no number of passes loses; five would gain up to 15 % from 150 K on.  Beyond it the splitters take 0.62 to 0.80 of
// the time from 3 M on, in fp32 and fp64, orders 2 to 4, sorted or not.  Above 110 M a bucket would need more parts than there are ways.
constexpr int64_t kSplitMin = 200000, kSplitWork = 700000, kSplitMax = 110000000;

int bucket_count(int64_t nnz) {
    int k = 16;
    while (k < kMaxBuckets && (int64_t)k * 100 * kPartMean < nnz) k <<= 1;
    return k;
}

// Where everything lies in the arena.
struct Layout {
    size_t cleared, bytes;
    size_t result, cursor, part_count, chunk_of, samples, bucket_split, bucket_cells, per_bucket, part_split, part_cells, part_owner, large_parts,
        part_nodes, bucket_nodes, chunk_owner, jobs, infos, keys1, vals1, keys2, vals2;
    int buckets, chunk_rows;
    uint32_t max_chunks, max_parts;
    Layout(int64_t nnz, size_t vsize) {
        buckets = bucket_count(nnz);
        max_chunks = (uint32_t)(nnz / kChunk + buckets + 1);
        max_parts = (uint32_t)(nnz / kPartMean + buckets + 1);
        chunk_rows = (int)std::min<int64_t>(max_chunks, 8 * (nnz / kChunk / buckets) + 8);
        bytes = 0;
        auto put = [&](size_t b) { const size_t o = bytes; bytes += (b + 255) / 256 * 256; return o; };
        result = put(256);
        cursor = put(4 * (size_t)buckets * kCursorGap);
        part_count = put(4 * (size_t)max_parts);
        chunk_of = put(4 * (size_t)buckets * chunk_rows);
        cleared = bytes;
        samples = put(8 * (size_t)buckets * kOverBuckets);
        bucket_split = put(8 * (size_t)buckets);
        bucket_cells = put(4 * kCells);
        per_bucket = put(2 * 4 * (size_t)buckets);
        part_split = put(8 * (size_t)buckets * kMaxParts);
        part_cells = put(4 * (size_t)buckets * kCells);
        part_owner = put(4 * (size_t)max_parts);
        large_parts = put(4 * (size_t)max_parts);
        part_nodes = put(4 * (size_t)max_parts * (kMaxOrder - 1));
        bucket_nodes = put(4 * (size_t)buckets * (kMaxOrder - 1));
        chunk_owner = put(8 * (size_t)max_chunks);
        jobs = put(sizeof(PartJob) * (size_t)max_parts);
        infos = put(sizeof(PartInfo) * (size_t)max_parts);
        keys1 = put(8 * (size_t)max_chunks * kChunk);
        vals1 = put(vsize * max_chunks * kChunk);
        keys2 = put(8 * (size_t)max_parts * kPartRoom);
        vals2 = put(vsize * max_parts * kPartRoom);
    }
};

template <typename K>
cudaError_t allow_smem(K kernel, size_t bytes, PerDeviceOnce &once) {
    return once_per_device(once, [&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); });
}

template <typename V, int ORDER>
const_status_t queue_tile(const char *name, unsigned blocks, const PackArgs &pa, const Tables &t, const uint64_t *kin, const V *vin,
                          uint64_t *kout, V *vout, cudaStream_t stream) {
    constexpr size_t smem = kTile * (sizeof(uint64_t) + sizeof(V) + sizeof(uint16_t));
    static PerDeviceOnce once;                                           // per template instance
    CB_CUDA(allow_smem(split_tile<V, ORDER>, smem, once));
    const DebugKnobs knobs = debug_knobs();
    const int spins = knobs.spin_limit > 0 ? knobs.spin_limit : kSpinLimit, withhold = knobs.withhold;
    // Blocks that stay for several tiles wait for an empty machine: started early they lie unevenly on the SMs, for good (build of
    // 77 M: 2735 us against 2509; of 5 M: 224 against 226).
    const bool stays = ORDER > 0 && (int64_t)blocks * kTile < t.n;
    cudaError_t e = cudaSuccess;
    CB_LAUNCH(name, stream, if (stays) split_tile<V, ORDER><<<blocks, kThreads, smem, stream>>>(pa, t, kin, vin, kout, vout, spins, withhold);
                            else e = launch_early(split_tile<V, ORDER>, dim3(blocks), kThreads, smem, stream, pa, t, kin, vin, kout, vout, spins, withhold));
    return e == cudaSuccess ? CONST_OK : CONST_ERR_CUDA;
}

template <typename V, int ORDER>
const_status_t queue_sort(const PackArgs &pa, const KeyLayout &k, const LevelShifts &ls, const Layout &at, unsigned char *arena, const Tables &t,
                          const V *vals, V *vals_out, int32_t *leaf_crd, cudaStream_t stream) {
    const uint32_t samples = (uint32_t)at.buckets * kOverBuckets;
    uint64_t *keys1 = reinterpret_cast<uint64_t *>(arena + at.keys1), *keys2 = reinterpret_cast<uint64_t *>(arena + at.keys2);
    V *vals1 = reinterpret_cast<V *>(arena + at.vals1), *vals2 = reinterpret_cast<V *>(arena + at.vals2);
    CB_LAUNCH("split_sample", stream, split_sample<ORDER><<<(samples + kThreads - 1) / kThreads, kThreads, 0, stream>>>(pa, t, samples));
    static PerDeviceOnce once_rank, once_sample, once_sort, once_large;
    CB_CUDA(allow_smem(split_rank, sizeof(uint64_t) * kMaxBuckets * kOverBuckets, once_rank));
    CB_LAUNCH("split_rank", stream,
              CB_CUDA(launch_early(split_rank, dim3(samples / (kThreads / 8)), kThreads, sizeof(uint64_t) * samples, stream, t, samples)));
    const_status_t s = queue_tile<V, ORDER>("split_buckets", (unsigned)std::min<int64_t>((t.n + kTile - 1) / kTile, 148 * tile_blocks(true)), pa, t, nullptr, vals, keys1, vals1, stream);
    if (s != CONST_OK) return s;
    // keys' pad, bins and their starts (see sort_block)
    constexpr auto with_bins = [](size_t bytes, int bins) { return bytes + kPad * sizeof(uint64_t) + (bins + 4) * sizeof(uint32_t) + (bins + 8) * sizeof(uint16_t); };
    constexpr size_t smem_sample = with_bins(kSampleThreads * kItems * sizeof(uint64_t), kBins<kSampleThreads>);
    CB_CUDA(allow_smem(split_sample2, smem_sample, once_sample));
    CB_LAUNCH("split_sample2", stream,
              CB_CUDA(launch_early(split_sample2, dim3((unsigned)at.buckets), kSampleThreads, smem_sample, stream, t, (const uint64_t *)keys1)));
    s = queue_tile<V, 0>("split_parts", at.max_chunks, pa, t, keys1, vals1, keys2, vals2, stream);
    if (s != CONST_OK) return s;
    constexpr size_t smem = with_bins(kTile * (sizeof(uint64_t) + sizeof(V)), kBins<kThreads>);
    constexpr size_t smem_large = with_bins(kPartRoom * (sizeof(uint64_t) + sizeof(V)), kBins<kWide>);
    CB_CUDA(allow_smem(part_sort<V, ORDER, kThreads>, smem, once_sort));
    CB_CUDA(allow_smem(part_sort<V, ORDER, kWide>, smem_large, once_large));
    uint32_t *pos1 = reinterpret_cast<uint32_t *>(vals1);
    const int withhold = debug_knobs().withhold;
    CB_LAUNCH("part_jobs", stream, CB_CUDA(launch_early(part_jobs, dim3((unsigned)at.buckets), kWide, 0, stream, t)));
    CB_LAUNCH("part_sort_large", stream,
              CB_CUDA(launch_early(part_sort<V, ORDER, kWide>, dim3(148), kWide, smem_large, stream, t, ls, (int)k.bits[ORDER - 1],
                                   (const uint64_t *)keys2, (const V *)vals2, vals_out, leaf_crd, keys1, pos1, withhold)));
    CB_LAUNCH("part_sort", stream,
              CB_CUDA(launch_early(part_sort<V, ORDER, kThreads>, dim3(at.max_parts), kThreads, smem, stream, t, ls, (int)k.bits[ORDER - 1],
                                   (const uint64_t *)keys2, (const V *)vals2, vals_out, leaf_crd, keys1, pos1, withhold)));
    CB_LAUNCH("part_scan", stream, CB_CUDA(launch_early(part_scan<ORDER>, dim3((unsigned)at.buckets), kWide, 0, stream, t, ls)));
    CB_CUDA(cudaGetLastError());
    return CONST_OK;
}

template <typename V>
const_status_t queue_order(const PackArgs &pa, const KeyLayout &k, const LevelShifts &ls, const Layout &at, unsigned char *arena, const Tables &t,
                           const void *vals, void *vals_out, int32_t *leaf_crd, cudaStream_t stream) {
    const V *in = static_cast<const V *>(vals);
    V *out = static_cast<V *>(vals_out);
    switch (pa.order) {
        case 2: return queue_sort<V, 2>(pa, k, ls, at, arena, t, in, out, leaf_crd, stream);
        case 3: return queue_sort<V, 3>(pa, k, ls, at, arena, t, in, out, leaf_crd, stream);
        default: return queue_sort<V, 4>(pa, k, ls, at, arena, t, in, out, leaf_crd, stream);
    }
}

}  // namespace

bool split_covers(int64_t nnz, const KeyLayout &k) {
    const int path = debug_knobs().build_path;
    if (nnz < 1 || nnz > kSplitMax || path == 1) return false;
    return path >= 2 || (nnz >= kSplitMin && nnz * (k.digits.passes - 2) >= kSplitWork);
}

size_t split_bytes(int64_t nnz, const_dtype_t dtype) { return Layout(nnz, dtype == CONST_F32 ? 4 : 8).bytes; }

const_status_t split_sort(const PackArgs &pa, const KeyLayout &k, int64_t nnz, const void *vals, const_dtype_t dtype, void *vals_out,
                          int32_t *leaf_crd, unsigned char *arena, cudaStream_t stream, SplitSort *out) {
    const Layout at(nnz, dtype == CONST_F32 ? 4 : 8);
    Tables t;
    auto u32 = [&](size_t o) { return reinterpret_cast<uint32_t *>(arena + o); };
    t.result = u32(at.result);
    t.arrived = t.result + 32;
    t.next_chunk = t.result + 48;
    t.large = t.result + 56;
    t.ready = t.result + 60;
    t.large_parts = u32(at.large_parts);
    t.cursor = u32(at.cursor);
    t.part_count = u32(at.part_count);
    t.chunk_of = u32(at.chunk_of);
    t.samples = reinterpret_cast<uint64_t *>(arena + at.samples);
    t.bucket_split = reinterpret_cast<uint64_t *>(arena + at.bucket_split);
    t.part_split = reinterpret_cast<uint64_t *>(arena + at.part_split);
    t.bucket_cells = u32(at.bucket_cells);
    t.part_cells = u32(at.part_cells);
    t.jobs = reinterpret_cast<PartJob *>(arena + at.jobs);
    t.part_base = u32(at.per_bucket);
    t.bucket_parts = t.part_base + at.buckets;
    t.part_owner = u32(at.part_owner);
    t.part_nodes = u32(at.part_nodes);
    t.bucket_nodes = u32(at.bucket_nodes);
    t.chunk_owner = reinterpret_cast<uint2 *>(arena + at.chunk_owner);
    t.infos = reinterpret_cast<PartInfo *>(arena + at.infos);
    t.key_max = 0;
    for (int l = 0; l < pa.order; ++l) t.key_max |= (uint64_t)(pa.dim[l] - 1) << pa.shift[l];
    t.n = nnz;
    t.buckets = at.buckets;
    t.bucket_shift = std::max(0, k.total_bits - 10);
    t.chunk_rows = at.chunk_rows;
    t.max_chunks = at.max_chunks;
    LevelShifts ls;
    ls.order = pa.order;
    for (int l = 0; l < kMaxOrder; ++l) ls.shift[l] = k.shift[l];
    CB_CUDA(cudaMemsetAsync(arena, 0, at.cleared, stream));
    const const_status_t s = dtype == CONST_F32 ? queue_order<uint32_t>(pa, k, ls, at, arena, t, vals, vals_out, leaf_crd, stream)
                                                : queue_order<unsigned long long>(pa, k, ls, at, arena, t, vals, vals_out, leaf_crd, stream);
    if (s != CONST_OK) return s;
    out->list_keys = reinterpret_cast<const uint64_t *>(arena + at.keys1);
    out->list_pos = u32(at.vals1);
    out->infos = t.infos;
    out->part_base = t.part_nodes;
    out->bucket_base = t.bucket_nodes;
    out->part_owner = t.part_owner;
    out->result = t.result;
    out->order = pa.order;
    out->ls = ls;
    out->nnz = nnz;
    return CONST_OK;
}

const_status_t split_scatter(const SplitSort &s, const CsfArrays &out, int32_t *slice_ptr, int64_t parts, cudaStream_t stream) {
    const PartInfo *infos = static_cast<const PartInfo *>(s.infos);
    CB_LAUNCH("part_nodes", stream, {
        switch (s.order) {
            case 2: part_nodes<2><<<(unsigned)parts, kNodeThreads, 0, stream>>>(infos, s.part_base, s.bucket_base, s.part_owner, s.list_keys, s.list_pos, (uint32_t)s.nnz, s.ls, out, slice_ptr); break;
            case 3: part_nodes<3><<<(unsigned)parts, kNodeThreads, 0, stream>>>(infos, s.part_base, s.bucket_base, s.part_owner, s.list_keys, s.list_pos, (uint32_t)s.nnz, s.ls, out, slice_ptr); break;
            default: part_nodes<4><<<(unsigned)parts, kNodeThreads, 0, stream>>>(infos, s.part_base, s.bucket_base, s.part_owner, s.list_keys, s.list_pos, (uint32_t)s.nnz, s.ls, out, slice_ptr); break;
        }
    });
    CB_CUDA(cudaGetLastError());
    return CONST_OK;
}

}  // namespace cb
