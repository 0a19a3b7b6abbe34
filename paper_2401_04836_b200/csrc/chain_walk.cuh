// Leaf-balanced walk of a CSF chain, shared by the fused chain kernels (chain_kernels.cu).
//
// The leaves of the tensor are cut into contiguous chunks of equal cost or equal length (cut_leaves), one per warp, whatever the
// slices look like; a warp searches for the place of its first leaf once and walks from there.  It proceeds in windows of leaves
// that do not cross a slice.  A window is staged by the whole warp with coalesced loads: every lane turns the
// node ends it has read (pos arrays) into bits of a leaf mask, so that a leaf knows the ordinal of its node by
// a population count and no lane ever follows a chain of dependent loads.  The staged record of a leaf is
//   row   the leaf's coordinate (row of the leaf factor)
//   val   its value
//   tag2  order 4: coordinate of its level-2 node if the leaf ends that node's part of a run, else -1
//   tag1  what ends with the leaf at level 1: the ordinal of the piece, or the level-1 coordinate; else -1
// Lane groups then work through equal runs of records.  A run that begins or ends inside a node sums a part of
// it (a piece): every contraction of the chain is linear in its intermediate, so pieces need no merging.
#pragma once
#include <algorithm>

#include "common.cuh"

namespace cb {
namespace walk {

constexpr unsigned kAll = 0xffffffffu;

// Two neighbouring entries.  fp32 pairs go through the packed multiply-add (two fused multiply-adds, each rounded as
// the scalar one, in one instruction): the kernels issue half as many.
template <typename T> struct Pair;
template <> struct Pair<float> {
    unsigned long long bits;
    __device__ __forceinline__ float lo() const { return __uint_as_float((unsigned)bits); }
    __device__ __forceinline__ float hi() const { return __uint_as_float((unsigned)(bits >> 32)); }
};
template <> struct Pair<double> {
    double x, y;
    __device__ __forceinline__ double lo() const { return x; }
    __device__ __forceinline__ double hi() const { return y; }
};
__device__ __forceinline__ Pair<float> make_pair(float x, float y) {
    Pair<float> p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p.bits) : "f"(x), "f"(y));
    return p;
}
__device__ __forceinline__ Pair<double> make_pair(double x, double y) { return Pair<double>{x, y}; }
__device__ __forceinline__ void fma2(Pair<float> &t, const Pair<float> &x, const Pair<float> &v) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(t.bits) : "l"(x.bits), "l"(v.bits));
}
__device__ __forceinline__ void fma2(Pair<double> &t, const Pair<double> &x, const Pair<double> &v) {
    t.x = fma(x.x, v.x, t.x);
    t.y = fma(x.y, v.y, t.y);
}

// 16 bytes of a factor row or of an intermediate
template <typename T> struct Vec {
    static constexpr int N = 16 / sizeof(T);
    Pair<T> p[N / 2];
    __device__ __forceinline__ T at(int i) const { return i & 1 ? p[i / 2].hi() : p[i / 2].lo(); }
};
__device__ __forceinline__ Vec<float> make_vec(const float4 &v) { return Vec<float>{{make_pair(v.x, v.y), make_pair(v.z, v.w)}}; }
__device__ __forceinline__ Vec<double> make_vec(const double2 &v) { return Vec<double>{{make_pair(v.x, v.y)}}; }
__device__ __forceinline__ Vec<float> load_vec(const float *p) { return make_vec(__ldg(reinterpret_cast<const float4 *>(p))); }
__device__ __forceinline__ Vec<double> load_vec(const double *p) { return make_vec(__ldg(reinterpret_cast<const double2 *>(p))); }
__device__ __forceinline__ Vec<float> peek_vec(const float *p) { return make_vec(*reinterpret_cast<const float4 *>(p)); }     // shared memory
__device__ __forceinline__ Vec<double> peek_vec(const double *p) { return make_vec(*reinterpret_cast<const double2 *>(p)); }
__device__ __forceinline__ Pair<float> load_pair(const float *p) {
    const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
    return make_pair(v.x, v.y);
}
__device__ __forceinline__ Pair<double> load_pair(const double *p) { return load_vec(p).p[0]; }
__device__ __forceinline__ void store_vec(float *p, const Vec<float> &v) {
    *reinterpret_cast<float4 *>(p) = make_float4(v.p[0].lo(), v.p[0].hi(), v.p[1].lo(), v.p[1].hi());
}
__device__ __forceinline__ void store_vec(double *p, const Vec<double> &v) {
    *reinterpret_cast<double2 *>(p) = make_double2(v.p[0].x, v.p[0].y);
}
// Adds 16 aligned bytes of entries atomically, each on its own (fp32: one vector reduction, a quarter of the operations
// on the lines of a slice that many warps share).
__device__ __forceinline__ void add_vec(float *p, const Vec<float> &v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};"
                 :: "l"(p), "f"(v.p[0].lo()), "f"(v.p[0].hi()), "f"(v.p[1].lo()), "f"(v.p[1].hi()) : "memory");
}
__device__ __forceinline__ void add_vec(double *p, const Vec<double> &v) {
    atomicAdd(p, v.p[0].x);
    atomicAdd(p + 1, v.p[0].y);
}
template <typename T>
__device__ __forceinline__ Vec<T> zero_vec() {
    Vec<T> z;
#pragma unroll
    for (int i = 0; i < Vec<T>::N / 2; ++i) z.p[i] = make_pair(T(0), T(0));
    return z;
}
template <typename T>
__device__ __forceinline__ void axpy(Vec<T> &t, const Pair<T> &xx, const Vec<T> &v) {      // xx: the factor, twice
#pragma unroll
    for (int i = 0; i < Vec<T>::N / 2; ++i) fma2(t.p[i], xx, v.p[i]);
}
template <typename T>
__device__ __forceinline__ void mul_add(Vec<T> &t, const Vec<T> &x, const Vec<T> &v) {
#pragma unroll
    for (int i = 0; i < Vec<T>::N / 2; ++i) fma2(t.p[i], x.p[i], v.p[i]);
}

// Asynchronous copy of 16 bytes of global memory into shared memory, and the wait for all of a thread's copies.
__device__ __forceinline__ void copy16(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Starts copying the factor rows (R entries each) of the window's pieces to dst.
template <typename T, int R>
__device__ __forceinline__ void fetch_rows(T *dst, const T *factor, const int32_t *j, int pieces, int lane) {
    constexpr int PER = R * sizeof(T) / 16;             // 16-byte parts per row
    for (int i = lane; i < pieces * PER; i += 32)
        copy16(dst + i * Vec<T>::N, factor + (size_t)j[i / PER] * R + (i % PER) * Vec<T>::N);
}

// The sum of the parts that the block's warps have left, `apart` entries apart.
template <int WARPS, typename T>
__device__ __forceinline__ Vec<T> add_parts(const T *parts, int apart) {
    Vec<T> sum = peek_vec(parts);
#pragma unroll
    for (int w = 1; w < WARPS; ++w) {
        const Vec<T> v = peek_vec(parts + w * apart);
#pragma unroll
        for (int c = 0; c < Vec<T>::N / 2; ++c) sum.p[c] = make_pair(sum.p[c].lo() + v.p[c].lo(), sum.p[c].hi() + v.p[c].hi());
    }
    return sum;
}

template <typename T, int ORDER>
struct Chain {                                          // level l: pos[l], crd[l]
    const int32_t *pos[ORDER], *crd[ORDER];
    const int32_t *slice_ptr;                           // [n[0] + 1] first leaf of every slice
    int32_t n[ORDER];
    const T *vals;
};

// Largest x in [lo, hi) with pos[x] <= target, by the whole warp: 128 probes a step (pos[lo] <= target), so that 16 384
// candidates take two dependent loads.
__device__ __forceinline__ int32_t warp_find(const int32_t *__restrict__ pos, int32_t lo, int32_t hi, int32_t target, int lane) {
    while (hi - lo > 1) {
        const int32_t step = (int32_t)(((int64_t)hi - lo + 127) / 128);
        int32_t p[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t at = lo + (int64_t)(32 * k + lane) * step;
            p[k] = at < hi ? __ldg(pos + at) : 0x7fffffff;          // (a target is below that)
        }
        int32_t c = -1;
#pragma unroll
        for (int k = 0; k < 4; ++k) c += __popc(__ballot_sync(kAll, p[k] <= target));
        lo += c * step;
        hi = hi - lo < step ? hi : lo + step;
    }
    return lo;
}

// Where a warp stands: the node of every inner level that contains a leaf.
template <int ORDER>
struct Place {
    int32_t node[ORDER - 1];
};

// Largest x in [lo, hi) with key(x) <= target, by the whole warp, for two targets at once (key(lo) <= target; key does not fall).
template <class Key>
__device__ __forceinline__ void warp_find2(Key key, int32_t (&lo)[2], int32_t (&hi)[2], const int64_t (&target)[2], int lane) {
    while (hi[0] - lo[0] > 1 || hi[1] - lo[1] > 1) {
        bool below[2][4];
        int32_t step[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            step[t] = (int32_t)(((int64_t)hi[t] - lo[t] + 127) / 128);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t at = lo[t] + (int64_t)(32 * k + lane) * step[t];
                below[t][k] = at < hi[t] && key((int32_t)at) <= target[t];
            }
        }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            int32_t c = -1;
#pragma unroll
            for (int k = 0; k < 4; ++k) c += __popc(__ballot_sync(kAll, below[t][k]));
            lo[t] += c * step[t];
            hi[t] = hi[t] - lo[t] < step[t] ? hi[t] : lo[t] + step[t];
        }
    }
}

// Root first (slice: the leaf's, where it is known, or -1), so that every search below is over one slice only: few steps, each a
// dependent load.
template <typename T, int ORDER>
__device__ __forceinline__ Place<ORDER> place_of(const Chain<T, ORDER> &x, int32_t leaf, int lane, int32_t slice = -1) {
    Place<ORDER> p;
    p.node[0] = slice >= 0 ? slice : warp_find(x.slice_ptr, 0, x.n[0], leaf, lane);
    const int32_t f0 = __ldg(x.pos[1] + p.node[0]), f1 = __ldg(x.pos[1] + p.node[0] + 1);
    if constexpr (ORDER == 3) {
        p.node[1] = warp_find(x.pos[2], f0, f1, leaf, lane);
    } else {
        p.node[2] = warp_find(x.pos[3], __ldg(x.pos[2] + f0), __ldg(x.pos[2] + f1), leaf, lane);
        p.node[1] = warp_find(x.pos[2], f0, f1, p.node[2], lane);
    }
    return p;
}

template <typename T>
struct __align__(16) Rec {
    int32_t row, tag1;
    T val;
};
template <>
struct __align__(16) Rec<float> {
    int32_t row, tag1;
    float val;
    int32_t tag2;
};

// The records of a window are run-major interleaved: record i of run g is at i * G + g, so that the G groups of a
// warp read consecutive records at every step.

// What a window needs of the tensor, as read: entry lane + 32 m of the leaf arrays from the window's first leaf on, and
// of the inner levels from the node on that holds it.  Requested one window ahead of its use.
template <typename T, int ORDER, int W>
struct Ahead {
    static constexpr int NW = W / 32;
    int32_t row[NW], end1[NW], j[NW];
    T val[NW];
    int32_t end2[ORDER == 4 ? NW : 1], k[ORDER == 4 ? NW : 1];
};

// Requests the window that starts at leaf e; leaves from e1 on are not wanted.
template <typename T, int ORDER, int W>
__device__ __forceinline__ void request(const Chain<T, ORDER> &x, const Place<ORDER> &place, int32_t e, int32_t e1, int lane,
                                        Ahead<T, ORDER, W> &a) {
    constexpr int LEAF = ORDER - 1;
#pragma unroll
    for (int m = 0; m < W / 32; ++m) {
        const int r = lane + 32 * m;
        const bool in = r < e1 - e;
        a.row[m] = in ? __ldg(x.crd[LEAF] + e + r) : 0;
        a.val[m] = in ? __ldg(x.vals + e + r) : T(0);
        const bool in1 = in && r < x.n[1] - place.node[1];
        a.end1[m] = in1 ? __ldg(x.pos[2] + place.node[1] + 1 + r) : 0x7fffffff;
        a.j[m] = in1 ? __ldg(x.crd[1] + place.node[1] + r) : 0;
        if constexpr (ORDER == 4) {
            const bool in2 = in && r < x.n[2] - place.node[2];
            a.end2[m] = in2 ? __ldg(x.pos[3] + place.node[2] + 1 + r) : 0x7fffffff;
            a.k[m] = in2 ? __ldg(x.crd[2] + place.node[2] + r) : 0;
        }
    }
}

// Bit r of the mask: a node ends with leaf r of the window.  b[m] is the window-relative last leaf of node
// lane + 32 m; node k ends at leaf k or later, so word w needs the nodes below 32 (w + 1) only.
template <int NW>
__device__ __forceinline__ void end_mask(int (&b)[NW], int cnt, unsigned (&mask)[NW]) {
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        unsigned v = 0;
#pragma unroll
        for (int m = 0; m <= w; ++m)
            if (b[m] < cnt && (b[m] >> 5) == w) v |= 1u << (b[m] & 31);
        mask[w] = __reduce_or_sync(kAll, v);
    }
}

// Shared-memory tables of one staged window.
template <typename T, int ORDER, int W>
struct Stage {
    Rec<T> rec[W];
    int32_t tag2[(ORDER == 4 && sizeof(T) == 8) ? W : 1];
    int32_t j[W];                        // level-1 coordinate of the window's fibres, then of its pieces (PIECES)
    int32_t k[ORDER == 4 ? W : 1];       // level-2 coordinate of the window's level-2 nodes
    int32_t last[ORDER == 4 ? W : 1];    // last leaf of those nodes
    __device__ __forceinline__ void put(int at, int32_t row, T val, int32_t tag1, int32_t t2) {
        Rec<T> r;
        r.row = row;
        r.tag1 = tag1;
        r.val = val;
        if constexpr (sizeof(T) == 4) r.tag2 = t2;
        else if constexpr (ORDER == 4) tag2[at] = t2;
        rec[at] = r;
    }
    __device__ __forceinline__ int32_t second_tag(int at, const Rec<T> &r) const {
        if constexpr (sizeof(T) == 4) return r.tag2;
        else if constexpr (ORDER == 4) return tag2[at];
        else return -1;
    }
};

// Stages the requested window's first cnt leaves (from leaf e0) as G runs of `run` records and moves `place` past
// them; returns the number of pieces.  PIECES: tag1 is the ordinal of the piece, whose level-1 coordinate goes to
// st.j; otherwise tag1 is that coordinate itself.  Records between cnt and G * run are neutral.
// flat: every level-2 node of the window has one leaf (order 4).
template <typename T, int ORDER, int W, int G, bool PIECES>
__device__ __forceinline__ int stage_window(const Ahead<T, ORDER, W> &a, Place<ORDER> &place, int32_t e0, int cnt, int run,
                                            int lane, Stage<T, ORDER, W> &st, bool &flat) {
    constexpr int NW = W / 32;
    static_assert(W <= 256 && W % 32 == 0, "r / run by multiplication; whole words");
    unsigned fm[NW], nm[NW];
    int b[NW];
    __syncwarp();                                                   // the tables of the window before are used up
#pragma unroll
    for (int m = 0; m < NW; ++m) st.j[lane + 32 * m] = a.j[m];
    if constexpr (ORDER == 4) {
#pragma unroll
        for (int m = 0; m < NW; ++m) {
            b[m] = a.end2[m] - 1 - e0;
            st.last[lane + 32 * m] = b[m];
            st.k[lane + 32 * m] = a.k[m];
        }
        end_mask<NW>(b, cnt, nm);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < NW; ++m) {                              // level-1 ends are node numbers: look their last leaf up
            const int o = a.end1[m] - 1 - place.node[ORDER - 2];
            b[m] = o < W ? st.last[o] : 0x7fffffff;
        }
    } else {
#pragma unroll
        for (int m = 0; m < NW; ++m) b[m] = a.end1[m] - 1 - e0;
    }
    end_mask<NW>(b, cnt, fm);
    __syncwarp();
    const unsigned below = (1u << lane) - 1u;
    const unsigned inv = (65536u + run - 1) / run;                  // r / run == r * inv >> 16 for r < 256
    int fibre = 0, node = 0, pieces = 0;
    int32_t ends[NW], jp[NW];                                       // ordinal of the piece the leaf ends, its coordinate
#pragma unroll
    for (int m = 0; m < NW; ++m) {
        const int r = lane + 32 * m;
        ends[m] = -1;
        if (32 * m < G * run) {
            const bool in = r < cnt;
            const int g = (int)((r * inv) >> 16), i = r - g * run;
            const bool cut = in && (i == run - 1 || r == cnt - 1);  // the run ends here, whatever it is inside of
            const bool end1 = cut || ((fm[m] >> lane) & 1u);
            const unsigned pm = __ballot_sync(kAll, end1);
            int32_t tag1 = -1, tag2 = -1;
            if (end1) {
                jp[m] = st.j[fibre + __popc(fm[m] & below)];
                ends[m] = pieces + __popc(pm & below);
                tag1 = PIECES ? ends[m] : jp[m];
            }
            if constexpr (ORDER == 4)
                if (cut || ((nm[m] >> lane) & 1u)) tag2 = st.k[node + __popc(nm[m] & below)];
            if (g < G) st.put(i * G + g, a.row[m], in ? a.val[m] : T(0), tag1, tag2);
            pieces += __popc(pm);
        }
        fibre += __popc(fm[m]);
        if constexpr (ORDER == 4) node += __popc(nm[m]);
    }
    if (PIECES) {
        __syncwarp();                                               // every fibre's coordinate has been read
#pragma unroll
        for (int m = 0; m < NW; ++m)
            if (ends[m] >= 0) st.j[ends[m]] = jp[m];
    }
    place.node[1] += fibre;
    if constexpr (ORDER == 4) place.node[ORDER - 2] += node;
    flat = ORDER == 4 && node == cnt;
    __syncwarp();
    return pieces;
}

// The leaves of one warp, and the end of those of its block.
struct Share {
    int32_t e0, e1, block_end;
    int32_t slice = -1, begin, end;                      // slice of leaf e0 and its leaves, where the search has met them
    Share() = default;
    __device__ __forceinline__ Share(int32_t nnz, int32_t chunk, int warps) {
        const int64_t b0 = (int64_t)blockIdx.x * warps * chunk, b1 = b0 + (int64_t)warps * chunk;
        const int64_t w0 = b0 + (int64_t)(threadIdx.x >> 5) * chunk;
        block_end = b1 < nnz ? (int32_t)b1 : nnz;
        e0 = w0 < nnz ? (int32_t)w0 : nnz;
        e1 = nnz - e0 < chunk ? nnz : e0 + chunk;
    }
    // Equal costs instead: a slice counts as `weight` leaves more than it has (weight = 0: equal leaves, no search).  Every warp of
    // the block has to call this.
    template <typename T, int ORDER>
    __device__ __forceinline__ Share(const Chain<T, ORDER> &x, int32_t chunk, int32_t weight, int warps, int lane) : Share(x.n[ORDER - 1], chunk, warps) {
        if (!weight) return;
        const int64_t c0 = ((int64_t)blockIdx.x * warps + (threadIdx.x >> 5)) * chunk, target[2] = {c0, c0 + chunk};
        int32_t lo[2] = {0, 0}, hi[2] = {x.n[0], x.n[0]};
        warp_find2([&](int32_t s) { return (int64_t)__ldg(x.slice_ptr + s) + (int64_t)weight * s; }, lo, hi, target, lane);
        int32_t at[2][3], e[2];
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int k = 0; k < 3; ++k) at[t][k] = __ldg(x.slice_ptr + (lo[t] + k < x.n[0] ? lo[t] + k : x.n[0]));
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int64_t in = target[t] - at[t][0] - (int64_t)weight * lo[t];
            e[t] = in < at[t][1] - at[t][0] ? at[t][0] + (int32_t)in : at[t][1];
        }
        e0 = e[0];
        e1 = e[1];
        const bool next = e0 == at[0][1];                // behind the slice's leaves: the next one's first
        slice = lo[0] + next;
        begin = next ? at[0][1] : at[0][0];
        end = next ? at[0][2] : at[0][1];
        __shared__ int32_t s_end;
        if (threadIdx.x == 32 * (warps - 1)) s_end = e1;
        __syncthreads();
        block_end = s_end;
    }
};

// Walks the warp's leaves: window(place, e, limit) consumes some leaves of [e, limit), all in one slice, moves the place
// and returns how many; flush(slice, whole) ends a slice or the warp's part of it (whole: the warp had all of it).
// find(e) is the place of leaf e; start(place) is called once, at the place of the first leaf.  Returns the slice that the whole block lies in, not
// flushed, or -1: the parts of such a slice are to be added up in the block first, which keeps the number of atomic
// additions to one row of the result (and the rounding errors they add) down where a slice is shared by many warps.
// Every warp of the block has to call this.
template <typename T, int ORDER, class Find, class Start, class Window, class Flush>
__device__ __forceinline__ int32_t walk_chunk(const Chain<T, ORDER> &x, const Share &own, Find find, Start start, Window window, Flush flush) {
    __shared__ int32_t first_slice;                      // where the block's first leaf lies
    Place<ORDER> place;
    place.node[0] = 0;
    int32_t e = own.e0, end = 0;
    bool from_start = false;
    if (e < own.e1) {
        place = find(e);
        start(place);
        from_start = (own.slice >= 0 ? own.begin : __ldg(x.slice_ptr + place.node[0])) == e;
        end = own.slice >= 0 ? own.end : __ldg(x.slice_ptr + place.node[0] + 1);
    }
    after_last_kernel();                                 // the result is cleared; everything up to here only read the tensor
    if (threadIdx.x == 0) first_slice = place.node[0];
    const bool joint = __syncthreads_or(threadIdx.x < 32 && end >= own.block_end) != 0;
    while (e < own.e1) {
        const int32_t limit = end < own.e1 ? end : own.e1;
        while (e < limit) e += window(place, e, limit);
        if (joint) break;                                // the slice goes on to the end of the block
        flush(place.node[0], from_start && end <= own.e1);
        from_start = true;
        ++place.node[0];
        if (e < own.e1) end = __ldg(x.slice_ptr + place.node[0] + 1);
    }
    return joint ? first_slice : -1;
}

// Leaves of the run of one lane group: the window's leaves dealt out evenly, rounded up to the unroll factor.
template <int W, int G, int UNROLL>
__device__ __forceinline__ int run_length(int cnt) {
    static_assert(W % (G * UNROLL) == 0, "G rounded runs of at most W leaves have to fit the W records of a stage");
    return (((cnt + G - 1) / G) + UNROLL - 1) / UNROLL * UNROLL;
}

// Host side
template <typename T, int ORDER>
inline Chain<T, ORDER> chain_of(const const_csf *X) {
    Chain<T, ORDER> x;
    for (int l = 0; l < ORDER; ++l) {
        x.pos[l] = X->pos[l];
        x.crd[l] = X->crd[l];
        x.n[l] = (int32_t)X->n[l];
    }
    x.slice_ptr = X->slice_ptr;
    x.vals = static_cast<const T *>(X->vals);
    return x;
}

// Leaves per warp: as many whole waves of the `fit` warps that an SM holds as keep a chunk below `most` leaves (finding a place
// and handing over a slice part are paid once per chunk, a wave that is not full leaves SMs idle), in multiples of 64.
// A tensor that gives no warp 64 leaves is dealt out to one wave as it is: windows end with their slice, so
// a warp with many short slices goes through as many windows one after the other (TTMc 8 x 8, 3000 leaves in slices of
// one: 103 us at 64 leaves a warp, 14.5 here; 30 000 in slices of four: 62 and 25), and more warps than fit start late
// (the latter with twice as many: 29).  But in chunks of half a slice on average where slices are longer than that: more
// parts of a slice mean more atomic additions and more rounding, and gain nothing (30 000 in slices of 64: 15.0 us, in
// chunks of 13 leaves 15.9, of 64 18.4; 20 000 in slices of 100: relative error 7.5e-8, in chunks of 9 leaves 8.3e-8).  Little more than
// a window of 64 a warp would be two (one_window): rather one, and a few warps that start late (TTMc 23 x 32 in fp64, 40 000 leaves:
// 27.7, in chunks of 128 34.6).
inline int32_t chunk_leaves(int64_t nnz, int64_t slices, int64_t most, int fit, bool one_window = false) {
    const int64_t wave = 148 * (int64_t)fit, waves = (nnz + wave * most - 1) / (wave * most);
    const int64_t c = (nnz + wave * waves - 1) / (wave * waves);
    if (c < 64) return (int32_t)std::min<int64_t>(std::max((nnz + 148 * fit - 1) / (148 * fit), nnz / (2 * slices)), 64);
    return one_window && c < 96 ? 64 : (int32_t)((c + 63) / 64 * 64);
}

// How the leaves are cut: cost per warp, and what a slice costs beyond its leaves (Share).  A slice's last window is not full and its
// result is handed over: with Zipf-sized slices the warps that got the many short ones took several times as long as the
// others.  Equal leaves against this, us: slices Zipf 1.1, TTMc 8 x 8, 1.5 M leaves in slices of 40: 219 / 77, 6 M of 400: 162 /
// 106, 20 M of 333: 453 / 334; 32 x 32: 256 / 149, 406 / 353, 1124 / 954; order 4: 387 / 129, 407 / 301, 1080 / 853; MTTKRP rank 32: 119 / 56,
// 122 / 103, 382 / 288; slices of equal size: within 1 % from 6 M on, below that 0.88 to 0.99 of the time
// by family, but up to a tenth slower where equal leaves are just whole windows (8 x 32, 300 000 leaves in slices of 400: 17.6 / 19.3; Zipf
// 1.1: 25.4 / 23.3) and in very short slices (order-4 MTTKRP, 50 000 in slices of five: 17.5 / 20.7; 300 000: 0.8 of the time).  Not where slices are long anyway, 3000 leaves (from 4000 leaves on it gained
// 1 to 3 % under Zipf 1.1 and lost 1 to 2 % on equal ones), nor where a chunk would cost less than `least`, which is no less than
// `weight` (a warp may end up without leaves, a block may not).  Short chunks, equal leaves against this, us: 10 x 12, 200 000 leaves in
// slices of 143, equal / Zipf 1.1: 25.9 / 28.6 against 21.3 / 19.8; fp64 18 x 23, 40 000 of 133: 35.2 / 33.9 against 24.9 / 23.6; order 4, TTMc,
// 150 000: 0.93 of the time on average.  MTTKRP of order 3 keeps a longer `least` where slices are long: 400 000 equal ones of 100 in
// chunks of 138 17.6 / 19.8.
// Where a wave is few warps, one of long chunks leaves slices of different density uneven: up to `even` waves then, in chunks of no less
// than 448 leaves each (equal leaves: in any number of waves).
struct Cut { int32_t chunk, weight; };
inline Cut cut_leaves(int64_t nnz, int64_t slices, int64_t most, int fit, int32_t weight, int least, bool one_window = false, int even = 1) {
    constexpr int64_t kShort = 448;
    const int64_t wave = 148 * (int64_t)fit, cost = nnz + weight * slices;
    const int64_t waves = std::max<int64_t>((cost + wave * most - 1) / (wave * most), std::min<int64_t>(even, (nnz + wave * kShort - 1) / (wave * kShort)));
    const int64_t c = (cost + wave * waves - 1) / (wave * waves);
    if (c >= least && nnz < 3000 * slices) return Cut{(int32_t)((c + 7) / 8 * 8), weight};
    return Cut{chunk_leaves(nnz, slices, even > 1 ? kShort : most, fit, one_window), 0};
}

// Clears `out` ("R[*] = 0" precedes the nest; bytes = 0: the launch before has done that) and launches the kernel so that it starts while the clearing still runs: it
// looks its place in the tensor up meanwhile and waits (after_last_kernel) before it writes.  Clearing by a kernel of the
// library instead of a memset is what allows that (20 000 nonzeros at rank 8, device time bound by the two launches:
// 14.2 -> 13.9 us a call).
template <class Args>
inline const_status_t launch_on_cleared(const char *name, void (*kernel)(Args), const Args &args, dim3 grid, int threads, size_t smem,
                                        void *out, size_t bytes, cudaStream_t stream) {
    if (bytes) CB_CUDA(clear_result(out, bytes, stream));
    cudaError_t e = cudaSuccess;
    CB_LAUNCH(name, stream, e = launch_early(kernel, grid, threads, smem, stream, args));
    return e == cudaSuccess ? CONST_OK : CONST_ERR_CUDA;
}

}  // namespace walk
}  // namespace cb
