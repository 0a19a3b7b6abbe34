// Fused kernels of the "chain" family: one CSF tensor contracted leaf level first with one dense factor per level
// (TTMc, Sec. 5.3; MTTKRP, Sec. 5.2), executed as the fused loop nest of Fig. 4(b):
//
//   for i (slice)                     -- root level, fused
//     for j (fibre)                   -- level 1, fused
//       t[*] = 0                      -- order-1 intermediate, reset per fibre
//       for k: t[b] += X[i,j,k] * V[k,b]            (producer contraction)
//       for a,b: Y[i,a,b] += U[j,a] * t[b]          (consumer contraction; MTTKRP: A[i,r] += B[j,r] * t[r])
// and, for order 4, with one more producer: P[c] += X[i,j,k,l] * W[l,c];  Q[b,c] += V[k,b] * P[c].
//
// Every warp owns a run of the tensor's leaves -- of equal cost, a slice counting as some leaves beyond its own, or of equal
// leaves (cut_leaves) -- and walks it in windows that it stages as flat records
// (chain_walk.cuh), on its own: no work list, no slice too large or too small.  The warps of a block meet only where the
// whole block lies in one slice, to add up their results.
//   producer   Lane groups (one 128-bit load per lane and factor row) work through equal runs of the window's
//     records, four row gathers in flight per lane.  Where a record ends a fibre, the group has the finished t.
//   consumer, MTTKRP   The group multiplies t with the row of B whose coordinate the record carries (requested
//     together with the row gathers) into its own accumulator of the slice.
//   consumer, TTMc   The group parks t in shared memory, with the fibre's j.  After the window the warp holds the
//     R2 x R3 slice result as RW x 16-byte register blocks; the lanes that cover one result work on one parked
//     t, so a warp consumes 32 / ((R2 / RW)(R3 / V)) of them per step.
// The slice result stays in registers and leaves the warp once per slice: stored if the warp had the whole slice, added
// atomically otherwise (once per block where the whole block lies in one slice).
//
// What bounds them, and what they measured on a B200 (before: one block or warp per slice from the work lists): the
// gathers are served by L2 (hit rate 80-90 %, DRAM below 10 %), and the kernels are held by L2 latency and by the
// instructions per leaf (9-12; order 4: 29), not by a bandwidth.  MTTKRP, 100 M leaves, rank 32: 1.79 -> 1.34 ms (gather
// ceiling 1.0 ms; 64 registers for 32 warps per SM matter: 72 registers cost 13 % more); TTMc 8 x 32, 8 M leaves in fibres of
// 1.6: 499 -> 284 us; order-4 TTMc, 50 M leaves: 4.57 ms on these pipes, 3.11 ms with the last contraction on the tensor
// cores -> 2.28 ms here (the factor rows of the consumer copied to shared memory behind the producer -0.4 ms, parked Q
// laid out free of bank conflicts -0.3 ms, leaf arrays requested one window ahead -0.1 ms; the latter costs more
// registers than it gains in the order-3 kernels).
#include <algorithm>
#include <type_traits>

#include "chain_walk.cuh"

namespace cb {
namespace {

using namespace walk;

constexpr int kWarps = 4;                             // warps per block; they meet where a slice covers the block
constexpr int kUnroll = 4;                            // row gathers in flight per lane

// blocks an SM holds: what the registers are cut for, or the shared memory (warp_bytes per warp) allows
constexpr int blocks_that_fit(int by_registers, size_t warp_bytes) {
    return std::min(by_registers, (int)(227 * 1024 / (warp_bytes * kWarps + 1024)));
}

template <typename T>
__device__ __forceinline__ void put_entry(T *dst, T v, bool whole) {
    if (whole) *dst = v;
    else atomicAdd(dst, v);
}

// writes entries [0, n) of a vector; n >= Vec::N and aligned: one 16-byte access
template <typename T>
__device__ __forceinline__ void put_vec(T *dst, const Vec<T> &v, int n, bool whole) {
    if (n >= Vec<T>::N && (reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
        if (whole) store_vec(dst, v);
        else add_vec(dst, v);
        return;
    }
#pragma unroll
    for (int i = 0; i < Vec<T>::N; ++i)
        if (i < n) put_entry(dst + i, v.at(i), whole);
}

// The block's warps have left their parts of one slice's result, [rows][cols] each, `apart` entries apart: adds them up
// and adds the sum to out, whose rows have real_cols entries (real_rows of them).
template <typename T>
__device__ __forceinline__ void add_joint(const T *parts, int apart, int rows, int cols, T *out, int real_rows, int real_cols) {
    constexpr int N = Vec<T>::N;
    __syncthreads();
    for (int i = threadIdx.x * N; i < rows * cols; i += kWarps * 32 * N) {
        const Vec<T> sum = add_parts<kWarps>(parts + i, apart);
        const int r = i / cols, c = i % cols;
        if (r < real_rows) put_vec(out + (size_t)r * real_cols + c, sum, real_cols - c, false);
    }
}

// sum of the pair over lanes that differ in the lane-number bits from `from` up
template <typename T>
__device__ __forceinline__ void reduce_pair(Pair<T> &p, int from) {
    T x = p.lo(), y = p.hi();
    for (int off = from; off < 32; off <<= 1) {
        x += __shfl_xor_sync(kAll, x, off);
        y += __shfl_xor_sync(kAll, y, off);
    }
    p = make_pair(x, y);
}

// ---------------------------------------------------------------------------------------------- MTTKRP
template <typename T, int ORDER, int RP>
struct MttkrpShape {
    static constexpr int N = Vec<T>::N;
    static constexpr int LPR = RP / N;                // lanes per factor row
    static constexpr int G = 32 / LPR;                // lane groups per warp
    static constexpr int W = 128;                     // leaves per window
    static constexpr int BLOCKS = sizeof(T) == 4 ? (ORDER == 3 ? 8 : 6) : 4;          // resident blocks the registers are cut for
    static constexpr int FIT = (sizeof(T) == 8 && ORDER == 3 ? 6 : BLOCKS) * kWarps;  // warps an SM holds (fp64, order 3: 80 registers)
    static_assert(LPR >= 1 && LPR <= 32, "rank tile");
};

// F[m]: factor of level m + 1, rows of `stride` entries, columns [RP * blockIdx.y, ...) taken here; R = real rank
template <typename T, int ORDER>
struct MttkrpArgs {
    Chain<T, ORDER> x;
    const T *F[ORDER - 1];
    T *out;
    size_t out_bytes;
    int32_t stride, R;
    int32_t chunk, weight;                            // cost per warp, and of a slice beyond its leaves (set by the launch)
};

template <typename T, int ORDER, int RP>
__global__ void __launch_bounds__(kWarps * 32, MttkrpShape<T, ORDER, RP>::BLOCKS) mttkrp_kernel(const __grid_constant__ MttkrpArgs<T, ORDER> a) {
    using S = MttkrpShape<T, ORDER, RP>;
    constexpr int N = S::N;
    __shared__ Stage<T, ORDER, S::W> stages[kWarps];
    const int lane = threadIdx.x & 31, g = lane / S::LPR, q = lane % S::LPR;
    const Share own(a.x, a.chunk, a.weight, kWarps, lane);
    Stage<T, ORDER, S::W> &st = stages[threadIdx.x >> 5];
    const int col = blockIdx.y * RP + q * N;
    const T *leaf = a.F[ORDER - 2] + col, *mid = ORDER == 4 ? a.F[1] + col : nullptr, *top = a.F[0] + col;
    Vec<T> acc = zero_vec<T>();
    const int32_t joint = walk_chunk(a.x, own, [&](int32_t e) { return place_of(a.x, e, lane, own.slice); },
        [](const Place<ORDER> &) {},
        [&](Place<ORDER> &place, int32_t e, int32_t limit) {
            const int cnt = limit - e < S::W ? limit - e : S::W;
            const int run = run_length<S::W, S::G, kUnroll>(cnt);
            bool flat;
            Ahead<T, ORDER, S::W> ahead;
            request<T, ORDER, S::W>(a.x, place, e, limit, lane, ahead);
            stage_window<T, ORDER, S::W, S::G, false>(ahead, place, e, cnt, run, lane, st, flat);
            Vec<T> t = zero_vec<T>(), s = zero_vec<T>();
            for (int i = 0; i < run; i += kUnroll) {
                Rec<T> r[kUnroll];
                Vec<T> v[kUnroll], u[kUnroll], w[kUnroll];
                int32_t k[kUnroll];
#pragma unroll
                for (int z = 0; z < kUnroll; ++z) {
                    r[z] = st.rec[(i + z) * S::G + g];
                    v[z] = load_vec(leaf + (size_t)r[z].row * a.stride);
                    if constexpr (ORDER == 4) {
                        k[z] = st.second_tag((i + z) * S::G + g, r[z]);
                        if (k[z] >= 0) w[z] = load_vec(mid + (size_t)k[z] * a.stride);
                    }
                    if (r[z].tag1 >= 0) u[z] = load_vec(top + (size_t)r[z].tag1 * a.stride);
                }
#pragma unroll
                for (int z = 0; z < kUnroll; ++z) {
                    axpy(t, make_pair(r[z].val, r[z].val), v[z]);
                    if constexpr (ORDER == 4) {
                        if (k[z] >= 0) { mul_add(s, t, w[z]); t = zero_vec<T>(); }
                        if (r[z].tag1 >= 0) { mul_add(acc, s, u[z]); s = zero_vec<T>(); }
                    } else {
                        if (r[z].tag1 >= 0) { mul_add(acc, t, u[z]); t = zero_vec<T>(); }
                    }
                }
            }
            return cnt;
        },
        [&](int32_t slice, bool whole) {
#pragma unroll
            for (int i = 0; i < N / 2; ++i) reduce_pair(acc.p[i], S::LPR);
            if (g == 0) put_vec(a.out + (size_t)__ldg(a.x.crd[0] + slice) * a.R + col, acc, a.R - col, whole);
            acc = zero_vec<T>();
        });
    if (joint >= 0) {
        T *part = reinterpret_cast<T *>(st.rec);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < N / 2; ++i) reduce_pair(acc.p[i], S::LPR);
        if (g == 0) store_vec(part + q * N, acc);
        const int c0 = blockIdx.y * RP;
        add_joint(reinterpret_cast<const T *>(stages[0].rec), (int)(sizeof(stages[0]) / sizeof(T)), 1, RP,
                  a.out + (size_t)__ldg(a.x.crd[0] + joint) * a.R + c0, 1, a.R - c0);
    }
}

// ---------------------------------------------------------------------------------------------- TTMc, order 3
template <typename T, int R2, int R3>
struct Ttmc3Shape {
    static constexpr int N = Vec<T>::N;
    static constexpr int LPR = R3 / N, G = 32 / LPR;
    static constexpr int W = 64;                      // leaves per window
    static constexpr int RW = (R2 / 8) * (R3 / N) <= 32 ? 8 : 16;      // rows of a register block
    static constexpr int LPF = (R2 / RW) * (R3 / N), FPW = 32 / LPF;   // lanes per parked t, parked t per step
    static constexpr int BLOCKS = sizeof(T) == 4 ? 5 : 3;              // resident blocks the registers are cut for
    struct __align__(16) Smem {
        Stage<T, 3, W> st;
        T t[W * R3];                                  // parked t, one row per piece
        T u[W * R2];                                  // the factor row that goes with it
    };
    static constexpr int FIT = blocks_that_fit(BLOCKS, sizeof(Smem)) * kWarps;       // warps an SM holds
};

template <typename T>
struct Ttmc3Args {
    Chain<T, 3> x;
    const T *U, *V;                                   // rows of R2 and R3 (padded) entries
    T *out;
    size_t out_bytes;
    int32_t R2, R3;                                   // real ranks
    int32_t chunk, weight;                            // cost per warp, and of a slice beyond its leaves (set by the launch)
};

template <typename T, int R2, int R3>
__global__ void __launch_bounds__(kWarps * 32, Ttmc3Shape<T, R2, R3>::BLOCKS) ttmc3_kernel(const __grid_constant__ Ttmc3Args<T> a) {
    using S = Ttmc3Shape<T, R2, R3>;
    constexpr int N = S::N;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, g = lane / S::LPR, q = lane % S::LPR;
    const Share own(a.x, a.chunk, a.weight, kWarps, lane);
    typename S::Smem &sm = reinterpret_cast<typename S::Smem *>(smem)[threadIdx.x >> 5];
    const T *V = a.V + q * N;
    // consumer: the lane owns rows rg .. rg + RW - 1 and columns cg .. cg + N - 1 of the slice result; acc[i][c]: rows
    // rg + 2 i and rg + 2 i + 1 of column cg + c
    const int slot = lane / S::LPF, rg = (lane % S::LPF) / (R3 / N) * S::RW, cg = (lane % S::LPF) % (R3 / N) * N;
    Pair<T> acc[S::RW / 2][N];
    auto clear = [&]() {
#pragma unroll
        for (int i = 0; i < S::RW / 2; ++i)
#pragma unroll
            for (int c = 0; c < N; ++c) acc[i][c] = make_pair(T(0), T(0));
    };
    clear();
    // adds the slots up and hands every row of the lane's block to put
    auto gather = [&](auto put) {
#pragma unroll
        for (int i = 0; i < S::RW / 2; ++i) {
            Vec<T> lo, hi;
#pragma unroll
            for (int c = 0; c < N; ++c) reduce_pair(acc[i][c], S::LPF);
#pragma unroll
            for (int c = 0; c < N / 2; ++c) {
                lo.p[c] = make_pair(acc[i][2 * c].lo(), acc[i][2 * c + 1].lo());
                hi.p[c] = make_pair(acc[i][2 * c].hi(), acc[i][2 * c + 1].hi());
            }
            put(rg + 2 * i, lo);
            put(rg + 2 * i + 1, hi);
        }
    };
    const int32_t joint = walk_chunk(a.x, own, [&](int32_t e) { return place_of(a.x, e, lane, own.slice); },
        [](const Place<3> &) {},
        [&](Place<3> &place, int32_t e, int32_t limit) {
            const int cnt = limit - e < S::W ? limit - e : S::W;
            const int run = run_length<S::W, S::G, kUnroll>(cnt);
            bool flat;
            Ahead<T, 3, S::W> ahead;
            request<T, 3, S::W>(a.x, place, e, limit, lane, ahead);
            const int pieces = stage_window<T, 3, S::W, S::G, true>(ahead, place, e, cnt, run, lane, sm.st, flat);
            fetch_rows<T, R2>(sm.u, a.U, sm.st.j, pieces, lane);
            Vec<T> t = zero_vec<T>();
            for (int i = 0; i < run; i += kUnroll) {
                Rec<T> r[kUnroll];
                Vec<T> v[kUnroll];
#pragma unroll
                for (int z = 0; z < kUnroll; ++z) {
                    r[z] = sm.st.rec[(i + z) * S::G + g];
                    v[z] = load_vec(V + (size_t)r[z].row * R3);
                }
#pragma unroll
                for (int z = 0; z < kUnroll; ++z) {
                    axpy(t, make_pair(r[z].val, r[z].val), v[z]);
                    if (r[z].tag1 >= 0) { store_vec(sm.t + r[z].tag1 * R3 + q * N, t); t = zero_vec<T>(); }
                }
            }
            copies_done();
            __syncwarp();
#pragma unroll 2
            for (int p = slot; p < pieces; p += S::FPW) {
                const T *row = sm.u + p * R2 + rg;
                const Vec<T> tv = peek_vec(sm.t + p * R3 + cg);
                Vec<T> u[S::RW / N];
#pragma unroll
                for (int i = 0; i < S::RW / N; ++i) u[i] = peek_vec(row + i * N);
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    const Pair<T> tt = make_pair(tv.at(c), tv.at(c));
#pragma unroll
                    for (int i = 0; i < S::RW / 2; ++i) fma2(acc[i][c], u[i * 2 / N].p[i % (N / 2)], tt);
                }
            }
            return cnt;
        },
        [&](int32_t slice, bool whole) {
            T *dst = a.out + (size_t)__ldg(a.x.crd[0] + slice) * a.R2 * a.R3 + cg;
            gather([&](int row, const Vec<T> &v) {
                if (slot == 0 && row < a.R2) put_vec(dst + row * a.R3, v, a.R3 - cg, whole);
            });
            clear();
        });
    if (joint >= 0) {
        __syncwarp();
        gather([&](int row, const Vec<T> &v) {
            if (slot == 0) store_vec(sm.t + row * R3 + cg, v);
        });
        add_joint(reinterpret_cast<typename S::Smem *>(smem)[0].t, (int)(sizeof(sm) / sizeof(T)), R2, R3,
                  a.out + (size_t)__ldg(a.x.crd[0] + joint) * a.R2 * a.R3, a.R2, a.R3);
    }
}

// ---------------------------------------------------------------------------------------------- TTMc, order 4, ranks up to 8
template <typename T>
struct Ttmc4Shape {
    static constexpr int N = Vec<T>::N;
    static constexpr int R = 8, SL = 4, G = 32 / SL;  // lanes per producer group, groups per warp
    static constexpr int W = 64, P = 40;              // leaves per window, parked Q (a window that would need more is halved)
    static constexpr int BLOCKS = sizeof(T) == 4 ? 3 : 1;              // resident blocks the registers are cut for
    static constexpr int QROW = R * R + 16;           // 16 spare entries: neighbouring pieces start in other banks
    // A lane of a producer group holds 2 R entries of Q as chunks of 16 bytes; chunk c of lane h is parked at
    // (c * SL + h) * 16 bytes, so that the lanes of a group write neighbouring chunks.
    struct __align__(16) Smem {
        Stage<T, 4, W> st;
        T q[P * QROW];                                // parked Q
        T u[P * R];                                   // the factor row that goes with it
    };
    static constexpr int FIT = blocks_that_fit(BLOCKS, sizeof(Smem)) * kWarps;
};

template <typename T>
struct Ttmc4Args {
    Chain<T, 4> x;
    const T *U, *V, *W;                               // rows of 8 entries
    T *out;
    size_t out_bytes;
    int32_t R2, R3, R4;                               // real ranks
    int32_t chunk, weight;                            // cost per warp, and of a slice beyond its leaves (set by the launch)
};

template <typename T>
__global__ void __launch_bounds__(kWarps * 32, Ttmc4Shape<T>::BLOCKS) ttmc4_kernel(const __grid_constant__ Ttmc4Args<T> a) {
    using S = Ttmc4Shape<T>;
    constexpr int N = S::N, R = S::R, NV = R / N;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, g = lane / S::SL, h = lane % S::SL;
    const Share own(a.x, a.chunk, a.weight, kWarps, lane);
    typename S::Smem &sm = reinterpret_cast<typename S::Smem *>(smem)[threadIdx.x >> 5];
    const T *V = a.V + 2 * h;
    // consumer: 16 lanes cover the 8 x 8 x 8 result; the lane owns every a for one b and four c; acc[i][c]: a = 2 i, 2 i + 1
    // (numbered so that neighbouring lanes read neighbouring chunks of the parked Q)
    const int slot = lane >> 4, b = 2 * (lane & 3) + ((lane >> 3) & 1), ch = (lane & 4);
    const int chunk = (b & 1) * NV + ch / N;
    Pair<T> acc[R / 2][4];
    auto clear = [&]() {
#pragma unroll
        for (int i = 0; i < R / 2; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[i][c] = make_pair(T(0), T(0));
    };
    clear();
    // adds the two slots up and hands the lane's part of every plane a = i to put, 16 bytes (from column c) at a time
    auto gather = [&](auto put) {
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
#pragma unroll
            for (int c = 0; c < 4; ++c) reduce_pair(acc[i][c], 16);
#pragma unroll
            for (int c = 0; c < 4; c += N) {
                Vec<T> lo, hi;
#pragma unroll
                for (int n = 0; n < N / 2; ++n) {
                    lo.p[n] = make_pair(acc[i][c + 2 * n].lo(), acc[i][c + 2 * n + 1].lo());
                    hi.p[n] = make_pair(acc[i][c + 2 * n].hi(), acc[i][c + 2 * n + 1].hi());
                }
                put(2 * i, ch + c, lo);
                put(2 * i + 1, ch + c, hi);
            }
        }
    };
    Ahead<T, 4, S::W> ahead;
    const int32_t joint = walk_chunk(a.x, own, [&](int32_t e) { return place_of(a.x, e, lane, own.slice); },
        [&](const Place<4> &place) {
            request<T, 4, S::W>(a.x, place, own.e0, own.e1, lane, ahead);
        },
        [&](Place<4> &place, int32_t e, int32_t limit) {
            int cnt = limit - e < S::W ? limit - e : S::W;
            const Place<4> from = place;
            int run = run_length<S::W, S::G, kUnroll>(cnt);
            bool flat;
            int pieces = stage_window<T, 4, S::W, S::G, true>(ahead, place, e, cnt, run, lane, sm.st, flat);
            if (pieces > S::P) {                      // uniform over the warp
                cnt = 32;
                place = from;
                run = run_length<S::W, S::G, kUnroll>(cnt);
                pieces = stage_window<T, 4, S::W, S::G, true>(ahead, place, e, cnt, run, lane, sm.st, flat);
            }
            request<T, 4, S::W>(a.x, place, e + cnt, own.e1, lane, ahead);
            fetch_rows<T, R>(sm.u, a.U, sm.st.j, pieces, lane);
            Vec<T> p[NV], q0[NV], q1[NV];             // P; rows b = 2 h and 2 h + 1 of Q
#pragma unroll
            for (int c = 0; c < NV; ++c) p[c] = q0[c] = q1[c] = zero_vec<T>();
            auto produce = [&](auto one_leaf_per_node) {
                constexpr bool FLAT = decltype(one_leaf_per_node)::value;
                for (int i = 0; i < run; i += kUnroll) {
                    Rec<T> r[kUnroll];
                    Vec<T> w[kUnroll][NV];
                    T v0[kUnroll], v1[kUnroll];
                    int32_t k[kUnroll];
#pragma unroll
                    for (int z = 0; z < kUnroll; ++z) {
                        const int at = (i + z) * S::G + g;
                        r[z] = sm.st.rec[at];
                        k[z] = sm.st.second_tag(at, r[z]);
#pragma unroll
                        for (int c = 0; c < NV; ++c) w[z][c] = load_vec(a.W + (size_t)r[z].row * R + c * N);
                        v0[z] = v1[z] = T(0);
                        if (k[z] >= 0) {
                            const Pair<T> v = load_pair(V + (size_t)k[z] * R);
                            v0[z] = v.lo();
                            v1[z] = v.hi();
                        }
                    }
#pragma unroll
                    for (int z = 0; z < kUnroll; ++z) {
                        if constexpr (FLAT) {         // Q[b, :] += V[k, b] (X W[l, :]), multiplied in the schedule's order
#pragma unroll
                            for (int c = 0; c < NV; ++c) {
                                Vec<T> x = zero_vec<T>();
                                axpy(x, make_pair(r[z].val, r[z].val), w[z][c]);
                                axpy(q0[c], make_pair(v0[z], v0[z]), x);
                                axpy(q1[c], make_pair(v1[z], v1[z]), x);
                            }
                        } else {                      // P[:] += X W[l, :];  Q[b, :] += V[k, b] P[:]
#pragma unroll
                            for (int c = 0; c < NV; ++c) axpy(p[c], make_pair(r[z].val, r[z].val), w[z][c]);
                            if (k[z] >= 0) {
#pragma unroll
                                for (int c = 0; c < NV; ++c) {
                                    axpy(q0[c], make_pair(v0[z], v0[z]), p[c]);
                                    axpy(q1[c], make_pair(v1[z], v1[z]), p[c]);
                                    p[c] = zero_vec<T>();
                                }
                            }
                        }
                        if (r[z].tag1 >= 0) {
                            T *dst = sm.q + r[z].tag1 * S::QROW + h * N;
#pragma unroll
                            for (int c = 0; c < NV; ++c) {
                                store_vec(dst + c * S::SL * N, q0[c]);
                                store_vec(dst + (NV + c) * S::SL * N, q1[c]);
                                q0[c] = q1[c] = zero_vec<T>();
                            }
                        }
                    }
                }
            };
            if (flat) produce(std::true_type());
            else produce(std::false_type());
            copies_done();
            __syncwarp();
#pragma unroll 2
            for (int s = slot; s < pieces; s += 2) {
                const T *row = sm.u + s * R;
                Vec<T> u[NV], q[4 / N];
#pragma unroll
                for (int i = 0; i < NV; ++i) u[i] = peek_vec(row + i * N);
#pragma unroll
                for (int i = 0; i < 4 / N; ++i) q[i] = peek_vec(sm.q + s * S::QROW + ((chunk + i) * S::SL + (lane & 3)) * N);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const Pair<T> qq = make_pair(q[c / N].at(c % N), q[c / N].at(c % N));
#pragma unroll
                    for (int i = 0; i < R / 2; ++i) fma2(acc[i][c], u[i * 2 / N].p[i % (N / 2)], qq);
                }
            }
            return cnt;
        },
        [&](int32_t slice, bool whole) {
            T *dst = a.out + (size_t)__ldg(a.x.crd[0] + slice) * a.R2 * a.R3 * a.R4;
            gather([&](int i, int c, const Vec<T> &v) {
                if (slot == 0 && b < a.R3 && i < a.R2) put_vec(dst + ((size_t)i * a.R3 + b) * a.R4 + c, v, a.R4 - c, whole);
            });
            clear();
        });
    if (joint >= 0) {
        __syncwarp();
        gather([&](int i, int c, const Vec<T> &v) {
            if (slot == 0) store_vec(sm.q + (i * R + b) * R + c, v);
        });
        T *dst = a.out + (size_t)__ldg(a.x.crd[0] + joint) * a.R2 * a.R3 * a.R4;
        const T *parts = reinterpret_cast<typename S::Smem *>(smem)[0].q;
        __syncthreads();
        for (int i = threadIdx.x * N; i < R * R * R; i += kWarps * 32 * N) {
            const Vec<T> sum = add_parts<kWarps>(parts + i, (int)(sizeof(sm) / sizeof(T)));
            const int a2 = i / (R * R), b2 = i / R % R, c2 = i % R;
            if (a2 < a.R2 && b2 < a.R3) put_vec(dst + ((size_t)a2 * a.R3 + b2) * a.R4 + c2, sum, a.R4 - c2, false);
        }
    }
}

// ---------------------------------------------------------------------------------------------- host side
template <class Args, typename T, int ORDER>
unsigned cut_blocks(Args &a, const Chain<T, ORDER> &x, const Cut &cut) {
    a.chunk = cut.chunk;
    a.weight = cut.weight;
    const int64_t warps = (x.n[ORDER - 1] + (int64_t)cut.weight * x.n[0] + cut.chunk - 1) / cut.chunk;
    return (unsigned)((warps + kWarps - 1) / kWarps);
}

template <typename T, int ORDER, int RP>
const_status_t launch_mttkrp(MttkrpArgs<T, ORDER> a, int tiles, cudaStream_t stream) {
    using S = MttkrpShape<T, ORDER, RP>;
    const int64_t nnz = a.x.n[ORDER - 1], slices = a.x.n[0];
    // (fp64, rank 32, order 4, slices Zipf 1.1 of 25 leaves, 800 000 of them, weights 32 / 48 / 64, us: 77 / 92 / 108; fp32, rank 8: 61 / 55 / 53)
    constexpr int32_t weight = RP >= 32 && (ORDER == 4 || sizeof(T) == 8) ? 32 : RP >= 16 || sizeof(T) == 8 ? 48 : 64;
    const int32_t least = ORDER == 4 ? 96 : nnz < 200 * slices ? 4 * weight : 5 * S::W;
    const dim3 grid(cut_blocks(a, a.x, cut_leaves(nnz, slices, 4096, S::FIT, weight, least)), (unsigned)tiles);
    return launch_on_cleared("chain3_kernel", mttkrp_kernel<T, ORDER, RP>, a, grid, kWarps * 32, 0, a.out, a.out_bytes, stream);
}

template <typename T, int R2, int R3>
const_status_t launch_ttmc3(Ttmc3Args<T> a, cudaStream_t stream) {
    constexpr int fit = Ttmc3Shape<T, R2, R3>::FIT;
    // Only four warps fit (fp64, 32 x 32): six waves, nine where slices are long.  Chunks that cost 448 throughout / equal leaves in
    // chunks of 256 to 3072 / this, us: slices of equal size, 1.5 M leaves in slices of 5 2147 / 1928 / 1941, 8 M of 100 2265 / 2079 /
    // 2070, 8 M of 1000 1661 / 1510 / 1529; slices Zipf 1.1, 400 000 of 25 196 / 272 / 178, 8 M of 1000 1163 / 1351 / 1166 (in six
    // waves 1232); geometric mean over 258 tensors, this to 448 0.97, to equal leaves 0.84.
    const int even = fit > 4 ? 1 : a.x.n[2] >= 700 * (int64_t)a.x.n[0] ? 9 : 6;
    // The more a leaf costs, the less a slice counts.  Slices Zipf 1.1, fp64, weights 32 / 64 / 96, us: 20 x 27, 400 000 leaves in slices of 100
    // 106 / 118 / 127; 8 x 32, in slices of 25 61 / 76 / 93, but 4 M in slices of 400 and fibres of several leaves 225 / 212 / -; fp32, 16 x 8,
    // 800 000 in slices of 25 73 / 64 / 61.
    constexpr bool wide = R3 >= 32 || R2 * R3 >= 512;
    constexpr int32_t weight = sizeof(T) == 8 && R2 * R3 > 64 ? (wide ? 48 : 80) : wide ? 64 : 96;
    const dim3 grid(cut_blocks(a, a.x, cut_leaves(a.x.n[2], a.x.n[0], 3072, fit, weight, 96, true, even)));
    constexpr size_t dyn = sizeof(typename Ttmc3Shape<T, R2, R3>::Smem) * kWarps;
    static PerDeviceOnce attr_once;                     // per template instance
    CB_CUDA(once_per_device(attr_once, [&] { return cudaFuncSetAttribute(ttmc3_kernel<T, R2, R3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn); }));
    return launch_on_cleared("chain3_kernel", ttmc3_kernel<T, R2, R3>, a, grid, kWarps * 32, dyn, a.out,
                             a.out_bytes, stream);
}

// r2, r3: 8, 16 or 32
template <typename T>
const_status_t dispatch_ttmc3(const Ttmc3Args<T> &a, int r2, int r3, cudaStream_t s) {
    switch (r2 * 100 + r3) {
        case 808: return launch_ttmc3<T, 8, 8>(a, s);
        case 816: return launch_ttmc3<T, 8, 16>(a, s);
        case 832: return launch_ttmc3<T, 8, 32>(a, s);
        case 1608: return launch_ttmc3<T, 16, 8>(a, s);
        case 1616: return launch_ttmc3<T, 16, 16>(a, s);
        case 1632: return launch_ttmc3<T, 16, 32>(a, s);
        case 3208: return launch_ttmc3<T, 32, 8>(a, s);
        case 3216: return launch_ttmc3<T, 32, 16>(a, s);
        case 3232: return launch_ttmc3<T, 32, 32>(a, s);
    }
    return CONST_ERR_UNSUPPORTED;
}

template <typename T, int ORDER>
const_status_t dispatch_mttkrp(const MttkrpArgs<T, ORDER> &a, int rp, int tiles, cudaStream_t s) {
    switch (rp) {
        case 4: return launch_mttkrp<T, ORDER, 4>(a, tiles, s);
        case 8: return launch_mttkrp<T, ORDER, 8>(a, tiles, s);
        case 16: return launch_mttkrp<T, ORDER, 16>(a, tiles, s);
        case 32: return launch_mttkrp<T, ORDER, 32>(a, tiles, s);
    }
    return CONST_ERR_UNSUPPORTED;
}

template <typename T>
const_status_t launch_ttmc4(Ttmc4Args<T> a, cudaStream_t stream) {
    const dim3 grid(cut_blocks(a, a.x, cut_leaves(a.x.n[3], a.x.n[0], 4096, Ttmc4Shape<T>::FIT, 64, 64)));
    constexpr size_t dyn = sizeof(typename Ttmc4Shape<T>::Smem) * kWarps;
    static PerDeviceOnce attr_once;                     // per template instance
    CB_CUDA(once_per_device(attr_once, [&] { return cudaFuncSetAttribute(ttmc4_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn); }));
    return launch_on_cleared("ttmc4_kernel", ttmc4_kernel<T>, a, grid, kWarps * 32, dyn, a.out,
                             a.out_bytes, stream);
}

// The result, set to zero by all blocks of a launch of 256 threads each.
struct Clear {
    uint4 *out;
    int64_t n16;
    uint32_t *tail;
    int32_t tail_words;
    Clear(void *p, size_t bytes)
        : out(static_cast<uint4 *>(p)), n16((int64_t)(bytes / 16)), tail(reinterpret_cast<uint32_t *>(out + n16)), tail_words((int32_t)(bytes % 16 / 4)) {}
    int blocks() const { return (int)std::max<int64_t>(1, std::min<int64_t>((n16 + 1023) / 1024, 148 * 8)); }
    __device__ __forceinline__ void run() const {
        for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n16; i += (int64_t)gridDim.x * 256) out[i] = make_uint4(0, 0, 0, 0);
        if (blockIdx.x == 0 && (int)threadIdx.x < tail_words) tail[threadIdx.x] = 0;
    }
};

__global__ void __launch_bounds__(256) clear_kernel(const __grid_constant__ Clear c) {
    start_next_kernel();
    c.run();
}

// Factors whose rank is not a width of the kernels are copied to rows of that width, zeros behind the rank, by the
// launch that clears the result.
template <typename T>
struct PadArgs {
    const T *src[3];
    T *dst[3];
    int64_t first[4];                                   // elements of the padded factors before factor m
    int32_t rank[3], width[3];
};

template <typename T>
__global__ void __launch_bounds__(256) pad_factors(const __grid_constant__ PadArgs<T> a, const __grid_constant__ Clear result) {
    start_next_kernel();
    result.run();
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < a.first[3]; e += (int64_t)gridDim.x * 256) {
#pragma unroll
        for (int m = 0; m < 3; ++m)
            if (e >= a.first[m] && e < a.first[m + 1]) {
                const int64_t i = e - a.first[m], row = i / a.width[m];
                const int32_t c = (int32_t)(i - row * a.width[m]);
                a.dst[m][i] = c < a.rank[m] ? __ldg(a.src[m] + row * a.rank[m] + c) : T(0);
            }
    }
}

int width_of(int rank) { return rank <= 8 ? 8 : rank <= 16 ? 16 : 32; }

template <typename T>
const_status_t run_any(const const_csf *X, bool mttkrp, const void *const *factors, const int *ranks, T *out, size_t bytes,
                       cudaStream_t stream) {
    const int m = X->order - 1;
    PadArgs<T> pad;
    const T *F[3] = {nullptr, nullptr, nullptr};
    int width[3] = {0, 0, 0};
    int64_t total = 0;
    bool padded = false;
    for (int f = 0; f < 3; ++f) {
        pad.first[f] = total;
        pad.src[f] = nullptr;
        pad.rank[f] = pad.width[f] = 1;
        if (f >= m) continue;
        F[f] = static_cast<const T *>(factors[f]);
        width[f] = mttkrp ? (ranks[f] <= 4 ? 4 : ranks[f] <= 32 ? width_of(ranks[f]) : (ranks[f] + 31) / 32 * 32)
                          : X->order == 4 ? 8 : width_of(ranks[f]);
        if (width[f] == ranks[f]) continue;
        pad.src[f] = F[f];
        pad.rank[f] = ranks[f];
        pad.width[f] = width[f];
        total += X->dims[X->mode_order[f + 1]] * width[f];
        padded = true;
    }
    pad.first[3] = total;
    // A factor is copied whole, whatever the nonzeros read of it.  Where that is more than the contraction is worth, the
    // generic executor does the work: it reads only the rows that occur and needs no scratch.  A padded entry costs 3.9e-6 us,
    // a nonzero of short fibres 1.1e-3 to 2.1e-3 us there (fp32 and fp64; TTMc 10 x 12, extents 1000 x 1e7 x 1e7, 3.2e8
    // padded entries: 1270 us of copying; the generic executor takes 31 us for 1e4 nonzeros, 177 for 1e5, 1470 for 1e6).
    if (total > 256 * X->nnz) return CONST_ERR_UNSUPPORTED;
    T *scratch = nullptr;
    if (padded) {
        if (scratch_alloc((void **)&scratch, sizeof(T) * total, stream) != cudaSuccess) {
            (void)cudaGetLastError();                   // the caller goes on without: the next launch must not find this error
            return CONST_ERR_UNSUPPORTED;
        }
        for (int f = 0; f < 3; ++f) {
            pad.dst[f] = scratch + pad.first[f];
            if (pad.src[f]) F[f] = pad.dst[f];
        }
        const Clear clear(out, bytes);
        const int blocks = std::max(clear.blocks(), (int)std::min<int64_t>((total + 255) / 256, 148 * 8));
        CB_LAUNCH("pad_factors", stream, pad_factors<T><<<blocks, 256, 0, stream>>>(pad, clear));
        bytes = 0;                                      // cleared
        if (cudaGetLastError() != cudaSuccess) {
            cudaFreeAsync(scratch, stream);
            return CONST_ERR_CUDA;
        }
    }
    const_status_t rc;
    const int rp = width[0] > 32 ? 32 : width[0];
    if (mttkrp && X->order == 3)
        rc = dispatch_mttkrp<T, 3>({chain_of<T, 3>(X), {F[0], F[1]}, out, bytes, width[0], ranks[0]}, rp, width[0] / rp, stream);
    else if (mttkrp)
        rc = dispatch_mttkrp<T, 4>({chain_of<T, 4>(X), {F[0], F[1], F[2]}, out, bytes, width[0], ranks[0]}, rp, width[0] / rp, stream);
    else if (X->order == 3)
        rc = dispatch_ttmc3<T>({chain_of<T, 3>(X), F[0], F[1], out, bytes, ranks[0], ranks[1]}, width[0], width[1], stream);
    else
        rc = launch_ttmc4<T>({chain_of<T, 4>(X), F[0], F[1], F[2], out, bytes, ranks[0], ranks[1], ranks[2]}, stream);
    if (scratch) cudaFreeAsync(scratch, stream);
    return rc;
}

}  // namespace

cudaError_t clear_result(void *out, size_t bytes, cudaStream_t stream) {
    const Clear c(out, bytes);
    CB_LAUNCH("clear_result", stream, clear_kernel<<<c.blocks(), 256, 0, stream>>>(c));
    return cudaGetLastError();
}

bool chain_covers(int order, bool mttkrp, const int *ranks) {
    if (mttkrp) return ranks[0] <= 1024;
    for (int f = 0; f + 1 < order; ++f)
        if (ranks[f] > (order == 4 ? 8 : 32)) return false;
    return true;
}

const_status_t run_chain_any(const const_csf *X, bool mttkrp, const void *const *factors, const int *ranks, const_dtype_t dtype,
                             void *out, int64_t out_elems, cudaStream_t stream) {
    const size_t bytes = (dtype == CONST_F32 ? 4 : 8) * (size_t)out_elems;
    if (X->nnz == 0) return clear_result(out, bytes, stream) == cudaSuccess ? CONST_OK : CONST_ERR_CUDA;
    return dtype == CONST_F32 ? run_any<float>(X, mttkrp, factors, ranks, (float *)out, bytes, stream)
                              : run_any<double>(X, mttkrp, factors, ranks, (double *)out, bytes, stream);
}

const_status_t run_ttmc3(const const_csf *X, const float *U, const float *V, int R2, int R3, float *Y,
                         int64_t n_rows, int32_t *, cudaStream_t stream) {
    const size_t bytes = sizeof(float) * R2 * R3 * n_rows;
    if (X->nnz == 0) return clear_result(Y, bytes, stream) == cudaSuccess ? CONST_OK : CONST_ERR_CUDA;
    // Short fibres go to the record walk, whose cost is per leaf; chain3_kernel pays per fibre, but less per leaf of a long
    // one and less to start.  Measured, walk against chain3_kernel (us): 20 M leaves in fibres of one, 16 x 16: 607 / 886;
    // of two: 405 / 470; of four: 362 / 354; 32 x 32 in fibres of two: 939 / 880; 1 M leaves in fibres of one: 68 / 79, of
    // two: 46 / 43.  Below a million leaves only where the slices fill a few windows, with fibres of little more than one and not
    // at R2 = 32: 100 000 leaves in fibres of one, 16 x 16, slices of 1 / 4 / 16 / 64: 106 / 95, 51 / 51, 23 / 27, 17.4 / 18.3;
    // 300 000: 351 / 264, 143 / 128, 47 / 54, 27 / 30; 32 x 32, 300 000: 612 / 407, 238 / 168, 83 / 69, 49 / 42; 493 000 in
    // fibres of 2.3 and slices of 425: 8 x 8 18.6 / 17.3, 8 x 32 29.3 / 25.3, 32 x 16 31.8 / 26.3.
    // With slices counted at their cost on both sides: slices of less than a hundred leaves, 16 x 16, walk / chain3_kernel, slices of 40,
    // 4 M in fibres of 11: 174 / 228 (Zipf 1.1: 171 / 185; but slices of 25, 9 M of 12, 8 x 16, Zipf 1.1: 504 / 479), 1 M of 18, Zipf 1.1: 50 / 52; slices of 85, of 11, 1 M: 37.1 / 35.9 (Zipf 1.1:
    // 34.6 / 41.0), 4 M: 117 / 123; at 32 x 8 slices of 600, 4 M of 1.6: 102 / 101, of 2.2: 97 / 86, 1 M of 1.6: 36 / 33, of 2.2, Zipf
    // 1.1: 33 / 34; long slices, 16 M in fibres of 3.2: 8 x 8 262 / 240, 16 x 16 333 / 354, 8 x 32
    // 418 / 483, 32 x 8 379 / 307; of 4.1: 258 / 205, 313 / 305, 393 / 410, 365 / 265.
    const double per_fibre = (double)X->nnz / (double)X->n[1], per_slice = (double)X->nnz / (double)X->n[0];
    const bool middle = X->nnz >= 100000 && per_slice >= 16 && R2 < 32;
    double line = middle ? 1.5 : 0.0;
    if (X->nnz >= 1000000) {
        line = 2.5;
        if (R2 * R3 >= 1024) line = 1.8;
        else if (R2 == 32 && R3 == 8) line = 1.9;
        else if (R2 < 32 && R3 < 32 && per_slice < 100) line = per_slice < 64 ? 20.0 : 8.0;
        else if (R2 < 32 && X->nnz >= 3000000) line = R3 == 32 || R2 * R3 == 256 ? 3.5 : 2.5;
    }
    if (per_fibre > line) return run_ttmc3_fibres(X, U, V, R2, R3, Y, n_rows, stream);
    return dispatch_ttmc3<float>({chain_of<float, 3>(X), U, V, Y, bytes, R2, R3}, R2, R3, stream);
}

const_status_t run_mttkrp3(const const_csf *X, const float *B, const float *C, int R, float *A, int64_t n_rows,
                           int32_t *, cudaStream_t stream) {
    const size_t bytes = sizeof(float) * R * n_rows;
    if (X->nnz == 0) return clear_result(A, bytes, stream) == cudaSuccess ? CONST_OK : CONST_ERR_CUDA;
    return dispatch_mttkrp<float, 3>({chain_of<float, 3>(X), {B, C}, A, bytes, R, R}, R, 1, stream);
}

const_status_t run_ttmc4(const const_csf *X, const float *U, const float *V, const float *W, int rank, float *Y,
                         int64_t n_rows, int32_t *, cudaStream_t stream) {
    if (rank != 8) return CONST_ERR_UNSUPPORTED;
    const size_t bytes = sizeof(float) * 512 * n_rows;
    if (X->nnz == 0) return clear_result(Y, bytes, stream) == cudaSuccess ? CONST_OK : CONST_ERR_CUDA;
    return launch_ttmc4<float>({chain_of<float, 4>(X), U, V, W, Y, bytes, rank, rank, rank}, stream);
}

}  // namespace cb
