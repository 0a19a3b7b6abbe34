// Fused order-3 TTMc (Sec. 5.3) for tensors of long fibres:
//   for i, for j (fused):  t[*] = 0;  for k: t[b] += X[i,j,k] * V[k,b];  for a,b: Y[i,a,b] += U[j,a] * t[b]      (Fig. 4(b))
//
// Every warp owns a run of the tensor's leaves, whatever the slices look like (equal runs, or runs of equal cost, see
// run_ttmc3_fibres), and alternates between two phases over windows of a few dozen fibres, on its own:
//   phase 1 (producer)  A factor row of R3 floats is read by R3/4 neighbouring lanes with one 128-bit load each.  The
//     nonzeros of the window are dealt out to the lane groups as equal contiguous runs of 4-aligned blocks, independent
//     of fibre lengths: a block's four coordinates and four values arrive with one 128-bit load each and the four row
//     gathers are issued together, one block ahead of the multiply-adds.  A group stores its partial t when its run
//     leaves a fibre (or hands it over, for a fibre begun by its neighbour).  The finished t of every fibre of the
//     window is thus parked in shared memory (the reduced-order intermediate, one row per fibre), with the fibre's j.
//   phase 2 (consumer)  The R2 x R3 slice result is cut into 8 x 4 register blocks; the lanes that cover one result
//     work on one fibre, so a warp consumes 32 / ((R2/8)(R3/4)) fibres per step: t comes from shared memory, U[j, 8 rows]
//     from global memory with two 128-bit loads, followed by 16 packed multiply-adds per lane.
// Against the record walk of chain_kernels.cu it needs fewer instructions per leaf of a long fibre and more per fibre.
// The slice result lives in registers and leaves the warp once per slice: stored if the warp had all of it, added
// atomically otherwise.
#include "chain_walk.cuh"

namespace cb {
namespace {

using walk::Chain;
using walk::Pair;
using walk::Place;
using walk::Vec;
using walk::axpy;
using walk::load_vec;
using walk::make_pair;
using walk::peek_vec;
using walk::store_vec;
using walk::zero_vec;

constexpr int kWarps = 4;             // warps per block; they meet where a slice covers the block
constexpr int kStreamAhead = 256;   // nonzeros between the L2 prefetch of a line of the leaf arrays and its use

__device__ __forceinline__ void fma4(Vec<float> &t, float x, const Vec<float> &v) { axpy(t, make_pair(x, x), v); }

template <int R2, int R3>
struct Shape {
    // phase 1
    static constexpr int LPR1 = R3 / 4;                 // lanes per factor row
    static constexpr int G1 = 32 / LPR1;                // lane groups per warp
    static constexpr int WINDOW = R3 >= 32 ? 64 : 128;  // fibres parked per warp
    // phase 2: register block of RW rows x 4 columns per lane
    static constexpr int RW = 8;
    static constexpr int LPF = (R2 / 8) * (R3 / 4);     // lanes that cover one fibre
    static constexpr int FPW = 32 / LPF;                // fibres per warp and step
    static constexpr int TILE = R2 * R3;                // floats of one output row (slice)
    static_assert(LPF >= 1 && LPF <= 32 && WINDOW % FPW == 0, "unsupported rank combination");
};

// Producer for a window of cnt fibres; fibre f holds leaves [Ps[f], Ps[f + 1]).  Parks their t in shared memory.
// A fibre that starts inside a group's run gets its row stored by that group; the part of a fibre
// that a group finds already begun (its run starts in the middle of it) goes to a per-group "head"
// slot and is added to the row afterwards, one group after the other, so no atomics and no clearing
// of the rows are needed.
template <int R2, int R3, bool ROUNDS>
__device__ __forceinline__ void phase1(const Chain<float, 3> &x, const float *__restrict__ F2, int cnt,
                                       int lane, float *__restrict__ Ts, const int32_t *__restrict__ Ps, float *__restrict__ Hs, int32_t *__restrict__ Hf) {
    using S = Shape<R2, R3>;
    const int g = lane / S::LPR1, q = lane % S::LPR1;
    const float *F2q = F2 + 4 * q;
    const int32_t P0 = Ps[0], P1 = Ps[cnt];
    const int32_t A0 = P0 & ~3;                                   // 4-aligned blocks of the leaf arrays
    const int32_t blocks = (P1 - A0 + 3) >> 2;
    const int32_t per_group = (blocks + S::G1 - 1) / S::G1;
    const int32_t ba = A0 + g * per_group * 4;
    const int32_t bb = ba + per_group * 4;
    const int32_t pa = ba > P0 ? ba : P0;                         // nonzeros of this group: [pa, pb)
    const int32_t pb = bb < P1 ? bb : P1;
    int32_t head_fibre = -1;
    if (pa < pb) {
        int lo = 0, hi = cnt - 1;                                 // fibre holding nonzero pa
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (Ps[mid] <= pa) lo = mid; else hi = mid - 1;
        }
        int f = lo;
        int32_t fend = Ps[f + 1];
        bool head = Ps[f] < pa;                                   // fibre f was begun by an earlier group
        // ROUNDS: in two levels, sum the rounds of 32 leaves before and t the present one.  Parts of equal cost are long, and the
        // rounding errors of a sum grow with its length (77 M, 16 x 16: relative error 3.8e-7 in one level, 2.6e-7 in two, for
        // 1 % of the time; a test of its own in every block of four, or for sums without a round: 3 to 6 %).
        Vec<float> t = zero_vec<float>(), sum = zero_vec<float>();
        auto round_off = [&]() {
            axpy(sum, make_pair(1.f, 1.f), t);
            t = zero_vec<float>();
        };
        auto park = [&]() {                                       // hand the partial t of fibre f over
            if constexpr (ROUNDS) {
                round_off();
                t = sum;
            }
            if (head) {
                store_vec(Hs + g * R3 + 4 * q, t);
                head_fibre = f;
                head = false;
            } else {
                store_vec(Ts + f * R3 + 4 * q, t);
            }
        };
        auto leave_fibre = [&]() {                                // the run leaves fibre f
            park();
            t = zero_vec<float>();
            if constexpr (ROUNDS) sum = t;
            ++f;
            fend = Ps[f + 1 <= cnt ? f + 1 : cnt];
        };

        auto partial_block = [&](int32_t p) {                     // first or last block of the run
            const int4 kk = __ldg(reinterpret_cast<const int4 *>(x.crd[2] + p));
            const float4 xx = __ldg(reinterpret_cast<const float4 *>(x.vals + p));
            const int32_t k[4] = {kk.x, kk.y, kk.z, kk.w};
            const float xv[4] = {xx.x, xx.y, xx.z, xx.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (p + u >= pa && p + u < pb) {
                    fma4(t, xv[u], load_vec(F2q + (size_t)k[u] * R3));
                    if (p + u + 1 == fend) leave_fibre();
                }
            }
        };

        // whole blocks [m0, m1) run through a software pipeline: coordinates two blocks ahead,
        // row gathers one block ahead of the multiply-adds
        const int32_t m0 = pa > ba ? ba + 4 : ba;
        const int32_t m1 = pb & ~3;
        if (pa > ba) partial_block(ba);
        if (m0 < m1) {
            int4 kn = __ldg(reinterpret_cast<const int4 *>(x.crd[2] + m0));
            float4 xc = __ldg(reinterpret_cast<const float4 *>(x.vals + m0));
            Vec<float> v0 = load_vec(F2q + (size_t)kn.x * R3), v1 = load_vec(F2q + (size_t)kn.y * R3);
            Vec<float> v2 = load_vec(F2q + (size_t)kn.z * R3), v3 = load_vec(F2q + (size_t)kn.w * R3);
            float4 xn = xc;
            if (m0 + 4 < m1) {
                kn = __ldg(reinterpret_cast<const int4 *>(x.crd[2] + m0 + 4));
                xn = __ldg(reinterpret_cast<const float4 *>(x.vals + m0 + 4));
            }
            for (int32_t p = m0; p < m1; p += 4) {
                if (((p >> 2) & 7) == 0) {                        // once per 128-byte line of the leaf arrays
                    if (q == 0 && p + kStreamAhead < m1) {
                        asm volatile("prefetch.global.L2 [%0];" :: "l"(x.crd[2] + p + kStreamAhead));
                        asm volatile("prefetch.global.L2 [%0];" :: "l"(x.vals + p + kStreamAhead));
                    }
                    if constexpr (ROUNDS) round_off();
                }
                Vec<float> w0 = v0, w1 = v1, w2 = v2, w3 = v3;
                float4 xw = xn;
                if (p + 4 < m1) {                                 // gathers of the next block
                    w0 = load_vec(F2q + (size_t)kn.x * R3); w1 = load_vec(F2q + (size_t)kn.y * R3);
                    w2 = load_vec(F2q + (size_t)kn.z * R3); w3 = load_vec(F2q + (size_t)kn.w * R3);
                }
                if (p + 8 < m1) {                                 // coordinates of the block after it
                    kn = __ldg(reinterpret_cast<const int4 *>(x.crd[2] + p + 8));
                    xn = __ldg(reinterpret_cast<const float4 *>(x.vals + p + 8));
                }
                fma4(t, xc.x, v0);
                if (p + 1 == fend) leave_fibre();
                fma4(t, xc.y, v1);
                if (p + 2 == fend) leave_fibre();
                fma4(t, xc.z, v2);
                if (p + 3 == fend) leave_fibre();
                fma4(t, xc.w, v3);
                if (p + 4 == fend) leave_fibre();
                v0 = w0; v1 = w1; v2 = w2; v3 = w3; xc = xw;
            }
        }
        if (m1 >= m0 && m1 < pb) partial_block(m1);
        if (f < cnt && pb > Ps[f]) park();                        // the run ends inside fibre f
    }
    if (q == 0) Hf[g] = head_fibre;
    __syncwarp();
    if (g == 0) {                                                 // add the heads, in group order
        for (int gg = 1; gg < S::G1; ++gg) {
            const int32_t hf = Hf[gg];
            if (hf >= 0) {
                float4 *row = reinterpret_cast<float4 *>(Ts + hf * R3 + 4 * q);
                const float4 h = *reinterpret_cast<const float4 *>(Hs + gg * R3 + 4 * q);
                float4 r = *row;
                r.x += h.x; r.y += h.y; r.z += h.z; r.w += h.w;
                *row = r;
            }
        }
    }
    __syncwarp();
}

// Consumer for the parked window: acc += (factor row of j) (x) t.  acc[r][c]: rows 2 r and 2 r + 1 of column c.
template <int R2, int R3>
__device__ __forceinline__ void phase2(const float *__restrict__ F1, int cnt, int lane, const float *__restrict__ Ts,
                                       const int32_t *__restrict__ Js, Pair<float> (&acc)[4][4]) {
    using S = Shape<R2, R3>;
    const int slot = lane / S::LPF, inner = lane % S::LPF;
    // lane owns rows 8*rg .. 8*rg+7 and columns 4*cg .. 4*cg+3 of the fibre in its slot
    const int rg = inner / (R3 / 4), cg = inner % (R3 / 4);
    const float *F1g = F1 + 8 * rg;
    for (int e = slot; e < cnt; e += S::FPW) {
        const float *up = F1g + (size_t)Js[e] * R2;
        const Vec<float> u0 = load_vec(up), u1 = load_vec(up + 4);
        const Vec<float> tv = peek_vec(Ts + e * R3 + 4 * cg);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const Pair<float> tt = make_pair(tv.at(c), tv.at(c));
            fma2(acc[0][c], u0.p[0], tt);
            fma2(acc[1][c], u0.p[1], tt);
            fma2(acc[2][c], u1.p[0], tt);
            fma2(acc[3][c], u1.p[1], tt);
        }
    }
    __syncwarp();
}

struct Args {
    Chain<float, 3> x;                                               // crd[2] and vals are readable up to the next multiple of 4
    const float *F1, *F2;
    float *out;
    int32_t chunk;                                                   // cost per warp: a leaf costs one,
    int32_t weight, slice_weight;                                    // a fibre so much, a slice so much, beyond what is in it
};

// The part of the tensor between two costs: its leaves [e0, e1), and the place of the first.  Root first, as walk::place_of; both
// ends in one search.
__device__ __forceinline__ void deal_weighted(const Args &a, int64_t cost, int lane, Place<3> &from, int32_t &e0, int32_t &e1) {
    const int64_t w = a.weight, v = a.slice_weight, total = a.x.n[2] + w * a.x.n[1] + v * a.x.n[0];
    int64_t target[2] = {cost < total ? cost : total - 1, cost + a.chunk < total ? cost + a.chunk : total - 1};
    int32_t lo[2] = {0, 0}, hi[2] = {a.x.n[0], a.x.n[0]}, slice_end[2];
    walk::warp_find2([&](int32_t s) { return __ldg(a.x.slice_ptr + s) + w * __ldg(a.x.pos[1] + s) + v * s; }, lo, hi, target, lane);
    from.node[0] = lo[0];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        target[t] -= v * lo[t];
        slice_end[t] = __ldg(a.x.slice_ptr + lo[t] + 1);
        hi[t] = __ldg(a.x.pos[1] + lo[t] + 1);
        lo[t] = __ldg(a.x.pos[1] + lo[t]);
    }
    const int32_t next_fibre = hi[0];
    walk::warp_find2([&](int32_t f) { return __ldg(a.x.pos[2] + f) + w * f; }, lo, hi, target, lane);
    from.node[1] = lo[0];
    int32_t e[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {                                    // the cost of a fibre is paid before its first leaf, of a slice behind its last
        const int32_t p = __ldg(a.x.pos[2] + lo[t]);
        const int64_t behind = target[t] - (p + w * lo[t]) - w;
        e[t] = behind >= slice_end[t] - p ? slice_end[t] : behind > 0 ? max(p, (p + (int32_t)behind) & ~3) : p;   // on a block of four leaves, inside a fibre
    }
    if (e[0] == slice_end[0]) {
        ++from.node[0];
        from.node[1] = next_fibre;
    }
    e0 = cost < total ? e[0] : a.x.n[2];
    e1 = cost + a.chunk < total ? e[1] : a.x.n[2];
}

template <int R2, int R3>
struct __align__(16) Smem {
    using S = Shape<R2, R3>;
    float t[S::WINDOW * R3], heads[S::G1 * R3];
    int32_t j[S::WINDOW], p[S::WINDOW + 1], head_fibre[S::G1];
};

template <int R2, int R3, bool WEIGHED>
__global__ void __launch_bounds__(kWarps * 32, 4) chain3_kernel(const __grid_constant__ Args a) {
    using S = Shape<R2, R3>;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    Smem<R2, R3> &sm = reinterpret_cast<Smem<R2, R3> *>(smem)[threadIdx.x >> 5];
    walk::Share own;
    Place<3> from;
    if constexpr (!WEIGHED) {
        own = walk::Share(a.x, a.chunk, a.slice_weight, kWarps, lane);
    } else {
        __shared__ int32_t block_end;
        deal_weighted(a, ((int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5)) * a.chunk, lane, from, own.e0, own.e1);
        if (threadIdx.x == kWarps * 32 - 1) block_end = own.e1;
        __syncthreads();
        own.block_end = block_end;
    }
    Pair<float> pairs[4][4];
    auto clear = [&]() {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) pairs[r][c] = make_pair(0.f, 0.f);
    };
    clear();
    // adds the slots up and hands row 8 rg + r, columns 4 cg .. 4 cg + 3 of the slice result to put
    const int rg = lane % S::LPF / (R3 / 4), cg = lane % S::LPF % (R3 / 4);
    auto gather = [&](auto put) {
        float acc[S::RW * 4];                                        // row-major 8 x 4 block
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                acc[8 * r + c] = pairs[r][c].lo();
                acc[8 * r + 4 + c] = pairs[r][c].hi();
            }
#pragma unroll
        for (int off = S::LPF; off < 32; off <<= 1)
#pragma unroll
            for (int i = 0; i < S::RW * 4; ++i) acc[i] += __shfl_xor_sync(walk::kAll, acc[i], off);
        if (lane < S::LPF)
#pragma unroll
            for (int r = 0; r < 8; ++r)
                put((8 * rg + r) * R3 + 4 * cg, walk::make_vec(make_float4(acc[4 * r], acc[4 * r + 1], acc[4 * r + 2], acc[4 * r + 3])));
    };
    const int32_t joint = walk::walk_chunk(a.x, own,
        [&](int32_t e) {
            if constexpr (WEIGHED) return from;
            else return walk::place_of(a.x, e, lane, own.slice);
        },
        [](const Place<3> &) {},
        [&](Place<3> &place, int32_t e, int32_t limit) {
            // fibres of the window: those of the next WINDOW that begin before `limit` (all in one slice)
            constexpr int NW = S::WINDOW / 32;
            int32_t p[NW], j[NW], last = 0x7fffffff;
#pragma unroll
            for (int m = 0; m < NW; ++m) {
                const int f = 32 * m + lane;
                const bool known = f < a.x.n[1] - place.node[1];
                p[m] = known ? __ldg(a.x.pos[2] + place.node[1] + f) : 0x7fffffff;
                j[m] = known ? __ldg(a.x.crd[1] + place.node[1] + f) : 0;
            }
            if (S::WINDOW <= a.x.n[1] - place.node[1]) last = __ldg(a.x.pos[2] + place.node[1] + S::WINDOW);
            int cnt = 0;
#pragma unroll
            for (int m = 0; m < NW; ++m) {
                sm.j[32 * m + lane] = j[m];
                sm.p[32 * m + lane] = p[m] < e ? e : p[m] < limit ? p[m] : limit;
                cnt += __popc(__ballot_sync(walk::kAll, p[m] < limit));
            }
            if (lane == 0) sm.p[S::WINDOW] = last < limit ? last : limit;
            __syncwarp();
            const int32_t end = sm.p[cnt];
            phase1<R2, R3, WEIGHED>(a.x, a.F2, cnt, lane, sm.t, sm.p, sm.heads, sm.head_fibre);
            phase2<R2, R3>(a.F1, cnt, lane, sm.t, sm.j, pairs);
            place.node[1] += cnt;
            return end - e;
        },
        [&](int32_t slice, bool whole) {
            float *dst = a.out + (size_t)__ldg(a.x.crd[0] + slice) * S::TILE;
            gather([&](int at, const Vec<float> &v) {
                if (whole) store_vec(dst + at, v);
                else walk::add_vec(dst + at, v);
            });
            clear();
        });
    if (joint >= 0) {                                                // the block's parts of one slice: added up first
        gather([&](int at, const Vec<float> &v) { store_vec(sm.t + at, v); });
        __syncthreads();
        float *dst = a.out + (size_t)__ldg(a.x.crd[0] + joint) * S::TILE;
        for (int i = threadIdx.x * 4; i < S::TILE; i += kWarps * 32 * 4)
            walk::add_vec(dst + i, walk::add_parts<kWarps>(reinterpret_cast<Smem<R2, R3> *>(smem)[0].t + i, (int)(sizeof(sm) / sizeof(float))));
    }
}

template <int R2, int R3, bool WEIGHED>
const_status_t launch_form(const Args &a, int64_t n_rows, cudaStream_t stream) {
    constexpr size_t dyn = sizeof(Smem<R2, R3>) * kWarps;
    static PerDeviceOnce attr_once;                     // per template instance
    CB_CUDA(once_per_device(attr_once, [&] { return cudaFuncSetAttribute(chain3_kernel<R2, R3, WEIGHED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn); }));
    const int64_t cost = (int64_t)a.x.n[2] + (int64_t)a.weight * a.x.n[1] + (int64_t)a.slice_weight * a.x.n[0], warps = (cost + a.chunk - 1) / a.chunk;
    return walk::launch_on_cleared("chain3_kernel", chain3_kernel<R2, R3, WEIGHED>, a, dim3((unsigned)((warps + kWarps - 1) / kWarps)), kWarps * 32, dyn,
                                   a.out, sizeof(float) * R2 * R3 * n_rows, stream);
}

template <int R2, int R3>
const_status_t launch_chain3(const Args &a, int64_t n_rows, cudaStream_t stream) {
    return a.weight ? launch_form<R2, R3, true>(a, n_rows, stream) : launch_form<R2, R3, false>(a, n_rows, stream);
}

}  // namespace

// Same contraction as the leaf-balanced walk of chain_kernels.cu.
const_status_t run_ttmc3_fibres(const const_csf *X, const float *U, const float *V, int R2, int R3, float *Y, int64_t n_rows,
                                cudaStream_t s) {
    // From three million leaves on the warps get equal costs instead of equal leaves: a leaf of a short fibre costs several
    // times one of a long fibre, so that with Zipf-sized slices equal leaves took unequal time, and chunks small enough to
    // even that out paid for their searches.  A fibre counts as six leaves (four and eight are worse by 3 to 10 % on most rank
    // pairs).  Whole waves of parts of at most 8192, 4096 or 2048, as 8, 2 or 1 fibres are consumed side by side: larger ones are
    // up to 5 % faster, but longer sums round more (21 M in fibres of 3.9, 16 x 32, relative error 2.9e-7 at 8192, 2.3e-7 at
    // 4096, 2.8e-7 in leaf chunks).  Leaf chunks of 1536 against this, us (work lists):
    // 10.5 M, slices Zipf 1.1, 8 x 8: 212 / 161 (152), 16 x 16: 324 / 231 (255), 32 x 32: 535 / 406 (453);
    // 77 M, 16 x 16: 1100 / 1041 (1140); uniform, 20 M in fibres of 33, 8 x 8: 161 / 142 (176), 32 x 32: 307 / 311 (324).
    // Equal leaves where they are as good: smaller tensors (2 M in fibres of 25: 24.4 / 25.7, 300 000: 17.8 / 19.5, the longer
    // search), fibres of less than three (6 M in fibres of 2.6, 8 x 16: 110 / 117, 16 x 16: 137 / 144), and slices of more than
    // 1024 fibres, whose sums would get longer (19 M in fibres of 3, 8 x 16, 4260 a slice: 329 / 328 us, error 1.8e-7 / 2.1e-7).
    constexpr int32_t kWeight = 6, kSliceWeight = 64, kResident = 16;
    constexpr int64_t kWave = 148 * kResident;
    // A slice counts as 64 leaves in either form (its result is handed over, its last window is not full): slices Zipf 1.1, 16 x 16, 281 000
    // leaves in slices of 38: 67 / 26, 3 M of 49: 383 / 153, 12 M of 195: 320 / 283; slices of equal size within 1 %.
    const int64_t cost = X->nnz + kWeight * X->n[1] + kSliceWeight * X->n[0], most = R2 * R3 >= 1024 ? 2048 : R2 * R3 >= 512 ? 4096 : 8192;
    const int64_t parts = (cost + kWave * most - 1) / (kWave * most) * kWave;
    Args a{walk::chain_of<float, 3>(X), U, V, Y, (int32_t)((cost + parts - 1) / parts), kWeight, kSliceWeight};
    if (X->nnz < 3000000 || X->nnz < 3 * X->n[1] || X->n[1] > 1024ll * X->n[0]) {
        const walk::Cut cut = walk::cut_leaves(X->nnz, X->n[0], 1536, kResident, kSliceWeight, 96);
        a.chunk = cut.chunk;
        a.weight = 0;
        a.slice_weight = cut.weight;
    }
    switch (R2 * 100 + R3) {
        case 808: return launch_chain3<8, 8>(a, n_rows, s);
        case 816: return launch_chain3<8, 16>(a, n_rows, s);
        case 832: return launch_chain3<8, 32>(a, n_rows, s);
        case 1608: return launch_chain3<16, 8>(a, n_rows, s);
        case 1616: return launch_chain3<16, 16>(a, n_rows, s);
        case 1632: return launch_chain3<16, 32>(a, n_rows, s);
        case 3208: return launch_chain3<32, 8>(a, n_rows, s);
        case 3216: return launch_chain3<32, 16>(a, n_rows, s);
        case 3232: return launch_chain3<32, 32>(a, n_rows, s);
    }
    return CONST_ERR_UNSUPPORTED;
}

}  // namespace cb
