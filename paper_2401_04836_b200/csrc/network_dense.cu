// The two-contraction network  Z[i,m] = sum_{j,k,l} U[i,j,k] V[j,l] W[k,l,m]  (Sec. 1) on the fp64 matrix pipe, for operands
// with locality: every slice i of U touches a short range of j, every slice l of W a short range of m, and the ranges are
// reasonably full (the paper's quantum-chemistry tensors; a band in the benchmark).
//
// Why.  In the gather form (network_kernels.cu) every multiply-add needs a fresh 8-byte operand from shared memory, which
// caps it at a quarter of the fp64 rate, and its bookkeeping costs more than that.  Written out densely over its ranges an
// operand that is a quarter full costs four times the multiply-adds, but in the form of matrix tiles (mma m8n8k4, 256
// multiply-adds per instruction, one operand load each), which run near the fp64 peak.
//
// Two kernels per chunk of slices i, fused over i in chunks: the intermediate T[i,l,k] exists for one chunk at a time.
//   t_kernel   block = one slice s of U (a tile of up to 128 k) x a share of l.  U_s is written out densely in shared memory,
//     [j in range][k]; a warp owns eight l and all k:  T[l, k] = sum_j V[j, l] U_s[j, k].  V comes straight from global
//     memory (each entry is used once per warp, rows of 64 bytes), U_s from shared memory, conflict-free.
//   z_kernel   block = four slices l of W x 64 slices i.  W_l is written out in shared memory, [k][m in range]; a warp owns
//     eight i and the whole range of m and keeps Z in registers over the four l:  Z[i, m] += sum_k T[i, l, k] W_l[k, m];  T
//     comes straight from global memory (L2), each entry used once.  The sums are added to Z atomically.
//
// Whether the operands qualify is found on the device (shape_kernel) and left in a mode word that every later kernel reads:
// nothing waits on the host.  Zeros written out where the tensor has no entry must not meet an infinity or a NaN, which the
// sparse sum would never touch: t_kernel checks that every T it computed is finite and otherwise sets the mode word, too;
// the gather kernel, launched last, then clears Z and does the work.
//
// Measured, 1024 x 1024 x 128, band 32, a quarter full: 4771 us in the gather form; here t_kernel 660 us (dense work at the
// fp64 peak of 37 TFLOP/s: 480) and z_kernel 820 us (540), 1499 us together with clearing and shape.  z_kernel is held by
// writing its slices out between the products: walking the fibres for it 1196 us, from places computed once 979, with the
// next slice's entries on their way meanwhile 889, without a test per product 820.  331 x 331 x 61, band 17: 162 -> 95 us;
// 700, 100, band 21: 1194 -> 471.
//
// The launches are short ones at the small end, so they are few and start early (launch_early): clearing Z and the mode word,
// ranges and places in one kernel, t and z once per chunk, the gather kernel.  Ranges and places in two kernels, the mode word
// cleared apart and ordinary launches: 15 us more at 331 and 1024; and 25 us instead of 8 for operands that do not qualify.
#include <algorithm>

#include "common.cuh"

namespace cb {
namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kRangeJ = 96;           // most j of a slice of U: two blocks of t_kernel share the memory of an SM
constexpr int kRangeM = 80;           // most m of a group of slices of W: so do two blocks of z_kernel with the staged entries
constexpr int kTileK = 128;           // k per tile
constexpr int kNodes = 4;             // slices of W per z_kernel block
constexpr int kRows = 8 * kWarps;     // slices of U per z_kernel block
constexpr int kMaxDilution = 8;       // dense multiply-adds per sparse one up to which the dense form is taken
constexpr int kModeWords = 16;        // words of Net::mode

struct Csf3d {
    const int32_t *crd0, *pos1, *crd1, *pos2, *crd2;
    const double *vals;
    int32_t n0, n1;
};

struct Net {
    Csf3d u, w;                       // levels (i, k, j) and (l, m, k)
    const double *V;
    double *Z, *T;
    int32_t *mode;                    // [0] nonzero: the gather kernel does the work (2: from the start, 1: T was not finite); [2..3] dense multiply-adds (64 bits); [4] blocks done
    int32_t *jmin, *jlen;             // per slice of U: first j, length of the range of j
    int32_t *mmin, *mlen;             // per group of slices of W: the same of m
    uint32_t *u_place, *w_place;      // per entry (shape_kernel)
    int32_t n_k, n_l, n_j, n_m, tk;   // tk: n_k rounded up to 8
    int32_t s0, s1;                   // chunk of slices of U
};

__device__ __forceinline__ void mma884(double &c0, double &c1, double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}

__device__ __forceinline__ int round_up(int x, int to) { return (x + to - 1) / to * to; }

// Z, and the words that steer the kernels behind, set to zero
__global__ void __launch_bounds__(256) clear_kernel(const __grid_constant__ Net a, int64_t n) {
    start_next_kernel();
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) a.Z[i] = 0.0;
    if (blockIdx.x == 0 && threadIdx.x < kModeWords) a.mode[threadIdx.x] = 0;
}

// A block goes through slices of U and groups of slices of W: their ranges, the dense work, whether they fit, and where every
// entry goes when its slice is written out: (place in the range) << 12 | k.  The kernels below write a slice out many times
// (once per share of l, once per 64 slices of U); with the place beside the value they do it from two coalesced streams,
// without walking the fibres.  The first range that does not fit ends the block's work.
__global__ void __launch_bounds__(kThreads) shape_kernel(const __grid_constant__ Net a, int32_t units, unsigned long long sparse) {
    __shared__ int lows[2][kWarps], highs[2][kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long work = 0;
    for (int32_t at = blockIdx.x, turn = 0; at < units; at += gridDim.x, turn ^= 1) {
        const bool of_u = at < a.u.n0;
        const int unit = of_u ? at : at - a.u.n0;
        const Csf3d &x = of_u ? a.u : a.w;
        const int node0 = of_u ? unit : unit * kNodes, node1 = of_u ? unit + 1 : min(node0 + kNodes, x.n0);
        const int32_t f0 = __ldg(x.pos1 + node0), f1 = __ldg(x.pos1 + node1);
        int lo = 0x7fffffff, hi = -1;
        for (int32_t f = f0 + threadIdx.x; f < f1; f += kThreads) {
            if (of_u) {
                lo = min(lo, __ldg(x.crd2 + __ldg(x.pos2 + f)));
                hi = max(hi, __ldg(x.crd2 + __ldg(x.pos2 + f + 1) - 1));
            } else {
                const int m = __ldg(x.crd1 + f);
                lo = min(lo, m);
                hi = max(hi, m);
            }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) {
            lows[turn][warp] = lo;
            highs[turn][warp] = hi;
        }
        __syncthreads();
        if (at == (int32_t)blockIdx.x) after_last_kernel();               // nothing has been written so far
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            lo = min(lo, lows[turn][w]);
            hi = max(hi, highs[turn][w]);
        }
        const int len = hi - lo + 1;
        if (len > (of_u ? kRangeJ : kRangeM)) {
            if (threadIdx.x == 0) a.mode[0] = 2;
            break;
        }
        if (threadIdx.x == 0) {
            (of_u ? a.jmin : a.mmin)[unit] = lo;
            (of_u ? a.jlen : a.mlen)[unit] = len;
        }
        work += of_u ? (unsigned long long)round_up(len, 4) * a.tk * a.n_l : (unsigned long long)round_up(len, 8) * a.tk * kNodes * a.u.n0;
        uint32_t *to = of_u ? a.u_place : a.w_place;
        const int h = threadIdx.x & 7;                                    // eight lanes per fibre
        for (int32_t f = f0 + (threadIdx.x >> 3); f < f1; f += kThreads / 8) {
            const uint32_t y = __ldg(x.crd1 + f);                         // k of a U fibre, m of a W fibre
            const int32_t p1 = __ldg(x.pos2 + f + 1);
            for (int32_t p = __ldg(x.pos2 + f) + h; p < p1; p += 8) {
                const uint32_t z = __ldg(x.crd2 + p);
                to[p] = of_u ? (z - lo) << 12 | y : (y - lo) << 12 | z;
            }
        }
    }
    // the last block compares the dense work with that of the gather form: it has to be worth it
    if (threadIdx.x != 0) return;
    unsigned long long *total = reinterpret_cast<unsigned long long *>(a.mode + 2);
    atomicAdd(total, work);
    __threadfence();
    const bool last = atomicAdd(a.mode + 4, 1) == (int)gridDim.x - 1;
    if (last && atomicAdd(total, 0ull) > kMaxDilution * sparse) a.mode[0] = 2;
}

constexpr int kAhead = 8;             // entries per thread requested ahead of their use

struct Entries {                      // this thread's entries p, p + kThreads, ... below `end` of a slice
    uint32_t place[kAhead];
    double v[kAhead];
    int32_t p, end;
    __device__ __forceinline__ void request(const uint32_t *places, const double *vals, int32_t first, int32_t last) {
        p = first + threadIdx.x;
        end = last;
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            const int32_t at = p + q * kThreads;
            place[q] = at < end ? __ldg(places + at) : 0xffffffffu;
            v[q] = at < end ? __ldg(vals + at) : 0.0;
        }
    }
    // put(place in the range, k - k0, value) for the entries of tile [k0, k0 + kt)
    template <class Put>
    __device__ __forceinline__ void write(const uint32_t *places, const double *vals, int k0, int kt, Put put) const {
        auto one = [&](uint32_t pl, double val) {
            const int k = (int)(pl & 4095u) - k0;
            if ((unsigned)k < (unsigned)kt) put((int)(pl >> 12), k, val);
        };
#pragma unroll
        for (int q = 0; q < kAhead; ++q)
            if (p + q * kThreads < end) one(place[q], v[q]);
        for (int32_t at = p + kAhead * kThreads; at < end; at += kThreads) one(__ldg(places + at), __ldg(vals + at));
    }
};

__device__ __forceinline__ void clear_shared(double *d, int n) {         // n even, d 16-byte aligned
    for (int i = threadIdx.x; i < n / 2; i += kThreads) reinterpret_cast<double2 *>(d)[i] = make_double2(0.0, 0.0);
}

__global__ void __launch_bounds__(kThreads, 2) t_kernel(const __grid_constant__ Net a, int l_tiles_per_block) {
    extern __shared__ __align__(16) double u_dense[];                     // [range of j][tile of k + 4]
    __shared__ int skip;                                                  // one reading for the block: others may set it meanwhile
    after_last_kernel();
    if (threadIdx.x == 0) skip = *a.mode;
    __syncthreads();
    if (skip) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int s = a.s0 + blockIdx.x, k0 = blockIdx.y * kTileK;
    const int kt = min(kTileK, a.tk - k0), ld = kt + 4;                  // ld = 4 or 12 modulo 16: the loads below meet no bank twice
    const int j0 = a.jmin[s], steps = round_up(a.jlen[s], 4) / 4;
    {
        Entries e;
        e.request(a.u_place, a.u.vals, __ldg(a.u.pos2 + __ldg(a.u.pos1 + s)), __ldg(a.u.pos2 + __ldg(a.u.pos1 + s + 1)));
        clear_shared(u_dense, steps * 4 * ld);
        __syncthreads();
        e.write(a.u_place, a.u.vals, k0, kt, [&](int j, int k, double v) { u_dense[j * ld + k] = v; });
        __syncthreads();
    }
    const int r = lane >> 2, c = lane & 3, tiles = kt / 8;
    const int last = min((int)(blockIdx.z + 1) * l_tiles_per_block, (a.n_l + 7) / 8);
    bool finite = true;
    for (int lt = blockIdx.z * l_tiles_per_block + warp; lt < last; lt += kWarps) {
        const int l = lt * 8 + r;
        double acc[kTileK / 8][2];
#pragma unroll
        for (int t = 0; t < kTileK / 8; ++t) acc[t][0] = acc[t][1] = 0.0;
        auto v_at = [&](int st) {
            const int j = j0 + st * 4 + c;
            return l < a.n_l && j < a.n_j && st < steps ? __ldg(a.V + (size_t)j * a.n_l + l) : 0.0;
        };
        double v[4];
#pragma unroll
        for (int z = 0; z < 4; ++z) v[z] = v_at(z);
        for (int st = 0; st < steps; st += 4) {
            double next[4];
#pragma unroll
            for (int z = 0; z < 4; ++z) next[z] = v_at(st + 4 + z);
#pragma unroll
            for (int z = 0; z < 4; ++z) {
                if (st + z >= steps) break;                               // uniform
                const double *row = u_dense + ((st + z) * 4 + c) * ld + r;
#pragma unroll
                for (int t = 0; t < kTileK / 8; ++t)
                    if (t < tiles) mma884(acc[t][0], acc[t][1], v[z], row[t * 8]);
            }
#pragma unroll
            for (int z = 0; z < 4; ++z) v[z] = next[z];
        }
        if (l < a.n_l) {
            double *dst = a.T + ((size_t)(s - a.s0) * a.n_l + l) * a.tk + k0 + 2 * c;
#pragma unroll
            for (int t = 0; t < kTileK / 8; ++t)
                if (t < tiles) {
                    finite = finite && isfinite(acc[t][0]) && isfinite(acc[t][1]);
                    *reinterpret_cast<double2 *>(dst + t * 8) = make_double2(acc[t][0], acc[t][1]);
                }
        }
    }
    if (!finite) atomicExch(a.mode, 1);
}

constexpr int kStaged = 2048;         // entries of a slice of W that wait in shared memory

// Entries of the next slice on their way into shared memory while the matrix tiles of this one run.
struct Staged {
    double v[kStaged];
    uint32_t place[kStaged];
    __device__ __forceinline__ void request(const uint32_t *places, const double *vals, int32_t first, int32_t last) {
        const int n = min(last - first, kStaged);
        for (int i = threadIdx.x; i < n; i += kThreads) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"((uint32_t)__cvta_generic_to_shared(place + i)), "l"(places + first + i) : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" :: "r"((uint32_t)__cvta_generic_to_shared(v + i)), "l"(vals + first + i) : "memory");
        }
    }
    // the caller has waited (own copies) and synchronised (the other threads')
    template <class Put>
    __device__ __forceinline__ void write(const uint32_t *places, const double *vals, int32_t first, int32_t last, int k0, int kt, Put put) const {
        for (int32_t p = first + threadIdx.x; p < last; p += kThreads) {
            const int i = p - first;
            const uint32_t pl = i < kStaged ? place[i] : __ldg(places + p);
            const int k = (int)(pl & 4095u) - k0;
            if ((unsigned)k < (unsigned)kt) put((int)(pl >> 12), k, i < kStaged ? v[i] : __ldg(vals + p));
        }
    }
};

// Products of kRows slices of U with the kNodes slices of W of one group, whose m span N tiles of eight.  Sums run over one
// tile of k at a time and then join those before: in one chain over all four slices the error was a quarter above the gather
// form's (1024: 4.3e-16 against 3.35e-16 relative 2-norm; so 2.9e-16).  N is a constant because asking at each product
// whether its tile is there costs as much as the additions gain: 1583 us an execute at 1024 and 297 a step at 331 with up to
// ten tiles and a test each, 1499 and 279 so.
template <int N>
__device__ __forceinline__ void z_group(const Net &a, int group, Staged &staged, double *w_dense) {
    constexpr int ld = N * 8 + 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = lane >> 2, c = lane & 3;
    const int m0 = a.mmin[group], len = a.mlen[group];
    const int s = a.s0 + blockIdx.y * kRows + warp * 8 + r;              // this lane's slice of U
    const bool have = s < a.s1;
    double acc[N][2];
#pragma unroll
    for (int t = 0; t < N; ++t) acc[t][0] = acc[t][1] = 0.0;
    const int n0 = group * kNodes, n1 = min(n0 + kNodes, a.w.n0);
    int32_t leaf = __ldg(a.w.pos2 + __ldg(a.w.pos1 + n0)), leaf1 = __ldg(a.w.pos2 + __ldg(a.w.pos1 + n0 + 1));
    staged.request(a.w_place, a.w.vals, leaf, leaf1);
    for (int node = n0; node < n1; ++node) {
        const int l = __ldg(a.w.crd0 + node);
        const int32_t leaf2 = node + 1 < n1 ? __ldg(a.w.pos2 + __ldg(a.w.pos1 + node + 2)) : leaf1;
        const double *t_row = a.T + ((size_t)(have ? s - a.s0 : 0) * a.n_l + l) * a.tk + c;
        for (int k0 = 0; k0 < a.tk; k0 += kTileK) {
            const int kt = min(kTileK, a.tk - k0), steps = kt / 4;       // steps is even
            auto t_at = [&](int st) { return have && st < steps ? __ldg(t_row + k0 + st * 4) : 0.0; };
            double x[4], part[N][2];
#pragma unroll
            for (int z = 0; z < 4; ++z) x[z] = t_at(z);
            if (k0 == 0) asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();                                              // the tile before is used up, the entries are here
            clear_shared(w_dense, kt * ld);
            __syncthreads();
            staged.write(a.w_place, a.w.vals, leaf, leaf1, k0, kt, [&](int m, int k, double v) { w_dense[k * ld + m] = v; });
            __syncthreads();
            if (k0 + kTileK >= a.tk && node + 1 < n1) staged.request(a.w_place, a.w.vals, leaf1, leaf2);
#pragma unroll
            for (int t = 0; t < N; ++t) part[t][0] = part[t][1] = 0.0;
            for (int st = 0; st < steps; st += 4) {
                double next[4];
#pragma unroll
                for (int z = 0; z < 4; ++z) next[z] = t_at(st + 4 + z);
#pragma unroll
                for (int z = 0; z < 4; ++z) {
                    if (st + z >= steps) break;                           // uniform
                    const double *row = w_dense + ((st + z) * 4 + c) * ld + r;
#pragma unroll
                    for (int t = 0; t < N; ++t) mma884(part[t][0], part[t][1], x[z], row[t * 8]);
                }
#pragma unroll
                for (int z = 0; z < 4; ++z) x[z] = next[z];
            }
#pragma unroll
            for (int t = 0; t < N; ++t) {
                acc[t][0] += part[t][0];
                acc[t][1] += part[t][1];
            }
        }
        leaf = leaf1;
        leaf1 = leaf2;
    }
    if (!have) return;
    double *z = a.Z + (size_t)__ldg(a.u.crd0 + s) * a.n_m + m0 + 2 * c;
#pragma unroll
    for (int t = 0; t < N; ++t) {
        if (t * 8 + 2 * c < len) atomicAdd(z + t * 8, acc[t][0]);
        if (t * 8 + 2 * c + 1 < len) atomicAdd(z + t * 8 + 1, acc[t][1]);
    }
}

__global__ void __launch_bounds__(kThreads, 2) z_kernel(const __grid_constant__ Net a) {
    extern __shared__ __align__(16) double z_smem[];
    Staged &staged = *reinterpret_cast<Staged *>(z_smem);
    double *w_dense = z_smem + sizeof(Staged) / sizeof(double);           // [tile of k][range of m + 4]
    __shared__ int skip;
    after_last_kernel();
    if (threadIdx.x == 0) skip = *a.mode;
    __syncthreads();
    if (skip) return;
    const int group = blockIdx.x;
    static_assert(kRangeM == 80, "one case per number of tiles");
    switch (round_up(a.mlen[group], 8) / 8) {
        case 1: return z_group<1>(a, group, staged, w_dense);
        case 2: return z_group<2>(a, group, staged, w_dense);
        case 3: return z_group<3>(a, group, staged, w_dense);
        case 4: return z_group<4>(a, group, staged, w_dense);
        case 5: return z_group<5>(a, group, staged, w_dense);
        case 6: return z_group<6>(a, group, staged, w_dense);
        case 7: return z_group<7>(a, group, staged, w_dense);
        case 8: return z_group<8>(a, group, staged, w_dense);
        case 9: return z_group<9>(a, group, staged, w_dense);
        case 10: return z_group<10>(a, group, staged, w_dense);
        default: return;                                                  // no entries
    }
}

// Z back to zero where the gather kernel takes over after products have been added to it
__global__ void __launch_bounds__(256) reclear_kernel(const int32_t *mode, double *Z, int64_t n) {
    after_last_kernel();
    if (*mode != 1) return;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) Z[i] = 0.0;
}

constexpr int64_t kScratchBytes = 256ll << 20;       // T of one chunk

}  // namespace

// On CONST_OK with *mode_out set, the work is queued, behind the clearing of Z, and *mode_out (device) says, once the stream
// gets there, whether the gather kernel still has to do it; *mode_out null: nothing was queued.  cudaFreeAsync(*scratch_out)
// afterwards.
const_status_t run_network_dense(const const_csf *U, const double *V, const const_csf *W, double *Z, int64_t n_i, int64_t n_j,
                                 int64_t n_k, int64_t n_l, int64_t n_m, int32_t **mode_out, void **scratch_out, cudaStream_t stream) {
    *mode_out = nullptr;
    *scratch_out = nullptr;
    const int64_t tk = (n_k + 7) / 8 * 8;
    const double sparse = (double)U->nnz * n_l + (double)W->nnz * U->n[0];
    const int64_t row_bytes = n_l * tk * 8;
    const int64_t n0 = U->n[0], groups = (W->n[0] + kNodes - 1) / kNodes;
    // Small networks stay with the gather kernel; so does one whose T would leave fewer than 64 slices to a chunk.  Where the
    // line lies (multiply-adds of the gather form): at 1.1e8 the band at 331 takes 162 us in the gather form and 95 here,
    // operands that then do not qualify pay about 8 us: 3 % of a call at 1.2e8, 4 % at 7e7.
    if (sparse < 6e7 || n_k > 4096 || kScratchBytes / row_bytes < std::min<int64_t>(n0, 64)) return CONST_OK;
    if (n_l > (1 << 24) || n_m > (1 << 24) || groups > 65535 * 8ll || n0 + W->n[0] > 0x7fffffffll) return CONST_OK;
    int64_t chunk = std::min<int64_t>({n0, kScratchBytes / row_bytes, 65535ll * kRows});       // what T may take, and the rows of a grid
    const int64_t chunks = (n0 + chunk - 1) / chunk;
    chunk = ((n0 + chunks - 1) / chunks + kRows - 1) / kRows * kRows;     // even chunks of whole blocks, never more than fit
    if (chunk * row_bytes > kScratchBytes) chunk = kScratchBytes / row_bytes;
    chunk = std::min<int64_t>(chunk, n0);
    const size_t small = kModeWords * sizeof(int32_t) + sizeof(int32_t) * (2 * (size_t)(n0 + groups) + (size_t)(U->nnz + W->nnz));
    const size_t small_pad = (small + 255) / 256 * 256;
    unsigned char *scratch = nullptr;
    if (scratch_alloc((void **)&scratch, small_pad + (size_t)(chunk * row_bytes), stream) != cudaSuccess) {
        (void)cudaGetLastError();                                         // no room: the gather kernel needs none
        return CONST_OK;
    }
    auto queue = [&]() -> const_status_t {
        Net a;
        auto csf = [](const const_csf *c) {
            return Csf3d{c->crd[0], c->pos[1], c->crd[1], c->pos[2], c->crd[2], static_cast<const double *>(c->vals), (int32_t)c->n[0], (int32_t)c->n[1]};
        };
        a.u = csf(U);
        a.w = csf(W);
        a.V = V;
        a.Z = Z;
        a.mode = reinterpret_cast<int32_t *>(scratch);
        a.jmin = a.mode + kModeWords;
        a.jlen = a.jmin + n0;
        a.mmin = a.jlen + n0;
        a.mlen = a.mmin + groups;
        a.u_place = reinterpret_cast<uint32_t *>(a.mlen + groups);
        a.w_place = a.u_place + U->nnz;
        a.T = reinterpret_cast<double *>(scratch + small_pad);
        a.n_k = (int32_t)n_k;
        a.n_l = (int32_t)n_l;
        a.n_j = (int32_t)n_j;
        a.n_m = (int32_t)n_m;
        a.tk = (int32_t)tk;
        a.s0 = a.s1 = 0;
        const int clear_blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n_i * n_m + 1023) / 1024, 148 * 8));
        CB_LAUNCH("clear_result", stream, clear_kernel<<<clear_blocks, 256, 0, stream>>>(a, n_i * n_m));
        CB_LAUNCH("network_shape", stream, CB_CUDA(launch_early(shape_kernel, dim3((unsigned)std::min<int64_t>(n0 + groups, 148 * 4)), kThreads, 0, stream, a, (int32_t)(n0 + groups), (unsigned long long)sparse)));
        const int kt = (int)std::min<int64_t>(kTileK, tk);
        const size_t t_smem = sizeof(double) * kRangeJ * (kt + 4), z_smem = sizeof(Staged) + sizeof(double) * kt * (kRangeM + 4);
        static PerDeviceOnce once;
        CB_CUDA(once_per_device(once, [] {
            const int most = (int)(sizeof(Staged) + sizeof(double) * std::max(kRangeJ * (kTileK + 4), kTileK * (kRangeM + 4)));
            cudaError_t e = cudaFuncSetAttribute(t_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
            return e == cudaSuccess ? cudaFuncSetAttribute(z_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most) : e;
        }));
        const int l_tiles = (int)((n_l + 7) / 8), k_tiles = (int)((tk + kTileK - 1) / kTileK);
        for (int64_t s0 = 0; s0 < n0; s0 += chunk) {
            a.s0 = (int32_t)s0;
            a.s1 = (int32_t)std::min<int64_t>(n0, s0 + chunk);
            const int rows = a.s1 - a.s0;
            // shares of l: about seven blocks for every SM, a multiple of the warps' tiles each
            const int want = std::max(1, (148 * 7 + rows * k_tiles - 1) / (rows * k_tiles));
            const int per = std::max(kWarps, ((l_tiles + want - 1) / want + kWarps - 1) / kWarps * kWarps);
            const dim3 tg((unsigned)rows, (unsigned)k_tiles, (unsigned)((l_tiles + per - 1) / per));
            CB_LAUNCH("network_t", stream, CB_CUDA(launch_early(t_kernel, tg, kThreads, t_smem, stream, a, per)));
            const dim3 zg((unsigned)groups, (unsigned)((rows + kRows - 1) / kRows));
            CB_LAUNCH("network_z", stream, CB_CUDA(launch_early(z_kernel, zg, kThreads, z_smem, stream, a)));
        }
        if (chunks > 1)          // (with one chunk every T has been looked at before the first product is added)
            CB_LAUNCH("network_shape", stream, CB_CUDA(launch_early(reclear_kernel, dim3(148), 256, 0, stream, a.mode, Z, n_i * n_m)));
        CB_CUDA(cudaGetLastError());
        return CONST_OK;
    };
    const const_status_t rc = queue();
    if (rc != CONST_OK) {
        cudaFreeAsync(scratch, stream);
        return rc;
    }
    *mode_out = reinterpret_cast<int32_t *>(scratch);
    *scratch_out = scratch;
    return CONST_OK;
}

}  // namespace cb
