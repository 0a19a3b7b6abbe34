// What the two sorts of the CSF builder share: the radix sort (csf_build.cu) and the splitter sort (csf_split.cu).
#pragma once
#include "common.cuh"

namespace cb {

struct PackArgs {
    const int32_t *c[kMaxOrder];   // coordinates of the mode stored at level l
    int64_t dim[kMaxOrder];
    int shift[kMaxOrder];
    int order;
};

constexpr int kRsMaxBits = 9;                     // widest digit of a radix pass
constexpr int kRsMaxBins = 1 << kRsMaxBits;
constexpr int kMaxPasses = 8;

// Digits of the radix passes.  A pass sorts on `bits[p]` key bits starting at `shift[p]`; the widths
// are 8 or 9 bits (the width the pass kernel is instantiated for), chosen so that the key is covered
// in as few passes as possible.
struct DigitPlan { int shift[kMaxPasses]; int bits[kMaxPasses]; int passes; };

struct KeyLayout { int bits[kMaxOrder]; int shift[kMaxOrder]; int total_bits; DigitPlan digits; };

struct LevelShifts { int shift[kMaxOrder]; int order; };

struct CsfArrays {
    int32_t *pos[kMaxOrder];
    int32_t *crd[kMaxOrder];
    int bits[kMaxOrder];
};

#ifdef __CUDACC__
__device__ __forceinline__ void report(int32_t *status, int32_t code) { atomicCAS(status, 0, code); }

// True in the block that is the last of its grid to arrive (`arrived` starts at zero); what the other blocks wrote before
// is visible to it.
__device__ __forceinline__ bool last_block(uint32_t *arrived) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(arrived, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Exclusive scan of one number per thread over a block of NT threads; the block's total in `total`.
template <int NT = 256>
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t &total) {
    __shared__ uint32_t sums[NT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += t;
    }
    __syncthreads();                                  // the sums of a scan before are used up
    if (lane == 31) sums[warp] = inc;
    __syncthreads();
    uint32_t before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        if (w < warp) before += sums[w];
        total += sums[w];
    }
    return before + inc - v;
}
#endif

// csf_split.cu
struct SplitSort {                 // what the splitter sort leaves behind for split_scatter
    const uint64_t *list_keys = nullptr;
    const uint32_t *list_pos = nullptr;
    const void *infos = nullptr;
    const uint32_t *part_base = nullptr, *bucket_base = nullptr, *part_owner = nullptr;
    const uint32_t *result = nullptr;        // device: totals at [0..3), parts at [3], status at [16], gave up at [17]
    int order = 0;
    LevelShifts ls;
    int64_t nnz = 0;
};
// Whether the splitter sort is the faster one (and can take the call at all).
bool split_covers(int64_t nnz, const KeyLayout &k);
size_t split_bytes(int64_t nnz, const_dtype_t dtype);
// Queues everything up to the level sizes; `arena` holds split_bytes(...) bytes.
const_status_t split_sort(const PackArgs &pa, const KeyLayout &k, int64_t nnz, const void *vals, const_dtype_t dtype, void *vals_out,
                          int32_t *leaf_crd, unsigned char *arena, cudaStream_t stream, SplitSort *out);
const_status_t split_scatter(const SplitSort &s, const CsfArrays &out, int32_t *slice_ptr, int64_t parts, cudaStream_t stream);

}  // namespace cb
