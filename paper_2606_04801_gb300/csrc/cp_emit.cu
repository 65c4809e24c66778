// The start of a call (outside vertices), the essential classes of calls whose
// pairs are not emitted in k_order, and K5: the backward scatter.
#include "cp_common.cuh"
#include "cp_kernels.h"
#include "cp_pairs.cuh"

namespace cp {
namespace {

constexpr int kT = 256;
constexpr int kIT = 256;  // k_init

// The counters and the order's bucket counts (zero_bytes from ctr on, a
// multiple of 16) to zero, by all blocks but the first, which takes the counters
// and then sets what starts elsewhere: one outside vertex per item, the oldest
// dual vertex (Sec. 3.1), never paired (Appendix A.4), with dual root id = item
// index.  (A memset before this kernel took longer than both together.)
__global__ void __launch_bounds__(kIT) k_init(const __grid_constant__ ItemTable tab, Counters* ctr, size_t zero_bytes, uint32_t* uft,
                                              uint64_t* aget, uint64_t* rest, TreeNode* nodet) {
    constexpr size_t kHead = (sizeof(Counters) + 15) / 16;
    uint4* z = reinterpret_cast<uint4*>(ctr);
    const uint4 zero = make_uint4(0, 0, 0, 0);
    if (blockIdx.x > 0) {
        for (size_t i = kHead + size_t(blockIdx.x - 1) * kIT + threadIdx.x; i < zero_bytes / 16; i += size_t(gridDim.x - 1) * kIT)
            z[i] = zero;
        return;
    }
    for (size_t i = threadIdx.x; i < kHead; i += kIT) z[i] = zero;
    __syncthreads();
    for (int i = threadIdx.x; i < tab.n; i += kIT) {
        const Item& it = tab.it[i];
        uft[it.toff + it.T] = kTag | uint32_t(i);
        aget[i] = ~0ull;
        rest[i] = 0;
        if (nodet) nodet[i] = TreeNode{~0ull, uint64_t(i), 0, uint64_t(i)};  // older than every top cell
        ctr->gmin[i] = ~0ull;
    }
    if (threadIdx.x == 0) ctr->n_rt = uint32_t(tab.n);
}

// The essential H0 class of each item.
__global__ void k_essential(const __grid_constant__ ItemTable tab, Counters* ctr, cp_pair* pairs, uint32_t cap) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    cp_pair p;
    if (i >= tab.n || !essential_pair(tab, ctr, i, p)) return;
    const uint32_t pos = atomicAdd(&ctr->n_pairs, 1u);
    if (pos < cap) pairs[pos] = p;
    else set_status(ctr, kStCapacity);
}

__global__ void k_scatter(const cp_pair* __restrict__ pairs, int64_t n, const float* __restrict__ gb,
                          const float* __restrict__ gd, const int64_t* __restrict__ offs, double* acc,
                          int64_t n_pixels) {
    for (int64_t i = int64_t(blockIdx.x) * kT + threadIdx.x; i < n; i += int64_t(gridDim.x) * kT) {
        const cp_pair& p = pairs[i];
        int64_t off = offs ? offs[p.item] : 0;
        if (p.birth_pixel >= 0) {
            int64_t q = off + p.birth_pixel;
            if (q < n_pixels) atomicAdd(acc + q, double(gb[i]));
        }
        if (p.death_pixel >= 0) {
            int64_t q = off + p.death_pixel;
            if (q < n_pixels) atomicAdd(acc + q, double(gd[i]));
        }
    }
}

// Total-persistence loss of the pairs above a persistence threshold and its
// gradient: dL/ddeath = 2 (d - b), dL/dbirth = -2 (d - b).  The loss is summed
// in a fixed order (per-block partials, then one ordered pass), so it is
// identical from run to run.
constexpr int kLossBlocks = 256;

__global__ void __launch_bounds__(kT) k_loss_scatter(const cp_pair* __restrict__ pairs, int64_t n,
                                                     const int64_t* d_n, float tau,
                                                     const int64_t* __restrict__ offs, double* acc, int64_t n_pixels,
                                                     double* partials) {
    __shared__ double red[kT / 32];
    double local = 0.0;
    if (d_n) n = *d_n < n ? *d_n : n;
    for (int64_t i = int64_t(blockIdx.x) * kT + threadIdx.x; i < n; i += int64_t(gridDim.x) * kT) {
        const cp_pair& p = pairs[i];
        if (p.death_pixel < 0) continue;
        double pers = double(p.death) - double(p.birth);
        if (!(pers > double(tau))) continue;
        local += pers * pers;
        int64_t off = offs ? offs[p.item] : 0;
        int64_t qd = off + p.death_pixel, qb = off + p.birth_pixel;
        if (qd < n_pixels) atomicAdd(acc + qd, 2.0 * pers);
        if (qb >= 0 && qb < n_pixels) atomicAdd(acc + qb, -2.0 * pers);
    }
    for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xFFFFFFFFu, local, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = local;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kT / 32; ++w) t += red[w];
        partials[blockIdx.x] = t;
    }
}

// Sparse accumulation: only the birth and death pixels of the pairs carry
// gradient, so the accumulators of those pixels alone are cleared, filled and
// rounded; the output is zeroed as a whole first.  kLoss: only those of the
// pairs in the loss (few of a smooth field's: bound by the scattered sectors,
// the two passes took 13 and 16 us over all pairs of 512^3 and take 5 and 8).
template <bool kLoss>
__device__ __forceinline__ bool in_loss(const cp_pair& p, float tau) {
    return !kLoss || (p.death_pixel >= 0 && double(p.death) - double(p.birth) > double(tau));
}

template <bool kLoss>
__global__ void k_touch_clear(const cp_pair* __restrict__ pairs, int64_t n, const int64_t* d_n, float tau,
                              const int64_t* __restrict__ offs, double* acc, int64_t n_pixels) {
    if (d_n) n = *d_n < n ? *d_n : n;
    for (int64_t i = int64_t(blockIdx.x) * kT + threadIdx.x; i < n; i += int64_t(gridDim.x) * kT) {
        const cp_pair& p = pairs[i];
        if (!in_loss<kLoss>(p, tau)) continue;
        int64_t off = offs ? offs[p.item] : 0;
        int64_t qb = off + p.birth_pixel, qd = off + p.death_pixel;
        if (p.birth_pixel >= 0 && qb < n_pixels) acc[qb] = 0.0;
        if (p.death_pixel >= 0 && qd < n_pixels) acc[qd] = 0.0;
    }
}

// The first block also sums the loss: one warp, in a fixed order and with the
// additions' rounding errors carried along, so that the order costs no accuracy
// (a launch of its own that summed them one after the other took 15 us).
template <bool kLoss>
__global__ void k_touch_round(const cp_pair* __restrict__ pairs, int64_t n, const int64_t* d_n, float tau,
                              const int64_t* __restrict__ offs, const double* __restrict__ acc,
                              float* __restrict__ grad, int64_t n_pixels, const double* __restrict__ partials, double* loss) {
    if (kLoss && blockIdx.x == 0 && threadIdx.x < 32) {
        double hi = 0.0, lo = 0.0;  // the sum and what its additions round off (two-sum)
        auto add = [&](double v, double rest) {
            const double t = hi + v, b = t - hi;
            lo += ((hi - (t - b)) + (v - b)) + rest;
            hi = t;
        };
#pragma unroll
        for (int i = 0; i < kLossBlocks; i += 32) add(partials[i + threadIdx.x], 0.0);
        for (int o = 16; o > 0; o >>= 1) add(__shfl_down_sync(0xFFFFFFFFu, hi, o), __shfl_down_sync(0xFFFFFFFFu, lo, o));
        if (threadIdx.x == 0) *loss = hi + lo;
    }
    if (d_n) n = *d_n < n ? *d_n : n;
    for (int64_t i = int64_t(blockIdx.x) * kT + threadIdx.x; i < n; i += int64_t(gridDim.x) * kT) {
        const cp_pair& p = pairs[i];
        if (!in_loss<kLoss>(p, tau)) continue;
        int64_t off = offs ? offs[p.item] : 0;
        int64_t qb = off + p.birth_pixel, qd = off + p.death_pixel;
        if (p.birth_pixel >= 0 && qb < n_pixels) grad[qb] = float(acc[qb]);
        if (p.death_pixel >= 0 && qd < n_pixels) grad[qd] = float(acc[qd]);
    }
}

int grid_for(int64_t n) {
    int64_t b = (n + kT - 1) / kT;
    int64_t cap = int64_t(device_sm_count()) * 8;
    return int(b < 1 ? 1 : (b > cap ? cap : b));
}

// Test of the bounded-wait path: waits on a word that nothing sets.
__global__ void k_wait_flag(Counters* ctr, const uint32_t* flag, uint64_t limit_ns) {
    if (threadIdx.x == 0) bounded_wait_ne(flag, 0u, ctr, limit_ns);
}

}  // namespace

cudaError_t launch_wait_test(Counters* ctr, const uint32_t* flag, uint64_t limit_ns, cudaStream_t s) {
    k_wait_flag<<<1, 32, 0, s>>>(ctr, flag, limit_ns);
    note_launches(1);
    return cudaGetLastError();
}

int loss_partials() { return kLossBlocks; }

cudaError_t launch_loss_backward(const cp_pair* pairs, int64_t n, const int64_t* d_n, float tau, const int64_t* offs,
                                 double* acc, double* partials, int nparts, double* d_loss, float* grad,
                                 int64_t n_pixels, cudaStream_t s) {
    if (nparts < kLossBlocks) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(grad, 0, sizeof(float) * size_t(n_pixels), s);
    if (e != cudaSuccess) return e;
    k_touch_clear<true><<<grid_for(n), kT, 0, s>>>(pairs, n, d_n, tau, offs, acc, n_pixels);
    k_loss_scatter<<<kLossBlocks, kT, 0, s>>>(pairs, n, d_n, tau, offs, acc, n_pixels, partials);
    k_touch_round<true><<<grid_for(n), kT, 0, s>>>(pairs, n, d_n, tau, offs, acc, grad, n_pixels, partials, d_loss);
    note_launches(3);
    return cudaGetLastError();
}

cudaError_t launch_init(const ItemTable& tab, Counters* ctr, size_t zero_bytes, uint32_t* uft, uint64_t* aget, uint64_t* rest,
                        TreeNode* nodet, cudaStream_t s) {
    const size_t blocks = 2 + zero_bytes / (16 * 2 * kIT);  // two stores per thread
    k_init<<<unsigned(blocks < 512 ? blocks : 512), kIT, 0, s>>>(tab, ctr, zero_bytes, uft, aget, rest, nodet);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_essential(const ItemTable& tab, Counters* ctr, cp_pair* pairs, uint32_t cap, cudaStream_t s) {
    k_essential<<<1, kMaxItems, 0, s>>>(tab, ctr, pairs, cap);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_backward(const cp_pair* pairs, int64_t n, const float* gb, const float* gd, const int64_t* offs,
                            double* acc, float* grad, int64_t n_pixels, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(grad, 0, sizeof(float) * size_t(n_pixels), s);
    if (e != cudaSuccess) return e;
    if (n > 0) {
        k_touch_clear<false><<<grid_for(n), kT, 0, s>>>(pairs, n, nullptr, 0.0f, offs, acc, n_pixels);
        k_scatter<<<grid_for(n), kT, 0, s>>>(pairs, n, gb, gd, offs, acc, n_pixels);
        k_touch_round<false><<<grid_for(n), kT, 0, s>>>(pairs, n, nullptr, 0.0f, offs, acc, grad, n_pixels, nullptr, nullptr);
        note_launches(3);
    }
    return cudaGetLastError();
}

}  // namespace cp
