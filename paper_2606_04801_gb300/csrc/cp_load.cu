// A batch's items copied to their places in one launch.
//
// What bounds it: memory bandwidth; 41.6 M floats in 72 items take 60 us, 5.5
// TB/s of reads and writes.  One copy per item took 351 us on the device
// (4.9 us each) behind 1,240 us of host time for issuing them.  One kernel
// takes all items in chunks of kChunk floats, spread over the chip by chunk
// and not by item, because the sizes are uneven.
// Items start anywhere in the packed destination, so most have source and
// destination on different 16-byte phases: those go as single floats, eight
// loads in flight per thread, the others as float4.
#include "cp_common.cuh"
#include "cp_kernels.h"

namespace cp {
namespace {

constexpr int kLT = 256;
constexpr int kPer = 16;             // floats per thread and chunk
constexpr int kChunk = kLT * kPer;

__global__ void __launch_bounds__(kLT) k_load_items(const __grid_constant__ LoadItems t) {
    for (int c = int(blockIdx.x); c < t.chunks; c += int(gridDim.x)) {
        int lo = 0, hi = t.n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (t.chunk0[mid] <= c) lo = mid;
            else hi = mid - 1;
        }
        const int64_t first = int64_t(c - t.chunk0[lo]) * kChunk;
        const int n = int(t.count[lo] - first < kChunk ? t.count[lo] - first : kChunk);
        const float* __restrict__ src = t.src[lo] + first;
        float* __restrict__ dst = t.dst[lo] + first;
        if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0) {
            float4 v[kPer / 4];
#pragma unroll
            for (int k = 0; k < kPer / 4; ++k) {
                const int i = 4 * (k * kLT + int(threadIdx.x));
                if (i + 3 < n) v[k] = __ldcs(reinterpret_cast<const float4*>(src + i));
            }
#pragma unroll
            for (int k = 0; k < kPer / 4; ++k) {
                const int i = 4 * (k * kLT + int(threadIdx.x));
                if (i + 3 < n) *reinterpret_cast<float4*>(dst + i) = v[k];
            }
            const int tail = (n & ~3) + int(threadIdx.x);
            if (tail < n) dst[tail] = src[tail];
            continue;
        }
#pragma unroll
        for (int h = 0; h < kPer; h += 8) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int i = (h + k) * kLT + int(threadIdx.x);
                if (i < n) v[k] = src[i];
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int i = (h + k) * kLT + int(threadIdx.x);
                if (i < n) dst[i] = v[k];
            }
        }
    }
}

}  // namespace

cudaError_t launch_load_items(LoadItems& t, cudaStream_t s) {
    int64_t chunks = 0;
    for (int i = 0; i < t.n; ++i) {
        t.chunk0[i] = int(chunks);
        chunks += (t.count[i] + kChunk - 1) / kChunk;
    }
    if (chunks == 0) return cudaSuccess;
    if (chunks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    t.chunks = int(chunks);
    const int64_t most = int64_t(device_sm_count()) * 8;
    k_load_items<<<unsigned(chunks < most ? chunks : most), kLT, 0, s>>>(t);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace cp
