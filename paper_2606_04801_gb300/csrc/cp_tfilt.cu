// T-filtration by duality.
//
// Under the T-construction (Sec. 2.2) the pixel values sit on the top cells
// of the lattice complex and every other cell takes the smallest value of the
// top cells that contain it.  The paper leaves this filtration to future work
// (Sec. 6), noting that its duality argument carries over.  This file computes
// it with the V-filtration pipeline, through the duality between the
// T-complex of an image I and the V-complex of
//     J = -I, flipped along every axis, padded with a one-voxel frame whose
//         value lies below every value of -I.
// A T-cell of dimension k is dual to a V-cell of J of dimension d-k (a T top
// cell to a J vertex, a T vertex to a J top cell); f_T(s) = -f_V(s*), and with
// the flip, increasing order in one complex is decreasing order in the other,
// ties included (the top cell a T-cell enters with is the vertex of J that
// its dual cell enters with; the doubled-grid indices reverse).  So:
//   - the T-filtration's H0 union-find (Kruskal over T-edges) is the dual
//     union-find of the V top dimension on J (J top cells = T vertices,
//     J facets = T edges); its last merge, into the outside through a frame
//     facet, is the T essential class;
//   - the T top-dimension dual union-find (T top cells + outside) is the V
//     H0 union-find on J (J vertices = T top cells, the frame = the outside);
//     the frame's own class is the V essential class and is dropped.
// A V pair (b, d) becomes the T pair (-d, -b) with its cells and pixels
// exchanged and mapped back: doubled coordinate a of J becomes 2n+1-a of the
// T grid, vertex coordinate c of J becomes pixel n-c of I.
//
// Kernels: J itself (with a check that every pixel lies below the largest
// finite float, so that the frame comes first), and the frame's links.  The V
// pairs are mapped where they are put in order (cp_order.cu).
#include "cp_common.cuh"
#include "cp_kernels.h"
#include "cp_walk.cuh"

namespace cp {
namespace {

constexpr int kTT = 256;
// The frame value: below every value of -I as long as every pixel is below
// the largest finite float (a pixel at that float, or above it, is flagged).
constexpr float kFrame = kTFrame;

// J four rows at a time, item blockIdx.y (consecutive threads write
// consecutive x and read consecutive, reversed, pixels of the mirrored rows of
// the image; four loads in flight per thread).  Bound by memory: 510^3 moves
// 1,068 MB in 188 us (5.7 TB/s; 227 us with eight rows), 254 x 256 x 250 131 MB
// in 37 us; with 64-bit divisions for each row it was bound by those, 60 us.
constexpr int kTRows = 4;

__global__ void __launch_bounds__(kTT) k_t_build(const __grid_constant__ TItems t, uint32_t* bad) {
    const int item = blockIdx.y;
    const TDims& d = t.d[item];
    const float* __restrict__ img = t.img[item];
    float* __restrict__ J = t.J[item];
    // (J has at most 2^27 vertices, so rows and positions fit 32 bits)
    const uint32_t W = uint32_t(d.W), H = uint32_t(d.H), D = d.ndim == 3 ? uint32_t(d.D) : 0u;
    const uint32_t Dj = d.ndim == 3 ? D + 2u : 1u, Hj = H + 2u, Wj = W + 2u, rows = Dj * Hj;
    bool flag = false;
    for (uint32_t r0 = blockIdx.x * kTRows; r0 < rows; r0 += gridDim.x * kTRows) {
        uint32_t in[kTRows];
        uint32_t live = 0;  // image rows (else a frame row, or past the end)
        uint32_t z = r0 / Hj, y = r0 - z * Hj;
#pragma unroll
        for (int k = 0; k < kTRows; ++k) {
            if (r0 + k < rows && y != 0 && y != Hj - 1u && (d.ndim != 3 || (z != 0 && z != Dj - 1u))) live |= 1u << k;
            in[k] = ((d.ndim == 3 ? D - z : 0u) * H + (H - y)) * W + W;  // read only when live, at - x
            if (++y == Hj) {
                y = 0;
                ++z;
            }
        }
        for (uint32_t x = threadIdx.x; x < Wj; x += kTT) {
            const bool inner = x > 0 && x < Wj - 1u;
            float a[kTRows];
#pragma unroll
            for (int k = 0; k < kTRows; ++k) a[k] = ((live >> k) & 1u) && inner ? __ldg(img + (in[k] - x)) : 0.0f;
#pragma unroll
            for (int k = 0; k < kTRows; ++k) {
                if (r0 + k >= rows) break;
                float v = kFrame;
                if (((live >> k) & 1u) && inner) {
                    flag |= !(a[k] < 3.40282347e38f);  // NaN, +inf, the largest float: the frame would not lie below
                    v = -a[k];
                }
                J[(r0 + k) * Wj + x] = v;
            }
        }
    }
    if (__any_sync(0xFFFFFFFFu, flag) && (threadIdx.x & 31u) == 0) atomicOr(bad, 1u);
}

// After the pruning pass: every frame vertex of J points straight at J's
// vertex 0, the frame's root.  The frame is one tree of equal values in which
// the pruning pass links each vertex to an earlier neighbour; its chains
// along y and x run the whole length of a face, and every walk from a basin
// that drains to the border would otherwise follow them.  Vertex 0 is an
// ancestor of every frame vertex (every frame vertex but 0 has an earlier
// neighbour in the frame, and equal values order by index), so the shortcut
// changes no root.  Item blockIdx.y.
__global__ void __launch_bounds__(kTT) k_t_flatten(uint8_t* __restrict__ code, const __grid_constant__ TItems t) {
    const int item = blockIdx.y;
    const TDims& d = t.d[item];
    uint8_t* __restrict__ cd = code + t.coff[item];
    const int64_t Dj = d.ndim == 3 ? d.D + 2 : 1, Hj = d.H + 2, Wj = d.W + 2;
    Item j;  // the shape that code_at2 and code_at3 want
    j.W = int32_t(Wj);
    j.bands = t.bands[item];
    auto code_at = [&](int64_t z, int64_t y, int64_t x) {
        return d.ndim == 3 ? code_at3(j, int(z), int(y), int(x)) : code_at2(j, int(y), int(x));
    };
    const uint8_t frame = d.ndim == 3 ? 7u : 15u;
    // whole frame rows, a thread per vertex (a long row takes the whole grid: with
    // a block per row the two rows of a 1 x 2^21 image took 3 ms): both y faces of
    // every plane, and the two z faces (3D)
    const uint32_t zf = d.ndim == 3 ? uint32_t(2 * Hj) : 0u;  // rows of the two z faces
    const uint32_t frame_rows = zf + 2u * (d.ndim == 3 ? uint32_t(Dj - 2) : 1u);
    const uint32_t n_frame = frame_rows * uint32_t(Wj);  // (J has at most 2^27 vertices)
    for (uint32_t k = blockIdx.x * kTT + threadIdx.x; k < n_frame; k += gridDim.x * kTT) {
        const uint32_t f = k / uint32_t(Wj);
        const int64_t x = k - f * uint32_t(Wj);
        int64_t z, y;
        if (f < zf) {
            z = f < uint32_t(Hj) ? 0 : Dj - 1;
            y = f % uint32_t(Hj);
        } else {
            const uint32_t g = f - zf;
            z = d.ndim == 3 ? 1 + g / 2 : 0;
            y = (g & 1) ? Hj - 1 : 0;
        }
        if (z != 0 || y != 0 || x != 0) cd[code_at(z, y, x)] |= frame;
    }
    // the two x faces of the other rows
    const int64_t zi = d.ndim == 3 ? Dj - 2 : 1, yi = Hj - 2;
    const int64_t nside = 2 * zi * yi;
    for (int64_t k = int64_t(blockIdx.x) * kTT + threadIdx.x; k < nside; k += int64_t(gridDim.x) * kTT) {
        const int64_t q = k >> 1;
        const int64_t z = d.ndim == 3 ? 1 + q / yi : 0, y = 1 + q % yi;
        const int64_t x = (k & 1) ? Wj - 1 : 0;
        cd[code_at(z, y, x)] |= frame;
    }
}

}  // namespace

cudaError_t launch_t_build(const TItems& t, uint32_t* bad, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    if (t.n < 1 || t.n > kMaxItems) return cudaErrorInvalidValue;
    const int gx = (device_sm_count() * 16 + t.n - 1) / t.n;
    k_t_build<<<dim3(gx, t.n), kTT, 0, s>>>(t, bad);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_t_flatten(uint8_t* code, const TItems& t, cudaStream_t s) {
    if (t.n < 1 || t.n > kMaxItems) return cudaErrorInvalidValue;
    const int gx = (device_sm_count() * 8 + t.n - 1) / t.n;
    k_t_flatten<<<dim3(gx, t.n), kTT, 0, s>>>(code, t);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace cp
