// K4: the pairs, in the canonical output order (item, dim, birth cell), in one
// cooperative launch: emission from the merge trees (calls without H1 and
// without sorted union-finds), a bucket sort on the output position, the
// gather.
//
// Every pair has a place of its own among all cells that could be born: the
// item's cells of lower dimension classes first, then its birth cell.  Places
// fall into buckets of 2^shift; a pair counts itself in its bucket, the
// counts' prefix sums place the buckets, and a pair's rank in its bucket is the
// number of members with a smaller place (a bucket holds a few pairs: at most
// one per place, and the birth cells of one class are sparse).
//
// Bound by three grid barriers and a handful of dependent L2 reads.  It
// replaces emission, key building, a histogram, its scan, four to six radix
// passes and a gather, eleven launches: 2048^2 (7,000 pairs) 50 -> 17 us, 128^3
// noise (380,000) 124 -> 36 us, 512^3 (170,000) 91 -> 30 us.
#include "cp_common.cuh"
#include "cp_grid.cuh"
#include "cp_kernels.h"
#include "cp_pairs.cuh"

namespace cp {
namespace {

constexpr int kOT = 1024;        // one CTA per SM: the grid barriers cost least (512 x 2: the same, 256 x 4: slower)
constexpr int kMaxChunks = 128;  // chunks of buckets, each scanned by a CTA (at most kOT)

// The T pair of a V pair of the dual image J (see cp_tfilt.cu): doubled
// coordinate a of J becomes 2n+1-a of the T grid, vertex coordinate c of J
// pixel n-c of I; cells and pixels trade places.
__device__ __forceinline__ int32_t t_cell(const TDims& t, int32_t vc) {
    if (vc < 0) return -1;
    const int64_t GWv = 2 * (t.W + 2) - 1, GHv = 2 * (t.H + 2) - 1;
    const int64_t X = vc % GWv, Y = (vc / GWv) % GHv, Z = vc / (GWv * GHv);
    const int64_t GWt = 2 * t.W + 1, GHt = 2 * t.H + 1, GDt = t.ndim == 3 ? 2 * t.D + 1 : 1;
    const int64_t tx = GWt - X, ty = GHt - Y, tz = t.ndim == 3 ? GDt - Z : 0;
    if (tx < 0 || tx >= GWt || ty < 0 || ty >= GHt || tz < 0 || tz >= GDt) return -1;  // a frame cell
    return int32_t((tz * GHt + ty) * GWt + tx);
}
__device__ __forceinline__ int32_t t_pixel(const TDims& t, int32_t vp) {
    if (vp < 0) return -1;
    const int64_t Wj = t.W + 2, Hj = t.H + 2;
    const int64_t x = vp % Wj, y = (vp / Wj) % Hj, z = vp / (Wj * Hj);
    const int64_t iz = t.ndim == 3 ? t.D - z : 0;
    return int32_t((iz * t.H + (t.H - y)) * t.W + (t.W - x));
}
__device__ __forceinline__ float neg_canon(float v) {
    const float r = -v;
    return r == 0.0f ? 0.0f : r;  // -0.0 reads as +0.0
}
__device__ __forceinline__ cp_pair t_pair(const TDims& t, const cp_pair& p) {
    const int top = t.ndim - 1;
    cp_pair q;
    q.item = p.item;
    q.birth = neg_canon(p.death);
    q.birth_cell = t_cell(t, p.death_cell);
    q.birth_pixel = t_pixel(t, p.death_pixel);
    if (p.dim == top && p.birth == kTFrame) {
        // the last merge into the outside, through a frame facet: the T
        // essential class, born at the T vertex dual to the dying top cell
        q.dim = 0;
        q.death = __int_as_float(0x7F800000);
        q.death_cell = -1;
        q.death_pixel = -1;
    } else {
        q.dim = p.dim == 0 ? top : 0;
        q.death = neg_canon(p.birth);
        q.death_cell = t_cell(t, p.birth_cell);
        q.death_pixel = t_pixel(t, p.birth_pixel);
    }
    return q;
}

__device__ __forceinline__ uint64_t place_of(const OrderArgs& a, const cp_pair& p) {
    const uint32_t c = a.classes == 3 ? uint32_t(p.dim) : (p.dim > 0 ? 1u : 0u);
    return a.base[p.item] + uint64_t(c) * a.cells[p.item] + uint32_t(p.birth_cell);
}

// The number of pairs to the caller (one thread of the grid), or none (any CTA
// that gives up): a CTA that gives up flags the call before it writes 0, and
// the number is taken back if the flag shows after it, so a failed call never
// reports pairs.
__device__ __forceinline__ void put_count(const OrderArgs& a, int64_t n) {
    volatile int64_t* c = &a.ctr->out_count;
    volatile int64_t* d = a.d_out_count;
    *c = n;
    if (d) *d = n;
}

// Grid barrier on the call's own counter (zero at the start of the call).
// False: the wait gave up and the CTA has to leave, since what other CTAs were
// to write may not be there.  It then arrives at no later barrier, so no CTA
// gets past one with another's part missing.
__device__ __forceinline__ bool order_barrier(const OrderArgs& a, uint32_t& epoch) {
    __syncthreads();
    ++epoch;
    bool late = false;
    if (threadIdx.x == 0) {
        const uint32_t target = epoch * gridDim.x + a.absent;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&a.ctr->order_bar) : "memory");
        const uint64_t t0 = global_timer_ns();
        while (!late && ld_acquire_u32(&a.ctr->order_bar) < target) late = global_timer_ns() - t0 > a.limit_ns;
        if (late) {
            set_status(a.ctr, kStTimeout);
            __threadfence();
            put_count(a, 0);
        }
    }
    return !__syncthreads_or(late);
}

// Pair i of the list: mapped (T calls), counted in its bucket.
__device__ __forceinline__ void count_pair(const OrderArgs& a, uint32_t i, const cp_pair& p) {
    const uint64_t b = place_of(a, p) >> a.shift;
    if (!CP_IN(b, a.buckets, a.ctr)) return;
    __stcg(a.slot + i, atomicAdd(a.count + b, 1u));
}

// Exclusive scan over the CTA; sh[kOT / 32] receives the total.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* sh) {
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= unsigned(o)) incl += u;
    }
    if (lane == 31) sh[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < kOT / 32 ? sh[lane] : 0u;
        uint32_t s = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, s, o);
            if (lane >= unsigned(o)) s += u;
        }
        if (lane < kOT / 32) sh[lane] = s - w;
        if (lane == 31) sh[kOT / 32] = s;
    }
    __syncthreads();
    return sh[warp] + incl - v;
}

__global__ void __launch_bounds__(kOT) k_order(const __grid_constant__ OrderArgs a) {
    Counters* ctr = a.ctr;
    __shared__ uint32_t sh_warp[kOT / 32 + 1], sh_n, sh_chunk[kMaxChunks];
    const uint32_t gtid = blockIdx.x * kOT + threadIdx.x, gsize = gridDim.x * kOT;
    uint32_t epoch = 0;
    // a bounded wait that gave up, or non-finite input: the call fails anyway
    // (set by the launches before: every CTA reads the same)
    if (ld_acquire_u32(&ctr->status) & (kStTimeout | kStNonfinite)) {
        if (gtid == 0) put_count(a, 0);
        return;
    }
    // ---- the pairs, each counted in its bucket
    if (a.from_trees) {
        const uint32_t r0 = min(ctr->n_r0, a.n_rids[0]), r1 = min(ctr->n_rt, a.n_rids[1]), n = r0 + r1;
        for (uint32_t g0 = blockIdx.x * kOT; g0 < n + uint32_t(a.tab.n); g0 += gsize) {
            const uint32_t g = g0 + threadIdx.x;
            bool emit = false;
            cp_pair pr;
            if (g < n) {
                const int q = g >= r0 ? 1 : 0;
                emit = tree_pair(a.tab, a.node[q][q ? g - r0 : g], q, nullptr, pr);
            } else if (g < n + uint32_t(a.tab.n) && !a.t_mode) {
                emit = essential_pair(a.tab, ctr, int(g - n), pr);
            }
            if (emit && a.t_mode) pr = t_pair(a.t[pr.item], pr);
            const uint32_t pp = warp_append(&ctr->n_pairs, emit);
            if (emit) {
                if (pp < a.pair_cap) {
                    a.pairs[pp] = pr;
                    count_pair(a, pp, pr);
                } else {
                    set_status(ctr, kStCapacity);
                }
            }
        }
    } else {
        const uint32_t n = min(ctr->n_pairs, a.pair_cap);
        for (uint32_t i = gtid; i < n; i += gsize) {
            cp_pair p = a.pairs[i];
            if (a.t_mode) {
                p = t_pair(a.t[p.item], p);
                a.pairs[i] = p;
            }
            count_pair(a, i, p);
        }
    }
    if (!order_barrier(a, epoch)) return;
    // ---- where each bucket starts within its chunk of 2^chunk_shift buckets
    // (a chunk per CTA at a time), and the chunks' totals
    if (threadIdx.x == 0) sh_n = min(ld_acquire_u32(&ctr->n_pairs), a.pair_cap);
    __syncthreads();
    const uint32_t n = sh_n;
    const uint32_t nchunks = (a.buckets + (1u << a.chunk_shift) - 1u) >> a.chunk_shift;  // <= kMaxChunks
    for (uint32_t k = blockIdx.x; k < nchunks; k += gridDim.x) {
        const uint32_t first = k << a.chunk_shift, last = min(a.buckets, first + (1u << a.chunk_shift));
        uint32_t run = 0;
        // four buckets per thread and turn (the arrays are padded to a multiple of 4)
        for (uint32_t b0 = first; b0 < last; b0 += 4 * kOT) {
            const uint32_t b = b0 + 4 * threadIdx.x;
            uint4 c = make_uint4(0, 0, 0, 0);
            if (b < last) c = __ldcg(reinterpret_cast<const uint4*>(a.count + b));
            const uint32_t at = run + block_scan(c.x + c.y + c.z + c.w, sh_warp);
            if (b < last)
                __stcg(reinterpret_cast<uint4*>(a.start + b), make_uint4(at, at + c.x, at + c.x + c.y, at + c.x + c.y + c.z));
            run += sh_warp[kOT / 32];
            __syncthreads();
        }
        if (threadIdx.x == 0) __stcg(a.chunk + k, run);
    }
    if (!order_barrier(a, epoch)) return;
    {
        const uint32_t c = threadIdx.x < nchunks ? __ldcg(a.chunk + threadIdx.x) : 0u;
        const uint32_t at = block_scan(c, sh_warp);
        if (threadIdx.x < kMaxChunks) sh_chunk[threadIdx.x] = at;
        __syncthreads();
    }
    // ---- the pairs' indices in bucket order
    for (uint32_t i = gtid; i < n; i += gsize) {
        const cp_pair* p = a.pairs + i;
        const int4 w = __ldcg(reinterpret_cast<const int4*>(p) + 1), u = __ldcg(reinterpret_cast<const int4*>(p));
        cp_pair q;
        q.birth_cell = u.z;
        q.dim = w.z;
        q.item = w.w;
        const uint64_t place = place_of(a, q), b = place >> a.shift;
        if (!CP_IN(b, a.buckets, ctr)) continue;
        const uint32_t at = sh_chunk[b >> a.chunk_shift] + __ldcg(a.start + b) + __ldcg(a.slot + i);
        if (CP_IN(at, n, ctr))
            __stcg(a.sorted + at, make_uint2(uint32_t(place & ((uint64_t(1) << a.shift) - 1u)), i));
    }
    if (!order_barrier(a, epoch)) return;
    // the count, by a thread that has a pair to place only if all have
    if (gtid == gsize - 1u) {
        put_count(a, int64_t(n));
        __threadfence();
        if (ld_acquire_u32(&ctr->status) & kStTimeout) put_count(a, 0);
        if (int64_t(n) > a.out_cap) set_status(ctr, kStCapacity);
        if (a.t_bad && *a.t_bad) set_status(ctr, kStNonfinite);
    }
    // ---- each to its place: the bucket's start and its rank among the members
    for (uint32_t d = gtid; d < n; d += gsize) {
        const uint2 e = __ldcg(a.sorted + d);
        const uint32_t i = CP_IN(e.y, n, ctr) ? e.y : 0u;
        const int4 u = __ldcg(reinterpret_cast<const int4*>(a.pairs + i)),
                   w = __ldcg(reinterpret_cast<const int4*>(a.pairs + i) + 1);
        cp_pair q;
        q.birth_cell = u.z;
        q.dim = w.z;
        q.item = w.w;
        const uint64_t b = place_of(a, q) >> a.shift;
        if (!CP_IN(b, a.buckets, ctr)) continue;
        const uint32_t s = sh_chunk[b >> a.chunk_shift] + __ldcg(a.start + b), m = __ldcg(a.count + b);
        uint32_t rank = s;
        for (uint32_t j = s; j < s + m; ++j) rank += __ldcg(a.sorted + j).x < e.x ? 1u : 0u;
        if (int64_t(rank) < a.out_cap) {
            if (a.out16) {
                int4* o = reinterpret_cast<int4*>(a.out + rank);
                o[0] = u;
                o[1] = w;
            } else {
                int32_t* o = reinterpret_cast<int32_t*>(a.out + rank);
                o[0] = u.x, o[1] = u.y, o[2] = u.z, o[3] = u.w;
                o[4] = w.x, o[5] = w.y, o[6] = w.z, o[7] = w.w;
            }
        }
    }
}

}  // namespace

void plan_order(uint64_t places, int* shift, int* chunk_shift, uint32_t* buckets) {
    // buckets of up to 1,024 places, some 65,000 to 131,000 of them while they
    // are smaller
    int s = 0, c = 9;
    while (s < 10 && (places >> s) > 131071u) ++s;
    *buckets = uint32_t(places >> s) + 1u;
    while (((*buckets - 1u) >> c) >= uint32_t(kMaxChunks)) ++c;
    *shift = s;
    *chunk_shift = c;
}

size_t order_chunks() { return kMaxChunks; }

cudaError_t launch_order(const OrderArgs& a, int max_ctas, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    const int blocks = device_cached(kCacheOrder, [] {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_order, kOT, 0);
        return per_sm > 0 ? device_sm_count() : -1;
    });
    if (blocks <= 0) return cudaErrorLaunchOutOfResources;
    cfg.gridDim = dim3(unsigned(max_ctas > 0 && max_ctas < blocks ? max_ctas : blocks));
    cfg.blockDim = dim3(kOT);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    note_launches(1);
    return cudaLaunchKernelEx(&cfg, k_order, a);
}

}  // namespace cp
