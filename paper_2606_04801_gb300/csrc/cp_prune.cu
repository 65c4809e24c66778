// K1: fused lookup + local pruning (Sec. 3.2, Sec. 3.3, Sec. 4.1 steps 1-2,
// Sec. 4.2 steps 1-3 before the union-finds).
//
// Per vertex v:
//   1. the mask of the neighbours that precede v (value, then index): 8 in 2D,
//      26 in 3D;
//   2. what it says about the lower star of v, by closed forms on words of 32
//      vertices, with a lookup (2D: 256 entries, 3D: a perfect hash) for the
//      vertices that leave survivors or a root;
//   3. the H0 forest link of v (first edge of L(v)), or v as an H0 root (local
//      minimum);
//   4. the dual forest link of each top cell, from its largest corner's lower
//      star: the top cell across the facet where it dies locally, the outside
//      vertex, or itself as a dual root;
//   5. the surviving edges and facets as 64-bit order keys.
// Planes (3D) ahead are brought into shared memory asynchronously; positions
// outside the image hold values that precede nothing.
#include "cp_common.cuh"
#include "cp_kernels.h"
#include "cp_mask3.cuh"
#include "cp_walk.cuh"
#include "cp_words3.cuh"

#include <type_traits>

namespace cp {

// Lookup tables in global memory, read through the read-only cache (lanes of
// a warp look up different entries, which constant memory would serialise).
// 2D: direct (3 bits) | h0_surv << 3 (6) | dual_surv << 9 (12) of each mask.
__device__ uint32_t g_lut2d[256];
// 3D: the perfect hash of the relevant masks (bucket -> displacement -> slot),
// and per slot h0_surv | dual_surv << 6, read for event vertices only (the
// links come from closed forms, cp_words3.cuh).
__device__ uint16_t g_disp3d[1 << 12];
__device__ uint32_t g_surv3d[1 << 14];

namespace {

struct Outs {
    uint32_t* uf0;
    uint32_t* uft;
    uint8_t* code;
    uint64_t n_code;
    uint64_t* s0;
    uint64_t* st;
    uint64_t* age0;
    uint64_t* res0;
    uint64_t* aget;
    uint64_t* rest;
    TreeNode* node0;  // merge-tree nodes, or nullptr (then age / res are written)
    TreeNode* nodet;
    uint32_t cap_s, cap_r0, cap_rt;
    Counters* ctr;
    uint32_t n_uf0, n_uft;  // forest sizes (bounds-checked build)
};

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long t = __shfl_xor_sync(0xFFFFFFFFu, v, o);
        v = t < v ? t : v;
    }
    return v;
}

__device__ __forceinline__ int tile_item(const ItemTable& t, int first, int last, int tile) {
    int lo = first, hi = last;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (t.it[mid].tile0 <= tile) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Root g (of cap) of a forest: its tagged word, and its node or its age and
// reservation words.  Beyond the capacity: a bare tag keeps the forest well
// formed (the call is flagged).
__device__ __forceinline__ void put_root(uint32_t* word, uint32_t g, uint32_t cap, uint64_t age, TreeNode* node,
                                         uint64_t* ages, uint64_t* res, bool dual, int item) {
    if (g >= cap) {
        *word = kTag;
        return;
    }
    if (node) {
        node[g] = TreeNode{~0ull, uint64_t(g), dual ? ~age : age, uint64_t(item)};
    } else {
        ages[g] = age;
        res[g] = 0;
    }
    *word = kTag | g;
}

// Room for a warp's survivors (H0, dual) and roots (the same) in their arrays:
// lanes 0 and 1 add to the two pairs of counters.  (All of a noise volume's
// events come through these: four atomics instead of two held them up.)
__device__ __forceinline__ void reserve(const Outs& o, uint32_t s0, uint32_t st, uint32_t r0, uint32_t rt, uint32_t& b0,
                                        uint32_t& bt, uint32_t& br0, uint32_t& brt) {
    const unsigned lane = lane_id();
    const uint32_t lo = lane == 0 ? s0 : r0, hi = lane == 0 ? st : rt;
    unsigned long long base = 0;
    if (lane < 2 && (lo | hi)) {
        unsigned long long* c = reinterpret_cast<unsigned long long*>(lane == 0 ? &o.ctr->n_s0 : &o.ctr->n_r0);
        base = atomicAdd(c, (unsigned long long)hi << 32 | lo);
        if ((lo && uint32_t(base) + lo > (lane == 0 ? o.cap_s : o.cap_r0)) ||
            (hi && uint32_t(base >> 32) + hi > (lane == 0 ? o.cap_s : o.cap_rt)))
            set_status(o.ctr, kStCapacity);
    }
    const unsigned long long s = __shfl_sync(0xFFFFFFFFu, base, 0), r = __shfl_sync(0xFFFFFFFFu, base, 1);
    b0 = uint32_t(s), bt = uint32_t(s >> 32), br0 = uint32_t(r), brt = uint32_t(r >> 32);
}

// Perfect hash of the 15,935 relevant masks (device layout, cp_mask3.cuh):
// bucket -> displacement -> slot.
__device__ __forceinline__ uint32_t hash_slot3(uint32_t rel, const uint16_t* disp) {
    const uint32_t b = (rel * 0x9E3779B1u) >> (32 - 12);
    const uint32_t d = __ldg(disp + b);
    return ((rel ^ (d * 0x27D4EB2Fu)) * 0x85EBCA77u) >> (32 - 14);
}

}  // namespace

// ---------------------------------------------------------------- 3D
// A CTA of two warps marches along z through a tile of 60 x 29 columns.  A
// warp compares 32 x 32 vertices of a plane, of which it owns 30 x 29, and
// does all of it on words: lane = column, bit = row.
//
//   compare  of every vertex with the 13 neighbours after it in linear order:
//            the sign of a difference (exact: zero only for equal values),
//            shifted into the lane's word.  The neighbours to the left belong
//            to the next lane's vertex, whose value the lane has as well; the
//            other 13 neighbours' bits are the complements of their own.
//   logic    on those words, 32 x 32 vertices per instruction: the relevant
//            mask (the collapse of Sec. 3.3 is one AND per edge and two per
//            corner), the H0 link, the top cells in the lower stars and where
//            each dies, and the vertices that need more than a link (events).
//   output   one code byte per vertex with both links (cp_walk.cuh), a column
//            of a band in one 32-byte sector.
//   events   the vertices whose lower star holds a survivor or a root: each
//            lane takes its relevant masks from the words; 32 at a time, once
//            a warp has as many, the lookup, the keys and roots.
//
// Closed forms used by the logic (compared with the table's entry on all
// 15,935 classes, check_words3):
//   - the H0 link is the first face neighbour in L(v);
//   - a top cell in slot t of L(v) dies across +z for t < 4, +y for t = 4, 5,
//     +x for t = 6; the one in slot 7 dies towards the highest slot that is
//     not in L(v), and is a dual root if all eight are: its facets arrive in
//     descending order, and at each the other side is older or has died;
//   - L(v) has survivors or a root only if the lower link is not a disc: its
//     Euler characteristic is not 1 or it is not connected.
//
// Positions outside the image read NaN, which precedes nothing; the complement
// bits of such neighbours are masked.
//
// Bound by issue (63% of the slots, 12 warps per SM resident on average; a
// fifth of the warps' time is one waiting for the other at a plane): 86 warp
// instructions per 32 vertices at 384^3, 45 of them the differences and
// shifts, which share the FMA and ALU pipes.  Two warps per CTA because they
// wait for one another at every plane (eight: 44% of the time, 736 us at
// 512^3).  Against compares and ballots in four warps that handed words to two
// logic warps through shared memory: 512^3 smooth 673 -> 443 us, 256^3 smooth
// (254 x 256 x 250) 121 -> 91, 128^3 smooth 27.6 -> 23.6, 128^3 noise 202 ->
// 156.  Tried: slots freed by mbarriers instead of a CTA barrier (the same
// waits, 468 us), four or two rows per turn of the compare loop (451, 455).
constexpr int kWX3 = 2, kWY3 = 1;            // warps along x and y
constexpr int kW3 = kWX3 * kWY3, kT3 = kW3 * 32;
constexpr int kOWX = 30;                     // owned columns of a warp (owned rows: kBand3)
constexpr int kOX = kWX3 * kOWX, kOY = kWY3 * kBand3;  // owned by the CTA: 60 x 29
constexpr int kZC = 64;                      // default bound on the owned planes of a task
constexpr int kRS = 68;                      // ring row: columns x0-4 .. x0+63 (16-byte aligned; a TMA box row)
constexpr int kRX = 3;                       // column x0-1 within a ring row
constexpr int kRW = kOX + 3;                 // columns read: x0-1 .. x0+61
constexpr int kRH = kOY + 3;                 // rows y0-1 .. y0+30
constexpr int kSlot = kRH * kRS;             // ring slot in floats
constexpr int kRing = 3;                     // ring slots
constexpr int kQ = 64;                       // events of a warp that wait (fewer than 32, and up to 32 more)
static_assert(kSlot % 32 == 0, "slots start at 128-byte boundaries");

// One task's place and constants (uniform over the CTA).
struct Task3 {
    const float* img;
    int D, H, W, x0, y0, z0, z1, zlast;  // owned planes [z0, z1), zlast = z1 - 1
    uint32_t HW, W1, HW1, voff, toff;
    int item;                // its index in the call's table
    const CUtensorMap* map;  // nullptr: the planes come by cp.async
};

// Ring slot of plane z >= 0.
__device__ __forceinline__ int ring_slot(int z) { return int(unsigned(z) % unsigned(kRing)); }

struct Queue3 {
    uint32_t rel[kQ], at[kQ];  // relevant mask (device layout); plane of the task << 10 | row << 5 | lane
    float val[kQ];
};

struct Smem3 {
    Queue3 queue[kW3];         // (a slot's first row is read one row up, into what lies before, and not used)
    alignas(128) float ring[kRing][kSlot];  // TMA destinations
    uint64_t bar[kRing];       // mbarrier of each slot (TMA completion)
    Task3 t;
};
static_assert(sizeof(Queue3) * kW3 >= sizeof(float) * kRS, "room for a row before the first slot");

// ---- asynchronous copies into shared memory
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
    const uint32_t d = uint32_t(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait for a slot's copy; a copy that never lands flags the call.
__device__ __forceinline__ void mbar_wait(uint64_t* bar, uint32_t parity, Counters* ctr) {
    if (mbar_try_wait(bar, parity)) return;
    const uint64_t t0 = global_timer_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (global_timer_ns() - t0 > kWaitLimitNs) {
            set_status(ctr, kStTimeout);
            return;
        }
    }
}
__device__ __forceinline__ void tma_load_plane(float* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            smem_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// Plane z of the tile.  TMA: one thread's tensor copy, completing on the
// slot's mbarrier; cp.async: a warp per row (positions outside the image hold
// NaN for the whole task).
__device__ __forceinline__ bool plane_read(const Task3& t, int z) { return z <= t.zlast + 1 && z < t.D; }
__device__ __forceinline__ void issue_plane(Smem3& sm, const Task3& t, int z) {
    if (!plane_read(t, z)) return;
    float* plane = sm.ring[ring_slot(z)];
    if (t.map) {
        if (threadIdx.x != 0) return;
        uint64_t* bar = &sm.bar[ring_slot(z)];
        // earlier generic-proxy accesses of the slot come before the copy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar, uint32_t(kRH * kRS * sizeof(float)));
        tma_load_plane(plane, t.map, bar, t.x0 - 1 - kRX, t.y0 - 1, z);
        return;
    }
    const int lane = int(lane_id());
    const float* src = t.img + uint32_t(z) * t.HW;
    for (int r = threadIdx.x >> 5; r < kRH; r += kW3) {
        const int gy = t.y0 - 1 + r;
        if (unsigned(gy) >= unsigned(t.H)) continue;
        const float* row = src + uint32_t(gy) * uint32_t(t.W);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int c = lane + 32 * k, gx = t.x0 - 1 + c;
            if (c < kRW && unsigned(gx) < unsigned(t.W)) cp_async4(plane + r * kRS + kRX + c, row + gx);
        }
    }
    cp_async_commit();
}
// Before reading plane z (every thread).
__device__ __forceinline__ void wait_plane(Smem3& sm, const Task3& t, int z, uint32_t& par, Counters* ctr) {
    if (!plane_read(t, z)) return;
    if (!t.map) {
        cp_async_wait<0>();
        return;
    }
    const int slot = ring_slot(z);
    mbar_wait(&sm.bar[slot], (par >> slot) & 1u, ctr);
    par ^= 1u << slot;
}

// Compare words of a warp's rows in one plane: bit = row, set when the
// neighbour precedes.
struct Words3 {
    uint32_t r, d, dr, a;      // in the plane: right < v, below < v, lower right < v, below < right
    uint32_t c[3], p[3], m[3]; // the plane after, rows -1, 0, +1: same column < v, right < v, same column < right
};

// pl: this lane's column in the warp's first row; up: the same in the plane
// after.  Rows from the last to the first, so that a row's bit is its number.
__device__ __forceinline__ Words3 compare_rows(const float* pl, const float* up, int y_first, int H, float& bad) {
    Words3 w = {};
    // of row i + 1: v and right, up and right; of row i: up and right
    float vna = 0.0f, vnb = 0.0f, una = 0.0f, unb = 0.0f;
    float u0a = __fadd_rn(up[31 * kRS], 0.0f), u0b = __fadd_rn(up[31 * kRS + 1], 0.0f);  // -0 and +0 are equal
#pragma unroll 1
    for (int i0 = 24; i0 >= 0; i0 -= 8) {
#pragma unroll
        for (int k = 7; k >= 0; --k) {
            const int i = i0 + k;
            const float v = pl[i * kRS];
            if (unsigned(y_first + i) < unsigned(H)) bad = fmaf(v, 0.0f, bad);  // NaN from the first NaN or infinity on
            const float va = __fadd_rn(v, 0.0f), vb = __fadd_rn(pl[i * kRS + 1], 0.0f);
            const float ua = __fadd_rn(up[(i - 1) * kRS], 0.0f), ub = __fadd_rn(up[(i - 1) * kRS + 1], 0.0f);
            auto put = [](uint32_t& acc, float q, float c) {
                acc = __funnelshift_l(__float_as_uint(__fsub_rn(q, c)), acc, 1);
            };
            put(w.r, vb, va);
            put(w.d, vna, va);
            put(w.dr, vnb, va);
            put(w.a, vna, vb);
            put(w.c[0], ua, va);
            put(w.c[1], u0a, va);
            put(w.c[2], una, va);
            put(w.p[0], ub, va);
            put(w.p[1], u0b, va);
            put(w.p[2], unb, va);
            put(w.m[0], ua, vb);
            put(w.m[1], u0a, vb);
            put(w.m[2], una, vb);
            vna = va;
            vnb = vb;
            una = u0a;
            unb = u0b;
            u0a = ua;
            u0b = ub;
        }
    }
    return w;
}

// Eight words of 4 code bytes each |= plane b's bits of the word w.
template <int b>
__device__ __forceinline__ void spread(uint32_t (&acc)[8], uint32_t w) {
    const uint32_t nib[2] = {w & 0x0F0F0F0Fu, (w >> 4) & 0x0F0F0F0Fu};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t x = __byte_perm(nib[j & 1], 0, 0x4440u | (j >> 1));
        acc[j] |= (x * (0x00204081u << b)) & (0x01010101u << b);
    }
}

// What a warp keeps from one plane for the next.
struct Carry3 {
    uint32_t c[3], p[3], m[3];         // the compare words towards this plane (p: of the column to the left)
    uint32_t py, px, s0, s1, s2, s3;   // the plane's part for the top cells above it
};

// 32 queued events (n: how many of them there are) from queue position
// `first` of the warp tile at (yw, xw).  Keys, roots and ages go straight to
// the global arrays, with one atomic per array.
__device__ __noinline__ unsigned long long event_batch(Smem3& sm, const Outs& o, const Queue3& queue, uint32_t first, uint32_t n) {
    const Task3& t = sm.t;
    const unsigned lane = lane_id(), lt = (1u << lane) - 1u;
    const int warp = threadIdx.x >> 5;
    const bool live = lane < n;
    const uint32_t qi = (first + lane) & (kQ - 1), e = live ? queue.at[qi] : 0u, rel = live ? queue.rel[qi] : 0u;
    const int x = t.x0 - 1 + (warp % kWX3) * kOWX + int(e & 31u), y = t.y0 - 1 + (warp / kWX3) * kBand3 + int((e >> 5) & 31u),
              z = t.z0 + int(e >> 10);
    const uint32_t sv = live ? __ldg(g_surv3d + hash_slot3(rel, g_disp3d)) : 0u;
    const uint32_t ord = live ? ord_bits(queue.val[qi]) : 0u;
    const uint32_t vl = uint32_t(z) * t.HW + uint32_t(y) * uint32_t(t.W) + uint32_t(x);
    const bool root0 = live && (rel & kM3Faces) == 0u, rootT = rel == kM3All;
    const uint32_t vg = t.voff + vl;
    const uint32_t h0s = sv & 0x3Fu, ds = sv >> 6;
    const unsigned m_r0 = __ballot_sync(0xFFFFFFFFu, root0);
    const unsigned m_rt = __ballot_sync(0xFFFFFFFFu, rootT);
    const uint32_t n0 = __reduce_add_sync(0xFFFFFFFFu, uint32_t(__popc(h0s)));
    const uint32_t nt = __reduce_add_sync(0xFFFFFFFFu, uint32_t(__popc(ds)));
    uint32_t b0, bt, g0, gt;
    reserve(o, n0, nt, __popc(m_r0), __popc(m_rt), b0, bt, g0, gt);
    g0 += __popc(m_r0 & lt);
    gt += __popc(m_rt & lt);
    unsigned long long gmin = ~0ull;
    if (root0 && CP_IN(vg, o.n_uf0, o.ctr)) {
        gmin = (unsigned long long)(uint64_t(ord) << 32 | vl);
        put_root(o.uf0 + vg, g0, o.cap_r0, make_key(ord, vg, 0), o.node0, o.age0, o.res0, false, t.item);
    }
    if (rootT) {  // the top cell whose smallest corner is this vertex, in slot 7 of its lower star
        const uint32_t self = t.toff + uint32_t(z) * t.HW1 + uint32_t(y) * t.W1 + uint32_t(x);
        if (CP_IN(self, o.n_uft, o.ctr))
            put_root(o.uft + self, gt, o.cap_rt, make_key(ord, vg, 26u), o.nodet, o.aget, o.rest, true, t.item);
    }
    uint32_t bits = __reduce_or_sync(0xFFFFFFFFu, h0s);
    while (bits) {
        const int s = __ffs(bits) - 1;
        bits &= bits - 1;
        const bool mine = (h0s >> s) & 1u;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, mine);
        const uint32_t q = b0 + __popc(m & lt);
        const uint32_t c = s == 0 ? 4u : (s == 1 ? 10u : (s == 2 ? 12u : (s == 3 ? 14u : (s == 4 ? 16u : 22u))));
        if (mine && q < o.cap_s) o.s0[q] = make_key(ord, vg, c);
        b0 += __popc(m);
    }
    bits = __reduce_or_sync(0xFFFFFFFFu, ds);
    while (bits) {
        const int f = __ffs(bits) - 1;
        bits &= bits - 1;
        const bool mine = (ds >> f) & 1u;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, mine);
        const uint32_t q = bt + __popc(m & lt);
        // facet slots 0..11 -> stencil bits 1,3,5,7,9,11,15,17,19,21,23,25
        const uint32_t c = f < 6 ? uint32_t(2 * f + 1) : uint32_t(2 * f + 3);
        if (mine && q < o.cap_s) o.st[q] = ~make_key(ord, vg, c);
        bt += __popc(m);
    }
    return gmin;
}

__device__ __forceinline__ void prune_task3d(Smem3& sm, const ItemTable& tab, const Outs& o, int ii, int ltask,
                                             const CUtensorMap* map, uint32_t& par) {
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int warp = threadIdx.x >> 5, lane = int(lane_id());
    const Item& it = tab.it[ii];
    // task order: x segment fastest, then y segment, then z chunk
    const int rest = ltask / it.tx;
    Task3 t;
    t.img = it.img;
    t.D = it.D;
    t.H = it.H;
    t.W = it.W;
    t.x0 = (ltask % it.tx) * kOX;
    t.y0 = (rest % it.ty) * kOY;
    t.z0 = (rest / it.ty) * it.zc;
    t.z1 = min(it.D, t.z0 + it.zc);
    t.zlast = t.z1 - 1;
    t.W1 = uint32_t(it.W) - 1u;
    t.HW = uint32_t(it.H) * uint32_t(it.W);
    t.HW1 = (uint32_t(it.H) - 1u) * t.W1;
    t.voff = uint32_t(it.voff);
    t.toff = uint32_t(it.toff);
    t.item = ii;
    t.map = map;
    __syncthreads();  // everything in shared memory may still be read by the previous task
    if (threadIdx.x == 0) sm.t = t;
    if (!map) {  // positions outside the image stay NaN for the whole task
        for (int i = threadIdx.x; i < kRH * kRW; i += kT3) {
            const int ly = i / kRW, c = i - ly * kRW;
            if (unsigned(t.y0 - 1 + ly) >= unsigned(it.H) || unsigned(t.x0 - 1 + c) >= unsigned(it.W))
                for (int s = 0; s < kRing; ++s) sm.ring[s][ly * kRS + kRX + c] = __int_as_float(0x7FFFFFFF);
        }
    } else if (threadIdx.x == 0) {
        // counted in blocks of 31 x 8 columns by the tuned number of planes, whatever the tile
        auto blocks = [](int lo, int hi, int n) { return uint32_t((hi + n - 1) / n - (lo + n - 1) / n); };
        atomicAdd(&o.ctr->tma_tasks, blocks(t.x0, min(t.x0 + kOX, it.W), 31) * blocks(t.y0, min(t.y0 + kOY, it.H), 8) *
                                         blocks(t.z0, t.z1, tab.zchunk3d));
    }
    // the warp's tile: columns xw .. xw + 31, rows yw .. yw + 31, the inner 30 x 29 owned
    const int wx = warp % kWX3, wy = warp / kWX3;
    const int x = t.x0 - 1 + wx * kOWX + lane, yw = t.y0 - 1 + wy * kBand3;
    const int band = (yw + 1) / kBand3;
    const bool idle = yw + 1 >= t.H || t.x0 + wx * kOWX >= t.W;  // owns nothing
    const bool own_x = lane >= 1 && lane <= kOWX && x < t.W;
    const int rows = t.H - (yw + 1);  // owned, if fewer than kBand3
    const uint32_t own = own_x ? (rows >= kBand3 ? (2u << kBand3) - 2u : (2u << max(rows, 0)) - 2u) : 0u;
    const uint32_t last_row = unsigned(rows) < 32u ? 1u << rows : 0u;  // the bit of row H - 1
    const uint32_t cube_xy = x < t.W - 1 ? own & ~last_row : 0u;
    const uint32_t mxm = x > 0 ? kAll : 0u, mxp = x < t.W - 1 ? kAll : 0u;  // columns with a neighbour on that side
    const uint32_t mym = yw < 0 ? ~2u : kAll, myp = ~last_row;              // rows likewise
    const uint32_t first_x = ~mxm, last_x = x == t.W - 2 ? kAll : 0u;
    const uint32_t last_y = last_row >> 1;  // the bit of row H - 2
    const int col = wy * kBand3 * kRS + kRX + wx * kOWX + lane;
    Carry3 cr = {};
    float bad = 0.0f;
    unsigned long long gmin = ~0ull;
    Queue3& queue = sm.queue[warp];
    uint32_t head = 0, tail = 0;  // events taken from the queue, put into it
    const unsigned lt = (1u << lane) - 1u;
    auto take = [&](uint32_t n) {
        __syncwarp();
        const unsigned long long g = event_batch(sm, o, queue, head, n);
        gmin = g < gmin ? g : gmin;
        head += n;
        __syncwarp();
    };
    // The code of a vertex holds the dual link of the top cell below it, which
    // needs the logic of the plane before, which needs the words of the plane
    // before that: planes first .. zlast + 1 are read.
    const int first = max(t.z0 - 2, 0);
    __syncthreads();
    issue_plane(sm, t, first);
    issue_plane(sm, t, first + 1);
    wait_plane(sm, t, first, par, o.ctr);
#pragma unroll 1
    for (int k = first; k <= t.zlast; ++k) {
        wait_plane(sm, t, k + 1, par, o.ctr);
        __syncthreads();  // plane k + 1 is there, plane k - 1 has been compared
        issue_plane(sm, t, k + 2);
        if (idle) continue;
        Words3 w = compare_rows(sm.ring[ring_slot(k)] + col, sm.ring[ring_slot(k + 1)] + col, yw, t.H, bad);
        if (k == t.D - 1) {  // no plane after
#pragma unroll
            for (int j = 0; j < 3; ++j) w.c[j] = w.p[j] = w.m[j] = 0u;
        }
        if (k >= t.z0 - 1) {
            Star3 st;
            {
                uint32_t n[27];
                n[13] = 0;
                const uint32_t mz = k > 0 ? kAll : 0u;
                const uint32_t yz[3] = {mym & mz, mz, myp & mz};
                n[14] = w.r;
                n[12] = ~__shfl_up_sync(kAll, w.r, 1) & mxm;
                n[16] = w.d;
                n[10] = ~(w.d << 1) & mym;
                n[17] = w.dr;
                n[9] = ~(__shfl_up_sync(kAll, w.dr, 1) << 1) & mxm & mym;
                n[15] = __shfl_up_sync(kAll, w.a, 1);
                n[11] = ~(w.a << 1) & mxp & mym;
#pragma unroll
                for (int dy = -1; dy <= 1; ++dy) {
                    n[22 + 3 * dy] = w.c[dy + 1];
                    n[23 + 3 * dy] = w.p[dy + 1];
                    n[21 + 3 * dy] = __shfl_up_sync(kAll, w.m[dy + 1], 1);
                    // the words of the row one up or down, towards this row
                    auto row = [&](uint32_t q) { return dy < 0 ? q << 1 : (dy > 0 ? q >> 1 : q); };
                    n[4 + 3 * dy] = ~row(cr.c[1 - dy]) & yz[dy + 1];
                    n[3 + 3 * dy] = ~row(cr.p[1 - dy]) & yz[dy + 1] & mxm;
                    n[5 + 3 * dy] = ~row(cr.m[1 - dy]) & yz[dy + 1] & mxp;
                }
                star_words3(n, st);
            }
            // the column to the right's slots 0, 2, 4, 6
            uint32_t xo[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) xo[j] = __shfl_down_sync(kAll, st.co[2 * j], 1);
            if (k >= t.z0) {
                // the top cells between planes k - 1 and k: the slot that its
                // largest corner sees it in.  Upper corners (slots 0..3 of plane
                // k's vertices) send it to +z; plane k - 1's part comes from its
                // own logic.
                const uint32_t cube = k > 0 ? cube_xy : 0u;
                const uint32_t up = st.co[3] | xo[1] | ((st.co[1] | xo[0]) >> 1);
                const uint32_t upi = k == t.D - 1 ? 0u : up, pyi = cr.py & ~last_y, pxi = cr.px & ~last_x;
                uint32_t acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                spread<0>(acc, st.h[0] >> 1);
                spread<1>(acc, st.h[1] >> 1);
                spread<2>(acc, st.h[2] >> 1);
                spread<3>(acc, (upi | pxi | cr.s0 | ~cube) >> 1);
                spread<4>(acc, (pyi | pxi | cr.s1 | ~cube) >> 1);
                spread<5>(acc, (cr.s2 | ~cube) >> 1);
                spread<6>(acc, (up | cr.py | cr.px | cr.s3 | ~cube) >> 1);
                const uint64_t at = uint64_t(it.coff) + ((uint64_t(k) * uint32_t(it.bands) + uint32_t(band)) * uint32_t(t.W) + uint32_t(x)) * 32u;
                if (own_x && CP_IN(at + 31u, o.n_code, o.ctr)) {
                    uint4* dst = reinterpret_cast<uint4*>(o.code + at);
                    dst[0] = make_uint4(acc[0], acc[1], acc[2], acc[3]);
                    dst[1] = make_uint4(acc[4], acc[5], acc[6], acc[7]);
                }
                // events: each lane's next one, to the queue
                uint32_t ev = st.event & own;
                for (;;) {
                    const unsigned have = __ballot_sync(kAll, ev != 0u);
                    if (!have) break;
                    const int row = ev ? __ffs(ev) - 1 : 0;
                    uint32_t rel = 0;
#pragma unroll
                    for (int n = 0; n < 27; ++n)
                        if (n != 13) rel |= ((relevant_plane(st, n) >> row) & 1u) << mask3_pos(n);
                    if (ev) {
                        const uint32_t q = (tail + __popc(have & lt)) & (kQ - 1);
                        queue.rel[q] = rel;
                        queue.at[q] = uint32_t(k - t.z0) << 10 | uint32_t(row) << 5 | uint32_t(lane);
                        queue.val[q] = sm.ring[ring_slot(k)][col + row * kRS];
                        ev &= ev - 1u;
                    }
                    tail += __popc(have);
                    if (tail - head >= 32u) take(32u);
                }
            }
            // plane k's part for the top cells above it
            uint32_t b0, b1, b2;
            slot7_target(st.co, b0, b1, b2);
            const uint32_t out = (~b0 & first_x) | (~b1 & ~mym) | (k == 0 ? ~b2 : 0u);
            const uint32_t self = st.co[7] & ~out;
            cr.py = (st.co[5] | xo[2]) >> 1;
            cr.px = xo[3];
            cr.s0 = self & b0;
            cr.s1 = self & b1;
            cr.s2 = self & b2;
            cr.s3 = st.co[7] & out;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            cr.c[j] = w.c[j];
            cr.p[j] = __shfl_up_sync(kAll, w.p[j], 1);
            cr.m[j] = w.m[j];
        }
    }
    if (tail != head) take(tail - head);
    if (!map) cp_async_wait<0>();
    if (!idle) {
        const bool in = unsigned(x) < unsigned(t.W);
        if (__any_sync(kAll, in && bad != bad) && lane == 0) set_status(o.ctr, kStNonfinite);
        gmin = warp_min_u64(gmin);
        if (lane == 0 && gmin != ~0ull) atomicMin(&o.ctr->gmin[ii], gmin);
    }
}

__global__ void __launch_bounds__(kT3, 8) k_prune3d(const __grid_constant__ ItemTable tab, const __grid_constant__ Outs o,
                                                    const __grid_constant__ TmaMaps maps) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem3& sm = *reinterpret_cast<Smem3*>(smem_raw);
    if (threadIdx.x == 0) {
        for (int s = 0; s < kRing; ++s) mbar_init(&sm.bar[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // TMA destinations must be 128-byte aligned; otherwise every item takes the cp.async path
    const bool tma_ok = (smem_u32(sm.ring) & 127u) == 0;
    uint32_t par = 0;  // phase parity of each slot's mbarrier (every thread waits on every TMA plane)
    for (int task = blockIdx.x; task < tab.tiles3d; task += gridDim.x) {
        const int ii = tile_item(tab, tab.n2d, tab.n - 1, task);
        const Item& it = tab.it[ii];
        prune_task3d(sm, tab, o, ii, task - it.tile0, tma_ok && it.tma >= 0 ? &maps.m[it.tma] : nullptr, par);
    }
}

// The words of every item's forests from its codes, links as ids (roots have
// theirs already).
__global__ void __launch_bounds__(256) k_expand(const __grid_constant__ ItemTable tab, const __grid_constant__ Outs o) {
    for (int j = 0; j < tab.n2d; ++j) {
        const Item& it = tab.it[j];
        const int64_t n = int64_t(it.H) * it.W;
        for (int64_t v = int64_t(blockIdx.x) * 256 + threadIdx.x; v < n; v += int64_t(gridDim.x) * 256) {
            const int y = int(v / it.W), x = int(v - int64_t(y) * it.W);
            const uint32_t c = o.code[it.coff + code_at2(it, y, x)];
            int dy, dx;
            if ((c & 15u) < 14u) {
                link_offset2(0, c & 15u, dy, dx);
                o.uf0[it.voff + v] = uint32_t(it.voff + v + int64_t(dy) * it.W + dx);
            }
            if (y >= it.H - 1 || x >= it.W - 1 || c >> 4 == 15u) continue;
            const int64_t self = it.toff + int64_t(y) * (it.W - 1) + x;
            link_offset2(1, c >> 4, dy, dx);
            o.uft[self] = c >> 4 == 9u ? uint32_t(it.toff + it.T) : uint32_t(self + int64_t(dy) * (it.W - 1) + dx);
        }
    }
    for (int j = tab.n2d; j < tab.n; ++j) {
        const Item& it = tab.it[j];
        const int64_t n = int64_t(it.D) * it.H * it.W;
        for (int64_t v = int64_t(blockIdx.x) * 256 + threadIdx.x; v < n; v += int64_t(gridDim.x) * 256) {
            const int x = int(v % it.W), y = int((v / it.W) % it.H), z = int(v / (int64_t(it.W) * it.H));
            const uint32_t c = o.code[it.coff + code_at3(it, z, y, x)];
            const uint32_t h = c & 7u, d = c >> 3;
            if (h < 6u) o.uf0[it.voff + v] = uint32_t(it.voff + v + link_offset3(0, h, it.H * it.W, it.W));
            if (z == 0 || y >= it.H - 1 || x >= it.W - 1 || d == 7u) continue;
            const int64_t self = it.toff + (int64_t(z - 1) * (it.H - 1) + y) * (it.W - 1) + x;
            o.uft[self] = d == 8u ? uint32_t(it.toff + it.T)
                                  : uint32_t(self + link_offset3(1, d, (it.H - 1) * (it.W - 1), it.W - 1));
        }
    }
}

// ---------------------------------------------------------------- 2D
// A warp takes a tile of 32 x 32 vertices, of which it owns the inner 30 x
// 30, and does all of it on words: lane = column, bit = row.
//
//   compare  of every vertex with its right, lower left, lower and lower
//            right neighbour: the sign of a difference (exact: zero only for
//            equal values), shifted into the lane's word.  The other four
//            neighbours' bits are the complements of their own.
//   logic    on those words, 32 x 32 vertices per instruction: the H0 link,
//            the top cells in the lower stars and where each dies, the events
//            (vertices whose lower star holds a survivor or a root: the lower
//            link is not one arc).
//   output   one code byte per vertex with both links (cp_walk.cuh), a
//            column of a tile in one 32-byte sector.
//   events   32 at a time: mask, table, and after one atomic per tile and
//            array the keys, roots and ages.
//
// Closed forms used by the logic (equal to the table's entries on all 256
// masks): the H0 link is the first of up, left, right, down in L(v); a top
// cell in quadrant 0 or 1 of L(v) dies across +y, in 2 across +x, in 3 towards
// the highest quadrant not in L(v), and is a dual root if all four are; there
// is an event unless exactly one face of L(v) is not followed, around v, by a
// quadrant of L(v).
//
// Small images are bound by a tile's events, which one warp takes 32 at a time:
// up to eight warps then take a tile together, each with all of its words but
// the events of its own rows.  Large ones are bound by issue.  Marching down a
// strip with a mask, a table read and two 32-bit links per vertex took 273 warp
// instructions per 32 vertices and wrote eight bytes per vertex instead of
// one: 4096^2 smooth 188 -> 40 us, 2048^2 49 -> 12, 2048^2 noise 113 -> 60,
// 769 x 1021 18 -> 7, 64^2 noise 10 -> 8.
constexpr int kW2 = 4;                   // warps per CTA (independent tiles)

struct Smem2 {
    uint32_t n[kW2][8][32];              // neighbour words: bit set = the neighbour precedes
    uint32_t queue[kW2][kTile2 * kTile2];  // events: row << 5 | lane; then | h0 << 10 | dual << 14 | roots << 18
};

struct Words2 {
    uint32_t r, d, dr, a;  // right < v, below < v, lower right < v, below < right
};

// The words of 32 rows from row y (the tile's first, y0 - 1) on; kIn: every
// position read lies inside the image.  Outside it, values are +inf.
template <bool kIn>
__device__ __forceinline__ Words2 words2(const float* __restrict__ img, int W, int H, int x, int y, float& bad) {
    constexpr int kB = 8;  // rows loaded at a time
    const float inf = __int_as_float(0x7F800000);
    const bool in0 = kIn || unsigned(x) < unsigned(W), in1 = kIn || unsigned(x + 1) < unsigned(W);
    const float* p = img + (int64_t(y) * W + x);
    auto get = [&](int i, float& a, float& b) {
        const bool row = kIn || unsigned(y + i) < unsigned(H);
        a = b = inf;
        if (row && in0) a = __ldg(p + int64_t(i) * W);
        if (row && in1) b = __ldg(p + int64_t(i) * W + 1);
    };
    auto check = [&](int i, float a) {  // NaN from the first NaN or infinity on
        if (kIn || (in0 && unsigned(y + i) < unsigned(H))) bad = fmaf(a, 0.0f, bad);
    };
    Words2 w = {0, 0, 0, 0};
    float a, b;
    get(0, a, b);
    check(0, a);
    a = __fadd_rn(a, 0.0f);  // -0 and +0 are equal: +0, so that their difference is +0
    b = __fadd_rn(b, 0.0f);
#pragma unroll 1
    for (int i0 = 1; i0 < 33; i0 += kB) {
        float c[kB], d[kB];
#pragma unroll
        for (int k = 0; k < kB; ++k) get(i0 + k, c[k], d[k]);
#pragma unroll
        for (int k = 0; k < kB; ++k) {
            check(i0 + k, c[k]);
            const float e = __fadd_rn(c[k], 0.0f), f = __fadd_rn(d[k], 0.0f);
            w.r = __funnelshift_l(__float_as_uint(__fsub_rn(b, a)), w.r, 1);
            w.d = __funnelshift_l(__float_as_uint(__fsub_rn(e, a)), w.d, 1);
            w.dr = __funnelshift_l(__float_as_uint(__fsub_rn(f, a)), w.dr, 1);
            w.a = __funnelshift_l(__float_as_uint(__fsub_rn(e, b)), w.a, 1);
            a = e;
            b = f;
        }
    }
    w.r = __brev(w.r);
    w.d = __brev(w.d);
    w.dr = __brev(w.dr);
    w.a = __brev(w.a);
    return w;
}

__global__ void __launch_bounds__(kW2 * 32) k_prune2d(const __grid_constant__ ItemTable tab, const __grid_constant__ Outs o,
                                                      const int parts) {
    __shared__ Smem2 sm;
    const int warp = threadIdx.x >> 5;
    const int lane = int(lane_id());
    const unsigned lt = (1u << lane) - 1u;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    wait_for_previous();
    for (int task = blockIdx.x * kW2 + warp; task < tab.tiles2d * parts; task += gridDim.x * kW2) {
        const int tile = task / parts, part = task - tile * parts;
        const int ii = tile_item(tab, 0, tab.n2d - 1, tile);
        const Item& it = tab.it[ii];
        const int ltask = tile - it.tile0;
        const int W = it.W, H = it.H, ty = ltask / it.tx;
        const int x0 = (ltask - ty * it.tx) * kTile2, y0 = ty * kTile2;
        const int x = x0 - 1 + lane;
        // ---- compare
        float bad = 0.0f;
        const bool inside = x0 > 0 && y0 > 0 && x0 + 31 < W && y0 + 31 < H;
        const Words2 w = inside ? words2<true>(it.img, W, H, x, y0 - 1, bad) : words2<false>(it.img, W, H, x, y0 - 1, bad);
        if (__any_sync(kAll, bad != bad) && lane == 0) set_status(o.ctr, kStNonfinite);
        // ---- logic: neighbours before in linear order by complement, from the row above and the lane to the left
        const uint32_t rl = __shfl_up_sync(kAll, w.r, 1), drl = __shfl_up_sync(kAll, w.dr, 1), al = __shfl_up_sync(kAll, w.a, 1);
        const uint32_t nul = ~(drl << 1), nu = ~(w.d << 1), nur = ~(w.a << 1), nl = ~rl, nr = w.r, ndl = al, nd = w.d, ndr = w.dr;
        const uint32_t q0 = nul & nu & nl, q1 = nur & nu & nr, q2 = ndl & nd & nl, q3 = ndr & nd & nr;
        const bool own_x = lane >= 1 && lane <= kTile2 && x < W;
        const uint32_t own = own_x ? (H - y0 >= kTile2 ? 0x7FFFFFFEu : (2u << (H - y0)) - 2u) : 0u;
        uint32_t ev;
        {
            const uint32_t a = nu & ~q1, b = nr & ~q3, c = nd & ~q2, d = nl & ~q0;
            const uint32_t two = (a & b) | (c & d) | ((a | b) & (c | d));
            // this part's rows
            const uint32_t rows = ((2u << ((part + 1) * kTile2 / parts)) - 1u) & ~((2u << (part * kTile2 / parts)) - 1u);
            ev = ~((a | b | c | d) & ~two) & own & rows;
        }
        // ---- code bytes: the byte of row i (bit i + 1) of the lane's column
        if (part == 0) {
            const uint32_t px = __shfl_down_sync(kAll, q2, 1), py = (q1 | __shfl_down_sync(kAll, q0, 1)) >> 1;
            const uint32_t last_x = x == W - 2 ? kAll : 0u, first_x = x == 0 ? kAll : 0u, first_y = y0 == 0 ? 2u : 0u;
            const int ly = H - 1 - y0;  // the bit of row H - 2
            const uint32_t last_y = unsigned(ly) < 32u ? 1u << ly : 0u;
            const uint32_t mx = q3 & ~q2, my = q3 & q2 & ~q1, dg = q3 & q2 & q1 & ~q0, root = q3 & q2 & q1 & q0;
            const uint32_t out = (px & last_x) | (py & last_y) | ((mx | dg) & first_x) | ((my | dg) & first_y);
            // runs of links up, and of links down (+y), at least 1, 2, 4, 8, 16 long
            const uint32_t u1 = nu & ~1u, u2 = u1 & (u1 << 1), u4 = u2 & (u2 << 2), u8 = u4 & (u4 << 4), u16 = u8 & (u8 << 8);
            const uint32_t d1 = py & ~out & 0x7FFFFFFEu, d2 = d1 & (d1 >> 1), d4 = d2 & (d2 >> 2), d8 = d4 & (d4 >> 4),
                           d16 = d8 & (d8 >> 8);
            // of the other links, at least 4 (and 16 along y) long; a lane whose own
            // link depends on what lies beyond the tile is in none
            auto four = [&](uint32_t q, bool left) {
                if (lane == (left ? 0 : 31)) q = 0u;
                q &= left ? __shfl_up_sync(kAll, q, 1) : __shfl_down_sync(kAll, q, 1);
                return q & (left ? __shfl_up_sync(kAll, q, 2) : __shfl_down_sync(kAll, q, 2));
            };
            const uint32_t hl = ~nu & nl, hr = ~nu & ~nl & nr, hd = ~nu & ~nl & ~nr & nd, h0 = ~(nu | nl | nr | nd);
            const uint32_t hl4 = four(hl, true), hr4 = four(hr, false);
            const uint32_t e1 = hd & 0x7FFFFFFEu, e2 = e1 & (e1 >> 1), hd4 = e2 & (e2 >> 2), e8 = hd4 & (hd4 >> 4),
                           hd16 = e8 & (e8 >> 8);
            const uint32_t cx = px & ~out, cm = mx & ~out, cy = my & ~out;
            const uint32_t cx4 = four(cx, false), cm4 = four(cm, true);
            const uint32_t g1 = cy & 0x7FFFFFFEu, g2 = g1 & (g1 << 1), cy4 = g2 & (g2 << 2), g8 = cy4 & (cy4 << 4),
                           cy16 = g8 & (g8 << 8);
            uint32_t acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            spread<0>(acc, ((u2 & ~u4) | (u8 & ~u16) | (hl & ~hl4) | hr4 | (hd & ~hd4) | hd16) >> 1);
            spread<1>(acc, ((u4 & ~u16) | (hr & ~hr4) | hd | h0) >> 1);
            spread<2>(acc, (u16 | (hl & ~hl4) | (hr & ~hr4) | (hd & ~hd4) | h0) >> 1);
            spread<3>(acc, (hl4 | hr4 | hd4 | h0) >> 1);
            spread<4>(acc, ((d2 & ~d4) | (d8 & ~d16) | (cx & ~cx4) | (cy & ~cy4) | cm4 | cy16 | out | root) >> 1);
            spread<5>(acc, ((d4 & ~d16) | cm | (cy & ~cy4) | cx4 | root) >> 1);
            spread<6>(acc, (d16 | (cx & ~cx4) | (cm & ~cm4) | cy | root) >> 1);
            spread<7>(acc, (dg | out | cx4 | cm4 | cy4 | root) >> 1);
            const uint64_t at = uint64_t(it.coff) + uint64_t(code_at2(it, y0, x));
            if (own_x && CP_IN(at + 31u, o.n_code, o.ctr)) {
                uint4* dst = reinterpret_cast<uint4*>(o.code + at);
                dst[0] = make_uint4(acc[0], acc[1], acc[2], acc[3]);
                dst[1] = make_uint4(acc[4], acc[5], acc[6], acc[7]);
            }
        }
        // ---- events
        uint32_t incl = __popc(ev);
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const uint32_t u = __shfl_up_sync(kAll, incl, s);
            if (lane >= s) incl += u;
        }
        const uint32_t total = __shfl_sync(kAll, incl, 31);
        if (total == 0) continue;
        uint32_t(*n)[32] = sm.n[warp];
        uint32_t* queue = sm.queue[warp];
        __syncwarp();  // the last tile's events have been read
        n[0][lane] = nul, n[1][lane] = nu, n[2][lane] = nur, n[3][lane] = nl;
        n[4][lane] = nr, n[5][lane] = ndl, n[6][lane] = nd, n[7][lane] = ndr;
        for (uint32_t at = incl - __popc(ev); ev; ev &= ev - 1u) queue[at++] = uint32_t(__ffs(ev) - 1) << 5 | uint32_t(lane);
        __syncwarp();
        uint32_t c_s = 0, c_r = 0;  // survivors (H0 | dual << 16), roots (the same)
#pragma unroll 2
        for (uint32_t e = lane; e < total; e += 32) {
            const uint32_t q = queue[e], l = q & 31u, row = q >> 5;
            uint32_t raw = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) raw |= ((n[k][l] >> row) & 1u) << k;
            const uint32_t en = __ldg(g_lut2d + raw);
            const uint32_t h0 = (en >> 3) & 15u, dual = (en >> 9) & 15u;
            const uint32_t r0 = (en & 7u) == 7u ? 1u : 0u, rt = raw == 255u ? 1u : 0u;
            queue[e] = q | h0 << 10 | dual << 14 | r0 << 18 | rt << 19;
            // cross-pruning: dual survivors that are also H0 survivors wait for the H0 union-find
            c_s += __popc(h0) | __popc(tab.cross2d ? dual & ~h0 : dual) << 16;
            c_r += r0 | rt << 16;
        }
        c_s = __reduce_add_sync(kAll, c_s);
        c_r = __reduce_add_sync(kAll, c_r);
        uint32_t b0, bt, br0, brt;
        reserve(o, c_s & 0xFFFFu, c_s >> 16, c_r & 0xFFFFu, c_r >> 16, b0, bt, br0, brt);
        unsigned long long gmin = ~0ull;
        __syncwarp();
        // a batch's values are loaded during the one before
        auto take = [&](uint32_t e, uint32_t& q, float& v) {
            q = e < total ? queue[e] : 0u;
            const int64_t at = int64_t(y0 - 1 + int((q >> 5) & 31u)) * W + (x0 - 1 + int(q & 31u));
            v = e < total ? __ldg(it.img + at) : 0.0f;
        };
        uint32_t q, q_next;
        float val, val_next;
        take(lane, q_next, val_next);
        for (uint32_t e0 = 0; e0 < total; e0 += 32) {
            q = q_next;
            val = val_next;
            take(e0 + 32 + lane, q_next, val_next);
            uint32_t h0 = (q >> 10) & 15u, dual = (q >> 14) & 15u;
            const uint32_t flg = tab.cross2d ? dual : 0u;
            if (tab.cross2d) dual &= ~h0;
            const bool root0 = (q >> 18) & 1u, rootT = (q >> 19) & 1u;
            const int ex = x0 - 1 + int(q & 31u), ey = y0 - 1 + int((q >> 5) & 31u);
            const uint32_t vl = uint32_t(ey) * uint32_t(W) + uint32_t(ex), vg = uint32_t(it.voff) + vl;
            const uint32_t mine = __popc(h0) | __popc(dual) << 16;  // at most 128 each in a warp
            uint32_t ex_s = mine;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const uint32_t u = __shfl_up_sync(kAll, ex_s, s);
                if (lane >= s) ex_s += u;
            }
            const uint32_t all = __shfl_sync(kAll, ex_s, 31);
            ex_s -= mine;
            const unsigned m0 = __ballot_sync(kAll, root0), mt = __ballot_sync(kAll, rootT);
            const uint32_t ord = ord_bits(val);
            for (uint32_t at = b0 + (ex_s & 0xFFFFu); h0; h0 &= h0 - 1u, ++at) {
                const uint32_t s = uint32_t(__ffs(h0) - 1);  // face slot s is stencil offset 2 s + 1; low bit: the dual waits
                if (at < o.cap_s) o.s0[at] = make_key(ord, vg, (2u * s + 1u) << 1 | ((flg >> s) & 1u));
            }
            for (uint32_t at = bt + (ex_s >> 16); dual; dual &= dual - 1u, ++at)
                if (at < o.cap_s) o.st[at] = ~make_key(ord, vg, (2u * uint32_t(__ffs(dual) - 1) + 1u) << 1);
            if (root0 && CP_IN(vg, o.n_uf0, o.ctr)) {
                const unsigned long long k = (unsigned long long)(uint64_t(ord) << 32 | vl);
                gmin = k < gmin ? k : gmin;
                put_root(o.uf0 + vg, br0 + __popc(m0 & lt), o.cap_r0, make_key(ord, vg, 0), o.node0, o.age0, o.res0, false, ii);
            }
            if (rootT) {  // the top cell in quadrant 3 of its largest corner
                const uint32_t self = uint32_t(it.toff) + uint32_t(ey) * uint32_t(W - 1) + uint32_t(ex);
                if (CP_IN(self, o.n_uft, o.ctr))
                    put_root(o.uft + self, brt + __popc(mt & lt), o.cap_rt, make_key(ord, vg, 16u), o.nodet, o.aget, o.rest, true, ii);
            }
            b0 += all & 0xFFFFu;
            bt += all >> 16;
            br0 += __popc(m0);
            brt += __popc(mt);
        }
        gmin = warp_min_u64(gmin);
        if (lane == 0 && gmin != ~0ull) atomicMin(&o.ctr->gmin[ii], gmin);
    }
}

// ---------------------------------------------------------------- host side
size_t prune_smem3d() { return sizeof(Smem3); }

bool encode_plane_map(CUtensorMap* map, const float* img, int64_t D, int64_t H, int64_t W) {
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = []() -> Encode {  // looked up once (thread-safe initialisation)
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<Encode>(fn);
        return nullptr;
    }();
    // row stride a multiple of 16 bytes, 16-byte aligned base, and planes that are worth it
    if (!encode || !img || (W & 3) != 0 || (reinterpret_cast<uintptr_t>(img) & 15u) != 0 || W < 40 || H < 11 || D < 2)
        return false;
    const cuuint64_t dim[3] = {cuuint64_t(W), cuuint64_t(H), cuuint64_t(D)};
    const cuuint64_t stride[2] = {cuuint64_t(W) * 4u, cuuint64_t(W) * cuuint64_t(H) * 4u};
    const cuuint32_t box[3] = {cuuint32_t(kRS), cuuint32_t(kRH), 1u};
    const cuuint32_t estride[3] = {1u, 1u, 1u};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(img), dim, stride, box, estride,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NAN_REQUEST_ZERO_FMA) == CUDA_SUCCESS;
}
int prune_tile_x() { return kTile2; }
int prune_tile_x3d() { return kOX; }
int g_rows2d = 64, g_zchunk3d = kZC, g_ctas3d = 0, g_cross2d = 0, g_uf_variant = 0;  // tuning (cp_set_tuning)
int prune_tile_y2d() { return kTile2; }
int prune_tile_y3d() { return kOY; }
int prune_zchunk3d() { return g_zchunk3d; }
int prune_cross2d() { return g_cross2d; }
int uf_variant() { return g_uf_variant; }

int set_tuning(int key, int value) {
    switch (key) {
        case 1:  // planes per 3D pruning task
            if (value < 4 || value > 4096) return -1;
            g_zchunk3d = value;
            return 0;
        case 2:  // 3D pruning CTAs per SM (0: as many as fit)
            if (value < 0 || value > 8) return -1;
            g_ctas3d = value;
            return 0;
        case 3:  // rows per 2D pruning task
            if (value < 4 || value > 4096) return -1;
            g_rows2d = value;
            return 0;
        case 5:  // 2D items: sequential cross-pruning (1) or H0 and the dual at once (0)
            if (value != 0 && value != 1) return -1;
            g_cross2d = value;
            return 0;
        case 7:  // union-find design: the merge tree (0) or Borůvka's forest and rounds over it (1)
            if (value != 0 && value != 1) return -1;
            g_uf_variant = value;
            return 0;
        default:
            return -1;
    }
}

int get_tuning(int key) {
    return key == 1 ? g_zchunk3d
           : key == 2 ? g_ctas3d
           : key == 3 ? g_rows2d
           : key == 5 ? g_cross2d
           : key == 7 ? g_uf_variant
                      : -1;
}

cudaError_t upload_luts(const uint64_t* lut2d, const uint16_t* disp3d, const uint64_t* entries3d,
                        const uint32_t* keys3d) {
    uint32_t p2[256];
    for (int i = 0; i < 256; ++i)
        p2[i] = uint32_t(lut2d[i] & 0x1FFu) | uint32_t((lut2d[i] >> 41) & 0xFFFu) << 9;
    cudaError_t e = cudaMemcpyToSymbol(g_lut2d, p2, sizeof(p2));
    if (e != cudaSuccess) return e;
    e = cudaMemcpyToSymbol(g_disp3d, disp3d, sizeof(uint16_t) * (1 << 12));
    if (e != cudaSuccess) return e;
    static uint32_t surv[1 << 14];
    for (int i = 0; i < (1 << 14); ++i)
        surv[i] = keys3d[i] == 0xFFFFFFFFu ? 0u
                                           : uint32_t((entries3d[i] >> 3) & 0x3Fu) | uint32_t((entries3d[i] >> 41) & 0xFFFu) << 6;
    return cudaMemcpyToSymbol(g_surv3d, surv, sizeof(surv));
}

static Outs outs_of(const PruneOuts& po) {
    Outs o;
    o.uf0 = po.uf0;
    o.uft = po.uft;
    o.code = po.code;
    o.n_code = po.n_code;
    o.s0 = po.s0;
    o.st = po.st;
    o.age0 = po.age0;
    o.res0 = po.res0;
    o.aget = po.aget;
    o.rest = po.rest;
    o.node0 = po.node0;
    o.nodet = po.nodet;
    o.cap_s = po.cap_s;
    o.cap_r0 = po.cap_r0;
    o.cap_rt = po.cap_rt;
    o.ctr = po.ctr;
    o.n_uf0 = po.n_uf0;
    o.n_uft = po.n_uft;
    return o;
}

cudaError_t launch_expand(const ItemTable& tab, const PruneOuts& po, cudaStream_t s) {
    k_expand<<<device_sm_count() * 8, 256, 0, s>>>(tab, outs_of(po));
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_prune(const ItemTable& tab, const PruneOuts& po, const TmaMaps& maps, cudaStream_t s) {
    const Outs o = outs_of(po);
    const int blocks3d = device_cached(kCachePrune3d, [] {
        cudaFuncSetAttribute(k_prune3d, cudaFuncAttributeMaxDynamicSharedMemorySize, int(prune_smem3d()));
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_prune3d, kT3, prune_smem3d());
        return device_sm_count() * (per_sm > 0 ? per_sm : 1);
    });
    const int blocks2d = device_cached(kCachePrune2d, [] {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_prune2d, kW2 * 32, 0);
        return device_sm_count() * (per_sm > 0 ? per_sm : 1);
    });
    if (tab.tiles2d > 0) {
        // warps per tile (its events' rows are split): as many as leave at most
        // 16 warps per SM; uniform noise, 1 -> 8 parts: 64^2 20.0 -> 7.8 us,
        // 480^2 20.5 -> 9.1; smooth, 2 parts: 769 x 1021 6.6 -> 7.0 us, 2048^2
        // (one part) 11.6 -> 18.2
        int parts = 8;
        while (parts > 1 && int64_t(tab.tiles2d) * parts > 2432) parts >>= 1;
        const int need2 = (tab.tiles2d * parts + kW2 - 1) / kW2;
        const cudaError_t e = launch_after(true, k_prune2d, need2 < blocks2d ? need2 : blocks2d, kW2 * 32, 0, s, tab, o, parts);
        if (e != cudaSuccess) return e;
    }
    if (tab.tiles3d > 0) {
        int cap = blocks3d;
        if (g_ctas3d > 0) cap = device_sm_count() * g_ctas3d < blocks3d ? device_sm_count() * g_ctas3d : blocks3d;
        int grid = tab.tiles3d < cap ? tab.tiles3d : cap;
        k_prune3d<<<grid, kT3, prune_smem3d(), s>>>(tab, o, maps);
        note_launches(1);
    }
    return cudaGetLastError();
}

}  // namespace cp
