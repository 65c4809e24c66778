// K1: fused lookup + local pruning (Sec. 3.2, Sec. 3.3, Sec. 4.1 steps 1-2,
// Sec. 4.2 steps 1-3 before the union-finds).
//
// Per vertex v:
//   1. the mask of the neighbours that precede v (value, then index): 8 in 2D,
//      26 in 3D;
//   2. what it says about the lower star of v: 2D by a direct 256-entry table,
//      3D by closed forms on words of 32 vertices, with a perfect-hash lookup
//      for the vertices that leave survivors;
//   3. the H0 forest link of v (first edge of L(v)), or v as an H0 root (local
//      minimum);
//   4. the dual forest link of each top cell, from its largest corner's lower
//      star: the top cell across the facet where it dies locally, the outside
//      vertex, or itself as a dual root;
//   5. the surviving edges and facets as 64-bit order keys.
// Rows (2D) and planes (3D) ahead are brought into shared memory
// asynchronously; positions outside the image hold values that precede
// nothing.
#include "cp_common.cuh"
#include "cp_kernels.h"
#include "cp_mask3.cuh"
#include "cp_walk.cuh"
#include "cp_words3.cuh"

#include <type_traits>

namespace cp {

// Lookup tables in global memory, read through the read-only cache (lanes of
// a warp look up different entries, which constant memory would serialise).
__device__ uint2 g_lut2d[256];  // same two-word entry layout as the 3D table
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

// Perfect hash of the 15,935 relevant masks (device layout, cp_mask3.cuh):
// bucket -> displacement -> slot.
__device__ __forceinline__ uint32_t hash_slot3(uint32_t rel, const uint16_t* disp) {
    const uint32_t b = (rel * 0x9E3779B1u) >> (32 - 12);
    const uint32_t d = __ldg(disp + b);
    return ((rel ^ (d * 0x27D4EB2Fu)) * 0x85EBCA77u) >> (32 - 14);
}

}  // namespace

// ---------------------------------------------------------------- 3D
// A CTA marches along z through a tile of 64 x 32 columns, of which it owns
// 60 x 29.  The lookup of a vertex is done 32 vertices at a time, on words
// that hold one bit per vertex:
//
//   compare  (4 warps, 8 rows each) of every vertex p of a plane and each of
//            the 13 neighbours q after it in linear order: does q precede p?
//            A warp does a row of 64 columns, two per lane (even columns give
//            one word, odd columns another): a compare and a ballot per
//            neighbour.  The other 13 neighbours' bits are the complements of
//            the neighbours' own.
//   logic    (2 warps: even and odd columns; lane = row) the relevant mask
//            (the collapse of Sec. 3.3 is one AND per edge and two per corner,
//            for 32 vertices), the H0 link, the top cells in the lower stars
//            and where each dies, and the vertices that need more than a link
//            (events); a code byte per vertex with both links (cp_walk.cuh).
//   output   (compare warps) the code bytes, two 4-byte stores per 8 columns.
//   events   (compare warps, 32 at a time once a warp each has some) the
//            vertices whose lower star holds a survivor or a root: their masks
//            from the image, the lookup, the keys and roots.
//
// The two kinds of warps hand planes on through named barriers, either a plane
// ahead of the other.
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
// Bound by the issue of compares, ballots and word logic (ALU pipe): 112 warp
// instructions per 32 vertices at 256^3 (halo and chunk lead-in included; 280
// with a 26-compare mask, a collapse and a table read per vertex, and links
// stored as words), 40 of them the compares and ballots.  One byte per vertex
// written instead of eight.  128^3 smooth 90 -> 28 us, 128^3 noise 282 -> 202
// us, 512^3 1,430 -> 673 us.  Tried: eight compare warps per CTA (72
// registers: spills, 1.2x the time), one logic warp (it bounds the step), a
// CTA barrier per plane instead of the named ones, the row loop unrolled fully
// (instruction cache misses), links as words with z chains (670 -> 840 us, and
// the walks miss L2).
constexpr int kW3 = 4;                     // compare warps per CTA (and two logic warps: even and odd columns)
constexpr int kT3 = kW3 * 32;              // threads of the compare warps
constexpr int kTX = 64, kTY = 32;          // compared columns / rows: x0-1 .. x0+62, y0-1 .. y0+30
constexpr int kOX = 60, kOY = 29;          // owned: x0 .. x0+59, y0 .. y0+28
constexpr int kRows = kTY / kW3;           // rows per warp
constexpr int kUnrollC = 4;                // rows per turn of the compare loop (all eight: instruction cache misses)
constexpr int kZC = 64;                    // default bound on the owned planes of a task
constexpr int kRW = kTX + 2, kRH = kTY + 2;  // plane tile read: cols x0-2 .. x0+63, rows y0-2 .. y0+31
constexpr int kRX = 2;                     // column x0-2 within a ring row (rows start at x0-4: 16-byte aligned)
constexpr int kRS = 72;                    // ring row stride in floats (a TMA box row)
constexpr int kSlot = 2464;                // ring slot in floats: kRH rows of kRS, padded to 128 bytes
constexpr int kFix = (2 * kRH + 2 * kRW + 31) / 32;  // border positions set per lane of a logic warp
constexpr int kRing = 3;                   // ring slots
constexpr int kWR = 28;                    // words per row: 26, padded (16-byte rows; LDS.128 without conflicts)
constexpr int kCR = 80;                    // code bytes per row: 64, padded
constexpr int kQ = 4096;                   // event queue (two planes of 1,740 while fewer than kQMin wait)
constexpr int kQMin = kT3;                 // events that a pass over the queue takes at least ...
constexpr int kQAge = 16;                  // ... unless the oldest is this many planes back (entries hold z mod 32)

// One task's place and constants (uniform over the CTA).
struct Task3 {
    const float* img;
    int D, H, W, x0, y0, z0, z1, zlast;  // owned planes [z0, z1), zlast = z1 - 1
    uint32_t HW, W1, HW1, voff, toff, pitch;
    int item;                // its index in the call's table
    uint8_t* code;           // the item's link codes
    const CUtensorMap* map;  // nullptr: the planes come by cp.async
    uint32_t own[2], cube[2];       // even / odd columns whose vertex / top cell the task owns
    uint32_t first_x[2], last_x[2]; // the columns x = 0 and x = W - 2
};

// Ring slot of plane z >= -1.
__device__ __forceinline__ int ring_slot(int z) { return int(unsigned(z + kRing) % unsigned(kRing)); }

struct Smem3 {
    float ring[kRing][kSlot];  // first: slots 128-byte aligned (TMA destinations)
    uint64_t bar[kRing];       // mbarrier of each slot (TMA completion)
    // compare words of a row: groups of {dx = -1, 0, +1} x {even, odd columns}
    // for (dz, dy) = (1,-1) (1,0) (1,1) (0,1), then (0,0,+1)
    alignas(16) uint32_t w[3][kTY][kWR];
    alignas(16) uint8_t code[2][kTY][kCR];  // columns 2, 4 .. 62 (and a pad), then 1, 3 .. 63; dual << 3 | H0
    // what the top cells below a plane need of the plane before, per row and parity
    uint32_t low[2][6][kTY];
    uint32_t xco[2][4][kTY], xev[2];  // between the two logic warps
    uint16_t queue[kQ];        // event vertices: (z mod 32) << 11 | row << 6 | column
    uint32_t tail[2];          // events queued up to the last even / odd plane
    Task3 t;
};

// raw |= kBit when the neighbour value u precedes the centre value c (kLe:
// the neighbour comes earlier in linear order, so it also precedes on a tie;
// NaN, the out-of-image fill, never precedes): a compare into a predicate and
// a predicated OR, two instructions per bit
template <uint32_t kBit, bool kLe>
__device__ __forceinline__ void or_if_precedes(uint32_t& raw, float u, float c) {
    if constexpr (kLe)
        asm("{\n\t.reg .pred p;\n\tsetp.le.f32 p, %1, %2;\n\t@p or.b32 %0, %0, %3;\n\t}"
            : "+r"(raw) : "f"(u), "f"(c), "n"(kBit));
    else
        asm("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %1, %2;\n\t@p or.b32 %0, %0, %3;\n\t}"
            : "+r"(raw) : "f"(u), "f"(c), "n"(kBit));
}

struct Nbr {
    float v[3][3];  // [row y-1, y, y+1][col x-1, x, x+1] of one plane
};

template <int n>
__device__ __forceinline__ void mask_bit(uint32_t& raw, const Nbr& A, const Nbr& B, const Nbr& C, float cv) {
    constexpr int a = n / 9, b = (n / 3) % 3, c = n % 3;
    const Nbr& P = a == 0 ? A : (a == 1 ? B : C);
    or_if_precedes<(1u << mask3_pos(n)), (n < 13)>(raw, P.v[b][c], cv);
}

// raw mask in the device layout (cp_mask3.cuh): the bit of canonical
// neighbour n = 9a + 3b + c set when the neighbour at plane a, row b, column
// c precedes the centre (ties: earlier linear index first)
__device__ __forceinline__ uint32_t mask26(const Nbr& A, const Nbr& B, const Nbr& C) {
    const float cv = B.v[1][1];
    uint32_t raw = 0;
    mask_bit<0>(raw, A, B, C, cv);
    mask_bit<1>(raw, A, B, C, cv);
    mask_bit<2>(raw, A, B, C, cv);
    mask_bit<3>(raw, A, B, C, cv);
    mask_bit<4>(raw, A, B, C, cv);
    mask_bit<5>(raw, A, B, C, cv);
    mask_bit<6>(raw, A, B, C, cv);
    mask_bit<7>(raw, A, B, C, cv);
    mask_bit<8>(raw, A, B, C, cv);
    mask_bit<9>(raw, A, B, C, cv);
    mask_bit<10>(raw, A, B, C, cv);
    mask_bit<11>(raw, A, B, C, cv);
    mask_bit<12>(raw, A, B, C, cv);
    mask_bit<14>(raw, A, B, C, cv);
    mask_bit<15>(raw, A, B, C, cv);
    mask_bit<16>(raw, A, B, C, cv);
    mask_bit<17>(raw, A, B, C, cv);
    mask_bit<18>(raw, A, B, C, cv);
    mask_bit<19>(raw, A, B, C, cv);
    mask_bit<20>(raw, A, B, C, cv);
    mask_bit<21>(raw, A, B, C, cv);
    mask_bit<22>(raw, A, B, C, cv);
    mask_bit<23>(raw, A, B, C, cv);
    mask_bit<24>(raw, A, B, C, cv);
    mask_bit<25>(raw, A, B, C, cv);
    mask_bit<26>(raw, A, B, C, cv);
    return raw;
}

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

// Named barriers between the compare warps and the logic warp, two of each
// kind (even and odd planes), so that either side can be a plane ahead.
constexpr int kBarWords = 1;  // + plane parity: the compare words of a plane are complete
constexpr int kBarCodes = 3;  // + plane parity: the codes of a plane are, and plane + 3 is in the ring
constexpr int kBarRows = 5;   // among the compare warps (cp.async planes)
constexpr int kBarLogic = 6;  // between the logic warps
__device__ __forceinline__ void bar_arrive(int id) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kT3 + 64) : "memory");
}
__device__ __forceinline__ void bar_sync(int id) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kT3 + 64) : "memory");
}

// max(m, |v|), NaN if either is
__device__ __forceinline__ float max_nan(float m, float v) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(m), "f"(fabsf(v)));
    return r;
}

// Plane z of the tile.  TMA: one thread's tensor copy, completing on the
// slot's mbarrier; positions outside the image read NaN (which precedes
// nothing), and those next to an image vertex are set to +inf once the plane
// has landed.  cp.async: a warp per row; +inf at positions outside the image,
// set once per task.
__device__ __forceinline__ void issue_tma(Smem3& sm, const Task3& t, int z) {  // one thread
    if (z > t.zlast + 1 || unsigned(z) >= unsigned(t.D)) return;
    uint64_t* bar = &sm.bar[ring_slot(z)];
    // earlier generic-proxy accesses of the slot come before the copy
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_expect_tx(bar, uint32_t(kRH * kRS * sizeof(float)));
    tma_load_plane(sm.ring[ring_slot(z)], t.map, bar, t.x0 - 2 - kRX, t.y0 - 2, z);
}
__device__ __forceinline__ void issue_rows(Smem3& sm, const Task3& t, int z) {  // the compare warps
    if (z > t.zlast + 1 || unsigned(z) >= unsigned(t.D)) return;
    float* plane = sm.ring[ring_slot(z)];
    const int lane = int(lane_id());
    const float* src = t.img + uint32_t(z) * t.HW;
    for (int r = threadIdx.x >> 5; r < kRH; r += kW3) {
        const int gy = t.y0 - 2 + r;
        if (unsigned(gy) >= unsigned(t.H)) continue;
        const float* row = src + uint32_t(gy) * uint32_t(t.W);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int c = lane + 32 * k, gx = t.x0 - 2 + c;
            if (c < kRW && unsigned(gx) < unsigned(t.W)) cp_async4(plane + r * kRS + kRX + c, row + gx);
        }
    }
}
// A plane outside the volume (z = D): every position +inf (the compare warps).
__device__ __forceinline__ void fill_plane(Smem3& sm, int z) {
    float* plane = sm.ring[ring_slot(z)];
    for (int i = threadIdx.x; i < kRH * kRS; i += kT3) plane[i] = __int_as_float(0x7F800000);
}

// Four code bytes.
__device__ __forceinline__ void put_code(const Outs& o, uint8_t* dst, uint32_t v) {
    if (CP_IN(dst + 3 - o.code, o.n_code, o.ctr)) *reinterpret_cast<uint32_t*>(dst) = v;
}

// Before reading plane z: wait for its TMA copy (cp.async planes are covered
// by the wait_group and the barrier of the step before).
__device__ __forceinline__ void wait_plane(Smem3& sm, const Task3& t, int z, uint32_t& par, Counters* ctr) {
    if (!t.map || unsigned(z) >= unsigned(t.D)) return;
    const int slot = ring_slot(z);
    mbar_wait(&sm.bar[slot], (par >> slot) & 1u, ctr);
    par ^= 1u << slot;
}

// Compare words of this warp's rows in one plane (pl; up: the plane after it).
// A position outside the image next to an image vertex holds +inf: everything
// precedes it, so its neighbours' reversed bits are zero.
// top_a, top_b: the largest magnitude of the two columns' values in image rows.
__device__ __forceinline__ void compare_rows(const float* pl, const float* up, uint32_t (*w)[kWR], int warp, int lane,
                                             float& top_a, float& top_b, int y_first, int H) {
    struct Row {
        float v[4];  // columns 2 lane - 1 .. 2 lane + 2 (tile columns)
    };
    auto read = [&](const float* p, int r) {
        Row q;
        const float2 a = *reinterpret_cast<const float2*>(p + r * kRS + kRX + 2 * lane);
        const float2 b = *reinterpret_cast<const float2*>(p + r * kRS + kRX + 2 * lane + 2);
        q.v[0] = a.x;
        q.v[1] = a.y;
        q.v[2] = b.x;
        q.v[3] = b.y;
        return q;
    };
    const int r0 = warp * kRows;
    Row cur = read(pl, r0 + 1), u0 = read(up, r0), u1 = read(up, r0 + 1);
#pragma unroll kUnrollC
    for (int i = 0; i < kRows; ++i) {
        const int r = r0 + i;
        const Row nx = read(pl, r + 2), u2 = read(up, r + 2);
        const float a = cur.v[1], b = cur.v[2];
        if (unsigned(y_first + i) < unsigned(H)) {
            top_a = max_nan(top_a, a);
            top_b = max_nan(top_b, b);
        }
        uint32_t m[26];
        auto put = [&](int k, const Row& q) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                m[k + 2 * d] = __ballot_sync(0xFFFFFFFFu, q.v[d] < a);
                m[k + 2 * d + 1] = __ballot_sync(0xFFFFFFFFu, q.v[d + 1] < b);
            }
        };
        put(0, u0);
        put(6, u1);
        put(12, u2);
        put(18, nx);
        m[24] = __ballot_sync(0xFFFFFFFFu, cur.v[2] < a);
        m[25] = __ballot_sync(0xFFFFFFFFu, cur.v[3] < b);
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < 24; k += 4)
                *reinterpret_cast<uint4*>(&w[r][k]) = make_uint4(m[k], m[k + 1], m[k + 2], m[k + 3]);
            *reinterpret_cast<uint2*>(&w[r][24]) = make_uint2(m[24], m[25]);
        }
        cur = nx;
        u0 = u1;
        u1 = u2;
    }
}

// Bits of the columns lo .. hi (tile columns) in the even (par 0) or odd word.
__device__ __forceinline__ uint32_t col_mask(int lo, int hi, int par) {
    const int l0 = max(0, (lo - par + 1) >> 1), l1 = min(31, (hi - par) >> 1);
    return l1 < l0 ? 0u : (0xFFFFFFFFu >> (31 - (l1 - l0))) << l0;
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

// The logic of plane p for the even (par = 0) or odd columns; one warp, lane =
// tile row.  wp, wl: the compare words of planes p and p - 1.  Returns the
// event queue's new end (the even columns' events come first).
template <int par>
__device__ __forceinline__ uint32_t logic_plane(Smem3& sm, int p, const uint32_t (*wp)[kWR], const uint32_t (*wl)[kWR],
                                                uint32_t tail) {
    const Task3& t = sm.t;
    const int r = int(lane_id()), rm = max(r - 1, 0), rp = min(r + 1, kTY - 1);
    const int y = t.y0 - 1 + r;
    const bool own_row = r >= 1 && r <= kOY && y < t.H, cube_row = own_row && y < t.H - 1;
    const bool last_y = y == t.H - 2, first_y = y == 0;
    Star3 st;
    {
        uint32_t n[27];
        n[13] = 0;
        // a row's word of one group for the column one to the left (dx = 1),
        // the same (0) or one to the right (-1) of this parity's columns
        auto at_col = [&](const uint32_t* g, int dx) -> uint32_t {
            const uint32_t* q = g + 2 * (dx + 1);
            if (dx == 0) return q[par];
            if (par == 0) return dx > 0 ? q[1] << 1 : q[1];
            return dx > 0 ? q[0] : q[0] >> 1;
        };
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
#pragma unroll
            for (int dy = -1; dy <= 1; ++dy) {
                n[13 + 9 + 3 * dy + dx] = wp[r][6 * (dy + 1) + 2 * (dx + 1) + par];
                n[13 - 9 - 3 * dy - dx] = ~at_col(&wl[dy < 0 ? rp : (dy > 0 ? rm : r)][6 * (dy + 1)], dx);
            }
            n[13 + 3 + dx] = wp[r][18 + 2 * (dx + 1) + par];
            n[13 - 3 - dx] = ~at_col(&wp[rm][18], dx);
        }
        n[14] = wp[r][24 + par];
        n[12] = ~(par == 0 ? wp[r][25] << 1 : wp[r][24]);
        star_words3(n, st);
    }
    const uint32_t own = own_row && p >= t.z0 ? t.own[par] : 0u;
    const uint32_t cube = cube_row && p > 0 ? t.cube[par] : 0u;
    uint32_t ev = st.event & own;
    const uint32_t nev = __popc(ev);
    uint32_t incl = nev;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (r >= o) incl += u;
    }
    // what the other parity's warp needs: its column one to the right is one of these
#pragma unroll
    for (int k = 0; k < 4; ++k) sm.xco[par][k][r] = st.co[2 * k];
    if (r == 31) sm.xev[par] = incl;
    asm volatile("bar.sync %0, 64;" ::"n"(kBarLogic) : "memory");
    uint32_t xo[4];  // slots 0, 2, 4, 6 of the column one to the right
#pragma unroll
    for (int k = 0; k < 4; ++k) xo[k] = par == 0 ? sm.xco[1][k][r] : sm.xco[0][k][r] >> 1;
    // ---- events, to the queue
    {
        uint32_t at = tail + (par == 0 ? 0u : sm.xev[0]) + incl - nev;
        while (ev) {
            const int l = __ffs(ev) - 1;
            ev &= ev - 1;
            sm.queue[at++ & (kQ - 1)] = uint16_t((p & 31) << 11 | r << 6 | (2 * l + par));
        }
        tail += sm.xev[0] + sm.xev[1];
    }
    // ---- the top cells between planes p - 1 and p: the slot that its largest
    // corner sees it in.  Upper corners (slots 0..3 of plane p's vertices) send
    // it to +z; plane p - 1's part comes from its own logic (sm.low).
    const bool last_z = p == t.D - 1;  // the top cells across +z lie outside
    const uint32_t up = st.co[3] | xo[1] | __shfl_down_sync(0xFFFFFFFFu, st.co[1] | xo[0], 1);
    const uint32_t py_new = __shfl_down_sync(0xFFFFFFFFu, st.co[5] | xo[2], 1);
    uint32_t* low = &sm.low[par][0][r];  // stride kTY
    const uint32_t py = low[0], px = low[kTY], s0 = low[2 * kTY], s1 = low[3 * kTY], s2 = low[4 * kTY],
                   s3 = low[5 * kTY];
    const uint32_t upi = last_z ? 0u : up, pyi = last_y ? 0u : py, pxi = px & ~t.last_x[par];
    uint32_t acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    // (the even columns' codes start at column 2, so that columns 1 + 8 k ..
    // 8 + 8 k are one aligned word of each parity)
    constexpr int sh = par == 0 ? 1 : 0;
    spread<0>(acc, st.h[0] >> sh);
    spread<1>(acc, st.h[1] >> sh);
    spread<2>(acc, st.h[2] >> sh);
    spread<3>(acc, (upi | pxi | s0 | ~cube) >> sh);
    spread<4>(acc, (pyi | pxi | s1 | ~cube) >> sh);
    spread<5>(acc, (s2 | ~cube) >> sh);
    spread<6>(acc, (up | py | px | s3 | ~cube) >> sh);
    uint4* dst = reinterpret_cast<uint4*>(&sm.code[p & 1][r][32 * par]);
    dst[0] = make_uint4(acc[0], acc[1], acc[2], acc[3]);
    dst[1] = make_uint4(acc[4], acc[5], acc[6], acc[7]);
    // plane p's part for the top cells above it
    uint32_t b0, b1, b2;
    slot7_target(st.co, b0, b1, b2);
    const uint32_t out = (~b0 & t.first_x[par]) | (first_y ? ~b1 : 0u) | (p == 0 ? ~b2 : 0u);
    const uint32_t self = st.co[7] & ~out;
    low[0] = py_new;
    low[kTY] = xo[3];
    low[2 * kTY] = self & b0;
    low[3 * kTY] = self & b1;
    low[4 * kTY] = self & b2;
    low[5 * kTY] = st.co[7] & out;
    return tail;
}

// 32 queued events (n: how many of them there are) from queue position `at`;
// k: a plane within 31 planes after theirs.  Keys, roots and ages go straight
// to the global arrays, with one atomic per array.
__device__ __noinline__ unsigned long long event_batch(Smem3& sm, const Outs& o, int k, uint32_t at, uint32_t n) {
    const Task3& t = sm.t;
    const unsigned lane = lane_id(), lt = (1u << lane) - 1u;
    const bool live = lane < n;
    const uint32_t e = live ? sm.queue[(at + lane) & (kQ - 1)] : 0u;
    const int x = t.x0 - 1 + int(e & 63u), y = t.y0 - 1 + int((e >> 6) & 31u), z = k - ((k - int(e >> 11)) & 31);
    bool root0 = false, rootT = false;
    uint32_t sv = 0, ord = 0, vl = 0;
    if (live) {
        vl = uint32_t(z) * t.HW + uint32_t(y) * uint32_t(t.W) + uint32_t(x);
        const float* c = t.img + vl;
        // neighbours outside the image: read the nearest inside, drop the bit
        const int dx[3] = {x > 0 ? -1 : 0, 0, x < t.W - 1 ? 1 : 0};
        const int64_t dy[3] = {y > 0 ? -int64_t(t.W) : 0, 0, y < t.H - 1 ? int64_t(t.W) : 0};
        const int64_t dz[3] = {z > 0 ? -int64_t(t.HW) : 0, 0, z < t.D - 1 ? int64_t(t.HW) : 0};
        Nbr P[3];
#pragma unroll
        for (int k = 0; k < 27; ++k) P[k / 9].v[(k / 3) % 3][k % 3] = __ldg(c + dz[k / 9] + dy[(k / 3) % 3] + dx[k % 3]);
        uint32_t raw = mask26(P[0], P[1], P[2]);
        if (z == 0) raw &= ~mask3_side(0, -1);
        if (z == t.D - 1) raw &= ~mask3_side(0, 1);
        if (y == 0) raw &= ~mask3_side(1, -1);
        if (y == t.H - 1) raw &= ~mask3_side(1, 1);
        if (x == 0) raw &= ~mask3_side(2, -1);
        if (x == t.W - 1) raw &= ~mask3_side(2, 1);
        const uint32_t rel = collapse3_lattice(raw);
        sv = __ldg(g_surv3d + hash_slot3(rel, g_disp3d));
        root0 = (rel & kM3Faces) == 0u;
        rootT = rel == kM3All;
        ord = ord_bits(P[1].v[1][1]);
    }
    const uint32_t vg = t.voff + vl;
    const uint32_t h0s = sv & 0x3Fu, ds = sv >> 6;
    const unsigned m_r0 = __ballot_sync(0xFFFFFFFFu, root0);
    const unsigned m_rt = __ballot_sync(0xFFFFFFFFu, rootT);
    const uint32_t n0 = __reduce_add_sync(0xFFFFFFFFu, uint32_t(__popc(h0s)));
    const uint32_t nt = __reduce_add_sync(0xFFFFFFFFu, uint32_t(__popc(ds)));
    // lanes 0 .. 3 take room in the four arrays
    uint32_t base = 0;
    {
        const uint32_t want = lane == 0 ? n0 : (lane == 1 ? nt : (lane == 2 ? __popc(m_r0) : __popc(m_rt)));
        uint32_t* c = lane == 0 ? &o.ctr->n_s0 : (lane == 1 ? &o.ctr->n_st : (lane == 2 ? &o.ctr->n_r0 : &o.ctr->n_rt));
        const uint32_t cap = lane < 2 ? o.cap_s : (lane == 2 ? o.cap_r0 : o.cap_rt);
        if (lane < 4 && want) {
            base = atomicAdd(c, want);
            if (base + want > cap) set_status(o.ctr, kStCapacity);
        }
    }
    uint32_t b0 = __shfl_sync(0xFFFFFFFFu, base, 0), bt = __shfl_sync(0xFFFFFFFFu, base, 1);
    const uint32_t g0 = __shfl_sync(0xFFFFFFFFu, base, 2) + __popc(m_r0 & lt);
    const uint32_t gt = __shfl_sync(0xFFFFFFFFu, base, 3) + __popc(m_rt & lt);
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
    t.pitch = uint32_t(it.pitch);
    t.item = ii;
    t.code = o.code + it.coff;
    t.map = map;
    __syncthreads();  // everything in shared memory may still be read by the previous task
    if (threadIdx.x == 0) {
        Task3 u = t;
        const int xm = u.W - u.x0;  // tile column of the last image column
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            u.own[k] = col_mask(1, min(kOX, xm), k);
            u.cube[k] = col_mask(1, min(kOX, xm - 1), k);
            u.first_x[k] = col_mask(1 - u.x0, 1 - u.x0, k);
            u.last_x[k] = col_mask(xm - 1, xm - 1, k);
        }
        sm.t = u;
        sm.tail[0] = sm.tail[1] = 0;
    }
    if (!map) {  // positions outside the image stay +inf for the whole task
        for (int i = threadIdx.x; i < kRH * kRW; i += kT3 + 64) {
            const int ly = i / kRW, c = i - ly * kRW;
            if (unsigned(t.y0 - 2 + ly) >= unsigned(it.H) || unsigned(t.x0 - 2 + c) >= unsigned(it.W))
                for (int s = 0; s < kRing; ++s) sm.ring[s][ly * kRS + kRX + c] = __int_as_float(0x7F800000);
        }
    } else if (threadIdx.x == 0) {
        // counted in blocks of 31 x 8 columns by the tuned number of planes, whatever the tile
        auto blocks = [](int lo, int hi, int n) { return uint32_t((hi + n - 1) / n - (lo + n - 1) / n); };
        atomicAdd(&o.ctr->tma_tasks, blocks(t.x0, min(t.x0 + kOX, it.W), 31) * blocks(t.y0, min(t.y0 + kOY, it.H), 8) *
                                         blocks(t.z0, t.z1, tab.zchunk3d));
    }
    __syncthreads();
    // The code of a vertex holds the dual link of the top cell below it, which
    // needs the logic of the plane before: planes first .. zlast are compared
    // and first + 1 .. zlast go through the logic, the first of them only for
    // the top cells above it.  Planes first .. zlast + 1 are read.
    const int first = max(t.z0 - 2, -1);
    //   compare warps, step k: wait for the codes of plane k - 2 (which come
    //     with plane k + 1 in the ring); output plane k - 2, events; compare
    //     plane k
    //   logic warps, step k: wait for the words of plane k (the compare of
    //     plane k was the last to read it); request plane k + 3 into its slot;
    //     logic of plane k; wait for plane k + 3 to land
    if (warp >= kW3) {
        const bool even = warp == kW3;  // this warp also brings the planes in
        // positions outside the image, next to it, are set to +inf in every
        // plane (TMA path): columns x = -1 and x = W, rows y = -1 and y = H
        const bool edge = t.x0 == 0 || t.y0 == 0 || t.x0 - 1 + kTX > t.W || t.y0 - 1 + kTY > t.H;
        auto request = [&](int z) {
            if (z <= t.zlast + 1 && unsigned(z) < unsigned(t.D) && map && even && lane == 0) issue_tma(sm, t, z);
        };
        auto landed = [&](int z) {
            if (z > t.zlast + 1) return;
            float* plane = sm.ring[ring_slot(z)];
            if (unsigned(z) >= unsigned(t.D)) {  // a plane outside the volume: every position +inf
                if (even)
                    for (int i = lane; i < kRH * kRS; i += 32) plane[i] = __int_as_float(0x7F800000);
            } else if (map) {
                wait_plane(sm, t, z, par, o.ctr);
                if (edge && even) {
#pragma unroll
                    for (int n = 0; n < kFix; ++n) {
                        const int i = lane + 32 * n, j = i - 2 * kRH;
                        const int c = j < 0 ? (i < kRH ? 1 - t.x0 : t.W + 2 - t.x0) : (j < kRW ? j : j - kRW);
                        const int r = j < 0 ? (i < kRH ? i : i - kRH) : (j < kRW ? 1 - t.y0 : t.H + 2 - t.y0);
                        if (j < 2 * kRW && unsigned(c) < unsigned(kRW) && unsigned(r) < unsigned(kRH))
                            plane[r * kRS + kRX + c] = __int_as_float(0x7F800000);
                    }
                }
            }
        };
#pragma unroll 1
        for (int z = first; z < first + 3; ++z) request(z);
#pragma unroll 1
        for (int z = first; z < first + 2; ++z) landed(z);
        bar_arrive(kBarCodes + (first & 1));
        landed(first + 2);
        bar_arrive(kBarCodes + ((first + 1) & 1));
        uint32_t tail = 0;
        int sc = 0;  // word slot of plane k
#pragma unroll 1
        for (int k = first; k <= t.zlast; ++k) {
            bar_sync(kBarWords + (k & 1));
            request(k + 3);
            if (k > first) {
                const uint32_t(*wl)[kWR] = sm.w[sc == 0 ? 2 : sc - 1];
                tail = even ? logic_plane<0>(sm, k, sm.w[sc], wl, tail) : logic_plane<1>(sm, k, sm.w[sc], wl, tail);
            }
            if (even && lane == 0) sm.tail[k & 1] = tail;
            landed(k + 3);
            bar_arrive(kBarCodes + (k & 1));
            sc = sc == 2 ? 0 : sc + 1;
        }
        return;
    }
    float top_a = 0.0f, top_b = 0.0f;  // largest magnitude of this lane's columns (NaN if one is)
    unsigned long long gmin = ~0ull;
    uint32_t head = 0;  // events taken from the queue
    int oldest = t.z0;  // no queued event lies before this plane
    int sc = 0;         // word slot of plane k
    if (!map) {
        for (int z = first; z < first + 2; ++z) issue_rows(sm, t, z);
        cp_async_commit();
    }
#pragma unroll 1
    for (int k = first; k <= t.zlast + 2; ++k) {
        const int p = k - 2;
        bar_sync(kBarCodes + (p & 1));
        if (!map) {
            asm volatile("bar.sync %0, %1;" ::"n"(kBarRows), "n"(kT3) : "memory");  // plane k - 1 has been compared
            issue_rows(sm, t, k + 2);                                               // into its slot
            cp_async_commit();
            cp_async_wait<1>();
            asm volatile("bar.sync %0, %1;" ::"n"(kBarRows), "n"(kT3) : "memory");  // plane k + 1 is there
        }
        const uint32_t tail = p >= t.z0 ? sm.tail[p & 1] : 0u;
        if (p >= t.z0) {
            // the codes of plane p: 8 columns (two words) of an owned row per thread and turn
            uint8_t* plane = t.code + uint64_t(uint32_t(p) * uint32_t(t.H)) * t.pitch + uint32_t(t.x0);
#pragma unroll 1
                for (int i = threadIdx.x; i < 8 * kOY; i += kT3) {
                    const int r = 1 + (i >> 3), c = i & 7, y = t.y0 - 1 + r;
                    const uint32_t ev = *reinterpret_cast<const uint32_t*>(&sm.code[p & 1][r][4 * c]);
                    const uint32_t od = *reinterpret_cast<const uint32_t*>(&sm.code[p & 1][r][32 + 4 * c]);
                    const uint32_t x = 8u * c;
                    uint8_t* dst = plane + uint64_t(uint32_t(y)) * t.pitch + x;
                    if (y < t.H && uint32_t(t.x0) + x < t.pitch) {
                        put_code(o, dst, __byte_perm(od, ev, 0x5140));
                        if (c < 7 && uint32_t(t.x0) + x + 4 < t.pitch) put_code(o, dst + 4, __byte_perm(od, ev, 0x7362));
                    }
                }
        }
        if (tail - head >= uint32_t(kQMin) || (tail != head && (k - oldest >= kQAge || k == t.zlast + 2))) {
            for (uint32_t at = head + 32u * warp; at < tail; at += kT3) {
                const unsigned long long g = event_batch(sm, o, k, at, min(32u, tail - at));
                gmin = g < gmin ? g : gmin;
            }
            head = tail;
        }
        if (tail == head) oldest = p + 1;
        if (k <= t.zlast) {
            if (k < 0) {  // a plane outside the volume: all ones
                wait_plane(sm, t, k + 1, par, o.ctr);
                for (int i = threadIdx.x; i < kTY * kWR; i += kT3) (&sm.w[sc][0][0])[i] = 0xFFFFFFFFu;
            } else {
                if (k == first) wait_plane(sm, t, k, par, o.ctr);
                wait_plane(sm, t, k + 1, par, o.ctr);
                compare_rows(sm.ring[ring_slot(k)], sm.ring[ring_slot(k + 1)], sm.w[sc], warp, lane, top_a, top_b,
                             t.y0 - 1 + warp * kRows, t.H);
            }
            bar_arrive(kBarWords + (k & 1));
            sc = sc == 2 ? 0 : sc + 1;
        }
    }
    if (!map) cp_async_wait<0>();
    const bool in_a = unsigned(t.x0 - 1 + 2 * lane) < unsigned(t.W), in_b = unsigned(t.x0 + 2 * lane) < unsigned(t.W);
    const bool bad = (in_a && !(top_a <= 3.40282347e38f)) || (in_b && !(top_b <= 3.40282347e38f));
    if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) set_status(o.ctr, kStNonfinite);
    gmin = warp_min_u64(gmin);
    if (lane == 0 && gmin != ~0ull) atomicMin(&o.ctr->gmin[ii], gmin);
}

__global__ void __launch_bounds__(kT3 + 64, 3) k_prune3d(const __grid_constant__ ItemTable tab, const __grid_constant__ Outs o,
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

// The words of a 3D item's forests from its codes, as the 2D pass writes them
// (roots have theirs already).
__global__ void __launch_bounds__(256) k_expand3d(const __grid_constant__ ItemTable tab, const __grid_constant__ Outs o) {
    for (int j = tab.n2d; j < tab.n; ++j) {
        const Item& it = tab.it[j];
        const int64_t n = int64_t(it.D) * it.H * it.W;
        for (int64_t v = int64_t(blockIdx.x) * 256 + threadIdx.x; v < n; v += int64_t(gridDim.x) * 256) {
            const int x = int(v % it.W), y = int((v / it.W) % it.H), z = int(v / (int64_t(it.W) * it.H));
            const uint32_t c = o.code[it.coff + (int64_t(z) * it.H + y) * it.pitch + x];
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
// Each warp marches down a strip of one image on its own (no block
// barriers): lane l handles column x0-1+l; lanes 1..31 own their columns (31
// per strip), lane 0 is a halo whose lookup codes the top cells of column
// x0-1 need.  The task owns rows [y0, y1) and computes lookups for rows
// [y0, min(y1, H-1)].
//
// Per row step y:
//  1. cp.async prefetch of row y+kAhead2 (columns x0-2 .. x0+31) into the
//     warp's 8-row shared-memory ring; out-of-image positions read +inf;
//  2. the 8-neighbour mask of (y, x) from registers (rows y-1, y) and the
//     ring (row y+1), direct table lookup, the H0 forest link (an up link
//     continues the chain of (y-1, x), the same lane's previous step) and
//     the survivors and H0 root of owned vertices;
//  3. the top cell whose smallest corner is (y-1, x): its largest corner m
//     among the 4 corner values holds, in its entry, where the top cell dies
//     locally; the codes of rows y-1 and y of column x+1 come by shuffle, so
//     each lane stores one coalesced dual forest link (or a dual root).
constexpr int kW2 = 8;                   // warps per CTA (independent tasks)
constexpr int kOX2 = 31;                 // owned columns per strip
constexpr int kRW2 = 34;                 // ring row: columns x0-2 .. x0+31
constexpr int kRing2 = 8, kAhead2 = 5;   // ring rows, rows in flight
constexpr int kCap2 = 32 * 4;            // staged keys per warp and kind (one step's maximum)
constexpr int kCapWR = 32;               // staged roots per warp and kind

struct WarpStage2 {
    uint64_t s0[kCap2];
    uint64_t st[kCap2];
    uint64_t r0age[kCapWR];
    uint64_t rtage[kCapWR];
    uint32_t r0node[kCapWR];
    uint32_t rtnode[kCapWR];
    uint8_t r0item[kCapWR];
    uint8_t rtitem[kCapWR];
};

struct Smem2 {
    uint2 lut[256];
    float ring[kW2][kRing2][kRW2];
    WarpStage2 ws[kW2];
};

struct WarpCounts {
    uint32_t s0, st, r0, rt;
};

template <class WS>
__device__ __forceinline__ void warp_flush(WS& ws, WarpCounts& c, const Outs& o) {
    __syncwarp();
    const unsigned lane = lane_id();
    uint32_t b0 = 0, bt = 0, br0 = 0, brt = 0;
    if (lane == 0) {
        if (c.s0) b0 = atomicAdd(&o.ctr->n_s0, c.s0);
        if (c.st) bt = atomicAdd(&o.ctr->n_st, c.st);
        if (c.r0) br0 = atomicAdd(&o.ctr->n_r0, c.r0);
        if (c.rt) brt = atomicAdd(&o.ctr->n_rt, c.rt);
        bool over = (c.s0 && b0 + c.s0 > o.cap_s) || (c.st && bt + c.st > o.cap_s) ||
                    (c.r0 && br0 + c.r0 > o.cap_r0) || (c.rt && brt + c.rt > o.cap_rt);
        if (over) set_status(o.ctr, kStCapacity);
    }
    b0 = __shfl_sync(0xFFFFFFFFu, b0, 0);
    bt = __shfl_sync(0xFFFFFFFFu, bt, 0);
    br0 = __shfl_sync(0xFFFFFFFFu, br0, 0);
    brt = __shfl_sync(0xFFFFFFFFu, brt, 0);
    for (uint32_t i = lane; i < c.s0; i += 32)
        if (b0 + i < o.cap_s) o.s0[b0 + i] = ws.s0[i];
    for (uint32_t i = lane; i < c.st; i += 32)
        if (bt + i < o.cap_s) o.st[bt + i] = ws.st[i];
    for (uint32_t i = lane; i < c.r0; i += 32)
        if (CP_IN(ws.r0node[i], o.n_uf0, o.ctr))
            put_root(o.uf0 + ws.r0node[i], br0 + i, o.cap_r0, ws.r0age[i], o.node0, o.age0, o.res0, false, ws.r0item[i]);
    for (uint32_t i = lane; i < c.rt; i += 32)
        if (CP_IN(ws.rtnode[i], o.n_uft, o.ctr))
            put_root(o.uft + ws.rtnode[i], brt + i, o.cap_rt, ws.rtage[i], o.nodet, o.aget, o.rest, true, ws.rtitem[i]);
    c.s0 = c.st = c.r0 = c.rt = 0;
    __syncwarp();
}

struct Row {
    float l, c, r;  // columns x-1, x, x+1
};

__device__ __forceinline__ void read_row(const float* slot, int lane, Row& R) {
    R.l = slot[lane];
    R.c = slot[lane + 1];
    R.r = slot[lane + 2];
}

struct RowPos {
    const float* img;
    uint32_t W, H;
    int gx0, gx1;     // image columns copied by this lane
    int idx1;         // ring position of the second column
    bool in0, in1;    // inside the image
};

// kCheck false: the caller knows that row y lies inside the image
template <bool kCheck = true>
__device__ __forceinline__ void issue_row(float (*ring)[kRW2], const RowPos& p, int lane, int y) {
    float* slot = ring[(y + kRing2) & (kRing2 - 1)];
    if (!kCheck || unsigned(y) < p.H) {
        const float* base = p.img + uint32_t(y) * p.W;
        if (p.in0) cp_async4(slot + lane + 1, base + p.gx0);
        if (p.in1) cp_async4(slot + p.idx1, base + p.gx1);
    } else {  // a row outside the image: every position +inf
        const float inf = __int_as_float(0x7F800000);
        if (p.in0) slot[lane + 1] = inf;
        if (p.in1) slot[p.idx1] = inf;
    }
    cp_async_commit();
}

__global__ void __launch_bounds__(kW2 * 32) k_prune2d(ItemTable tab, Outs o) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem2& sm = *reinterpret_cast<Smem2*>(smem_raw);
    const int warp = threadIdx.x >> 5;
    const int lane = int(lane_id());
    const unsigned lt = (1u << lane) - 1u;
    for (int i = threadIdx.x; i < 256; i += kW2 * 32) sm.lut[i] = g_lut2d[i];
    __syncthreads();
    WarpStage2& ws = sm.ws[warp];
    float(*ring)[kRW2] = sm.ring[warp];
    WarpCounts cnt = {0, 0, 0, 0};
    const float inf = __int_as_float(0x7F800000);
    for (int task = blockIdx.x * kW2 + warp; task < tab.tiles2d; task += gridDim.x * kW2) {
        const int ii = tile_item(tab, 0, tab.n2d - 1, task);
        const Item& it = tab.it[ii];
        const int ltask = task - it.tile0;
        const int x0 = (ltask % it.tx) * kOX2, y0 = (ltask / it.tx) * tab.rows2d;
        const int y1 = min(it.H, y0 + tab.rows2d);  // owned rows [y0, y1)
        const int ylast = min(y1, it.H - 1);        // lookups for rows [y0, ylast]
        const int x = x0 - 1 + lane;
        const uint32_t W = uint32_t(it.W), H = uint32_t(it.H), W1 = W - 1u;
        const uint32_t voff = uint32_t(it.voff), toff = uint32_t(it.toff), OUT = uint32_t(it.toff + it.T);
        const bool owned_x = lane >= 1 && x < it.W;
        const bool cube_x = lane <= 30 && x >= 0 && x < it.W - 1;
        RowPos rp;
        rp.img = it.img;
        rp.W = W;
        rp.H = H;
        rp.gx0 = x;
        rp.in0 = unsigned(x) < W;
        rp.gx1 = lane == 0 ? x0 - 2 : x0 + 31;
        rp.idx1 = lane == 0 ? 0 : kRW2 - 1;
        rp.in1 = (lane == 0 || lane == 31) && unsigned(rp.gx1) < W;
        const bool has1 = lane == 0 || lane == 31;
        __syncwarp();  // the ring may still be read by the previous task
#pragma unroll
        for (int s = 0; s < kRing2; ++s) {
            if (!rp.in0) ring[s][lane + 1] = inf;
            if (has1 && !rp.in1) ring[s][rp.idx1] = inf;
        }
#pragma unroll
        for (int k = -1; k < kAhead2; ++k) issue_row(ring, rp, lane, y0 + k);
        cp_async_wait<kAhead2 - 2>();  // rows y0-1 .. y0+1 have landed
        __syncwarp();
        Row A, B, C;
        read_row(ring[(y0 - 1 + kRing2) & (kRing2 - 1)], lane, A);
        read_row(ring[y0 & (kRing2 - 1)], lane, B);
        unsigned long long my_min = ~0ull;
        uint32_t far = 0, far_t = 0, cprev = 0;  // last H0 link / dual link written by this lane
        bool nonfinite = false;                   // an owned value is NaN or infinite (checked once per task)
        // interior: a std::integral_constant; true for a row with y >= y0 + 2 and
        // y + kAhead2 <= ylast, where no boundary row or end-of-task case arises
        auto step = [&](const int y, auto interior) {
            constexpr bool kIn = decltype(interior)::value;
            issue_row<!kIn>(ring, rp, lane, y + kAhead2);
            read_row(ring[(y + 1) & (kRing2 - 1)], lane, C);
            // ---- lookup of (y, x): bit i of the mask is stencil offset n = i (i < 4) or
            // i + 1 (i >= 4); offsets before the centre in linear order precede on ties
            const float cv = B.c;
            uint32_t raw = 0;
            or_if_precedes<1u << 0, true>(raw, A.l, cv);
            or_if_precedes<1u << 1, true>(raw, A.c, cv);
            or_if_precedes<1u << 2, true>(raw, A.r, cv);
            or_if_precedes<1u << 3, true>(raw, B.l, cv);
            or_if_precedes<1u << 4, false>(raw, B.r, cv);
            or_if_precedes<1u << 5, false>(raw, C.l, cv);
            or_if_precedes<1u << 6, false>(raw, C.c, cv);
            or_if_precedes<1u << 7, false>(raw, C.r, cv);
            const uint2 e = sm.lut[raw];
            const bool owned = owned_x && (kIn || y < y1);
            const uint32_t ord = ord_bits(cv);
            const uint32_t vl = uint32_t(y) * W + uint32_t(x);
            const uint32_t vg = voff + vl;
            const uint32_t direct = e.x & 7u;
            // H0: a local minimum becomes a root (registered in the staging block
            // below); otherwise the link along the first edge (face slots: up,
            // left, right, down), where a link up continues the chain that this
            // lane started one row before
            const bool root0 = owned && direct == 7u;
            nonfinite |= owned && !(fabsf(cv) <= 3.40282347e38f);
            {
                const uint32_t mag = (direct == 0u || direct == 3u) ? W : 1u;
                const uint32_t u = direct < 2u ? vg - mag : vg + mag;
                if (owned) far = root0 ? vg : ((direct == 0u && (kIn || y > y0)) ? far : u);
                if (owned && !root0 && CP_IN(vg, o.n_uf0, o.ctr)) o.uf0[vg] = far;
            }
            const uint32_t h0s = owned ? (e.x >> 3) & 0xFu : 0u;
            const uint32_t ds = owned ? (e.x >> 9) & 0xFu : 0u;
            // cross-pruning: dual survivors that are also H0 survivors wait for the
            // H0 union-find (flag bit of the H0 key); otherwise every dual survivor
            // goes to the dual list now (one that kills an H0 class closes a dual
            // cycle there: a no-op)
            const uint32_t flg = tab.cross2d ? ds : 0u;
            const uint32_t dn = tab.cross2d ? ds & ~h0s : ds;
            // ---- the top cell with smallest corner (y-1, x): its largest corner m
            // (value, then linear index) holds it; m's code field for it says where
            // it dies locally (8: a dual root, registered in the staging block
            // below; 15: not held, non-finite input only)
            const uint32_t cprev_r = __shfl_down_sync(0xFFFFFFFFu, cprev, 1);
            const uint32_t ccur_r = __shfl_down_sync(0xFFFFFFFFu, e.y, 1);
            const bool cube = cube_x && (kIn || y > y0);
            const float cvals[4] = {A.c, A.r, B.c, B.r};
            int k = 0;
            float best = cvals[0];
#pragma unroll
            for (int j = 1; j < 4; ++j) {
                const bool ge = cvals[j] >= best;
                best = ge ? cvals[j] : best;
                k = ge ? j : k;
            }
            const uint32_t word = k == 0 ? cprev : (k == 1 ? cprev_r : (k == 2 ? e.y : ccur_r));
            const uint32_t t = uint32_t(3 - k);  // quadrant of the top cell as seen from m
            const uint32_t code = (word >> (4u * t)) & 15u;
            const uint32_t self = toff + uint32_t(y - 1) * W1 + uint32_t(x);
            const bool rootT = cube && code == 8u;
            {
                // the top cell across: quadrant `code` of m, smallest corner m - (negative axes)
                const int my = y - 1 + (k >> 1), mx = x + (k & 1);
                const int ty = my - int(((code >> 1) & 1u) ^ 1u);
                const int tx = mx - int((code & 1u) ^ 1u);
                const bool out = unsigned(ty) >= H - 1u || unsigned(tx) >= W1;
                // a link to (y-2, x) continues the chain that this lane wrote for that top
                // cell in the previous step; a code of 15 writes a root tag to keep the
                // forest well formed
                const bool chain = ty == y - 2 && tx == x && (kIn || y - 1 > y0);
                const uint32_t tgt = code < 4u ? (out ? OUT : toff + uint32_t(ty) * W1 + uint32_t(tx)) : kTag;
                if (cube) far_t = rootT ? self : ((code < 4u && chain) ? far_t : tgt);
                if (cube && !rootT && CP_IN(self, o.n_uft, o.ctr)) o.uft[self] = far_t;
            }
            cprev = e.y;
            // ---- stage survivors and roots
            if (__any_sync(0xFFFFFFFFu, root0 || rootT || (h0s | dn) != 0u)) {
                const unsigned m_r0 = __ballot_sync(0xFFFFFFFFu, root0);
                const unsigned m_rt = __ballot_sync(0xFFFFFFFFu, rootT);
                const uint32_t or0 = __reduce_or_sync(0xFFFFFFFFu, h0s);
                const uint32_t ort = __reduce_or_sync(0xFFFFFFFFu, dn);
                const uint32_t n0 = __reduce_add_sync(0xFFFFFFFFu, uint32_t(__popc(h0s)));  // <= 32 * 4
                const uint32_t nt = __reduce_add_sync(0xFFFFFFFFu, uint32_t(__popc(dn)));   // <= 32 * 4
                if (cnt.s0 + n0 > uint32_t(kCap2) || cnt.st + nt > uint32_t(kCap2) ||
                    cnt.r0 + __popc(m_r0) > uint32_t(kCapWR) || cnt.rt + __popc(m_rt) > uint32_t(kCapWR))
                    warp_flush(ws, cnt, o);
                if (m_r0) {
                    if (root0) {
                        const uint32_t p = cnt.r0 + __popc(m_r0 & lt);
                        ws.r0node[p] = vg;
                        ws.r0item[p] = uint8_t(ii);
                        ws.r0age[p] = make_key(ord, vg, 0);
                        const unsigned long long kk = (unsigned long long)(uint64_t(ord) << 32 | vl);
                        my_min = kk < my_min ? kk : my_min;
                    }
                    cnt.r0 += __popc(m_r0);
                }
                if (m_rt) {
                    if (rootT) {
                        const uint32_t my = uint32_t(y - 1 + (k >> 1)), mx = uint32_t(x + (k & 1));
                        const uint32_t mg = voff + my * W + mx;
                        const uint32_t p = cnt.rt + __popc(m_rt & lt);
                        ws.rtnode[p] = self;
                        ws.rtitem[p] = uint8_t(ii);
                        ws.rtage[p] = make_key(ord_bits(best), mg, (6u * (t >> 1) + 2u * (t & 1u)) << 1);
                    }
                    cnt.rt += __popc(m_rt);
                }
                uint32_t bits = or0;
                while (bits) {
                    const int s = __ffs(bits) - 1;
                    bits &= bits - 1;
                    const bool mine = (h0s >> s) & 1u;
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, mine);
                    if (mine)  // face slot s is stencil offset 2s+1; low bit: the dual waits for it
                        ws.s0[cnt.s0 + __popc(m & lt)] = make_key(ord, vg, (uint32_t(2 * s + 1) << 1) | ((flg >> s) & 1u));
                    cnt.s0 += __popc(m);
                }
                bits = ort;
                while (bits) {
                    const int f = __ffs(bits) - 1;
                    bits &= bits - 1;
                    const bool mine = (dn >> f) & 1u;
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, mine);
                    if (mine) ws.st[cnt.st + __popc(m & lt)] = ~make_key(ord, vg, uint32_t(2 * f + 1) << 1);
                    cnt.st += __popc(m);
                }
                __syncwarp();
            }
            cp_async_wait<kAhead2 - 2>();  // row y+2 has landed (for the next step)
            __syncwarp();
            A = B;
            B = C;
        };
        // the first two rows and the last few take every check; the interior rows
        // are a second instantiation of the step without them
        int y = y0;
        for (; y <= ylast && y < y0 + 2; ++y) step(y, std::false_type());
        for (; y + kAhead2 <= ylast; ++y) step(y, std::true_type());
        for (; y <= ylast; ++y) step(y, std::false_type());
        if (__any_sync(0xFFFFFFFFu, nonfinite) && lane == 0) set_status(o.ctr, kStNonfinite);
        cp_async_wait<0>();
        const unsigned long long w = warp_min_u64(my_min);
        if (lane == 0 && w != ~0ull) atomicMin(&o.ctr->gmin[ii], w);
    }
    if (__any_sync(0xFFFFFFFFu, (cnt.s0 | cnt.st | cnt.r0 | cnt.rt) != 0)) warp_flush(ws, cnt, o);
}

// ---------------------------------------------------------------- host side
size_t prune_smem2d() { return sizeof(Smem2); }
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
int prune_tile_x() { return kOX2; }
int prune_tile_x3d() { return kOX; }
int g_rows2d = 64, g_zchunk3d = kZC, g_ctas3d = 0, g_cross2d = 0, g_uf_variant = 0;  // tuning (cp_set_tuning)
int prune_tile_y2d() { return g_rows2d; }
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
        case 7:  // union-find design: reservation rounds (0) or Borůvka's forest first (1)
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

// Table entry as two 32-bit words:
//   x: direct (3 bits) | h0_surv << 3 (6) | dual_surv << 9 (12) | in_l << 21 (8)
//   y: the eight 4-bit dual codes
static uint2 pack_entry(uint64_t v) {
    const uint32_t direct = uint32_t(v & 7u), h0s = uint32_t((v >> 3) & 0x3Fu);
    const uint32_t ds = uint32_t((v >> 41) & 0xFFFu), in_l = uint32_t((v >> 53) & 0xFFu);
    uint2 r;
    r.x = direct | (h0s << 3) | (ds << 9) | (in_l << 21);
    r.y = uint32_t((v >> 9) & 0xFFFFFFFFu);
    return r;
}

cudaError_t upload_luts(const uint64_t* lut2d, const uint16_t* disp3d, const uint64_t* entries3d,
                        const uint32_t* keys3d) {
    uint2 p2[256];
    for (int i = 0; i < 256; ++i) p2[i] = pack_entry(lut2d[i]);
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
    if (tab.n3d < 1) return cudaSuccess;
    k_expand3d<<<device_sm_count() * 8, 256, 0, s>>>(tab, outs_of(po));
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_prune(const ItemTable& tab, const PruneOuts& po, const TmaMaps& maps, cudaStream_t s) {
    const Outs o = outs_of(po);
    const int blocks3d = device_cached(kCachePrune3d, [] {
        cudaFuncSetAttribute(k_prune3d, cudaFuncAttributeMaxDynamicSharedMemorySize, int(prune_smem3d()));
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_prune3d, kT3 + 64, prune_smem3d());
        return device_sm_count() * (per_sm > 0 ? per_sm : 1);
    });
    const int blocks2d = device_cached(kCachePrune2d, [] {
        cudaFuncSetAttribute(k_prune2d, cudaFuncAttributeMaxDynamicSharedMemorySize, int(prune_smem2d()));
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_prune2d, kW2 * 32, prune_smem2d());
        return device_sm_count() * (per_sm > 0 ? per_sm : 1);
    });
    if (tab.tiles2d > 0) {
        const int need2 = (tab.tiles2d + kW2 - 1) / kW2;
        k_prune2d<<<need2 < blocks2d ? need2 : blocks2d, kW2 * 32, prune_smem2d(), s>>>(tab, o);
        note_launches(1);
    }
    if (tab.tiles3d > 0) {
        int cap = blocks3d;
        if (g_ctas3d > 0) cap = device_sm_count() * g_ctas3d < blocks3d ? device_sm_count() * g_ctas3d : blocks3d;
        int grid = tab.tiles3d < cap ? tab.tiles3d : cap;
        k_prune3d<<<grid, kT3 + 64, prune_smem3d(), s>>>(tab, o, maps);
        note_launches(1);
    }
    return cudaGetLastError();
}

}  // namespace cp
