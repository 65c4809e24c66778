// Walks through the pruned forests, from a survivor's two endpoints to the
// roots of their classes.
//
// Both are in a code byte per vertex; of the 32-bit arrays only a root's word
// is written (its root id).
//
// 3D items: 29 rows of a column of a plane at a time in one 32-byte sector
// (code_at3: a column of a pruning tile), bits 0-2 the vertex's H0 link (face slot 0..5, 6: a root, 7: a frame vertex of a T-filtration
// item, whose root is vertex 0), bits 3-6 the dual link of the top cell with
// its smallest corner one plane below, at (z - 1, y, x) (0..6: towards that
// slot as seen from that corner, 7: a root, 8: the outside, 9, 10, 11: +z, +y,
// +x).  A 512^3 volume's codes (134 MB) mostly stay in L2 between the pruning
// pass and the walks, where words (1,074 MB) did not.
//
// 2D items: 30 rows of a column at a time in one 32-byte sector (code_at2: a
// column of a pruning tile), bits 0-3 the H0 link (0..4: up by 1 << d rows, all
// of whose vertices but the last link up; 5, 6, 7: left, right, down by one, 8,
// 9, 10: by four, 11: down by 16, likewise; 14: a root, 15: the frame as above),
// bits 4-7 the dual link of the top cell with its smallest corner there (0..4:
// +y by 1 << d, likewise; 5..8: +x, -x, -y, both; 9: the outside; 10, 11, 12:
// +x, -x, -y by four, 13: -y by 16, likewise; 15: a root).  Runs end where the
// tile does.  The runs shorten long straight descents: with runs of links up
// and +y alone, the walks of 2048^2 straight valleys took 337 us (falling along
// +y) and 670 us (along x) and take 91 and 284; ordinary fields' differ little
// (2048^2 noise 89 -> 84 us, 4096^2 blurred 46 -> 39), and the pruning pass pays
// 2 us at 4096^2 for them.
#pragma once
#include "cp_common.cuh"

namespace cp {

// Offset of the 3D link with code field d (H0: 0..5; dual: 0..6, 9..11) between
// ids, with hp and p the plane's and the row's.
__host__ __device__ __forceinline__ int32_t link_offset3(int dual, uint32_t d, int32_t hp, int32_t p) {
    if (!dual) {
        const int32_t m = (d == 0u || d == 5u) ? hp : ((d == 1u || d == 4u) ? p : 1);
        return d < 3u ? -m : m;
    }
    if (d < 8u) return ((d & 4u) ? 0 : -hp) + ((d & 2u) ? 0 : -p) + ((d & 1u) ? 0 : -1);
    return d == 9u ? hp : (d == 10u ? p : 1);
}

constexpr int kTile2 = 30;  // rows (and columns) of a 2D pruning tile
constexpr int kBand3 = 29;  // rows of a warp's part of a 3D pruning tile

// Where vertex (y, x) of a 2D item has its code byte (its first byte is the
// item's).
__host__ __device__ __forceinline__ uint32_t code_at2(const Item& it, int y, int x) {
    const uint32_t t = uint32_t(y) / uint32_t(kTile2);
    return (t * uint32_t(it.W) + uint32_t(x)) * 32u + (uint32_t(y) - t * uint32_t(kTile2));
}

// The same for vertex (z, y, x) of a 3D item.
__host__ __device__ __forceinline__ uint32_t code_at3(const Item& it, int z, int y, int x) {
    const uint32_t b = uint32_t(y) / uint32_t(kBand3);
    return ((uint32_t(z) * uint32_t(it.bands) + b) * uint32_t(it.W) + uint32_t(x)) * 32u + (uint32_t(y) - b * uint32_t(kBand3));
}

// Offset of the 2D link with code field d (H0: 0..11; dual: 0..8, 10..13), a
// signed byte for each of the 16 fields (0: no step).
struct Offsets2 {
    uint32_t y[4], x[4];
};
__host__ __device__ __forceinline__ Offsets2 offsets2(int dual) {
    return dual ? Offsets2{{0x08040201u, 0xFF000010u, 0x000000FFu, 0x0000F0FCu}, {0u, 0x00FF0100u, 0xFC0400FFu, 0u}}
                : Offsets2{{0xF8FCFEFFu, 0x010000F0u, 0x10040000u, 0u}, {0u, 0x0001FF00u, 0x000004FCu, 0u}};
}
__host__ __device__ __forceinline__ void link_offset2(int dual, uint32_t d, int& dy, int& dx) {
    const Offsets2 o = offsets2(dual);
    dy = int8_t(o.y[d >> 2] >> (8u * (d & 3u)));
    dx = int8_t(o.x[d >> 2] >> (8u * (d & 3u)));
}

#ifdef __CUDACC__
struct Forest {
    const uint32_t* uf;    // root words
    const uint8_t* code;   // codes
    uint32_t n_nodes;      // entries of uf / code (bounds-checked build)
    uint64_t n_code;
    int dual;
};

// One endpoint's path in an item's codes: where it is, and whether it has
// reached the outside (which has no code).
struct Path {
    uint32_t at;
    bool out;
};

// What a link does, by its code field d, without branches, so that both paths
// of every lane have a load in flight all the time.  A code that is no step
// leaves the path where it is.  Bound by the latency of these loads (L2, or L1
// for steps along a sector); with a branch per kind of link and path, k_roots2
// took 185 us at 512^3 instead of 108, 84 instead of 59 for 128^3 noise.
//
// 3D: per unit of z, y and x, two bits at 2 d hold the offset + 1.
template <class... P>
constexpr uint32_t step_field(uint32_t w, uint32_t d, uint32_t v, P... rest) {
    w = (w & ~(3u << (2 * d))) | v << (2 * d);
    if constexpr (sizeof...(rest) > 0) return step_field(w, rest...);
    return w;
}
constexpr uint32_t kStay = 0x55555555u;
// H0: -z -y -x +x +y +z
constexpr uint32_t kStepZ0 = step_field(kStay, 0u, 0u, 5u, 2u), kStepY0 = step_field(kStay, 1u, 0u, 4u, 2u),
                   kStepX0 = step_field(kStay, 2u, 0u, 3u, 2u);
// dual: the corners of slots 0 .. 6, then +z +y +x
constexpr uint32_t kStepZ1 = step_field(kStay, 0u, 0u, 1u, 0u, 2u, 0u, 3u, 0u, 9u, 2u),
                   kStepY1 = step_field(kStay, 0u, 0u, 1u, 0u, 4u, 0u, 5u, 0u, 10u, 2u),
                   kStepX1 = step_field(kStay, 0u, 0u, 2u, 0u, 4u, 0u, 6u, 0u, 11u, 2u);
struct Step3 {
    uint32_t cz, cy, cx, shift, mask, hp, band;
    __device__ __forceinline__ Step3(int dual, const Item& it)
        : cz(dual ? kStepZ1 : kStepZ0), cy(dual ? kStepY1 : kStepY0), cx(dual ? kStepX1 : kStepX0), shift(dual ? 3u : 0u),
          mask(dual ? 15u : 7u), hp(32u * uint32_t(it.W) * uint32_t(it.bands)), band(32u * uint32_t(it.W)) {}
    __device__ __forceinline__ uint32_t field(uint32_t c) const { return (c >> shift) & mask; }
    __device__ __forceinline__ uint32_t next(uint32_t at, uint32_t d) const {
        const uint32_t s = 2u * d;
        at += ((cz >> s) & 3u) * hp + ((cx >> s) & 3u) * 32u + ((cy >> s) & 3u) - (hp + 33u);
        const uint32_t r = at & 31u;  // 29: one row below the band, 31: one above it (and a column to the left)
        if (r >= uint32_t(kBand3)) at += r == 31u ? uint32_t(kBand3) - band : band - uint32_t(kBand3);
        return at;
    }
    __device__ __forceinline__ bool ends(uint32_t d) const { return mask == 7u ? d >= 6u : (0xF180u >> d) & 1u; }
    __device__ __forceinline__ bool outside(uint32_t d) const { return mask == 15u && d == 8u; }
    __device__ __forceinline__ bool frame(uint32_t d) const { return mask == 7u && d == 7u; }
};
struct Step2 {
    uint32_t shift, band, end;  // end: the codes that are no step
    Offsets2 o;
    __device__ __forceinline__ Step2(int dual, int32_t W)
        : shift(dual ? 4u : 0u), band(32u * uint32_t(W)), end(dual ? 0x8200u : 0xC000u), o(offsets2(dual)) {}
    __device__ __forceinline__ uint32_t field(uint32_t c) const { return (c >> shift) & 15u; }
    // Byte d of the 16 in t, with its sign.
    static __device__ __forceinline__ uint32_t pick(const uint32_t (&t)[4], uint32_t d) {
        const uint32_t sel = (d & 7u) * 0x1111u | 0x8880u;
        uint32_t v;
        asm("prmt.b32 %0, %1, %2, %3;" : "=r"(v) : "r"(d < 8u ? t[0] : t[2]), "r"(d < 8u ? t[1] : t[3]), "r"(sel));
        return v;
    }
    __device__ __forceinline__ uint32_t next(uint32_t at, uint32_t d) const {
        at += pick(o.x, d) * 32u + pick(o.y, d);
        const uint32_t r = at & 31u;  // 30: one row below the tile, 31: one above it (and a column to the left)
        if (r >= uint32_t(kTile2)) at += r == 31u ? uint32_t(kTile2) - band : band - uint32_t(kTile2);
        return at;
    }
    __device__ __forceinline__ bool ends(uint32_t d) const { return (end >> d) & 1u; }
    __device__ __forceinline__ bool outside(uint32_t d) const { return end == 0x8200u && d == 9u; }
    __device__ __forceinline__ bool frame(uint32_t d) const { return end == 0xC000u && d == 15u; }
};

// Both paths in lockstep until neither has a link to follow.  False: the
// bounded walk gave up (a corrupted forest).
template <class Step>
__device__ __forceinline__ bool follow(const Forest& f, uint64_t coff, const Step& st, Counters* ctr, Path& a, Path& b,
                                       uint32_t& hops) {
    uint64_t t0 = 0;
    const uint8_t* code = f.code + coff;
    uint32_t da, db;
    (void)ctr;
    for (uint32_t n = 1;; ++n) {
        if (!CP_IN(coff + a.at, f.n_code, ctr)) a = Path{0, true};
        if (!CP_IN(coff + b.at, f.n_code, ctr)) b = Path{0, true};
        const uint32_t ca = __ldg(code + a.at), cb = __ldg(code + b.at);
        da = st.field(ca);
        db = st.field(cb);
        a.at = a.out ? 0u : st.next(a.at, da);
        b.at = b.out ? 0u : st.next(b.at, db);
        ++hops;
        if ((a.out || st.ends(da)) && (b.out || st.ends(db))) break;
        if ((n & 1023u) == 0) {
            const uint64_t now = global_timer_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > kWaitLimitNs) return false;
        }
    }
    // the frame of a T item is rooted at vertex 0
    if (!a.out && st.frame(da)) a.at = 0;
    if (!b.out && st.frame(db)) b.at = 0;
    a.out |= st.outside(da);
    b.out |= st.outside(db);
    return true;
}

__device__ __forceinline__ uint32_t root_id2(const Forest& f, const Item& it, int item, Counters* ctr, const Path& p) {
    if (p.out) return uint32_t(item);
    const uint32_t q = p.at >> 5, t = q / uint32_t(it.W), x = q - t * uint32_t(it.W);
    const uint32_t y = t * uint32_t(kTile2) + (p.at & 31u);
    const uint32_t node = f.dual ? uint32_t(it.toff) + y * uint32_t(it.W - 1) + x : uint32_t(it.voff) + y * uint32_t(it.W) + x;
    (void)ctr;
    return CP_IN(node, f.n_nodes, ctr) ? __ldg(f.uf + node) & ~kTag : 0u;
}

__device__ __forceinline__ uint32_t root_id3(const Forest& f, const Item& it, int item, Counters* ctr, const Path& p) {
    if (p.out) return uint32_t(item);
    const uint32_t q = p.at >> 5, t = q / uint32_t(it.W), x = q - t * uint32_t(it.W);
    const uint32_t z = t / uint32_t(it.bands), y = (t - z * uint32_t(it.bands)) * uint32_t(kBand3) + (p.at & 31u);
    const uint32_t node = f.dual ? uint32_t(it.toff) + ((z - 1u) * uint32_t(it.H - 1) + y) * uint32_t(it.W - 1) + x
                                 : uint32_t(it.voff) + (z * uint32_t(it.H) + y) * uint32_t(it.W) + x;
    (void)ctr;
    return CP_IN(node, f.n_nodes, ctr) ? __ldg(f.uf + node) & ~kTag : 0u;
}

// Root ids of the two endpoints of the survivor with key k (the key itself,
// not its complement), both paths in lockstep (two loads in flight); hops
// counts the steps.  False: a bounded walk gave up (a corrupted forest).
// kDim: the items are all 2D or all 3D (0: both kinds; in one kernel for all,
// the 3D walks take 2 to 5% longer).
template <int kDim = 0>
__device__ __forceinline__ bool walk_roots(const ItemTable& tab, const Forest& f, Counters* ctr, uint64_t k,
                                           uint32_t& ra, uint32_t& rb, uint32_t& hops) {
    const uint32_t vg = key_vertex(k);
    const int item = item_of_vertex(tab, vg);
    const Item& it = tab.it[item];
    int dz, dy, dx;
    stencil_off(it.ndim, int(key_n(k, it.ndim)), dz, dy, dx);
    const uint32_t local = vg - uint32_t(it.voff), W = uint32_t(it.W), H = uint32_t(it.H);
    const uint32_t row = local / W;
    const int x = int(local - row * W);
    if (kDim == 3 || (kDim == 0 && it.ndim == 3)) {
        const int y = int(row % H), z = int(row / H);
        Path a = {0, false}, b = a;
        if (!f.dual) {
            a.at = code_at3(it, z, y, x);
            b.at = code_at3(it, z + dz, y + dy, x + dx);
        } else {
            // the facet's zero coordinate picks the side: smallest corners of its two top cells
            const int cz = z + (dz < 0 ? -1 : 0), cy = y + (dy < 0 ? -1 : 0), cx = x + (dx < 0 ? -1 : 0);
            auto corner = [&](int s) {  // s: the zero coordinate's side (-1, +1)
                const int qz = dz == 0 && s < 0 ? z - 1 : cz, qy = dy == 0 && s < 0 ? y - 1 : cy,
                          qx = dx == 0 && s < 0 ? x - 1 : cx;
                const bool out = qz < 0 || qz >= it.D - 1 || qy < 0 || qy >= it.H - 1 || qx < 0 || qx >= it.W - 1;
                return Path{out ? 0u : code_at3(it, qz + 1, qy, qx), out};
            };
            a = corner(-1);
            b = corner(1);
        }
        if (!follow(f, uint64_t(it.coff), Step3(f.dual, it), ctr, a, b, hops)) {
            ra = rb = 0;
            return false;
        }
        ra = root_id3(f, it, item, ctr, a);
        rb = root_id3(f, it, item, ctr, b);
        return true;
    }
    const int y = int(row);
    Path a = {0, false}, b = a;
    if (!f.dual) {
        a.at = code_at2(it, y, x);
        b.at = code_at2(it, y + dy, x + dx);
    } else {
        // as in 3D
        const int cy = y + (dy < 0 ? -1 : 0), cx = x + (dx < 0 ? -1 : 0);
        auto corner = [&](int s) {
            const int qy = dy == 0 && s < 0 ? y - 1 : cy, qx = dx == 0 && s < 0 ? x - 1 : cx;
            const bool out = qy < 0 || qy >= it.H - 1 || qx < 0 || qx >= it.W - 1;
            return Path{out ? 0u : code_at2(it, qy, qx), out};
        };
        a = corner(-1);
        b = corner(1);
    }
    if (!follow(f, uint64_t(it.coff), Step2(f.dual, it.W), ctr, a, b, hops)) {
        ra = rb = 0;
        return false;
    }
    ra = root_id2(f, it, item, ctr, a);
    rb = root_id2(f, it, item, ctr, b);
    return true;
}
#endif

}  // namespace cp
