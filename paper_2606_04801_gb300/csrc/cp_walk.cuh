// Walks through the pruned forests, from a survivor's two endpoints to the
// roots of their classes.
//
// 2D items: a 32-bit word per vertex / top cell, the parent's id or a tagged
// root id.  3D items: a code byte per vertex, at (z H + y) pitch + x of the
// item's codes: bits 0-2 the vertex's H0 link (face slot 0..5, 6: a root, 7: a
// frame vertex of a T-filtration item, whose root is vertex 0), bits 3-6 the
// dual link of the top cell with its smallest corner one plane below, at
// (z - 1, y, x) (0..6: towards that slot as seen from that corner, 7: a root,
// 8: the outside, 9, 10, 11: +z, +y, +x).  Only a root's word of the 32-bit arrays is written for 3D items (its
// root id).  A 512^3 volume's codes (134 MB) mostly stay in L2 between the
// pruning pass and the walks, where words (1,074 MB) did not.
#pragma once
#include "cp_common.cuh"

namespace cp {

// Offset of the 3D link with code field d (H0: 0..5; dual: 0..6, 9..11) in the
// codes' index space.
__host__ __device__ __forceinline__ int32_t link_offset3(int dual, uint32_t d, int32_t hp, int32_t p) {
    if (!dual) {
        const int32_t m = (d == 0u || d == 5u) ? hp : ((d == 1u || d == 4u) ? p : 1);
        return d < 3u ? -m : m;
    }
    if (d < 8u) return ((d & 4u) ? 0 : -hp) + ((d & 2u) ? 0 : -p) + ((d & 1u) ? 0 : -1);
    return d == 9u ? hp : (d == 10u ? p : 1);
}

#ifdef __CUDACC__
struct Forest {
    const uint32_t* uf;    // 2D: links; 3D: root words
    const uint8_t* code;   // 3D items' codes
    uint32_t n_nodes;      // entries of uf / code (bounds-checked build)
    uint64_t n_code;
    int dual;
};

// One endpoint's path in a 3D item's codes.
struct Path3 {
    uint32_t at;
    bool live, out;
};

__device__ __forceinline__ void step3(const Forest& f, const Item& it, int32_t hp, Counters* ctr, Path3& p) {
    (void)ctr;
    const uint64_t i = uint64_t(it.coff) + p.at;
    if (!CP_IN(i, f.n_code, ctr)) {
        p.live = false;
        p.at = 0;
        return;
    }
    const uint32_t c = __ldg(f.code + i);
    const uint32_t d = f.dual ? c >> 3 : c & 7u;
    if (f.dual ? d == 7u : d == 6u) {
        p.live = false;
    } else if (f.dual ? d == 8u : d == 7u) {
        p.live = false;
        p.out = f.dual;  // else: the frame of a T item, rooted at vertex 0
        p.at = 0;
    } else {
        p.at += uint32_t(link_offset3(f.dual, d, hp, it.pitch));
    }
}

__device__ __forceinline__ uint32_t root_id3(const Forest& f, const Item& it, int item, Counters* ctr, const Path3& p) {
    if (p.out) return uint32_t(item);
    const uint32_t row = p.at / uint32_t(it.pitch), x = p.at - row * uint32_t(it.pitch);
    uint32_t node;
    if (!f.dual) {
        node = uint32_t(it.voff) + row * uint32_t(it.W) + x;
    } else {
        const uint32_t z = row / uint32_t(it.H), y = row - z * uint32_t(it.H);
        node = uint32_t(it.toff) + ((z - 1u) * uint32_t(it.H - 1) + y) * uint32_t(it.W - 1) + x;
    }
    (void)ctr;
    return CP_IN(node, f.n_nodes, ctr) ? __ldg(f.uf + node) & ~kTag : 0u;
}

// Root ids of the two endpoints of the survivor with key k (the key itself,
// not its complement), both paths in lockstep (two loads in flight); hops
// counts the steps.  False: a bounded walk gave up (a corrupted forest).
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
    uint64_t t0 = 0;
    uint32_t steps = 0;
    auto overdue = [&]() {
        if ((++steps & 1023u) != 0) return false;
        const uint64_t now = global_timer_ns();
        if (t0 == 0) t0 = now;
        return now - t0 > kWaitLimitNs;
    };
    if (it.ndim == 3) {
        const int32_t p = it.pitch, hp = int32_t(H) * p;
        Path3 a = {row * uint32_t(p) + uint32_t(x), true, false}, b = a;
        if (!f.dual) {
            b.at += uint32_t(dz * hp + dy * p + dx);
        } else {
            // the facet's zero coordinate picks the side: smallest corners of its two top cells
            const int y = int(row % H), z = int(row / H);
            const int cz = z + (dz < 0 ? -1 : 0), cy = y + (dy < 0 ? -1 : 0), cx = x + (dx < 0 ? -1 : 0);
            auto corner = [&](int s) {  // s: the zero coordinate's side (-1, +1)
                const int qz = dz == 0 && s < 0 ? z - 1 : cz, qy = dy == 0 && s < 0 ? y - 1 : cy,
                          qx = dx == 0 && s < 0 ? x - 1 : cx;
                Path3 q = {0, true, false};
                if (qz < 0 || qz >= it.D - 1 || qy < 0 || qy >= it.H - 1 || qx < 0 || qx >= it.W - 1) {
                    q.live = false;
                    q.out = true;
                } else {
                    q.at = uint32_t((qz + 1) * hp + qy * p + qx);
                }
                return q;
            };
            a = corner(-1);
            b = corner(1);
        }
        while (a.live || b.live) {
            if (a.live) step3(f, it, hp, ctr, a);
            if (b.live) step3(f, it, hp, ctr, b);
            ++hops;
            if (overdue()) {
                ra = rb = 0;
                return false;
            }
        }
        ra = root_id3(f, it, item, ctr, a);
        rb = root_id3(f, it, item, ctr, b);
        return true;
    }
    uint32_t na = vg, nb = uint32_t(int64_t(vg) + int64_t(dy) * W + dx);
    if (f.dual) {
        // the facet's zero coordinate picks the side
        const int y = int(row);
        na = top_of_octant(it, 0, y, x, -1, dy == 0 ? -1 : dy, dy == 0 ? dx : -1);
        nb = top_of_octant(it, 0, y, x, 1, dy == 0 ? 1 : dy, dy == 0 ? dx : 1);
    }
    uint32_t pa = CP_IN(na, f.n_nodes, ctr) ? __ldcg(f.uf + na) : kTag;
    uint32_t pb = CP_IN(nb, f.n_nodes, ctr) ? __ldcg(f.uf + nb) : kTag;
    while (!(pa & kTag) || !(pb & kTag)) {
        ++hops;
        if (!(pa & kTag)) pa = CP_IN(pa, f.n_nodes, ctr) ? __ldcg(f.uf + pa) : kTag;
        if (!(pb & kTag)) pb = CP_IN(pb, f.n_nodes, ctr) ? __ldcg(f.uf + pb) : kTag;
        if (overdue()) {
            ra = rb = 0;
            return false;
        }
    }
    ra = pa & ~kTag;
    rb = pb & ~kTag;
    return true;
}
#endif

}  // namespace cp
