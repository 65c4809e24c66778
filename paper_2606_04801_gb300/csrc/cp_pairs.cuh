// The pair that a union-find commit writes (shared by the union-find and
// the slab split's first stage).
#pragma once
#include "cp_common.cuh"
#include "cp_grid.cuh"
#include "cp_kernels.h"

namespace cp {

// The pair of a committed survivor with key `key` (the key itself, not its
// complement) of item `item`, whose dying class has age key a (the root
// vertex; for the dual the vertex whose lower star holds the dying top cell).  Returns false for a zero-persistence pair,
// which is omitted (Sec. 2.3).
__device__ __forceinline__ bool commit_pair(const ItemTable& tab, uint64_t a, int dual, uint64_t key, int item,
                                            cp_pair& out) {
    const Item& it = tab.it[item];
    const uint32_t young = key_vertex(a);
    uint32_t vg = key_vertex(key);
    int n = int(key_n(key, it.ndim));
    int dz, dy, dx;
    stencil_off(it.ndim, n, dz, dy, dx);
    const uint32_t W = uint32_t(it.W), H = uint32_t(it.H);
    auto corner = [&](uint32_t v, uint32_t& l, int& z, int& y, int& x) {  // local index and coordinates
        l = v - uint32_t(it.voff);
        const uint32_t row = l / W, pl = row / H;
        x = int(l - row * W);
        y = int(row - pl * H);
        z = int(pl);
    };
    uint32_t lv;
    int x, y, z;
    corner(vg, lv, z, y, x);
    float fv = ord_float(uint32_t(key >> 32));
    float fy = ord_float(uint32_t(a >> 32));
    if (!dual) {
        // H0: birth at the dying root vertex, death at the edge (value of its higher endpoint v)
        out.birth = fy;
        out.death = fv;
        uint32_t ly;
        int yx, yy, yz;
        corner(young, ly, yz, yy, yx);
        out.birth_cell = int32_t(doubled_index(it, yz, yy, yx, 0, 0, 0));
        out.death_cell = int32_t(doubled_index(it, z, y, x, dz, dy, dx));
        out.birth_pixel = int32_t(ly);
        out.death_pixel = int32_t(lv);
        out.dim = 0;
    } else {
        // top dimension: birth at the facet, death at the dying top cell
        uint32_t mg = key_vertex(a);
        int nt = int(key_n(a, it.ndim));
        int tz, ty, tx;
        stencil_off(it.ndim, nt, tz, ty, tx);
        uint32_t lm;
        int mx, my, mz;
        corner(mg, lm, mz, my, mx);
        out.birth = fv;
        out.death = fy;
        out.birth_cell = int32_t(doubled_index(it, z, y, x, dz, dy, dx));
        out.death_cell = int32_t(doubled_index(it, mz, my, mx, tz, ty, tx));
        out.birth_pixel = int32_t(lv);
        out.death_pixel = int32_t(lm);
        out.dim = it.ndim - 1;
    }
    out.item = it.user;
    return out.birth != out.death;
}

// The pair of merge-tree root nd (list q: H0, dual) if the tree connects it
// with an older one and it has persistence; h1flags as in UfParams.
__device__ __forceinline__ bool tree_pair(const ItemTable& tab, const TreeNode& nd, int q, uint32_t* h1flags,
                                          cp_pair& out) {
    if (nd.key == ~0ull) return false;
    const uint64_t key = q ? ~nd.key : nd.key;
    const int item = int(nd.item);
    if (h1flags && tab.it[item].ndim == 3) {
        const uint32_t id = cell_id3(tab.it[item], key, q != 0);
        atomicOr(h1flags + (id >> 5), 1u << (id & 31u));
    }
    return commit_pair(tab, q ? ~nd.age : nd.age, q, key, item, out);
}

// The essential H0 class of item i: born at its minimum, never dies.
__device__ __forceinline__ bool essential_pair(const ItemTable& tab, Counters* ctr, int i, cp_pair& p) {
    const Item& it = tab.it[i];
    const unsigned long long g = ctr->gmin[i];
    if (g == ~0ull) {
        set_status(ctr, kStInternal);
        return false;
    }
    const uint32_t v = uint32_t(g & 0xFFFFFFFFu);
    const int x = int(v % uint32_t(it.W)), y = int((v / uint32_t(it.W)) % uint32_t(it.H)),
              z = int(v / uint32_t(it.W * it.H));
    p.birth = ord_float(uint32_t(g >> 32));
    p.death = __int_as_float(0x7F800000);
    p.birth_cell = int32_t(doubled_index(it, z, y, x, 0, 0, 0));
    p.death_cell = -1;
    p.birth_pixel = int32_t(v);
    p.death_pixel = -1;
    p.dim = 0;
    p.item = it.user;
    return true;
}

}  // namespace cp
