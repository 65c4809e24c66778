// The 3D lower star (Sec. 3.3) of 32 vertices at a time, on words with one
// bit per vertex: what the pruning kernel needs of the lookup table's entry,
// in closed form.  Host code runs the same functions over every class of the
// table and compares (check_words3).
#pragma once
#include <cstdint>

#include "cp_mask3.cuh"

namespace cp {

struct Star3 {
    uint32_t h[3];   // planes of the H0 code: the first face slot of L(v) (0..5), 6: none (a local minimum)
    uint32_t co[8];  // octant t's top cell lies in L(v)
    uint32_t event;  // the lower link is not a disc (survivors or a root), or may not be
    // the relevant mask's other planes: the faces in slot order, and the edges
    // [dy][dx], [dz][dx], [dz][dy] (1: the positive side)
    uint32_t f[6], xy[2][2], xz[2][2], yz[2][2];
};

// The relevant mask's plane of the canonical neighbour n (n != 13).
CP_HD inline uint32_t relevant_plane(const Star3& s, int n) {
    const int dz = n / 9 - 1, dy = (n / 3) % 3 - 1, dx = n % 3 - 1;
    const int i = dz > 0, j = dy > 0, k = dx > 0;
    if (dz && dy && dx) return s.co[4 * i + 2 * j + k];
    if (!dz && dy && dx) return s.xy[j][k];
    if (dz && !dy && dx) return s.xz[i][k];
    if (dz && dy && !dx) return s.yz[i][j];
    return s.f[dz ? 5 * i : (dy ? 1 + 3 * j : 2 + k)];
}

CP_HD inline void full_add(uint32_t a, uint32_t b, uint32_t c, uint32_t& sum, uint32_t& carry) {
    sum = a ^ b ^ c;
    carry = (a & b) | (c & (a ^ b));
}

// r[n]: the canonical neighbour n = 9(dz+1) + 3(dy+1) + (dx+1) precedes v.
CP_HD inline void star_words3(const uint32_t (&r)[27], Star3& o) {
    // faces in slot order z-, y-, x-, x+, y+, z+; the opposite of slot s is 5 - s
    uint32_t(&f)[6] = o.f;
    f[0] = r[4], f[1] = r[10], f[2] = r[12], f[3] = r[14], f[4] = r[16], f[5] = r[22];
    // the collapse: an edge with both its faces, a corner with its three edges
    uint32_t(&xy)[2][2] = o.xy, (&xz)[2][2] = o.xz, (&yz)[2][2] = o.yz;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            xy[i][j] = r[13 + 3 * (2 * i - 1) + (2 * j - 1)] & f[i ? 4 : 1] & f[j ? 3 : 2];  // [dy][dx]
            xz[i][j] = r[13 + 9 * (2 * i - 1) + (2 * j - 1)] & f[i ? 5 : 0] & f[j ? 3 : 2];  // [dz][dx]
            yz[i][j] = r[13 + 9 * (2 * i - 1) + 3 * (2 * j - 1)] & f[i ? 5 : 0] & f[j ? 4 : 1];  // [dz][dy]
        }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int z = t >> 2, y = (t >> 1) & 1, x = t & 1;
        o.co[t] = r[13 + 9 * (2 * z - 1) + 3 * (2 * y - 1) + (2 * x - 1)] & xy[y][x] & xz[z][x] & yz[z][y];
    }
    // the lowest face
    o.h[0] = ~f[0] & (f[1] | (~f[2] & (f[3] | (~f[4] & f[5]))));
    o.h[1] = ~f[0] & ~f[1] & (f[2] | f[3] | (~f[4] & ~f[5]));
    o.h[2] = ~f[0] & ~f[1] & ~f[2] & ~f[3];
    // connected: what the lowest face reaches, two sweeps over the faces (a
    // longer way round is reported as an event; the lookup then settles it)
    auto edge = [&](int s, int t) -> uint32_t {  // s < t, not opposite
        const int az = s == 0 ? 0 : (t == 5 ? 1 : -1);  // z sign among the two, if any
        const int ay = (s == 1 || t == 1) ? 0 : ((s == 4 || t == 4) ? 1 : -1);
        const int ax = (s == 2 || t == 2) ? 0 : ((s == 3 || t == 3) ? 1 : -1);
        return az < 0 ? xy[ay][ax] : (ay < 0 ? xz[az][ax] : yz[az][ay]);
    };
    uint32_t reach[6], before = 0;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        reach[s] = f[s] & ~before;
        before |= f[s];
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int s = k < 6 ? k : 11 - k;
#pragma unroll
        for (int t = 0; t < 6; ++t)
            if (t != s && t != 5 - s) reach[s] |= reach[t] & (s < t ? edge(s, t) : edge(t, s));
    }
    uint32_t apart = 0;
#pragma unroll
    for (int s = 0; s < 6; ++s) apart |= f[s] & ~reach[s];
    // Euler characteristic faces - edges + corners, as the number of ones
    // among faces, absent edges and corners less 12: 1 exactly if that number
    // is 13 (5 modulo 8; it lies between 6 and 18)
    uint32_t in[26];
#pragma unroll
    for (int s = 0; s < 6; ++s) in[s] = f[s];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        in[6 + k] = ~xy[k >> 1][k & 1];
        in[10 + k] = ~xz[k >> 1][k & 1];
        in[14 + k] = ~yz[k >> 1][k & 1];
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) in[18 + t] = o.co[t];
    uint32_t two[13], four = 0, ones = in[0], twos;
#pragma unroll
    for (int k = 0; k < 12; ++k) full_add(ones, in[1 + 2 * k], in[2 + 2 * k], ones, two[k]);
    two[12] = ones & in[25];
    ones ^= in[25];
    twos = two[0];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        uint32_t c;
        full_add(twos, two[1 + 2 * k], two[2 + 2 * k], twos, c);
        four ^= c;
    }
    o.event = ~(ones & ~twos & four) | apart;
}

// Planes of the slot towards which a top cell in slot 7 of L(v) dies: the
// highest slot not in L(v), 7 if all are (a dual root).
CP_HD inline void slot7_target(const uint32_t (&c)[8], uint32_t& b0, uint32_t& b1, uint32_t& b2) {
    b0 = c[6] & (~c[5] | (c[4] & (~c[3] | (c[2] & (~c[1] | c[0])))));
    b1 = ~c[6] | (c[5] & c[4] & (~c[3] | ~c[2] | (c[1] & c[0])));
    b2 = ~(c[6] & c[5] & c[4]) | (c[3] & c[2] & c[1] & c[0]);
}

// Slot towards which the top cell in slot t < 7 of L(v) dies (+z, +y, +x).
CP_HD constexpr int slot_target(int t) { return t < 4 ? t + 4 : (t < 6 ? t + 2 : 7); }

}  // namespace cp
