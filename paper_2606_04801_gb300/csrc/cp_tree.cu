// K3: the elder-rule union-find over the survivors (H0: Sec. 4.1 step 3,
// Sec. 4.2 step 2; the dual graph: Sec. 3.1, Appendix A, Sec. 4.1 step 5,
// Sec. 4.2 step 3) as a merge tree that takes the survivors in any order: no
// sort, no rounds, no grid barrier.
//
// Every root class u of the pruned forests has one word T[u] = (s, v): u is
// connected with the older root v by survivors of key at most s; (infinity,
// u) while it is connected with nothing older.  A survivor (u, v, s) goes in
// as follows:
//   1. u: the younger of the two, v: the older.  The same root: the survivor
//      closes a cycle, done;
//   2. if T[u]'s key is below s, u becomes the older root in T[u]; back to 1;
//   3. else compare and swap T[u] from the word (t, w) just read to (s, v).
//      If another survivor changed it meanwhile, on with its new word at 2;
//   4. if t was infinity, done; else the displaced connection (u, w, t) is
//      still owed, and u ~ v at level s < t: go on with (v, w, t).
// Why this is the sequential elder rule.  The connections in T and those
// displaced ones still in some thread's hands connect, at every level a, what
// all survivors taken so far with keys at most a connect: step 3 replaces
// (u, w, t) by (u, v, s) and (v, w, t), and what step 1 drops is implied by
// the rest.  Every T[u] points to an older root.  When all survivors are
// in, a class of k roots at level a is a tree of T's connections of key at
// most a; each root gives at most one and the oldest none, so all but the
// oldest have T's key at most a: T[u]'s key is the level at which u stops
// being the oldest of its class, which is the survivor that kills it.  The
// keys (so the pairs) do not depend on the schedule; the parents may.
//
// Long climbs shorten their way: with u connected with p at s1 (u's word) and p
// with w at s2 < s1 (p's), u's word becomes (s1, w).  Its key stays, so the
// pairs do; w is older than p; and what the word said follows from it and the
// words of p, a root older than u: a connection displaced from or dropped at a
// root rests on words, present or past, of older roots alone, so no two rest
// on one another.
//
// This is the triplet merge tree of Smirnov and Morozov (TopoInVis 2017), in
// root-id space.
//
// Two threads could each drop a connection that the other's implies only if
// each had read the other's word from before its displacement after making
// its own: the full fence after a displacement rules that out (a connection
// taken from T by a swap is owed by one thread alone until it is back in T).
//
// What bounds it: dependent L2 reads and swaps of a node's 16-byte word, 4 to 7
// per survivor, with as many survivors in flight as threads fit.  Only the
// younger end's word is read: the older an end, the more survivors end there,
// and with both ends' words read the sectors of the oldest few roots held up
// the chip.  Ages never change, so they come through L1, and a word keeps the
// upper half of its parent's age with the parent, so that a climb reads one
// word per step (ages with equal upper halves are looked up).  Times, first
// with 8 radix passes over both lists and reservation rounds with two grid
// barriers each (cp_uf.cu), then with both ends climbed, now:
//   2048^2 blurred (97 K survivors)                46 -> 32 us
//   512^3 blurred (587 K survivors)         553 -> 244 -> 67 us
//   128^3 uniform noise (1.15 M survivors) 1110 -> 475 -> 127 us
//   2048^2 uniform noise (2.61 M survivors)       495 -> 257 us
// On a slope with noise (each basin drains into the one below it) the paths of
// a survivor's ends meet far down, and a climb is as long as that: shortened
// after 4, 8, 16, 32, 64 steps or never, 2048 x 8192 noise on a ramp takes
// 1.22, 1.26, 1.41, 1.55, 1.75 or 9.17 ms (sort and rounds: 5.9), 2048^2 valleys
// 88, 85, 88, 97, 121 or 908 us, but 128^3 noise, whose swaps it adds to, 192,
// 173, 152, 141, 138 or 137 us and 512^3 blurred 123, 113, 102, 97, 97 or 96.
// Tried and left out: the smallest survivor of each root put in first
// (Boruvka's first step; its atomics cost the walks what it saved here), words
// through L1 until the first swap (more swaps fail), fewer threads.
#include "cp_common.cuh"
#include "cp_grid.cuh"
#include "cp_kernels.h"
#include "cp_pairs.cuh"

namespace cp {
namespace {

constexpr int kTT = 256;
constexpr uint32_t kFar = 32;  // steps after which a climb shortens the paths it takes

// A node's word, read and swapped as 128 bits: {key, parent}.
struct Word {
    uint64_t key;     // infinity (~0): connected with nothing older yet
    uint64_t parent;  // root id | upper half of its age << 32 (unused while key is infinity)
};

__device__ __forceinline__ Word ld_word(const TreeNode* n) {
    Word w;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(w.key), "=l"(w.parent)
                 : "l"(n)
                 : "memory");
    return w;
}
__device__ __forceinline__ Word cas_word(TreeNode* n, Word expect, Word desired) {
    Word w;
    asm volatile(
        "{\n\t.reg .b128 t, e, d;\n\tmov.b128 e, {%3, %4};\n\tmov.b128 d, {%5, %6};\n\t"
        "atom.relaxed.gpu.global.cas.b128 t, [%2], e, d;\n\tmov.b128 {%0, %1}, t;\n\t}"
        : "=l"(w.key), "=l"(w.parent)
        : "l"(n), "l"(expect.key), "l"(expect.parent), "l"(desired.key), "l"(desired.parent)
        : "memory");
    return w;
}

// Both lists' survivors, in the order the pruning pass wrote them, one
// survivor per thread.
__global__ void __launch_bounds__(kTT) k_tree(const __grid_constant__ TreeArgs a) {
    Counters* ctr = a.ctr;
    wait_for_previous();
    // non-finite input, or walks that gave up: the call fails anyway
    if (ld_acquire_u32(&ctr->status) & (kStTimeout | kStNonfinite)) return;
    const uint32_t n0 = min(*a.l[0].d_n, a.cap), n1 = min(*a.l[1].d_n, a.cap), n = n0 + n1;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctr->rounds0 = n0 ? 1u : 0u;
        ctr->roundst = n1 ? 1u : 0u;
        ctr->trace_active[0][0] = n0;
        ctr->trace_active[1][0] = n1;
    }
    uint32_t hops = 0;
    for (uint32_t g = blockIdx.x * kTT + threadIdx.x; g < n; g += gridDim.x * kTT) {
        const int q = g >= n0 ? 1 : 0;
        const TreeList& L = a.l[q];
        const uint32_t i = q ? g - n0 : g;
        TreeNode* T = L.node;
        uint64_t s = L.keys[i];  // ascending order of the stored keys in both lists
        uint32_t u = __ldcg(L.ra + i), v = __ldcg(L.rb + i);
        uint64_t t0 = 0;
        uint32_t steps = 0;
        // every climb ends (parents are older) and a swap only fails when another
        // survivor went in; the wall-clock bound guards against a corrupted word
        auto overdue = [&]() {
            if ((++steps & 1023u) != 0) return false;
            const uint64_t now = global_timer_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 <= kWaitLimitNs) return false;
            set_status(ctr, kStTimeout);
            return true;
        };
        auto age = [&](uint32_t w) { return __ldg(&T[w].age); };
        if (u == v || !CP_IN(u, L.n_rids, ctr) || !CP_IN(v, L.n_rids, ctr)) continue;
        uint32_t hu = uint32_t(age(u) >> 32), hv = uint32_t(age(v) >> 32);
        while (u != v) {
            // u: the younger (ages: smaller is older)
            if (hu < hv || (hu == hv && age(u) < age(v))) {
                const uint32_t t = u, h = hu;
                u = v, hu = hv;
                v = t, hv = h;
            }
            Word w = ld_word(T + u);
            bool in = false, late = overdue();
            while (w.key > s && !in && !late) {
                const Word got = cas_word(T + u, w, Word{s, uint64_t(hv) << 32 | v});
                in = got.key == w.key && got.parent == w.parent;
                if (!in) {
                    w = got;
                    late = overdue();
                }
            }
            if (late) break;
            if (in) {
                if (w.key == ~0ull) break;
                asm volatile("fence.sc.gpu;" ::: "memory");
                s = w.key;
                u = v, hu = hv;
                v = uint32_t(w.parent), hv = uint32_t(w.parent >> 32);
                if (!CP_IN(v, L.n_rids, ctr)) break;
            } else {  // connected with an older root below s
                const uint32_t p = uint32_t(w.parent);
                if (!CP_IN(p, L.n_rids, ctr)) break;
                Word x = w;
                if (steps > kFar) {  // two steps at once, and one from now on if the second is below the first
                    x = ld_word(T + p);
                    if (x.key >= s) x = w;
                    else if (x.key < w.key) cas_word(T + u, w, Word{w.key, x.parent});
                }
                u = uint32_t(x.parent), hu = uint32_t(x.parent >> 32);
                if (!CP_IN(u, L.n_rids, ctr)) break;
            }
        }
        hops += steps;
    }
    for (int o = 16; o > 0; o >>= 1) hops += __shfl_xor_sync(0xFFFFFFFFu, hops, o);
    if (lane_id() == 0 && hops) atomicAdd(&ctr->trace_hops[0][1], (unsigned long long)hops);
}

// The pair of every root that the tree connects with an older one (calls with
// H1, whose reduction needs the committed survivors marked; the others emit in
// k_order).
__global__ void __launch_bounds__(kTT) k_tree_emit(const __grid_constant__ TreeEmitArgs a) {
    Counters* ctr = a.ctr;
    if (ld_acquire_u32(&ctr->status) & (kStTimeout | kStNonfinite)) return;
    const uint32_t r0 = min(ctr->n_r0, a.n_rids[0]), r1 = min(ctr->n_rt, a.n_rids[1]), n = r0 + r1;
    for (uint32_t g0 = blockIdx.x * kTT; g0 < n; g0 += gridDim.x * kTT) {
        const uint32_t g = g0 + threadIdx.x;
        bool emit = false;
        cp_pair pr;
        if (g < n) {
            const int q = g >= r0 ? 1 : 0;
            emit = tree_pair(a.tab, a.node[q][q ? g - r0 : g], q, a.h1flags[q], pr);
        }
        const uint32_t pp = warp_append(&ctr->n_pairs, emit);
        if (emit) {
            if (pp < a.pair_cap) a.pairs[pp] = pr;
            else set_status(ctr, kStCapacity);
        }
    }
}

}  // namespace

cudaError_t launch_tree(const TreeArgs& a, cudaStream_t s) {
    const int blocks = device_cached(kCacheTree, [] {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tree, kTT, 0);
        return device_sm_count() * (per_sm > 0 ? per_sm : 1);
    });
    return launch_after(true, k_tree, blocks, kTT, 0, s, a);
}

cudaError_t launch_tree_emit(const TreeEmitArgs& a, cudaStream_t s) {
    k_tree_emit<<<device_sm_count() * 4, kTT, 0, s>>>(a);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace cp
