// Hashing and the canonical form of a tree, by the 32 lanes of a warp.  pt_kernels.cu
// compiles it for the device; tests/canon_lanes.cpp runs the lanes on the host in every
// order that the warp's barriers allow.
#pragma once

#include <cstdint>

#include "pt_internal.h"

namespace pt {

// ---------------------------------------------------------------- hashing
// Split hash of the key definition: SplitMix64's output function applied as
//   h.lo = mix(lo ^ mix(hi + 0x9e3779b97f4a7c15)), h.hi = mix(hi ^ mix(lo + 0xd1b54a32d192ed03)).
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}
__device__ __forceinline__ unsigned __int128 split_hash(unsigned long long lo, unsigned long long hi) {
    unsigned long long a = mix64(lo ^ mix64(hi + 0x9e3779b97f4a7c15ull));
    unsigned long long b = mix64(hi ^ mix64(lo + 0xd1b54a32d192ed03ull));
    return ((unsigned __int128)b << 64) | a;
}
__device__ __forceinline__ bool less128(unsigned long long alo, unsigned long long ahi, unsigned long long blo,
                                        unsigned long long bhi) {
    return ahi < bhi || (ahi == bhi && alo < blo);
}

// ---------------------------------------------------------------- canonicaliser
// One warp per tree, everything in shared memory and by levels: the edges give the
// adjacency; a breadth-first pass from leaf 0 the parents and the levels; an upward
// pass over the levels smallest taxa, leaf sets, child order and the number of inner
// nodes below; a downward pass the canonical numbers (pre-order, so a node's first
// inner child follows it and the second comes after the first's inner nodes) and the
// places in the full-optimisation schedule.  Then the lanes write the arrays, hash
// the n-3 non-trivial splits, reduce the 128-bit key sum, and rank the splits.
// A level costs a few shared-memory round trips; lane 0 doing all this node by node,
// with half of it through global memory, took 61 us for 27 taxa.
struct CanonSmem {
    uint64_t bits[kMaxNode][2];
    int32_t deg[kMaxNode], par[kMaxNode];
    int32_t tail;
    int16_t nbr[kMaxNode][3];
    int16_t order[kMaxNode], lev[kMaxNode + 1];
    int16_t c0[kMaxNode], c1[kMaxNode];  // children of inner nodes, smallest taxon first
    int16_t inner[kMaxNode];             // inner nodes below and at v
    int16_t canon[kMaxNode], pos[kMaxNode];
    uint8_t mint[kMaxNode];
};

__device__ __forceinline__ void canon_tree(int n, int tree, int lane, const int32_t* __restrict__ edges,
                                           const double* __restrict__ lengths, const TreeSet& ts, int32_t* err,
                                           CanonSmem& s) {
    const unsigned all = 0xffffffffu;
    const int NN = 2 * n - 2, E = 2 * n - 3;
    const int32_t* ed = edges + (size_t)tree * 2 * E;
    int32_t* up = ts.up + (size_t)tree * NN;
    int32_t* ch = ts.ch + (size_t)tree * NN * 2;
    double* len = ts.len + (size_t)tree * NN;
    uint64_t* bits = ts.bits + (size_t)tree * NN * 2;
    int32_t* erank = ts.erank + (size_t)tree * NN;
    int32_t* sched = ts.sched + (size_t)tree * 3 * n;
    if (lengths)  // device-resident inputs are checked here: finite, non-negative lengths
        for (int e = lane; e < E; e += 32) {
            const double x = lengths[(size_t)tree * E + e];
            if (!(x >= 0.0 && x <= 1.7976931348623157e308)) atomicCAS(&err[kErrLen], 0, tree + 1);
        }
    // An edge list that is no tree is flagged and gets the key 0, which no tree has; a
    // caterpillar takes its place, as kernels queued behind this one follow its arrays
    // before the host reads the flag.
    bool bad = false;
    auto edge = [&](int e, int& a, int& b) {
        if (!bad) { a = ed[2 * e]; b = ed[2 * e + 1]; return; }
        a = e;
        b = e >= n ? e + 1 : e == 0 ? n : e == n - 1 ? NN - 1 : n + e - 1;
    };
    int levels;
    while (true) {
        bool ok = true;
        for (int v = lane; v < NN; v += 32) {
            s.deg[v] = 0;
            s.par[v] = -2;
        }
        if (lane == 0) s.tail = 1;
        __syncwarp();
        for (int e = lane; e < E; e += 32) {
            int a, b;
            edge(e, a, b);
            if (a < 0 || b < 0 || a >= NN || b >= NN || a == b) { ok = false; continue; }
            const int i = atomicAdd(&s.deg[a], 1), j = atomicAdd(&s.deg[b], 1);
            if (i < 3) s.nbr[a][i] = (int16_t)b;
            if (j < 3) s.nbr[b][j] = (int16_t)a;
        }
        __syncwarp();
        for (int v = lane; v < NN; v += 32) ok = ok && s.deg[v] == (v < n ? 1 : 3);
        ok = __all_sync(all, ok);
        levels = 0;
        if (ok) {
            if (lane == 0) {
                s.par[0] = -1;
                s.order[0] = 0;
                s.lev[0] = 0;
            }
            __syncwarp();
            for (int lo = 0, hi = 1; lo < hi && ok; ++levels) {
                for (int i = lo + lane; i < hi; i += 32) {
                    const int v = s.order[i], pv = s.par[v];
                    for (int k = 0; k < (v < n ? 1 : 3); ++k) {
                        const int c = s.nbr[v][k];
                        if (c == pv) continue;
                        if (atomicCAS(&s.par[c], -2, v) != -2) ok = false;  // a cycle
                        else s.order[atomicAdd(&s.tail, 1)] = (int16_t)c;
                    }
                }
                ok = __all_sync(all, ok);
                __syncwarp();
                lo = hi;
                hi = s.tail;
                if (lane == 0) s.lev[levels + 1] = (int16_t)lo;
                __syncwarp();  // every lane has read the tail before a lane of the next level moves it
            }
            ok = ok && s.tail == NN;
        }
        __syncwarp();
        if (ok || bad) break;
        bad = true;
        if (lane == 0) atomicCAS(&err[kErrTree], 0, tree + 1);
    }
    for (int l = levels - 1; l >= 0; --l) {  // upward
        for (int i = s.lev[l] + lane; i < s.lev[l + 1]; i += 32) {
            const int v = s.order[i];
            if (v < n) {
                s.mint[v] = (uint8_t)v;
                s.inner[v] = 0;
                s.bits[v][0] = v < 64 ? (1ull << v) : 0ull;
                s.bits[v][1] = v >= 64 ? (1ull << (v - 64)) : 0ull;
                continue;
            }
            const int p = s.par[v], x = s.nbr[v][0], y = s.nbr[v][1], z = s.nbr[v][2];
            int a = x == p ? y : x, b = z == p ? y : z;
            if (s.mint[b] < s.mint[a]) { const int t = a; a = b; b = t; }
            s.c0[v] = (int16_t)a;
            s.c1[v] = (int16_t)b;
            s.mint[v] = s.mint[a];
            s.inner[v] = (int16_t)(1 + s.inner[a] + s.inner[b]);
            s.bits[v][0] = s.bits[a][0] | s.bits[b][0];
            s.bits[v][1] = s.bits[a][1] | s.bits[b][1];
        }
        __syncwarp();
    }
    if (lane == 0) {
        s.canon[0] = 0;
        s.canon[s.nbr[0][0]] = (int16_t)n;
        s.pos[s.nbr[0][0]] = 0;
    }
    __syncwarp();
    for (int l = 1; l < levels; ++l) {  // downward; a subtree of I inner nodes has 3 I + 1 schedule entries
        for (int i = s.lev[l] + lane; i < s.lev[l + 1]; i += 32) {
            const int v = s.order[i], c = s.canon[v], p = s.pos[v];
            sched[p] = c;
            if (v < n) continue;
            const int a = s.c0[v], b = s.c1[v], I = s.inner[a];
            s.canon[a] = (int16_t)(a < n ? a : c + 1);
            s.canon[b] = (int16_t)(b < n ? b : c + 1 + I);
            s.pos[a] = (int16_t)(p + 1);
            s.pos[b] = (int16_t)(p + 2 + 3 * I);
            sched[p + 3 * s.inner[v]] = c | kUpd;
        }
        __syncwarp();
    }
    for (int k = 3 * n - 5 + lane; k < 3 * n; k += 32) sched[k] = -1;
    // canonical arrays
    for (int v = lane; v < NN; v += 32) {
        const int c = s.canon[v];
        up[c] = v == 0 ? -1 : s.canon[s.par[v]];
        ch[2 * c] = v < n ? -1 : s.canon[s.c0[v]];
        ch[2 * c + 1] = v < n ? -1 : s.canon[s.c1[v]];
        bits[2 * c] = s.bits[v][0];
        bits[2 * c + 1] = s.bits[v][1];
    }
    if (lane == 0) len[0] = 0.0;
    for (int e = lane; e < E; e += 32) {
        int a, b;
        edge(e, a, b);
        const int c = s.canon[s.par[a] == b ? a : b];
        len[c] = lengths && !bad ? lengths[(size_t)tree * E + e] : 0.1;
        if (ts.emap) ts.emap[(size_t)tree * E + e] = c;
    }
    // key = sum of split hashes over internal edges (inner nodes except the first)
    const int top = s.nbr[0][0];
    unsigned __int128 acc = 0;
    for (int v = n + lane; v < NN; v += 32)
        if (v != top) acc += split_hash(s.bits[v][0], s.bits[v][1]);
    unsigned long long lo = (unsigned long long)acc, hi = (unsigned long long)(acc >> 64);
    for (int off = 16; off; off >>= 1) {
        unsigned long long olo = __shfl_down_sync(all, lo, off);
        unsigned long long ohi = __shfl_down_sync(all, hi, off);
        unsigned long long nlo = lo + olo;
        hi = hi + ohi + (nlo < lo);
        lo = nlo;
    }
    if (lane == 0) {
        if (lo == 0 && hi == 0) lo = 1;
        ts.key[2 * tree] = bad ? 0 : lo;
        ts.key[2 * tree + 1] = bad ? 0 : hi;
    }
    // rank of every internal split among the tree's internal splits
    for (int v = lane; v < NN; v += 32) {
        int r = -1;
        if (v >= n && v != top) {
            const unsigned long long blo = s.bits[v][0], bhi = s.bits[v][1];
            r = 0;
            for (int w = n; w < NN; ++w)
                if (w != top && less128(s.bits[w][0], s.bits[w][1], blo, bhi)) ++r;
        }
        erank[s.canon[v]] = r;
    }
}

}  // namespace pt
