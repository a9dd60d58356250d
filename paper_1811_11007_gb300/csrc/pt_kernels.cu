// CUDA kernels of the PT hot path (sm_103a).
//
// Layout in HBM (per group of trees): partial-likelihood vectors in FP32 (mixed
// precision) or FP64.  A site's 4C values are ordered [state][category] and cut
// into 16-byte chunks, stored [slot][chunk][site][values of the chunk]
// (vec_index), so the 32 lanes of a warp read each chunk as one contiguous run,
// and in FP32 with four categories a chunk is one state's four categories: two
// register pairs that the packed FP32 instructions take as they are.
// Transition matrices are ordered [from][to][category] to match.
// Per-site power-of-two scaler counts [slot][site] int32.  Slots of a tree:
// D_v (the subtree below inner node v, at v) for every inner v, then U_v (the
// rest of the tree, at v's parent) for every inner v but the first.
//
// Parallel structure: a lane owns sites; a CTA or a cluster of up to eight owns a tree
// (full optimisation) or one NNI neighbour (proposal optimisation), as the number of
// items leaves room for.  Cross-thread traffic is only the per-evaluation reduction of
// d lnL/dt and d2 lnL/dt2 (FP32 pairs, or FP64) and the scores, so every pass over sites runs
// without barriers.
#include "pt_internal.h"
#include "pt_canon.h"
#include "pt_exchange.h"
#include "pt_gamma.h"
#include "pt_math.h"

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cmath>
#include <cstdint>
#include <type_traits>

namespace pt {

std::atomic<long long> g_launches{0};
long long launch_count() { return g_launches.load(); }

namespace {

constexpr double kLn2 = 0.69314718055994530942;

template <typename R> struct Prec;
template <> struct Prec<float> {
    // stored vectors are rescaled by 2^32 when every entry is below 2^-32, so a
    // product of two stored vectors stays far above the FP32 normal range
    static constexpr int kScaleExp = 32;
    __device__ static float thresh() { return 2.3283064365386963e-10f; }   // 2^-32
    __device__ static float mult() { return 4294967296.0f; }                // 2^32
    __device__ static float rcp(float x) { return rcp_rn(x); }
    __device__ static float mul(float x, float y) { return __fmul_rn(x, y); }  // never part of an FMA
};
template <> struct Prec<double> {
    static constexpr int kScaleExp = 256;
    __device__ static double thresh() { return 8.636168555094445e-78; }      // 2^-256
    __device__ static double mult() { return 1.157920892373162e+77; }        // 2^256
    __device__ static double rcp(double x) { return 1.0 / x; }
    __device__ static double mul(double x, double y) { return __dmul_rn(x, y); }
};

// ---------------------------------------------------------------- canonicaliser
constexpr int kCanonWarps = 4;
__global__ void k_canon(int n, DCount cnt, const int32_t* __restrict__ edges, const double* __restrict__ lengths,
                        TreeSet ts, int32_t* err) {
    __shared__ CanonSmem sm[kCanonWarps];
    const int warp = threadIdx.x >> 5, tree = blockIdx.x * kCanonWarps + warp;
    if (tree < dcount(cnt)) canon_tree(n, tree, threadIdx.x & 31, edges, lengths, ts, err, sm[warp]);
}

// ---------------------------------------------------------------- candidates
// Candidate c = (tree f, internal edge j, swap s): edge node v = n+1+j, its
// parent u, v's sibling B, v's children C < D.  Swap 0 exchanges B and C
// (new split B u D), swap 1 exchanges B and D (new split B u C); the key
// changes by H(new split) - H(C u D).
__global__ void k_enum(int n, DCount Fc, TreeSet fr, uint64_t* __restrict__ nkey, int32_t* __restrict__ cinfo) {
    const int m = 2 * (n - 3);
    const long long total = (long long)dcount(Fc) * m;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < total;
         c += (long long)gridDim.x * blockDim.x) {
        int f = (int)(c / m), r = (int)(c % m), j = r >> 1, sw = r & 1;
        const int NN = 2 * n - 2;
        const int32_t* up = fr.up + (size_t)f * NN;
        const int32_t* ch = fr.ch + (size_t)f * NN * 2;
        const uint64_t* bits = fr.bits + (size_t)f * NN * 2;
        int v = n + 1 + j, u = up[v];
        int sib = ch[2 * u] == v ? ch[2 * u + 1] : ch[2 * u];
        int keep = sw == 0 ? ch[2 * v + 1] : ch[2 * v];
        unsigned __int128 key = ((unsigned __int128)fr.key[2 * f + 1] << 64) | fr.key[2 * f];
        key -= split_hash(bits[2 * v], bits[2 * v + 1]);
        key += split_hash(bits[2 * sib] | bits[2 * keep], bits[2 * sib + 1] | bits[2 * keep + 1]);
        unsigned long long lo = (unsigned long long)key, hi = (unsigned long long)(key >> 64);
        if (!lo && !hi) lo = 1;
        nkey[2 * c] = lo;
        nkey[2 * c + 1] = hi;
        cinfo[4 * c + 0] = f;
        cinfo[4 * c + 1] = v;
        cinfo[4 * c + 2] = sw;
        cinfo[4 * c + 3] = fr.erank[(size_t)f * NN + v];
    }
}

// ---------------------------------------------------------------- visited table
constexpr int kMaxProbe = 1 << 14;

__device__ __forceinline__ size_t slot_hash(unsigned long long lo, unsigned long long hi, unsigned long long mask) {
    return (size_t)(mix64(lo ^ mix64(hi ^ 0x632be59bd9b4e019ull)) & mask);
}

// Finds or claims the slot of a key by linear probing with a 128-bit CAS.
// Returns the slot index and whether this call created it; -1 when the probe
// limit is reached.
__device__ long long table_find_or_claim(Slot* tab, int log2, unsigned long long lo, unsigned long long hi,
                                         bool* created) {
    const unsigned long long mask = (1ull << log2) - 1;
    const unsigned __int128 key = ((unsigned __int128)hi << 64) | lo;
    size_t h = slot_hash(lo, hi, mask);
    for (int p = 0; p < kMaxProbe; ++p) {
        size_t i = (h + p) & mask;
        unsigned __int128* kp = reinterpret_cast<unsigned __int128*>(&tab[i].klo);
        unsigned __int128 old = atomicCAS(kp, (unsigned __int128)0, key);
        if (old == 0) { *created = true; return (long long)i; }
        if (old == key) { *created = false; return (long long)i; }
    }
    return -1;
}

// A thread per 16 bytes, so a warp writes one run of memory (a thread per slot wrote
// 8 bytes at a time 64 bytes apart: 175 us for 2^22 slots).
__global__ void k_table_init(Slot* tab, size_t nslots) {
    ulonglong2* const q = reinterpret_cast<ulonglong2*>(tab);
    const unsigned long long nan = 0x7ff8000000000000ull;
    static_assert(sizeof(Slot) == 64, "chunks: key; tag, ahi; alo, lnl; alpha, pad");
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < 4 * nslots; i += (size_t)gridDim.x * blockDim.x) {
        const int c = (int)(i & 3);
        q[i] = c == 0   ? make_ulonglong2(0, 0)
               : c == 1 ? make_ulonglong2(kTagEmpty, kTagEmpty)
               : c == 2 ? make_ulonglong2(kTagEmpty, nan)
                        : make_ulonglong2(nan, 0);
    }
}

__global__ void k_cand_insert(Slot* tab, int log2, DCount nc, const uint64_t* __restrict__ nkey,
                              const int32_t* __restrict__ cinfo, TreeSet fr, DRound rd, int32_t* cslot,
                              int32_t* flag, int32_t* err, unsigned long long* stats) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int ncand = dcount(nc), round = dround(rd);
    int dup = 0;
    if (i >= ncand && i < nc.cap) { cslot[i] = -1; flag[i] = 0; }  // past the device count
    if (i < ncand && !(fr.key[2 * cinfo[4 * i]] | fr.key[2 * cinfo[4 * i] + 1])) {  // a refused tree proposes nothing
        cslot[i] = -1; flag[i] = 0;
    } else if (i < ncand) {
        bool created;
        long long s = table_find_or_claim(tab, log2, nkey[2 * i], nkey[2 * i + 1], &created);
        if (s < 0) {
            atomicExch(&err[kErrTable], 1);
            cslot[i] = -1; flag[i] = 0;
        } else {
            unsigned long long tag = created ? kTagEmpty : atomicAdd(&tab[s].tag, 0ull);
            if (tag != kTagEmpty && (int)(tag >> 48) < round) {
                cslot[i] = -1; flag[i] = 0; dup = 1;
            } else {
                int f = cinfo[4 * i];
                atomicMin(&tab[s].ahi, (unsigned long long)fr.key[2 * f + 1]);
                cslot[i] = (int32_t)s; flag[i] = 1;
            }
        }
    }
    unsigned b = __ballot_sync(0xffffffffu, dup);
    if ((threadIdx.x & 31) == 0 && b) atomicAdd(&stats[kStDup], (unsigned long long)__popc(b));
}

// phase 2: smallest low word of the parent key among proposers with the smallest high word;
// phase 3: smallest (edge rank, swap) among proposers with the smallest parent key;
// phase 4: flag = this candidate is the winner of its slot.
__global__ void k_cand_arb(int phase, Slot* tab, DCount nc, const int32_t* __restrict__ cinfo, TreeSet fr, DRound rd,
                           const int32_t* __restrict__ cslot, int32_t* flag) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= dcount(nc) || !flag[i]) return;
    const int round = dround(rd);
    Slot* sl = &tab[cslot[i]];
    int f = cinfo[4 * i];
    unsigned long long phi = fr.key[2 * f + 1], plo = fr.key[2 * f];
    unsigned long long me = ((unsigned long long)round << 48) | ((unsigned long long)cinfo[4 * i + 3] << 1) |
                            (unsigned long long)cinfo[4 * i + 2];
    if (phase == 2) {
        if (sl->ahi == phi) atomicMin(&sl->alo, plo);
    } else if (phase == 3) {
        if (sl->ahi == phi && sl->alo == plo) atomicMin(&sl->tag, me);
    } else {
        flag[i] = (sl->ahi == phi && sl->alo == plo && sl->tag == me) ? 1 : 0;
    }
}

__global__ void k_make_items(int ncand, const int32_t* __restrict__ flag, const int32_t* __restrict__ pos,
                             const int32_t* __restrict__ cinfo, const int32_t* __restrict__ cslot,
                             const uint64_t* __restrict__ nkey, Item* items, uint64_t* ikey) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ncand || !flag[i]) return;
    Item it;
    it.tree = cinfo[4 * i]; it.v = cinfo[4 * i + 1]; it.swap = cinfo[4 * i + 2]; it.slot = cslot[i];
    items[pos[i]] = it;
    ikey[2 * pos[i]] = nkey[2 * i];
    ikey[2 * pos[i] + 1] = nkey[2 * i + 1];
}

__global__ void k_compact_idx(int N, const int32_t* __restrict__ flag, const int32_t* __restrict__ pos, int32_t* idx) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N && flag[i]) idx[pos[i]] = i;
}

__global__ void k_fill_i32(int N, int32_t* a, int32_t va, int32_t* b, int32_t vb) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) {
        a[i] = va;
        if (b) b[i] = vb;
    }
}

// Hill-climb move choice: per tree f (items f*m .. f*m+m-1, every neighbour of
// the tree), the neighbour with the best proposal score, ties by the smallest
// key (high word first); a NaN score never wins.  One warp per tree.
__global__ void k_climb_best(int F, int m, const double* __restrict__ lnl, const uint64_t* __restrict__ ikey,
                             int32_t* best) {
    const int f = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (f >= F) return;
    double bl = -INFINITY;
    unsigned long long bhi = ~0ull, blo = ~0ull;
    int bi = -1;
    for (int r = lane; r < m; r += 32) {
        const int i = f * m + r;
        const double x = lnl[i];
        const unsigned long long hi = ikey[2 * i + 1], lo = ikey[2 * i];
        if (!(x == x)) continue;
        if (bi < 0 || x > bl || (x == bl && (hi < bhi || (hi == bhi && lo < blo)))) {
            bl = x; bhi = hi; blo = lo; bi = i;
        }
    }
    for (int o = 16; o; o >>= 1) {
        const double x = __shfl_xor_sync(0xffffffffu, bl, o);
        const unsigned long long hi = __shfl_xor_sync(0xffffffffu, bhi, o), lo = __shfl_xor_sync(0xffffffffu, blo, o);
        const int i = __shfl_xor_sync(0xffffffffu, bi, o);
        if (i >= 0 && (bi < 0 || x > bl || (x == bl && (hi < bhi || (hi == bhi && lo < blo))))) {
            bl = x; bhi = hi; blo = lo; bi = i;
        }
    }
    if (lane == 0) best[f] = bi < 0 ? f * m : bi;
}

// Enters whole trees (starts, or a caller's frontier) as visited.  Among
// equal keys the lowest index wins; status/lnl written by the winner.  A key
// already present from an earlier call is left as it is (winner = -1).
__global__ void k_insert_trees(Slot* tab, int log2, DCount cnt, TreeSet ts, const double* lnl, const int32_t* status,
                               int32_t* winner, int32_t* err) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= dcount(cnt)) return;
    if (!(ts.key[2 * i] | ts.key[2 * i + 1])) { winner[i] = -1; return; }  // a refused tree
    bool created;
    long long s = table_find_or_claim(tab, log2, ts.key[2 * i], ts.key[2 * i + 1], &created);
    if (s < 0) { atomicExch(&err[kErrTable], 1); winner[i] = -1; return; }
    // only slots claimed by this call (still untagged) take part; a key entered
    // earlier keeps its record
    unsigned long long tag = created ? kTagEmpty : atomicAdd(&tab[s].tag, 0ull);
    if (tag != kTagEmpty) { winner[i] = -1; return; }
    atomicMin(&tab[s].alo, (unsigned long long)i);
    winner[i] = (int32_t)s;
}

__global__ void k_insert_trees_fin(Slot* tab, DCount cnt, const double* lnl, const int32_t* status, DRound rd,
                                   int32_t* winner) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= dcount(cnt) || winner[i] < 0) return;
    const int round = dround(rd);
    Slot* sl = &tab[winner[i]];
    if (sl->alo != (unsigned long long)i) { winner[i] = -1; return; }
    sl->lnl = lnl ? lnl[i] : __longlong_as_double(0x7ff8000000000000ll);
    sl->tag = ((unsigned long long)round << 48) | (unsigned long long)(status ? status[i] : 2);
}

// lmax = max(lmax, max over masked lnl) (ordered-integer trick on doubles)
__device__ __forceinline__ long long ord_of(double x) {
    long long b = __double_as_longlong(x);
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffll);
}
__device__ __forceinline__ double of_ord(long long b) {
    return __longlong_as_double(b >= 0 ? b : (b ^ 0x7fffffffffffffffll));
}
__global__ void k_lmax(DCount cnt, const double* lnl, const int32_t* mask, double* lmax) {
    __shared__ long long best;
    const int count = dcount(cnt);
    if (threadIdx.x == 0) best = ord_of(*lmax);
    __syncthreads();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        if ((!mask || mask[i] >= 0) && lnl[i] == lnl[i]) atomicMax(&best, ord_of(lnl[i]));
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long* p = reinterpret_cast<unsigned long long*>(lmax);
        unsigned long long cur = *p;
        while (true) {
            double c = __longlong_as_double((long long)cur);
            if (ord_of(c) >= best) break;
            unsigned long long prev = atomicCAS(p, cur, (unsigned long long)__double_as_longlong(of_ord(best)));
            if (prev == cur) break;
            cur = prev;
        }
    }
}

// Visit decision of fully optimised trees: GOOD iff lnl >= lmax - thr.
__global__ void k_finalize_trees(Slot* tab, DCount cnt, const int32_t* slot_of, const double* lnl, const double* lmax,
                                 double thr, DRound rd, int32_t* good, unsigned long long* stats,
                                 const double* alpha) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int count = dcount(cnt), round = dround(rd);
    int g = 0;
    if (i < count) {
        g = lnl[i] >= *lmax - thr;
        good[i] = g;
        if (slot_of && slot_of[i] >= 0) {
            Slot* sl = &tab[slot_of[i]];
            sl->lnl = lnl[i];
            if (alpha) sl->alpha = alpha[i];
            sl->tag = ((unsigned long long)round << 48) | (unsigned long long)(g ? 2 : 3);
        }
    }
    unsigned b = __ballot_sync(0xffffffffu, g);
    if ((threadIdx.x & 31) == 0 && b) atomicAdd(&stats[kStGood], (unsigned long long)__popc(b));
}

__global__ void k_dump_flag(const Slot* tab, size_t nslots, int32_t* flag) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nslots; i += (size_t)gridDim.x * blockDim.x)
        flag[i] = (tab[i].klo | tab[i].khi) ? 1 : 0;
}
__global__ void k_dump_gather(const Slot* tab, size_t nslots, const int32_t* flag, const int32_t* pos, uint64_t* keys,
                              uint8_t* status, double* lnl) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nslots; i += (size_t)gridDim.x * blockDim.x) {
        if (!flag[i]) continue;
        int p = pos[i];
        keys[2 * p] = tab[i].klo; keys[2 * p + 1] = tab[i].khi;
        unsigned long long t = tab[i].tag;
        status[p] = (uint8_t)(t == kTagEmpty ? 0 : (t & 0xff));
        lnl[p] = tab[i].lnl;
    }
}

// ---------------------------------------------------------------- scheduling order
// Counting sort of the kept trees by predicted cost (one block): a histogram of
// the binned costs, bins in decreasing order, scatter with per-bin cursors.
__global__ void k_cost_order(DCount cnt, const int32_t* kidx, const float* cost, int32_t* order) {
    __shared__ int hist[65], start[65];
    const int K = dcount(cnt);
    for (int b = threadIdx.x; b < 65; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    auto bin = [&](int k) {
        const float x = cost[kidx[k]] * 32.f;
        return x == x ? 1 + (int)fminf(63.f, fmaxf(0.f, x)) : 64;  // NaN: first
    };
    for (int k = threadIdx.x; k < K; k += blockDim.x) atomicAdd(&hist[bin(k)], 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int b = 64; b >= 1; --b) { start[b] = acc; acc += hist[b]; }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) order[atomicAdd(&start[bin(k)], 1)] = k;
}

// ---------------------------------------------------------------- Gamma shape
// Shape of each frontier tree: the one its visit recorded in the visited table
// (read-only probe of the key), else the model's.
__global__ void k_frontier_alpha(TreeSet fr, int count, const Slot* tab, int log2, double base, double* alpha) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= count) return;
    const unsigned long long lo = fr.key[2 * f], hi = fr.key[2 * f + 1], mask = (1ull << log2) - 1;
    double a = base;
    size_t h = slot_hash(lo, hi, mask);
    for (int p = 0; p < kMaxProbe; ++p) {
        const Slot& sl = tab[(h + p) & mask];
        if (sl.klo == lo && sl.khi == hi) {
            if (sl.alpha == sl.alpha) a = sl.alpha;
            break;
        }
        if (!(sl.klo | sl.khi)) break;
    }
    alpha[f] = a;
}

// Category rates [t][kMaxCat] of tree t's shape alpha[t] (one thread per tree).
__global__ void k_gamma_rates(int count, int C, const double* alpha, double* rates) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < count) discrete_gamma(alpha[t], C, rates + (size_t)t * kMaxCat);
}

// ---------------------------------------------------------------- split frequencies
// Split table: 128-bit split bitset (side without taxon 0) -> summed weight.
// Tree i adds w_i = exp(lnl_i - max lnl) to each of its n-3 non-trivial splits
// (the leaf sets below its inner nodes other than the first; trees are rooted
// at leaf 0, so those sets never hold taxon 0).
__global__ void k_split_init(SplitSlot* tab, size_t nslots) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nslots; i += (size_t)gridDim.x * blockDim.x) {
        tab[i].klo = 0; tab[i].khi = 0; tab[i].w = 0.0; tab[i].trees = 0;
    }
}

__global__ void k_split_add(TreeSet ts, int count, const double* lnl, const double* lmax, SplitSlot* tab, int log2,
                            int32_t* err) {
    const int n = ts.n, NN = 2 * n - 2, per = n - 3;
    const long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (x >= (long long)count * per) return;
    const int t = (int)(x / per), v = n + 1 + (int)(x % per);
    const uint64_t* bits = ts.bits + ((size_t)t * NN + v) * 2;
    const unsigned long long lo = bits[0], hi = bits[1];
    const double w = exp(lnl[t] - *lmax);
    const unsigned long long mask = (1ull << log2) - 1;
    const unsigned __int128 key = ((unsigned __int128)hi << 64) | lo;
    size_t h = slot_hash(lo, hi, mask);
    for (int p = 0; p < kMaxProbe; ++p) {
        const size_t i = (h + p) & mask;
        unsigned __int128* kp = reinterpret_cast<unsigned __int128*>(&tab[i].klo);
        const unsigned __int128 old = atomicCAS(kp, (unsigned __int128)0, key);
        if (old == 0 || old == key) {
            atomicAdd(&tab[i].w, w);
            atomicAdd(&tab[i].trees, 1ull);
            return;
        }
    }
    atomicExch(&err[kErrTable], 1);
}

__global__ void k_split_flag(const SplitSlot* tab, size_t nslots, int32_t* flag) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nslots; i += (size_t)gridDim.x * blockDim.x)
        flag[i] = (tab[i].klo | tab[i].khi) ? 1 : 0;
}

__global__ void k_split_gather(const SplitSlot* tab, size_t nslots, const int32_t* flag, const int32_t* pos,
                               uint64_t* splits, double* w, unsigned long long* trees) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nslots; i += (size_t)gridDim.x * blockDim.x) {
        if (!flag[i]) continue;
        const int p = pos[i];
        splits[2 * p] = tab[i].klo;
        splits[2 * p + 1] = tab[i].khi;
        w[p] = tab[i].w;
        trees[p] = tab[i].trees;
    }
}

// ---------------------------------------------------------------- scan
__global__ void k_scan_block(const int32_t* in, int32_t* out, int N, int32_t* bsum) {
    __shared__ int32_t ws[32];
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    int x = i < N ? in[i] : 0, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int v = x;
    for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += y; }
    if (lane == 31) ws[w] = v;
    __syncthreads();
    if (w == 0) {
        int s = lane < (blockDim.x >> 5) ? ws[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(0xffffffffu, s, o); if (lane >= o) s += y; }
        ws[lane] = s;
    }
    __syncthreads();
    int pre = (w ? ws[w - 1] : 0) + v - x;
    if (i < N) out[i] = pre;
    if (threadIdx.x == blockDim.x - 1) bsum[blockIdx.x] = ws[(blockDim.x >> 5) - 1];
}
__global__ void k_scan_sums(int32_t* bsum, int nb) {
    __shared__ int32_t ws[32];
    __shared__ int32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nb; base += blockDim.x) {
        int i = base + threadIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        int x = i < nb ? bsum[i] : 0, v = x;
        for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += y; }
        if (lane == 31) ws[w] = v;
        __syncthreads();
        if (w == 0) {
            int s = lane < (blockDim.x >> 5) ? ws[lane] : 0;
            for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(0xffffffffu, s, o); if (lane >= o) s += y; }
            ws[lane] = s;
        }
        __syncthreads();
        int pre = carry + (w ? ws[w - 1] : 0) + v - x;
        if (i < nb) bsum[i] = pre;
        __syncthreads();
        if (threadIdx.x == 0) carry += ws[(blockDim.x >> 5) - 1];
        __syncthreads();
    }
}
__global__ void k_scan_add(int32_t* out, int N, const int32_t* bsum) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) out[i] += bsum[blockIdx.x];
}
__global__ void k_scan_total(const int32_t* in, const int32_t* out, int N, int32_t* total) {
    if (threadIdx.x == 0) *total = N > 0 ? out[N - 1] + in[N - 1] : 0;
}
__global__ void k_mul_counts(int na, const int* F, const int* m, int* ncand) {
    const int k = threadIdx.x;
    if (k < na) ncand[k] = F[k] * m[k];
}
__global__ void k_prefix_counts(int ng, const int* cnt, const int* perm, int* gstart) {
    if (threadIdx.x == 0) {
        int acc = 0;
        gstart[0] = 0;
        for (int g = 0; g < ng; ++g) { acc += cnt[perm ? perm[g] : g]; gstart[g + 1] = acc; }
    }
}

// ---------------------------------------------------------------- tree outputs
// Materialises NNI neighbours as edge lists in the parent's canonical
// numbering with the five optimised lengths; the canonicaliser renumbers them.
__global__ void k_materialize(int n, DCount nk, const int32_t* kidx, const Item* items, TreeSet fr, const double* len5,
                              int32_t* edges_out, double* lengths_out, int32_t* slot_of) {
    const int NN = 2 * n - 2, E = 2 * n - 3;
    const long long total = (long long)dcount(nk) * E;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i / E), w = (int)(i % E) + 1, ii = kidx ? kidx[k] : k;
        const Item it = items[ii];
        const int32_t* up = fr.up + (size_t)it.tree * NN;
        const int32_t* ch = fr.ch + (size_t)it.tree * NN * 2;
        const int v = it.v, u = up[v];
        const int sib = ch[2 * u] == v ? ch[2 * u + 1] : ch[2 * u];
        const int c0 = ch[2 * v], c1 = ch[2 * v + 1];
        const double* t5 = len5 + (size_t)ii * 5;
        int p = up[w];
        if (w == sib) p = v;
        if (w == (it.swap == 0 ? c0 : c1)) p = u;
        const double l = w == v     ? t5[0]
                         : w == u   ? t5[1]
                         : w == sib ? t5[2]
                         : w == c0  ? t5[3]
                         : w == c1  ? t5[4]
                                    : fr.len[(size_t)it.tree * NN + w];
        edges_out[2 * i] = w;
        edges_out[2 * i + 1] = p;
        lengths_out[i] = l;
        if (w == 1) slot_of[k] = it.slot;
    }
}

__global__ void k_len5_inherit(int n, DCount cnt, const Item* items, TreeSet fr, double* len5) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= dcount(cnt)) return;
    const int NN = 2 * n - 2;
    const Item it = items[o];
    const int32_t* up = fr.up + (size_t)it.tree * NN;
    const int32_t* ch = fr.ch + (size_t)it.tree * NN * 2;
    const double* len = fr.len + (size_t)it.tree * NN;
    const int v = it.v, u = up[v];
    const int sib = ch[2 * u] == v ? ch[2 * u + 1] : ch[2 * u];
    const int node[5] = {v, u, sib, ch[2 * v], ch[2 * v + 1]};
    for (int b = 0; b < 5; ++b) len5[(size_t)o * 5 + b] = len[node[b]];
}

__global__ void k_prop_full_finish(DCount cnt, const Item* items, const double* lnl, const double* lmax, double thr,
                                   DRound rd, Slot* tab, int32_t* kept) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= dcount(cnt)) return;
    const double f = lnl[o];
    const int k = f >= *lmax - thr;
    kept[o] = k;
    Slot* sl = &tab[items[o].slot];
    sl->lnl = f;
    sl->tag = ((unsigned long long)dround(rd) << 48) | (unsigned long long)(k ? 4 : 1);
}

__global__ void k_gather_i32(DCount cnt, const int32_t* idx, const int32_t* src, int32_t* dst) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < dcount(cnt)) dst[k] = src[idx[k]];
}

// Gathers trees idx[k] of a set into canonical edge lists + lengths + lnl + keys.
// A thread per tree and edge (a thread per tree walked its edges one by one, a line
// of memory apart from its neighbours': 95 us for the lengths of 256 trees of 64 taxa).
__global__ void k_gather_out(int n, DCount cnt, const int32_t* idx, TreeSet ts, const double* lnl, int32_t* edges_out,
                             double* lengths_out, double* lnl_out, uint64_t* keys_out) {
    const int NN = 2 * n - 2, E = 2 * n - 3;
    const long long total = (long long)dcount(cnt) * E;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(i / E), e = (int)(i % E), t = idx ? idx[k] : k;
        if (edges_out) {
            edges_out[2 * i] = e + 1;
            edges_out[2 * i + 1] = ts.up[(size_t)t * NN + e + 1];
        }
        if (lengths_out) lengths_out[i] = ts.len[(size_t)t * NN + e + 1];
        if (e == 0 && lnl_out) lnl_out[k] = lnl[t];
        if (e == 0 && keys_out) { keys_out[2 * k] = ts.key[2 * t]; keys_out[2 * k + 1] = ts.key[2 * t + 1]; }
    }
}

__global__ void k_lengths_to_input(int n, int count, TreeSet ts, double* lengths_out) {
    const int NN = 2 * n - 2, E = 2 * n - 3;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)count * E;
         i += (long long)gridDim.x * blockDim.x)
        lengths_out[i] = ts.len[(size_t)(i / E) * NN + ts.emap[i]];
}

// ---------------------------------------------------------------- likelihood arithmetic
// P_r(t)[i][j] = isqpi_i * sum_k R_ik exp(lam_k r t) R_jk * sqpi_j, one row
// (4 entries) per call, exponentials in FP64.
template <typename R>
__device__ __forceinline__ void pmat_row(const Model& M, double rt, int i, R* row, int stride = 1) {
    double e[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) e[k] = exp(M.lam[k] * rt);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) acc += M.R[i * 4 + k] * e[k] * M.R[j * 4 + k];
        row[j * stride] = (R)(acc * M.isqpi[i] * M.sqpi[j]);
    }
}

// ---------------------------------------------------------------- packed FP32
// Blackwell's FP32 pipe takes two FP32 operations per lane in one instruction
// (fma / mul / add .f32x2 on 64-bit register pairs, each half rounded as the
// scalar instruction rounds it).  With four categories every vector operation
// here runs on pairs of categories: the issue slots of the 4 x 4 products halve
// and every result keeps its bits.  With the chunked vectors it took a sum-table build
// of a proposal (27 taxa x 816 patterns) from 16.5 to 11 thousand cycles.
using f32x2 = float2;
__device__ __forceinline__ unsigned long long& b64(f32x2& x) { return reinterpret_cast<unsigned long long&>(x); }
__device__ __forceinline__ unsigned long long b64c(f32x2 x) {
    return reinterpret_cast<const unsigned long long&>(x);
}
__device__ __forceinline__ f32x2 pmul(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(b64(d)) : "l"(b64c(a)), "l"(b64c(b)));
    return d;
}
__device__ __forceinline__ f32x2 padd(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(b64(d)) : "l"(b64c(a)), "l"(b64c(b)));
    return d;
}
__device__ __forceinline__ f32x2 pfma(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(b64(d)) : "l"(b64c(a)), "l"(b64c(b)), "l"(b64c(c)));
    return d;
}
__device__ __forceinline__ f32x2 pneg(f32x2 a) { return make_float2(-a.x, -a.y); }
// a - b as one packed instruction (b * -1 is exact)
__device__ __forceinline__ f32x2 psub(f32x2 a, f32x2 b) { return pfma(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float pmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float padd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float pfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float pneg(float a) { return -a; }
__device__ __forceinline__ float psub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ f32x2 pair(const float* x) { return make_float2(x[0], x[1]); }

// Source of a 4C-wide vector at a site: a tip (code lookup, by the site pg) or a
// stored slot (`ld` sites per chunk, see vec_index; by the slot's index p).
template <typename R, int C>
struct Src {
    const R* clv;      // slot base (nullptr for a tip)
    const int32_t* scl;
    const uint8_t* tip;  // tip codes of the leaf (nullptr for a slot)
};

// A stored vector at site p of a slot of ld sites, x[state * C + category].
template <typename R, int C>
__device__ __forceinline__ void load_vec(const R* src, int ld, int p, R* x) {
    if constexpr (sizeof(R) == 4) {
#pragma unroll
        for (int q = 0; q < C; ++q) {
            const float4 v = reinterpret_cast<const float4*>(src)[(size_t)q * ld + p];
            x[4 * q] = v.x; x[4 * q + 1] = v.y; x[4 * q + 2] = v.z; x[4 * q + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 2 * C; ++q) {
            const double2 v = reinterpret_cast<const double2*>(src)[(size_t)q * ld + p];
            x[2 * q] = v.x; x[2 * q + 1] = v.y;
        }
    }
}

template <typename R, int C>
__device__ __forceinline__ void load_raw(const Src<R, C>& s, int ld, int p, int pg, R* x, int& cnt) {
    if (s.tip) {
        int code = s.tip[pg];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int r = 0; r < C; ++r) x[i * C + r] = (code >= 4 || code == i) ? R(1) : R(0);
        cnt = 0;
    } else {
        load_vec<R, C>(s.clv, ld, p, x);
        cnt = s.scl[p];
    }
}

// y_r = P_r x_r, P [16][C] ([from * 4 + to][category]), x and y [state][category].
template <typename R, int C>
__device__ __forceinline__ void apply_p_reg(const R* Pm, const R* x, R* y) {
    if constexpr (sizeof(R) == 4 && C == 4) {
        const float4* P4 = reinterpret_cast<const float4*>(Pm);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float4 w = P4[i * 4];
            f32x2 lo = pmul(make_float2(w.x, w.y), pair(x)), hi = pmul(make_float2(w.z, w.w), pair(x + 2));
#pragma unroll
            for (int j = 1; j < 4; ++j) {
                w = P4[i * 4 + j];
                lo = pfma(make_float2(w.x, w.y), pair(x + 4 * j), lo);
                hi = pfma(make_float2(w.z, w.w), pair(x + 4 * j + 2), hi);
            }
            y[4 * i] = lo.x; y[4 * i + 1] = lo.y; y[4 * i + 2] = hi.x; y[4 * i + 3] = hi.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            R w[4 * C];  // row i of every category: 4C consecutive values on a 16-byte boundary
#pragma unroll
            for (int q = 0; q < 4 * C * (int)sizeof(R) / 16; ++q) {
                if constexpr (sizeof(R) == 4) {
                    const float4 v = reinterpret_cast<const float4*>(Pm)[i * C + q];
                    w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
                } else {
                    const double2 v = reinterpret_cast<const double2*>(Pm)[i * 2 * C + q];
                    w[2 * q] = v.x; w[2 * q + 1] = v.y;
                }
            }
#pragma unroll
            for (int r = 0; r < C; ++r) {
                R acc = w[r] * x[r];
#pragma unroll
                for (int j = 1; j < 4; ++j) acc = fma(w[j * C + r], x[j * C + r], acc);
                y[i * C + r] = acc;
            }
        }
    }
}

// y_r = P_r x_r of a source; for a tip the product is a column of P (or all
// ones for a gap).
template <typename R, int C>
__device__ __forceinline__ void apply_p(const R* Pm, const Src<R, C>& s, int ld, int p, int pg, R* y, int& cnt) {
    if (s.tip) {
        int code = s.tip[pg];
        cnt = 0;
        if (code >= 4) {
#pragma unroll
            for (int q = 0; q < 4 * C; ++q) y[q] = R(1);
        } else if constexpr (sizeof(R) == 4 && C == 4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 v = reinterpret_cast<const float4*>(Pm)[i * 4 + code];
                y[4 * i] = v.x; y[4 * i + 1] = v.y; y[4 * i + 2] = v.z; y[4 * i + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int r = 0; r < C; ++r) y[i * C + r] = Pm[(i * 4 + code) * C + r];
        }
        return;
    }
    R x[4 * C];
    load_raw<R, C>(s, ld, p, pg, x, cnt);
    apply_p_reg<R, C>(Pm, x, y);
}

// y *= z, elementwise
template <typename R, int C>
__device__ __forceinline__ void mul_vec(R* y, const R* z) {
    if constexpr (sizeof(R) == 4) {
#pragma unroll
        for (int q = 0; q < 4 * C; q += 2) {
            const f32x2 t = pmul(pair(y + q), pair(z + q));
            y[q] = t.x; y[q + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4 * C; ++q) y[q] *= z[q];
    }
}

template <typename R, int C>
__device__ __forceinline__ void store_vec(R* dst, int ld, int p, const R* y) {
    if constexpr (sizeof(R) == 4) {
#pragma unroll
        for (int q = 0; q < C; ++q)
            reinterpret_cast<float4*>(dst)[(size_t)q * ld + p] =
                make_float4(y[4 * q], y[4 * q + 1], y[4 * q + 2], y[4 * q + 3]);
    } else {
#pragma unroll
        for (int q = 0; q < 2 * C; ++q)
            reinterpret_cast<double2*>(dst)[(size_t)q * ld + p] = make_double2(y[2 * q], y[2 * q + 1]);
    }
}

// ---------------------------------------------------------------- compensated FP32 (scores of the mixed path)
// The pair operations on T = float, or T = f32x2: two categories at once.
template <typename T>
struct F2T {
    T h, l;
};
template <typename T>
__device__ __forceinline__ F2T<T> t2_norm(T h, T l) {  // f2_norm
    const T s = padd(h, l);
    return F2T<T>{s, psub(l, psub(s, h))};
}
template <typename T>
__device__ __forceinline__ F2T<T> t2_mul(F2T<T> a, F2T<T> b) {  // f2_mul
    const T p = pmul(a.h, b.h);
    T e = pfma(a.h, b.h, pneg(p));
    e = pfma(a.h, b.l, e);
    e = pfma(a.l, b.h, e);
    return t2_norm<T>(p, e);
}
// The lanes of a C-category vector: pairs of categories, or the one category.
template <int C>
struct Lanes {
    using T = f32x2;
    static constexpr int n = C / 2, w = 2;
};
template <>
struct Lanes<1> {
    using T = float;
    static constexpr int n = 1, w = 1;
};
__device__ __forceinline__ void lane_get(const float* p, float& x) { x = *p; }
__device__ __forceinline__ void lane_get(const float* p, f32x2& x) { x = *reinterpret_cast<const f32x2*>(p); }
template <typename T>
__device__ __forceinline__ T lane_all(float x);
template <>
__device__ __forceinline__ float lane_all<float>(float x) { return x; }
template <>
__device__ __forceinline__ f32x2 lane_all<f32x2>(float x) { return make_float2(x, x); }

// y = P x for pairs on lane group g of the categories: P as (ph, pl) [16][C],
// x and y [4].  Every term is non-negative (probabilities times likelihoods);
// the exact products ph x_h are summed by two-sums, the small terms (product
// errors, ph x_l, pl x_h, the sums' errors) in a plain FP32 correction, kept
// negated (cn) so that each product's error takes one instruction.
template <int C>
__device__ __forceinline__ void f2_apply4(const float* ph, const float* pl, int g,
                                          const F2T<typename Lanes<C>::T>* x, F2T<typename Lanes<C>::T>* y) {
    using T = typename Lanes<C>::T;
    T nh[4], nl[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        nh[j] = pneg(x[j].h);
        nl[j] = pneg(x[j].l);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        T s{}, cn{};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            T a, b;
            lane_get(ph + (i * 4 + j) * C + g * Lanes<C>::w, a);
            lane_get(pl + (i * 4 + j) * C + g * Lanes<C>::w, b);
            const T p = pmul(a, x[j].h);
            const T e = pfma(a, nh[j], p);
            cn = j == 0 ? e : padd(cn, e);
            cn = pfma(a, nl[j], cn);
            cn = pfma(b, nh[j], cn);
            if (j == 0) {
                s = p;
            } else {
                const T t = padd(s, p), bb = psub(t, s);
                cn = padd(cn, padd(psub(psub(t, bb), s), psub(bb, p)));
                s = t;
            }
        }
        const T t = psub(s, cn);
        y[i] = F2T<T>{t, psub(psub(s, t), cn)};
    }
}

// x *= y for 4 pairs
template <typename T>
__device__ __forceinline__ void f2_mul4(F2T<T>* x, const F2T<T>* y) {
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = t2_mul<T>(x[i], y[i]);
}

__device__ __forceinline__ float lane_max(float x) { return x; }
__device__ __forceinline__ float lane_max(f32x2 x) { return fmaxf(x.x, x.y); }
// exact power-of-two scaling of 4 pairs to max h in [1, 2), each category on its
// own; the exponents removed, one per category
__device__ __forceinline__ float pow2_norm(float mx, int& e) {
    if (!(mx > 0.f)) { e = 0; return 1.f; }
    e = ((__float_as_int(mx) >> 23) & 0xff) - 127;
    if (e < -125) e = -125;
    return __int_as_float((127 - e) << 23);
}
__device__ __forceinline__ void f2_normalise4(F2T<float>* x, int* e) {
    const float m = pow2_norm(fmaxf(fmaxf(x[0].h, x[1].h), fmaxf(x[2].h, x[3].h)), e[0]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[i].h *= m;
        x[i].l *= m;
    }
}
__device__ __forceinline__ void f2_normalise4(F2T<f32x2>* x, int* e) {
    f32x2 m;
    m.x = pow2_norm(fmaxf(fmaxf(x[0].h.x, x[1].h.x), fmaxf(x[2].h.x, x[3].h.x)), e[0]);
    m.y = pow2_norm(fmaxf(fmaxf(x[0].h.y, x[1].h.y), fmaxf(x[2].h.y, x[3].h.y)), e[1]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[i].h = pmul(x[i].h, m);
        x[i].l = pmul(x[i].l, m);
    }
}
__device__ __forceinline__ F2 lane_of(F2T<float> x, int) { return F2{x.h, x.l}; }
__device__ __forceinline__ F2 lane_of(F2T<f32x2> x, int k) { return k ? F2{x.h.y, x.l.y} : F2{x.h.x, x.l.x}; }

// x * 2^-d for d >= 0 (0 when far below the FP32 range: negligible next to the other term)
__device__ __forceinline__ F2 f2_down(F2 x, int d) {
    if (d > 120) return F2{0.f, 0.f};
    const float m = __int_as_float((127 - d) << 23);
    return F2{x.h * m, x.l * m};
}

// acc * 2^E += x * 2^e (pairs with exponents; acc.h == 0 means empty)
__device__ __forceinline__ void f2_merge(F2& acc, int& E, F2 x, int e) {
    if (!(acc.h > 0.f)) { acc = x; E = e; return; }
    if (e > E) { acc = f2_down(acc, e - E); E = e; }
    else x = f2_down(x, E - e);
    acc = f2_add(acc, x);
}

// Source of a pair vector at a site: a tip (code lookup, exact) or a stored
// slot (h and l arrays of the same layout, one scaler count).
template <int C>
struct Src2 {
    const float* h;
    const float* l;
    const int32_t* scl;
    const uint8_t* tip;
};

// Lane group g of y = P x for a pair source (P: [16][C] pairs): slot index p of
// slots of ld sites, site pg of a tip row.
template <int C>
__device__ __forceinline__ void f2_apply_src4(const float* Ph, const float* Pl, const Src2<C>& s, int ld, int p, int pg, int g,
                                              F2T<typename Lanes<C>::T>* y) {
    using T = typename Lanes<C>::T;
    constexpr int w = Lanes<C>::w;
    if (s.tip) {
        const int code = s.tip[pg];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            T a, b;
            lane_get(Ph + (i * 4 + (code & 3)) * C + g * w, a);
            lane_get(Pl + (i * 4 + (code & 3)) * C + g * w, b);
            y[i] = code >= 4 ? F2T<T>{lane_all<T>(1.f), lane_all<T>(0.f)} : F2T<T>{a, b};
        }
        return;
    }
    F2T<T> x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        lane_get(s.h + vec_index<float>(ld, p, j * C + g * w), x[j].h);
        lane_get(s.l + vec_index<float>(ld, p, j * C + g * w), x[j].l);
    }
    f2_apply4<C>(Ph, Pl, g, x, y);
}

// One site of a stored pair vector: the join of two sources under P_a and P_b,
// rescaled by 2^32 when every h is below 2^-32 (as rescale()), and its scaler count.
template <int C>
__device__ __forceinline__ void f2_join(const float* Pah, const float* Pal, const Src2<C>& a, const float* Pbh,
                                        const float* Pbl, const Src2<C>& b, int ld, int p, int pg, float* dh, float* dl,
                                        int32_t* ds) {
    using T = typename Lanes<C>::T;
    constexpr int n = Lanes<C>::n, w = Lanes<C>::w;
    int kk = (a.tip ? 0 : a.scl[p]) + (b.tip ? 0 : b.scl[p]);
    F2T<T> y[n][4];
    float mx = 0.f;
#pragma unroll
    for (int g = 0; g < n; ++g) {
        F2T<T> z[4];
        f2_apply_src4<C>(Pah, Pal, a, ld, p, pg, g, y[g]);
        f2_apply_src4<C>(Pbh, Pbl, b, ld, p, pg, g, z);
        f2_mul4<T>(y[g], z);
#pragma unroll
        for (int i = 0; i < 4; ++i) mx = fmaxf(mx, lane_max(y[g][i].h));
    }
    if (mx < Prec<float>::thresh()) {
        const T m = lane_all<T>(Prec<float>::mult());
#pragma unroll
        for (int g = 0; g < n; ++g)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                y[g][i].h = pmul(y[g][i].h, m);
                y[g][i].l = pmul(y[g][i].l, m);
            }
        ++kk;
    }
    float h[4 * C], l[4 * C];
#pragma unroll
    for (int g = 0; g < n; ++g)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < w; ++k) {
                const F2 v = lane_of(y[g][i], k);
                h[i * C + g * w + k] = v.h;
                l[i * C + g * w + k] = v.l;
            }
    store_vec<float, C>(dh, ld, p, h);
    store_vec<float, C>(dl, ld, p, l);
    ds[p] = kk;
}

// ln of a pair site likelihood times 2^E, in FP64
__device__ __forceinline__ double f2_log(F2 L, int E) {
    return log((double)L.h + (double)L.l) + (double)E * kLn2;
}

// Entry q (< 16C, [16][C]) of P_r(t) of a branch as a pair (FP64 sum, split once):
// W[(i*4+j)*4+k] = isqpi_i sqpi_j R_ik R_jk, ex[k*C+r] = exp(lam_k rate_r t).
template <int C>
__device__ __forceinline__ void f2_pmat_entry(const double* W, const double* ex, int q, float* Ph, float* Pl) {
    const int r = q % C, ij = q / C;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) acc += W[ij * 4 + k] * ex[k * C + r];
    const F2 v = f2_of(acc);
    Ph[q] = v.h;
    Pl[q] = v.l;
}

// threshold rescale of a stored vector
template <typename R, int C>
__device__ __forceinline__ int rescale(R* y) {
    R mx = y[0];
#pragma unroll
    for (int q = 1; q < 4 * C; ++q) mx = fmax(mx, y[q]);
    if (mx < Prec<R>::thresh()) {
#pragma unroll
        for (int q = 0; q < 4 * C; ++q) y[q] *= Prec<R>::mult();
        return 1;
    }
    return 0;
}

// exact power-of-two normalisation to max in [1, 2); returns the exponent removed
template <typename R, int C>
__device__ __forceinline__ int normalise(R* y) {
    R mx = y[0];
#pragma unroll
    for (int q = 1; q < 4 * C; ++q) mx = fmax(mx, y[q]);
    if (!(mx > R(0))) return 0;
    int e;
    if constexpr (sizeof(R) == 4) {
        e = ((__float_as_int(mx) >> 23) & 0xff) - 127;
        if (e < -125) e = -125;  // keep the multiplier a normal number
        float m = __int_as_float((127 - e) << 23);
#pragma unroll
        for (int q = 0; q < 4 * C; ++q) y[q] *= m;
    } else {
        e = (int)((__double_as_longlong(mx) >> 52) & 0x7ff) - 1023;
        if (e < -1021) e = -1021;
        double m = __longlong_as_double((long long)(1023 - e) << 52);
#pragma unroll
        for (int q = 0; q < 4 * C; ++q) y[q] *= m;
    }
    return e;
}

// Sum-table of one branch at one site.  With M_ik = sqrt(pi_i) R_ik and
// x_k = (M^T X_r)_k, y_k = (M^T Y_r)_k, L_r(t) = sum_k exp(lam_k r t) x_k y_k.
// Eigenvector 0 is the stationary one (lam_0 = 0), and sum_k x_k y_k =
// sum_i pi_i X_i Y_i, so
//   L_r(t) = sum_i pi_i X_i Y_i + sum_{k>=1} expm1(lam_k r t) x_k y_k,
// a form without the cancellation of the plain spectral sum at short branches
// (which costs FP32 its accuracy).  Stored: s_{r,0} = sum_i pi_i X_i Y_i,
// s_{r,k} = x_k y_k for k >= 1.
// X, Y [state][category], s [k][category].
template <typename R, int C>
__device__ __forceinline__ void sumtable(const R* Mt, const R* pi, const R* X, const R* Y, R* s) {
    if constexpr (sizeof(R) == 4 && C == 4) {
#pragma unroll
        for (int g = 0; g < 4; g += 2) {
            f32x2 s0 = pmul(pmul(make_float2(pi[0], pi[0]), pair(X + g)), pair(Y + g));
#pragma unroll
            for (int i = 1; i < 4; ++i)
                s0 = pfma(pmul(make_float2(pi[i], pi[i]), pair(X + 4 * i + g)), pair(Y + 4 * i + g), s0);
            s[g] = s0.x; s[g + 1] = s0.y;
#pragma unroll
            for (int k = 1; k < 4; ++k) {
                f32x2 m = make_float2(Mt[k], Mt[k]);
                f32x2 x = pmul(m, pair(X + g)), y = pmul(m, pair(Y + g));
#pragma unroll
                for (int i = 1; i < 4; ++i) {
                    m = make_float2(Mt[i * 4 + k], Mt[i * 4 + k]);
                    x = pfma(m, pair(X + 4 * i + g), x);
                    y = pfma(m, pair(Y + 4 * i + g), y);
                }
                x = pmul(x, y);
                s[4 * k + g] = x.x; s[4 * k + g + 1] = x.y;
            }
        }
    } else {
#pragma unroll
        for (int r = 0; r < C; ++r) {
            R s0 = pi[0] * X[r] * Y[r];
#pragma unroll
            for (int i = 1; i < 4; ++i) s0 = fma(pi[i] * X[i * C + r], Y[i * C + r], s0);
            s[r] = s0;
#pragma unroll
            for (int k = 1; k < 4; ++k) {
                R x = Mt[k] * X[r], y = Mt[k] * Y[r];
#pragma unroll
                for (int i = 1; i < 4; ++i) {
                    x = fma(Mt[i * 4 + k], X[i * C + r], x);
                    y = fma(Mt[i * 4 + k], Y[i * C + r], y);
                }
                s[k * C + r] = x * y;
            }
        }
    }
}

// The sites of a CTA's threads.  Their FP32 Newton sums are rounded, so the sum
// over the sites is defined by a launch-independent geometry: vk shares of
// consecutive sites (cluster_sites), vt virtual threads per share, virtual
// thread t of a share adding its sites t, t + vt, t + 2 vt, ... in that order,
// and the virtual threads' sums added by one binary tree over their linear index
// (neighbours first).  A launch spreads the vk * vt virtual threads over a cluster
// of kp CTAs, each virtual thread over `lanes` neighbouring lanes that take its
// sites in turn: the same sums, bit for bit, with as many SMs per item as the
// number of items leaves room for.
struct Sites {
    int p0, step;    // site m of this thread: p0 + m * step,
    int pl0, pstep;  // stored at local index pl0 + m * pstep
    int cnt;         // this thread's sites
    int M;           // the largest cnt of any thread
    int lanes, jj;   // lanes per virtual thread, this thread's among them
    int nt;          // sites of the virtual thread
    int ld;          // local capacity
};
__device__ __forceinline__ Sites make_sites(int P, const Geo& g, int rank, int kp) {
    Sites x;
    const int Ps = cluster_sites(P, g.vk), pt = blockDim.x;
    const int gv = (rank * pt + (int)threadIdx.x) / g.lanes, jj = (int)threadIdx.x % g.lanes;
    const int vr = gv / g.vt, vt = gv - vr * g.vt;
    const int start = min(P, vr * Ps), len = min(P, start + Ps) - start;
    const int i0 = vt + g.vt * jj;
    x.step = g.vt * g.lanes;
    x.p0 = start + i0;
    x.cnt = i0 < len ? (len - i0 + x.step - 1) / x.step : 0;
    x.M = (Ps + x.step - 1) / x.step;
    x.pl0 = threadIdx.x;
    x.pstep = pt;
    x.lanes = g.lanes;
    x.jj = jj;
    x.nt = vt < len ? (len - vt + g.vt - 1) / g.vt : 0;
    x.ld = geo_local(P, g, pt);
    return x;
}

// Sum-table storage: chunk q (16 bytes: 4 values in FP32, 2 in FP64) of local
// site p at index q * pcap + p, so consecutive threads touch consecutive 16
// bytes; then the site weights, and in FP64 the rows' exponents (the mixed path
// scores from pairs, and its Newton ratios do not see a row's power of two).
template <typename R, int C>
struct STab {
    R* s;          // [nchunk][pcap] vec
    R* w;          // [pcap] site weights, set once per item
    int* e;        // [pcap] exponents (FP64)
    int pcap;
    __device__ __forceinline__ void init(unsigned char* base, int ld) {
        pcap = (ld + 3) & ~3;
        s = reinterpret_cast<R*>(base);
        w = s + (size_t)4 * C * pcap;
        e = reinterpret_cast<int*>(w + pcap);
    }
    __device__ __forceinline__ void put(int p, const R* v, int E) const {
        if constexpr (sizeof(R) == 4) {
#pragma unroll
            for (int q = 0; q < C; ++q)
                reinterpret_cast<float4*>(s)[(size_t)q * pcap + p] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        } else {
#pragma unroll
            for (int q = 0; q < 2 * C; ++q)
                reinterpret_cast<double2*>(s)[(size_t)q * pcap + p] = make_double2(v[2 * q], v[2 * q + 1]);
            e[p] = E;
        }
    }
    __device__ __forceinline__ void get(int p, R* v) const {
        if constexpr (sizeof(R) == 4) {
#pragma unroll
            for (int q = 0; q < C; ++q) {
                float4 x = reinterpret_cast<const float4*>(s)[(size_t)q * pcap + p];
                v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 2 * C; ++q) {
                double2 x = reinterpret_cast<const double2*>(s)[(size_t)q * pcap + p];
                v[2 * q] = x.x; v[2 * q + 1] = x.y;
            }
        }
    }
};

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_ctas() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Sets up the two exchange barriers of a cluster CTA (once per launch, before its
// first cluster barrier; thread 0): each phase takes one arrival per warp of the
// CTA (its local entry) and one from the leader, which arms the remote bytes.
template <typename NS>
__device__ __forceinline__ void cluster_exchange_init(NS& ns) {
    const unsigned nw = (blockDim.x + 31) >> 5;
    mbar_init(&ns.mbx[0], nw + 1);
    mbar_init(&ns.mbx[1], nw + 1);
    ns.abort_ = 0;
    mbar_fence_init();
}

// A branch length between the solves: an FP32 pair in mixed precision (the steps
// are taken on pairs; every FP64 instruction costs its warp some 60 cycles and the
// SM's one FP64 pipe 16, whoever issues it), FP64 in the FP64 path.
template <typename R> struct LenOf { using T = double; };
template <> struct LenOf<float> { using T = F2; };
template <typename R> using Len = typename LenOf<R>::T;
// A length past FP32's range (accepted, as every finite one) becomes its largest number: the
// pair of an infinity has no difference from the solved length, and the move went unnoticed.
template <typename R> __device__ __forceinline__ Len<R> len_of(double x) {
    if constexpr (sizeof(R) == 4) return f2_of(fmin(x, (double)FLT_MAX));
    else return x;
}
__device__ __forceinline__ double len_dbl(F2 x) { return (double)x.h + (double)x.l; }
__device__ __forceinline__ double len_dbl(double x) { return x; }

// Block-wide context for the Newton machinery.
template <typename R, int C>
struct NewtonSmem {
    alignas(16) R egh[3][4 * C];  // coefficients on the sum-table for L, dL/dt, d2L/dt2
    double red[2][32];     // per-warp partial sums of scores, two alternating slots
    double lr[4 * C];      // lam_k * rate_r, [k][r] (as every 4C array here)
    float lrf[4 * C];      // the same in FP32 (coefficients of the Newton derivatives)
    double ex[4 * C];      // exp(lam_k r t) for a P-matrix refresh
    Exp2Tab et;
    F2 lrp[4 * C];         // lr as pairs (mixed precision)
    F2 Wp[64];             // W as pairs; [.][0].h: the entry's p_entry_base
    F2 em[4 * C];          // exp(lam_k r t) - 1 for a P-matrix refresh from pairs
    float lr_min;          // the smallest |lr| but the zero ones
    double W[64];          // W[(i*4+j)*4+k] = isqpi_i sqpi_j R_ik R_jk: P_ij = sum_k W_ijk exp(lam_k r t)
    Len<R> tmin, tmax, tol, sweep_tol, prior;  // the solver's constants
    int moved_at;          // last sweep (from 1) of the item that moved a length by more than sweep_tol
    int done;
    int leader;            // the warp that takes the Newton steps
    // Newton sums: each warp's (d1 h, d2 h, d1 l, d2 l) in FP32 or (d1, d2) in FP64; in a
    // cluster every warp of every CTA pushes its entry into entry rank * nw + warp of
    // every CTA's slot, two alternating slots, each with an mbarrier that counts the
    // bytes it received
    alignas(16) float cxr[2][kMaxTeamWarps][4];
    alignas(8) unsigned long long mbx[2];
    int abort_;            // a wait on mbx ran out (reported by the kernel)
};

// The entries of the binary tree that one warp finishes: entry i of ne at
// index i of the linear order; lane j takes its `per` neighbouring entries, then
// the lanes are added neighbours first (entries past ne count as zero, exactly).
__device__ __forceinline__ int tree_per(int ne) { return ne > 64 ? 4 : ne > 32 ? 2 : 1; }

// Two sums at once as FP32 pairs (h, l) x (d1, d2), added by packed two-sums.
struct Sum2 {
    f32x2 h, l;
};
__device__ __forceinline__ Sum2 sum2_add(Sum2 a, Sum2 b) {
    const f32x2 t = padd(a.h, b.h), bb = psub(t, a.h);
    const f32x2 err = padd(psub(a.h, psub(t, bb)), psub(b.h, bb));
    return Sum2{t, padd(padd(a.l, b.l), err)};
}
__device__ __forceinline__ Sum2 sum2_xor(Sum2 a, int o) {
    return Sum2{make_float2(__shfl_xor_sync(0xffffffffu, a.h.x, o), __shfl_xor_sync(0xffffffffu, a.h.y, o)),
                make_float2(__shfl_xor_sync(0xffffffffu, a.l.x, o), __shfl_xor_sync(0xffffffffu, a.l.y, o))};
}
// Compensated warp sums of two FP32 partials (two-sums over the virtual threads of
// the warp, which lie `lanes` apart; neighbours first): every lane ends with both
// sums as unevaluated pairs, with no FP64 instruction.
template <int kLanes>
__device__ __forceinline__ Sum2 warp_sum_comp(float x, float y) {
    Sum2 a{make_float2(x, y), make_float2(0.f, 0.f)};
#pragma unroll
    for (int o = kLanes; o < 32; o <<= 1) a = sum2_add(a, sum2_xor(a, o));
    return a;
}
// The last levels of the tree: n lanes' sums (a power of two) into each of them.
template <int n>
__device__ __forceinline__ Sum2 sum2_lanes(Sum2 a) {
#pragma unroll
    for (int o = 1; o < n; o <<= 1) a = sum2_add(a, sum2_xor(a, o));
    return a;
}
__device__ __forceinline__ double warp_sum(double x, int lanes) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
        if (o >= lanes) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

template <typename R, int C>
__device__ __forceinline__ void init_newton_smem(const Model& M, const Cfg& cfg, NewtonSmem<R, C>& ns,
                                                 const double* rates) {
    for (int x = threadIdx.x; x < 64; x += blockDim.x) {
        int k = x & 3, ij = x >> 2, i = ij >> 2, j = ij & 3;
        auto W = [&](int q) { return M.isqpi[i] * M.sqpi[j] * M.R[i * 4 + q] * M.R[j * 4 + q]; };
        ns.W[x] = W(k);
        if (sizeof(R) == 4) {
            if (k == 0) {
                const double Wij[4] = {W(0), W(1), W(2), W(3)};
                ns.Wp[x] = F2{p_entry_base(i == j ? 1.0 : 0.0, Wij), 0.f};
            } else {
                ns.Wp[x] = f2_of(W(k));
            }
        }
    }
    if (threadIdx.x == 0) {
        // Leader warp: FP64 instructions issue slowly and only on the issuing warp's
        // scheduler, so blocks sharing an SM should not all lead from the same one.
        // Warp slots of a block are taken to be consecutive and schedulers to be
        // slot mod 4; a wrong guess costs time only.
        unsigned slot;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
        const int nw = (blockDim.x + 31) >> 5;
        const int want = (int)((slot / nw) & 3);
        int lead = 0;
        for (int w = 0; w < nw && w < 4; ++w)
            if ((int)((slot + w) & 3) == want) { lead = w; break; }
        ns.leader = lead;
        ns.moved_at = 0;
        ns.tmin = len_of<R>(cfg.tmin);
        ns.tmax = len_of<R>(cfg.tmax);
        ns.tol = len_of<R>(cfg.newton_tol);
        ns.sweep_tol = len_of<R>(cfg.sweep_tol);
        ns.prior = len_of<R>(cfg.prior_rate);
    }
    if (threadIdx.x < C) {  // the stationary slots' coefficients never change
        ns.egh[0][threadIdx.x] = (R)(1.0f / C);
        ns.egh[1][threadIdx.x] = R(0);
        ns.egh[2][threadIdx.x] = R(0);
    }
    for (int q = threadIdx.x; q < 4 * C; q += blockDim.x) {
        ns.lr[q] = M.lam[q / C] * rates[q % C];
        ns.lrf[q] = (float)ns.lr[q];
        if (sizeof(R) == 4) ns.lrp[q] = f2_of(ns.lr[q]);
    }
    if (threadIdx.x == 0) {
        double m = 1e30;
        for (int q = C; q < 4 * C; ++q) m = fmin(m, fabs(M.lam[q / C] * rates[q % C]));
        ns.lr_min = (float)m;
    }
}

// Coefficients at branch length t on the sum-table (see sumtable()): egh[0]
// gives L (1 for the stationary slot, expm1(lam r t) otherwise), egh[1] and
// egh[2] give dL/dt and d2L/dt2; all divided by C.  Called by the lanes q of one
// warp (the stationary slots q < C are set once, init_newton_smem), in the working
// precision's own exponentials; no FP64 instruction in FP32.
template <int C>
__device__ __forceinline__ void put_egh(F2 t, NewtonSmem<float, C>& ns, int q) {
    if (q >= C && q < 4 * C) {
        const float l = ns.lrf[q], x = l * t.h, e = expf(x) * (1.0f / C);
        ns.egh[0][q] = expm1f(x) * (1.0f / C);
        ns.egh[1][q] = l * e;
        ns.egh[2][q] = l * l * e;
    }
}
template <int C>
__device__ __forceinline__ void put_egh(double t, NewtonSmem<double, C>& ns, int q) {
    if (q >= C && q < 4 * C) {
        const double lr = ns.lr[q];
        ns.egh[0][q] = expm1(lr * t) / C;
        const double e = exp(lr * t) / C;
        ns.egh[1][q] = lr * e;
        ns.egh[2][q] = lr * lr * e;
    }
}

// Safeguarded Newton step: bracket [lo, hi]; Newton point when d2 < 0 and
// strictly inside, else sqrt(lo*hi).  Returns true when converged.
//
// Written for the one warp that takes the step while the rest of the block
// waits: FP64 instructions issue at a small fraction of the FP32 rate, so the
// comparisons are done on the IEEE bit patterns with integer instructions
// (t, lo, hi are positive and finite, so their patterns order like the
// values), and d1/d2 is a reciprocal seed refined by one Newton-Raphson
// correction of the quotient (Markstein's scheme: q = q0 + r (d1 - d2 q0)),
// accurate to about 2^-46 relative; NaN and infinite quotients fail the
// bracket test and fall back to the midpoint, as in plain IEEE arithmetic.
__device__ __forceinline__ bool dbl_pos(double x) {  // x > 0 (false for NaN)
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool dbl_neg(double x) {  // x < 0 (false for NaN, -0)
    const long long a = __double_as_longlong(x) & 0x7fffffffffffffffLL;
    return __double_as_longlong(x) < 0 && a != 0 && a <= 0x7ff0000000000000LL;
}
// d2f: an FP32 estimate of d2, available before d2 itself (the reciprocal
// seed then stays off the FP64 dependency chain); on the Newton branch the
// convergence test uses the increment itself.
__device__ __forceinline__ bool newton_step(double& t, double& lo, double& hi, double d1, double d2, float d2f,
                                            double tol) {
    const long long b1 = __double_as_longlong(d1);
    if ((b1 & 0x7fffffffffffffffLL) == 0) return true;  // d1 == 0
    if (dbl_pos(d1)) lo = t; else hi = t;
    double r = (double)__frcp_rn(d2f);
    double q0 = d1 * r;
    double e = fma(-d2, q0, d1);
    // a seed off by more than ~2^-10 (d2f lost to cancellation): reseed from d2 (rare)
    const int xe = (int)((__double_as_longlong(e) >> 52) & 0x7ff), x1 = (int)((b1 >> 52) & 0x7ff);
    if (xe > x1 - 10) {
        r = (double)__frcp_rn(__double2float_rn(d2));
        q0 = d1 * r;
        e = fma(-d2, q0, d1);
    }
    const double q = fma(e, r, q0);
    const double tn = t - q;
    const long long bt = __double_as_longlong(tn);
    if (dbl_neg(d2) && bt > __double_as_longlong(lo) && bt < __double_as_longlong(hi)) {
        t = tn;
        return (__double_as_longlong(q) & 0x7fffffffffffffffLL) <= __double_as_longlong(tol);
    }
    const double tm = sqrt(lo * hi);
    const bool conv = (__double_as_longlong(tm - t) & 0x7fffffffffffffffLL) <= __double_as_longlong(tol);
    t = tm;
    return conv;
}

// The same safeguarded step on FP32 pairs (F2): the mixed path's derivative
// sums arrive as pairs, and t, lo, hi are carried as pairs (~48 bits), so the
// step needs no FP64 instruction (a dependent FP64 operation costs 64 cycles on
// this part).  Quotient: one reciprocal seed, refined once (q = q0 + (d1 -
// q0 d2) / d2); square root of the bisection: sqrtf refined by one Heron step.
__device__ __forceinline__ bool f2_lt(F2 a, F2 b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }
__device__ __forceinline__ F2 f2_abs(F2 a) { return a.h < 0.f ? F2{-a.h, -a.l} : a; }
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
    const F2 d = f2_two_sum(a.h, -b.h);
    return f2_norm(d.h, __fadd_rn(d.l, __fsub_rn(a.l, b.l)));
}
__device__ __forceinline__ F2 f2_div(F2 a, F2 b) {
    const float rc = rcp_rn(b.h);
    const float q0 = __fmul_rn(a.h, rc);
    const float p = __fmul_rn(q0, b.h), pe = __fmaf_rn(q0, b.h, -p);
    // a - q0 b: a.h - p is exact (p lies within a factor 2 of a.h)
    const float r = __fadd_rn(__fsub_rn(__fsub_rn(a.h, p), pe), __fsub_rn(a.l, __fmul_rn(q0, b.l)));
    return f2_norm(q0, __fmul_rn(r, rc));
}
__device__ __forceinline__ F2 f2_sqrt(F2 x) {
    const float s0 = sqrtf(x.h);
    if (!(s0 > 0.f)) return F2{s0, 0.f};
    const float p = __fmul_rn(s0, s0), pe = __fmaf_rn(s0, s0, -p);
    const float r = __fadd_rn(__fsub_rn(__fsub_rn(x.h, p), pe), x.l);
    return f2_norm(s0, __fmul_rn(r, __fmul_rn(0.5f, rcp_rn(s0))));
}
__device__ __forceinline__ bool newton_step_f2(F2& t, F2& lo, F2& hi, F2 d1, F2 d2, F2 tol) {
    if (d1.h == 0.f) return true;  // d1 == 0 (a pair is zero iff its high part is)
    if (d1.h > 0.f) lo = t; else hi = t;
    const F2 q = f2_div(d1, d2);
    const F2 tn = f2_sub(t, q);
    if (d2.h < 0.f && f2_lt(lo, tn) && f2_lt(tn, hi)) {  // NaN fails the bracket test
        t = tn;
        return !f2_lt(tol, f2_abs(q));
    }
    const F2 tm = f2_sqrt(f2_mul(lo, hi));
    const bool conv = !f2_lt(tol, f2_abs(f2_sub(tm, t)));
    t = tm;
    return conv;
}

// Sum of the virtual threads' scores over the item, the same in every thread
// whatever the launch shape: the warps' sums in shared memory (red), then the
// cluster's kp x nw of them by the tree.  Every thread of every CTA must call it
// the same number of times; cseq alternates the slot, so a CTA writes one only
// after every CTA has passed the barrier of the exchange that last read it.
template <bool kClus>
__device__ __forceinline__ double team_sum(double acc, double (*red)[32], Team& tm, int lanes) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5, sl = tm.cseq++ & 1;
    acc = warp_sum(acc, lanes);
    if (lane == 0) red[sl][w] = acc;
    if constexpr (kClus) cooperative_groups::this_cluster().sync();
    else __syncthreads();
    const int ne = tm.kp * nw, per = tree_per(ne);
    double e[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = lane * per + k;
        if (k < per && i < ne) {
            if constexpr (kClus) e[k] = cooperative_groups::this_cluster().map_shared_rank(&red[sl][0], i / nw)[i % nw];
            else e[k] = red[sl][i];
        }
    }
    return warp_sum((e[0] + e[1]) + (e[2] + e[3]), 1);
}
// One site's score, added to the virtual thread's sum in site order; term of the
// lane's own site (0 where it has none this round).
__device__ __forceinline__ void add_score(double& acc, double term, int lanes) {
    if (lanes == 1) {
        acc = __dadd_rn(acc, term);
        return;
    }
    const int base = (threadIdx.x & 31) & ~(lanes - 1);
    for (int j = 0; j < lanes; ++j) acc = __dadd_rn(acc, __shfl_sync(0xffffffffu, term, base + j));
}

// lnL of the current sum-table at length t: sum_p w_p (ln L_p + E_p ln 2) (FP64;
// the mixed path scores from pairs).
template <int C, bool kClus>
__device__ double eval_lnl(const STab<double, C>& st, const Sites& sx, double t,
                           NewtonSmem<double, C>& ns, Team& tm) {
    put_egh<C>(t, ns, threadIdx.x);
    __syncthreads();
    double e[4 * C];
#pragma unroll
    for (int q = 0; q < 4 * C; ++q) e[q] = ns.egh[0][q];
    double acc = 0.0;
    for (int m = 0; m < sx.M; ++m) {
        double term = 0.0;
        if (m < sx.cnt) {
            const int pl = sx.pl0 + m * sx.pstep;
            double s[4 * C];
            st.get(pl, s);
            double L = e[0] * s[0];
#pragma unroll
            for (int z = 1; z < 4 * C; ++z) {
                const int q = (z & 3) * C + (z >> 2);  // categories outermost
                L = fma(e[q], s[q], L);
            }
            term = __dmul_rn(st.w[pl], log(L) + (double)st.e[pl] * kLn2);
        }
        add_score(acc, term, sx.lanes);
    }
    return team_sum<kClus>(acc, ns.red, tm, sx.lanes);
}

// One site's terms of the Newton sums: a = L'/L, c = L''/L - (L'/L)^2 and the site
// weight, from the sum-table at the coefficients e, g, h (the stationary slots,
// k = 0, have zero derivative coefficients).  A virtual thread takes its sites in
// pairs; the two of a pair (and a last single one) round c in two forms: first of a pair
// fma(-a, a, L''/L), else fma(L'', 1/L, -a a).  Neither is the better one: an earlier
// source left the contraction to the compiler, which chose these, and results that are
// stored or compared keep their bits only if they stay.
template <typename R, int C>
__device__ __forceinline__ void newton_site(const STab<R, C>& st, int p, const R* e, const R* g, const R* h, bool first,
                                            R& a, R& c, R& wt) {
    R s[4 * C];
    st.get(p, s);
    R L = e[0] * s[0], L1 = g[C] * s[C], L2 = h[C] * s[C];
#pragma unroll
    for (int z = 1; z < 4 * C; ++z) {
        const int q = (z & 3) * C + (z >> 2);  // categories outermost
        L = fma(e[q], s[q], L);
        if ((z & 3) != 0 && z != 1) {
            L1 = fma(g[q], s[q], L1);
            L2 = fma(h[q], s[q], L2);
        }
    }
    const R inv = Prec<R>::rcp(L);
    a = Prec<R>::mul(L1, inv);
    c = first ? fma(-a, a, Prec<R>::mul(L2, inv)) : fma(L2, inv, -Prec<R>::mul(a, a));
    wt = st.w[p];
}

// Sets up a solve from length t0 (the coefficients of its first evaluation) and
// returns t0 within the bounds; called before the sum-table is built, by every
// thread, after the last barrier of the solve before.
template <int C>
__device__ __forceinline__ F2 newton_begin(F2 t0, NewtonSmem<float, C>& ns) {
    F2 t = f2_lt(t0, ns.tmin) ? ns.tmin : t0;
    if (f2_lt(ns.tmax, t)) t = ns.tmax;
    put_egh<C>(t, ns, threadIdx.x);
    return t;
}
template <int C>
__device__ __forceinline__ double newton_begin(double t0, NewtonSmem<double, C>& ns) {
    const double t = fmin(fmax(t0, ns.tmin), ns.tmax);
    put_egh<C>(t, ns, threadIdx.x);
    return t;
}

// The warp's Newton sums at the coefficients in ns, in every lane: (d1 h, d2 h, d1 l,
// d2 l) in FP32, (d1, d2) in FP64.  One form per number of lanes: with the number a
// variable, its loops' branches were a tenth of an evaluation's chain.
template <typename R, int C, int kLanes>
__device__ __forceinline__ float4 site_sums(const STab<R, C>& st, const Sites& sx, const NewtonSmem<R, C>& ns) {
    R e[4 * C], g[4 * C], h[4 * C];
#pragma unroll
    for (int q = 0; q < 4 * C; ++q) { e[q] = ns.egh[0][q]; g[q] = ns.egh[1][q]; h[q] = ns.egh[2][q]; }
    R a1 = R(0), a2 = R(0);
    if constexpr (kLanes == 1) {
        // two sites per pass (their chains interleave), added in site order
        int m = 0, p = sx.pl0;
        for (; m + 1 < sx.cnt; m += 2, p += 2 * sx.pstep) {
            R a, c, wt, a_, c_, wt_;
            newton_site<R, C>(st, p, e, g, h, true, a, c, wt);
            newton_site<R, C>(st, p + sx.pstep, e, g, h, false, a_, c_, wt_);
            a1 = fma(wt, a, a1);
            a2 = fma(wt, c, a2);
            a1 = fma(wt_, a_, a1);
            a2 = fma(wt_, c_, a2);
        }
        if (m < sx.cnt) {
            R a, c, wt;
            newton_site<R, C>(st, p, e, g, h, false, a, c, wt);
            a1 = fma(wt, a, a1);
            a2 = fma(wt, c, a2);
        }
    } else {
        // the virtual thread's sites of this round lie in its lanes, in order:
        // every lane of the group adds all of them (the same sum as one thread's)
        const int base = (threadIdx.x & 31) & ~(kLanes - 1);
        for (int m = 0; m < sx.M; ++m) {
            R a = R(0), c = R(0), wt = R(0);
            const int k = sx.jj + m * kLanes;  // this lane's site among the virtual thread's
            if (m < sx.cnt)
                newton_site<R, C>(st, sx.pl0 + m * sx.pstep, e, g, h, !(k & 1) && k + 1 < sx.nt, a, c, wt);
#pragma unroll
            for (int j = 0; j < kLanes; ++j) {
                const R aj = __shfl_sync(0xffffffffu, a, base + j), cj = __shfl_sync(0xffffffffu, c, base + j),
                        wj = __shfl_sync(0xffffffffu, wt, base + j);
                a1 = fma(wj, aj, a1);
                a2 = fma(wj, cj, a2);
            }
        }
    }
    if constexpr (sizeof(R) == 4) {
        const Sum2 a = warp_sum_comp<kLanes>(a1, a2);
        return make_float4(a.h.x, a.h.y, a.l.x, a.l.y);
    } else {
        const double2 d = make_double2(warp_sum(a1, kLanes), warp_sum(a2, kLanes));
        return reinterpret_cast<const float4&>(d);
    }
}

// Below this t |lam r| (so off-diagonal entries of about 2^-17) the rounding test of
// p_entry_pair fails for one solve in ten or more, and the FP64 sum is taken at once.
constexpr float kPairMin = 3e-5f;

// Newton solve on the current sum-table from t (as newton_begin returned it).  Per
// evaluation: every thread sums w L'/L and w (L''/L - (L'/L)^2) over its sites, the
// warps reduce, and one warp alone takes the step and writes the coefficients of
// the next length.  After the last step that warp stores the length in *dst, notes
// in ns.moved_at whether it is more than sweep_tol from told (sweep number sweep),
// and P_r of the final length goes to Pdst [16][C]; all visible when the call
// returns.  Everything but the sums over sites is that warp's: what one warp does in
// FP64 or in a long chain holds up one scheduler, what every warp does, all of them.
// Bound by that chain: an evaluation of 816 patterns takes 2.5 to 2.9 thousand cycles
// on one or four CTAs (site 500, warp sums 300, exchange 250 to 600, tree 400, step 490,
// coefficients 400 to 570), a solve of three evaluations 11 to 14 thousand.
// kClus: the sum-table holds this CTA's share of a cluster's sites; each
// evaluation's derivative sums are exchanged over the cluster, and every CTA
// takes the same step.
template <typename R, int C, bool kClus>
__device__ __forceinline__ void newton_solve(const Cfg& cfg, const STab<R, C>& st, const Sites& sx, Len<R> t,
                                             Len<R> told, Len<R>* dst, int sweep, NewtonSmem<R, C>& ns, int& evals,
                                             bool& converged, R* Pdst, Team& tm) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    __syncthreads();  // the coefficients of newton_begin
    const int ld = ns.leader;
    Len<R> lo = ns.tmin, hi = ns.tmax;
    auto sums = [&] {
        return sx.lanes == 1   ? site_sums<R, C, 1>(st, sx, ns)
               : sx.lanes == 2 ? site_sums<R, C, 2>(st, sx, ns)
               : sx.lanes == 4 ? site_sums<R, C, 4>(st, sx, ns)
                               : site_sums<R, C, 8>(st, sx, ns);
    };
    auto step = [&](int cs, bool last) {
        // the rest of the tree over the kp x nw warp entries: every CTA adds the same
        // numbers in the same order
        const int ne = tm.kp * nw, per = tree_per(ne);
        bool done;
        if constexpr (sizeof(R) == 4) {
            // FP32 pairs, added by two-sums (~48 bits)
            auto entry = [&](int k) {
                const int i = lane * per + k;
                const float4 q = k < per && i < ne ? *reinterpret_cast<const float4*>(&ns.cxr[cs][i][0])
                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
                return Sum2{make_float2(q.x, q.y), make_float2(q.z, q.w)};
            };
            Sum2 q = entry(0);
            if (per > 1) q = sum2_add(q, entry(1));
            if (per > 2) q = sum2_add(q, sum2_add(entry(2), entry(3)));
            q = ne > 16 ? sum2_lanes<32>(q) : ne > 8 ? sum2_lanes<16>(q) : ne > 4 ? sum2_lanes<8>(q) : sum2_lanes<4>(q);
            // the butterfly leaves (h, l) unnormalised (l can reach a sizeable
            // fraction of h after cancellation): renormalise, so that the
            // quotient's reciprocal seed is taken from the rounded total
            // (lanes past ne hold partial sums: lane 0's are taken)
            F2 d1p = f2_two_sum(__shfl_sync(0xffffffffu, q.h.x, 0), __shfl_sync(0xffffffffu, q.l.x, 0));
            const F2 d2p = f2_two_sum(__shfl_sync(0xffffffffu, q.h.y, 0), __shfl_sync(0xffffffffu, q.l.y, 0));
            if (ns.prior.h != 0.f) d1p = f2_sub(d1p, ns.prior);  // MAP: the prior's slope
            done = newton_step_f2(t, lo, hi, d1p, d2p, ns.tol);
        } else {
            auto entry = [&](int k) {
                const int i = lane * per + k;
                return k < per && i < ne ? *reinterpret_cast<const double2*>(&ns.cxr[cs][i][0]) : make_double2(0.0, 0.0);
            };
            double2 q = entry(0);
            if (per > 1) {
                const double2 x = entry(1), y = entry(2), z = entry(3);
                q = make_double2((q.x + x.x) + (y.x + z.x), (q.y + x.y) + (y.y + z.y));
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                if (o >= ne) break;
                q.x += __shfl_xor_sync(0xffffffffu, q.x, o);
                q.y += __shfl_xor_sync(0xffffffffu, q.y, o);
            }
            double D1 = __shfl_sync(0xffffffffu, q.x, 0);
            const double D2 = __shfl_sync(0xffffffffu, q.y, 0);
            if (__double_as_longlong(ns.prior) != 0) D1 -= ns.prior;  // MAP: the prior's slope
            done = newton_step(t, lo, hi, D1, D2, (float)D2, ns.tol);
        }
        if (!done && !last) {
            put_egh<C>(t, ns, lane);
            return 0;
        }
        // for the P matrices below: pairs where their rounding test mostly passes
        // (off-diagonal entries not tiny), else FP64 exponentials
        bool pairs = false;
        if constexpr (sizeof(R) == 4) {
            pairs = t.h * ns.lr_min > kPairMin;
            if (pairs && lane < 4 * C) {
                const F2 x = f2_mul(ns.lrp[lane], t);
                ns.em[lane] = x.h > -80.f ? expm1_pair(x, ns.et) : F2{-1.f, 0.f};
            }
        }
        if (!pairs && lane < 4 * C) ns.ex[lane] = exp(ns.lr[lane] * len_dbl(t));
        if (lane == 0) {
            bool moved;
            if constexpr (sizeof(R) == 4) moved = f2_lt(ns.sweep_tol, f2_abs(f2_sub(t, told)));
            else moved = fabs(t - told) > ns.sweep_tol;
            if (moved) ns.moved_at = sweep;
            *dst = t;
        }
        return (done ? 1 : 2) | (pairs ? 4 : 0);
    };
    converged = false;
    evals = newton_evaluations<kClus>(cfg.newton_maxit, w, lane, nw, ld, ns, tm, sums, step);
    if (kClus && evals == 0) return;  // given up: the length stays
    // P matrices of the final length, rounded once from FP64 or from pairs to the
    // same bits (a dependent FP64 instruction takes some 60 cycles, exp() a thousand;
    // the pairs' chain a third of that)
    converged = (ns.done & 3) == 1;
    if (sizeof(R) == 4 && (ns.done & 4)) {
        bool sure = true;
        for (int x = threadIdx.x; x < 16 * C; x += blockDim.x) {
            const int r = x % C, ij = x / C;
            bool ok;
            const F2* const Wk = ns.Wp + ij * 4;
            Pdst[x] = p_entry_pair(ij % 5 == 0 ? 1.f : 0.f, Wk, ns.em + r, C, ok, Wk[0].h);
            sure = sure && ok;
        }
        if (!__syncthreads_or(!sure)) return;
        if (w == ld && lane < 4 * C) ns.ex[lane] = exp(ns.lr[lane] * len_dbl(t));
        __syncthreads();
    }
    for (int x = threadIdx.x; x < 16 * C; x += blockDim.x) {
        const int r = x % C, ij = x / C;
        double acc = ns.W[ij * 4];  // lam_0 = 0
#pragma unroll
        for (int k = 1; k < 4; ++k) acc = fma(ns.W[ij * 4 + k], ns.ex[k * C + r], acc);
        Pdst[x] = (R)acc;
    }
    __syncthreads();
}


// ---------------------------------------------------------------- pair scores (mixed precision)
// Scores of the mixed path, computed from pair partials (F2) category by
// category (each category normalised on its own, merged with its exponent):
// sum over the calling block's sites of w_p ln L_p, reduced over the block
// into red[32] (FP64) and returned in every thread.  Kept out of line so the
// FP32 Newton loops around them keep their registers.

// Proposal: the four members A, X2 (at u) and B, Y2 (at v) around the new
// edge (slots of ld sites), P matrices of the five final lengths as pairs (Ph/Pl
// [5][16*C]: central, A, B, C, D; mbr = each member's branch); L_p across the
// central branch.
template <int C, bool kClus>
__device__ __noinline__ double propose_score_f2(const Src2<C>* mem, const int* mbr, const float* Ph, const float* Pl,
                                                const double* pi, const int32_t* w, int ld, const Sites& sx,
                                                double (*red)[32], Team& tm) {
    float pih[4], pil[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const F2 x = f2_of(pi[i]);
        pih[i] = x.h;
        pil[i] = x.l;
    }
    double acc = 0.0;
    auto site = [&](int p) {
        int kk = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) kk += mem[b].tip ? 0 : mem[b].scl[p];
        F2 L{0.f, 0.f};
        int E = 0;
        using T = typename Lanes<C>::T;
#pragma unroll 1
        for (int g = 0; g < Lanes<C>::n; ++g) {
            F2T<T> x[4], y[4], t[4];
            f2_apply_src4<C>(Ph + mbr[0] * C * 16, Pl + mbr[0] * C * 16, mem[0], ld, p, p, g, x);
            f2_apply_src4<C>(Ph + mbr[1] * C * 16, Pl + mbr[1] * C * 16, mem[1], ld, p, p, g, t);
            f2_mul4<T>(x, t);
            f2_apply_src4<C>(Ph + mbr[2] * C * 16, Pl + mbr[2] * C * 16, mem[2], ld, p, p, g, y);
            f2_apply_src4<C>(Ph + mbr[3] * C * 16, Pl + mbr[3] * C * 16, mem[3], ld, p, p, g, t);
            f2_mul4<T>(y, t);
            int ex[Lanes<C>::w], ey[Lanes<C>::w];
            f2_normalise4(x, ex);
            f2_normalise4(y, ey);
            f2_apply4<C>(Ph, Pl, g, y, t);  // across the central branch (branch 0)
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = t2_mul<T>(x[i], t[i]);
#pragma unroll
            for (int k = 0; k < Lanes<C>::w; ++k) {
                F2 Lr{0.f, 0.f};
#pragma unroll
                for (int i = 0; i < 4; ++i) Lr = f2_add(Lr, f2_mul(lane_of(x[i], k), F2{pih[i], pil[i]}));
                f2_merge(L, E, Lr, ex[k] + ey[k]);
            }
        }
        L = F2{L.h * (1.0f / C), L.l * (1.0f / C)};  // 1/C is a power of two for C = 1, 2, 4
        return __dmul_rn((double)w[p], f2_log(L, E - Prec<float>::kScaleExp * kk));
    };
    for (int m = 0; m < sx.M; ++m) add_score(acc, m < sx.cnt ? site(sx.p0 + m * sx.step) : 0.0, sx.lanes);
    return team_sum<kClus>(acc, red, tm, sx.lanes);
}

// ---------------------------------------------------------------- tree scores (mixed precision)
// Scores of trees at their lengths: one pruning pass in pair arithmetic, nothing
// stored but the sums.  A thread owns one site and one lane group of its categories
// and walks the tree's inner nodes in post-order, the subtree that needs more of the
// stack first, so that at most log2(n) vectors wait (local memory); the node just
// made stays in registers.  The categories' groups are scaled apart and merged with
// their exponents at the root.  Sites are summed in units of kScoreUnit (a fixed
// tree), the units in a fixed order by k_score_sum: a score does not depend on the launch.
// Bound by FP32 issue (about 270 packed instructions per node, site and group) and,
// for few sites, by the FP64 exponentials of the P matrices, which each CTA makes
// once per tree, in parallel over edges and categories.  One tree of 27 taxa x 816
// patterns took 157 us as the last step of the full optimisation, whose nodes each
// waited for their own P matrices, and takes 38; 256 of 64 x 987 1129, now about 560.
constexpr int kScoreUnit = 64, kScoreStack = 9;
struct ScoreProg {
    uint8_t kind, a, b;  // kind 0: two tips, 1: tip a and the last result (edge b), 2: waiting result (edge a) and last (edge b)
};
__host__ __device__ inline size_t score_smem(int C, int nn) {
    return ((size_t)nn * 32 * C * 4 + (size_t)nn * (3 + 8) + 15) & ~size_t(15);
}
template <int C, int kThreads>
__global__ void __launch_bounds__(kThreads) k_score(const FullGroup* __restrict__ groups, const int* __restrict__ gstart,
                                               int ngroups, int nn_max, int t0, int t1, int chunks, int units_max,
                                               double* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char smraw[];
    using T = typename Lanes<C>::T;
    constexpr int S = Lanes<C>::n;  // threads per site
    float* const Ph = reinterpret_cast<float*>(smraw);
    float* const Pl = Ph + (size_t)nn_max * 16 * C;
    ScoreProg* const prog = reinterpret_cast<ScoreProg*>(Pl + (size_t)nn_max * 16 * C);
    uint8_t* const ch = reinterpret_cast<uint8_t*>(prog + nn_max);  // children; then need[] and two stacks
    uint8_t *const need = ch + 2 * nn_max, *const stk = need + nn_max;
    __shared__ double W[64], red[24];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int total = min(gstart[ngroups], t1) - t0;
    for (long long work = blockIdx.x; work < (long long)total * chunks; work += gridDim.x) {
        const int x = t0 + (int)(work / chunks), c = (int)(work % chunks);
        int k = 0;
        while (k + 1 < ngroups && gstart[k + 1] <= x) ++k;
        const FullGroup& G = groups[k];
        const int gi = G.order ? G.order[x - gstart[k]] : x - gstart[k];
        const Model& M = G.M;
        const Aln& A = G.A;
        const int n = G.ts.n, NN = 2 * n - 2, P = A.P, units = (P + kScoreUnit - 1) / kScoreUnit;
        const int u0 = (int)((long long)units * c / chunks), u1 = (int)((long long)units * (c + 1) / chunks);
        if (u0 == u1) continue;  // uniform over the block
        const int tree = G.first + gi;
        __syncthreads();  // the work item before is done with shared memory
        for (int z = threadIdx.x; z < 64; z += blockDim.x) {
            const int q = z & 3, ij = z >> 2, i = ij >> 2, j = ij & 3;
            W[z] = M.isqpi[i] * M.sqpi[j] * M.R[i * 4 + q] * M.R[j * 4 + q];
        }
        for (int v = threadIdx.x; v < 2 * NN; v += blockDim.x) ch[v] = (uint8_t)G.ts.ch[(size_t)tree * 2 * NN + v];
        __syncthreads();
        if (warp == 0) {
            if (lane == 0) {
                // post-order program; need[v]: results that wait while v's subtree is made
                for (int v = NN - 1; v >= n; --v) {
                    const int a = ch[2 * v], b = ch[2 * v + 1], na = a < n ? 0 : need[a], nb = b < n ? 0 : need[b];
                    need[v] = (uint8_t)(na == nb ? na + 1 : max(na, nb));
                }
                int sp = 0, np = 0;
                uint8_t* const done = stk + NN;
                stk[0] = (uint8_t)n;
                done[0] = 0;
                sp = 1;
                while (sp) {
                    const int v = stk[sp - 1], c0 = ch[2 * v], c1 = ch[2 * v + 1];
                    const bool swap = c1 >= n && (c0 < n || need[c1] > need[c0]);
                    const int a = swap ? c1 : c0, b = swap ? c0 : c1;  // a first; a tip only if both are
                    const int st = done[sp - 1]++;
                    if (st == 0 && a >= n) { stk[sp] = (uint8_t)a; done[sp++] = 0; continue; }
                    if (st <= 1 && b >= n) { done[sp - 1] = 2; stk[sp] = (uint8_t)b; done[sp++] = 0; continue; }
                    prog[np++] = a < n   ? ScoreProg{0, (uint8_t)a, (uint8_t)b}
                                 : b < n ? ScoreProg{1, (uint8_t)b, (uint8_t)a}
                                         : ScoreProg{2, (uint8_t)a, (uint8_t)b};
                    --sp;
                }
            }
        }
        const double* rr = G.rates ? G.rates + (size_t)gi * kMaxCat : M.rates;
        const double* glen = G.ts.len + (size_t)tree * NN;
        // warps other than the one with the program start on the matrices
        for (int z = ((int)threadIdx.x + (int)blockDim.x - 32) % (int)blockDim.x; z < (NN - 1) * C; z += blockDim.x) {
            const int v = 1 + z / C, r = z % C;
            double e[4] = {1.0, 0.0, 0.0, 0.0};  // lam_0 = 0
#pragma unroll
            for (int q = 1; q < 4; ++q) e[q] = exp(M.lam[q] * rr[r] * glen[v]);
#pragma unroll
            for (int ij = 0; ij < 16; ++ij) {
                double acc = 0.0;
#pragma unroll
                for (int q = 0; q < 4; ++q) acc += W[ij * 4 + q] * e[q];
                const F2 w = f2_of(acc);
                Ph[((size_t)v * 16 + ij) * C + r] = w.h;
                Pl[((size_t)v * 16 + ij) * C + r] = w.l;
            }
        }
        __syncthreads();
        F2 pi[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) pi[i] = f2_of(M.pi[i]);
        const int g = (int)threadIdx.x % S, per = (int)blockDim.x / (S * kScoreUnit);  // units per pass
        for (int ub = u0; ub < u1; ub += per) {
            const int u = ub + (int)threadIdx.x / (S * kScoreUnit);
            const int p = u * kScoreUnit + (int)threadIdx.x / S % kScoreUnit;
            const bool valid = u < u1 && p < P;
            double term = 0.0;
            F2 L{0.f, 0.f};
            int E = 0;
            if (valid) {
                F2T<T> acc[4], wait[kScoreStack][4];
                int kk = 0, wk[kScoreStack], sp = 0;
                auto tip = [&](int v, F2T<T>* y) {
                    const Src2<C> s{nullptr, nullptr, nullptr, A.tips + (size_t)v * P};
                    f2_apply_src4<C>(Ph + (size_t)v * 16 * C, Pl + (size_t)v * 16 * C, s, 0, 0, p, g, y);
                };
                for (int q = 0; q < n - 2; ++q) {
                    const ScoreProg o = prog[q];
                    F2T<T> y[4], z[4];
                    if (o.kind == 0) {
                        if (q > 0) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) wait[sp][i] = acc[i];
                            wk[sp++] = kk;
                        }
                        kk = 0;
                        tip(o.a, y);
                        tip(o.b, z);
                    } else {
                        f2_apply4<C>(Ph + (size_t)o.b * 16 * C, Pl + (size_t)o.b * 16 * C, g, acc, y);
                        if (o.kind == 1) {
                            tip(o.a, z);
                        } else {
                            kk += wk[--sp];
#pragma unroll
                            for (int i = 0; i < 4; ++i) acc[i] = wait[sp][i];
                            f2_apply4<C>(Ph + (size_t)o.a * 16 * C, Pl + (size_t)o.a * 16 * C, g, acc, z);
                        }
                    }
                    float mx = 0.f;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        acc[i] = t2_mul<T>(y[i], z[i]);
                        mx = fmaxf(mx, lane_max(acc[i].h));
                    }
                    if (mx < Prec<float>::thresh()) {
                        const T m = lane_all<T>(Prec<float>::mult());
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            acc[i].h = pmul(acc[i].h, m);
                            acc[i].l = pmul(acc[i].l, m);
                        }
                        ++kk;
                    }
                }
                const int code = A.tips[p];  // leaf 0, across the edge of node n
                F2T<T> t[4];
                int e[Lanes<C>::w];
                f2_normalise4(acc, e);
                f2_apply4<C>(Ph + (size_t)n * 16 * C, Pl + (size_t)n * 16 * C, g, acc, t);
#pragma unroll
                for (int w = 0; w < Lanes<C>::w; ++w) {
                    F2 Lr{0.f, 0.f};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (code >= 4 || code == i) Lr = f2_add(Lr, f2_mul(lane_of(t[i], w), pi[i]));
                    f2_merge(L, E, Lr, e[w] - Prec<float>::kScaleExp * kk);
                }
            }
            if constexpr (S == 2) {  // the site's other categories
                const F2 o{__shfl_xor_sync(0xffffffffu, L.h, 1), __shfl_xor_sync(0xffffffffu, L.l, 1)};
                const int oE = __shfl_xor_sync(0xffffffffu, E, 1);
                if (o.h > 0.f) f2_merge(L, E, o, oE);
            }
            if (valid && g == 0) {
                L = F2{L.h * (1.0f / C), L.l * (1.0f / C)};  // 1/C is a power of two
                term = __dmul_rn((double)A.w[p], f2_log(L, E));
            }
            // the unit's sum: its S * 2 warps
            term = warp_sum(term, 1);
            if (lane == 0) red[warp] = term;
            __syncthreads();
            if (threadIdx.x < per && ub + (int)threadIdx.x < u1) {
                double sum = 0.0;
#pragma unroll
                for (int w = 0; w < 2 * S; ++w) sum += red[threadIdx.x * 2 * S + w];
                part[(size_t)(x - t0) * units_max + ub + threadIdx.x] = sum;
            }
            __syncthreads();
        }
    }
}

// Sums a tree's units (lane l takes units l, l + 32, ..., then the lanes by a butterfly);
// with a prior, adds the log prior of its lengths.
__global__ void k_score_sum(const FullGroup* __restrict__ groups, const int* __restrict__ gstart, int ngroups, int t0,
                            int t1, int units_max, const double* __restrict__ part, double prior_rate,
                            double prior_log) {
    const int x = t0 + blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (x >= min(gstart[ngroups], t1)) return;
    int k = 0;
    while (k + 1 < ngroups && gstart[k + 1] <= x) ++k;
    const FullGroup& G = groups[k];
    const int gi = G.order ? G.order[x - gstart[k]] : x - gstart[k];
    const int units = (G.A.P + kScoreUnit - 1) / kScoreUnit, NN = 2 * G.ts.n - 2;
    double f = 0.0;
    for (int u = lane; u < units; u += 32) f += part[(size_t)(x - t0) * units_max + u];
    f = warp_sum(f, 1);
    if (lane == 0) {
        if (prior_rate != 0.0) {  // MAP: log prior of the lengths
            const double* len = G.ts.len + (size_t)(G.first + gi) * NN;
            double sum = 0.0;
            for (int w = 1; w < NN; ++w) sum += len[w];
            f += (double)(NN - 1) * prior_log - prior_rate * sum;
        }
        G.lnl_out[gi] = f;
    }
}

// ---------------------------------------------------------------- P matrices of tree sets
// Pm[tree][v][16][C] for v = 1..NN-1 (edge (v, up v)); a row of one category per thread.
// Pm_lo (FP32 only, may be null): the rounding residuals, P - Pm (pairs for the scores).
template <typename R>
__global__ void k_pmats(Model M, TreeSet ts, int first, DCount cnt, R* Pm, const double* rates, float* Pm_lo) {
    const int n = ts.n, NN = 2 * n - 2, C = M.C;
    long long total = (long long)dcount(cnt) * NN * C * 4;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total;
         x += (long long)gridDim.x * blockDim.x) {
        int i = (int)(x & 3);
        long long y = x >> 2;
        int r = (int)(y % C);
        y /= C;
        int v = (int)(y % NN);
        int t = (int)(y / NN);
        double l = ts.len[(size_t)(first + t) * NN + v];
        const double rr = rates ? rates[(size_t)(first + t) * kMaxCat + r] : M.rates[r];
        const size_t o = ((size_t)t * NN + v) * C * 16 + i * 4 * C + r;
        if (Pm_lo) {
            double row[4];
            pmat_row<double>(M, l * rr, i, row);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const F2 x = f2_of(row[j]);
                Pm[o + j * C] = (R)x.h;
                Pm_lo[o + j * C] = x.l;
            }
        } else {
            pmat_row<R>(M, l * rr, i, Pm + o, C);
        }
    }
}

// ---------------------------------------------------------------- partials (K1)
// grid (tree, site chunk).  All D_v bottom-up, then all U_v top-down.
template <typename R, int C>
__global__ void k_partials(Model M, Aln A, TreeSet ts, int first, DCount cnt, ClvGroup g, const R* __restrict__ Pm_all,
                           int with_up) {
    extern __shared__ __align__(16) unsigned char smraw[];
    R* Pm = reinterpret_cast<R*>(smraw);
    const int n = ts.n, NN = 2 * n - 2, P = A.P;
    const int gi = blockIdx.x, tree = first + gi;
    if (gi >= dcount(cnt)) return;  // uniform over the block
    const R* Psrc = Pm_all + (size_t)gi * NN * C * 16;
    for (int x = threadIdx.x; x < NN * C * 16; x += blockDim.x) Pm[x] = Psrc[x];
    __syncthreads();
    const int p = blockIdx.y * blockDim.x + threadIdx.x;
    if (p >= P) return;
    const int32_t* up = ts.up + (size_t)tree * NN;
    const int32_t* ch = ts.ch + (size_t)tree * NN * 2;
    R* clv = reinterpret_cast<R*>(g.clv) + (size_t)gi * g.tree_stride;
    int32_t* scl = g.scl + (size_t)gi * g.scl_stride;
    const size_t sstride = (size_t)P * 4 * C;
    auto srcD = [&](int v) {
        Src<R, C> s;
        if (v < n) { s.clv = nullptr; s.scl = nullptr; s.tip = A.tips + (size_t)v * P; }
        else { s.clv = clv + (size_t)(v - n) * sstride; s.scl = scl + (size_t)(v - n) * P; s.tip = nullptr; }
        return s;
    };
    for (int v = NN - 1; v >= n; --v) {
        R y0[4 * C], y1[4 * C];
        int c0cnt, c1cnt;
        int c0 = ch[2 * v], c1 = ch[2 * v + 1];
        apply_p<R, C>(Pm + (size_t)c0 * C * 16, srcD(c0), P, p, p, y0, c0cnt);
        apply_p<R, C>(Pm + (size_t)c1 * C * 16, srcD(c1), P, p, p, y1, c1cnt);
        mul_vec<R, C>(y0, y1);
        int sc = rescale<R, C>(y0);
        store_vec<R, C>(clv + (size_t)(v - n) * sstride, P, p, y0);
        scl[(size_t)(v - n) * P + p] = c0cnt + c1cnt + sc;
    }
    if (!with_up) return;
    for (int v = n + 1; v < NN; ++v) {
        int u = up[v];
        int sib = ch[2 * u] == v ? ch[2 * u + 1] : ch[2 * u];
        Src<R, C> a;
        if (u == n) { a.clv = nullptr; a.scl = nullptr; a.tip = A.tips; }
        else { a.clv = clv + (size_t)(n - 2 + u - n - 1) * sstride; a.scl = scl + (size_t)(n - 2 + u - n - 1) * P; a.tip = nullptr; }
        R y0[4 * C], y1[4 * C];
        int cs, ca;
        apply_p<R, C>(Pm + (size_t)sib * C * 16, srcD(sib), P, p, p, y0, cs);
        apply_p<R, C>(Pm + (size_t)u * C * 16, a, P, p, p, y1, ca);
        mul_vec<R, C>(y0, y1);
        int sc = rescale<R, C>(y0);
        const int slot = n - 2 + (v - n - 1);
        store_vec<R, C>(clv + (size_t)slot * sstride, P, p, y0);
        scl[(size_t)slot * P + p] = cs + ca + sc;
    }
}

// Partials of the mixed path as pairs (see F2): every D_v and U_v of a tree
// with its h part in g.clv (what the FP32 Newton iterations read) and its l
// part in g.clv_lo; grid and layout as k_partials.  P matrices: pairs from
// k_pmats (Pm_all h, Pm_lo l).
template <int C>
__global__ void k_partials_f2(Model M, Aln A, TreeSet ts, int first, DCount cnt, ClvGroup g,
                              const float* __restrict__ Pm_all, const float* __restrict__ Pm_lo, int with_up) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int n = ts.n, NN = 2 * n - 2, P = A.P;
    float* Ph = reinterpret_cast<float*>(smraw);
    float* Pl = Ph + (size_t)NN * C * 16;
    const int gi = blockIdx.x, tree = first + gi;
    if (gi >= dcount(cnt)) return;  // uniform over the block
    for (int x = threadIdx.x; x < NN * C * 16; x += blockDim.x) {
        Ph[x] = Pm_all[(size_t)gi * NN * C * 16 + x];
        Pl[x] = Pm_lo[(size_t)gi * NN * C * 16 + x];
    }
    __syncthreads();
    const int p = blockIdx.y * blockDim.x + threadIdx.x;
    if (p >= P) return;
    const int32_t* up = ts.up + (size_t)tree * NN;
    const int32_t* ch = ts.ch + (size_t)tree * NN * 2;
    float* clv = reinterpret_cast<float*>(g.clv) + (size_t)gi * g.tree_stride;
    float* clo = reinterpret_cast<float*>(g.clv_lo) + (size_t)gi * g.tree_stride;
    int32_t* scl = g.scl + (size_t)gi * g.scl_stride;
    const size_t sstride = (size_t)P * 4 * C;
    auto slot_src = [&](int slot) {
        return Src2<C>{clv + (size_t)slot * sstride, clo + (size_t)slot * sstride, scl + (size_t)slot * P, nullptr};
    };
    auto srcD = [&](int v) {
        return v < n ? Src2<C>{nullptr, nullptr, nullptr, A.tips + (size_t)v * P} : slot_src(v - n);
    };
    auto make = [&](int slot, int a, const Src2<C>& sa, int b, const Src2<C>& sb) {
        f2_join<C>(Ph + (size_t)a * C * 16, Pl + (size_t)a * C * 16, sa, Ph + (size_t)b * C * 16, Pl + (size_t)b * C * 16,
                   sb, P, p, p, clv + (size_t)slot * sstride, clo + (size_t)slot * sstride, scl + (size_t)slot * P);
    };
    for (int v = NN - 1; v >= n; --v) make(v - n, ch[2 * v], srcD(ch[2 * v]), ch[2 * v + 1], srcD(ch[2 * v + 1]));
    if (!with_up) return;
    for (int v = n + 1; v < NN; ++v) {
        const int u = up[v];
        const int sib = ch[2 * u] == v ? ch[2 * u + 1] : ch[2 * u];
        const Src2<C> above = u == n ? Src2<C>{nullptr, nullptr, nullptr, A.tips} : slot_src(n - 2 + u - n - 1);
        make(n - 2 + (v - n - 1), sib, srcD(sib), u, above);
    }
}

// ---------------------------------------------------------------- proposal optimisation (K4)
// One CTA or cluster per NNI neighbour (persistent loop).  The quartet around internal
// edge (u, v): A = the side of u towards leaf 0 (U_u, or leaf 0 itself when u
// is the first inner node), B = v's sibling, C < D = v's children.  After the
// swap u holds A and X2, v holds B and Y2 (swap 0: X2 = C, Y2 = D; swap 1:
// X2 = D, Y2 = C).  Branches 0..4 = central, A, B, C, D, optimised in that
// order per sweep.
template <typename R, int C>
struct ProposeSmem {
    R Pm[5][C * 16];
    R Mt[16];
    R pi[4];
    double T[5];         // the five lengths: inherited or learned, then the final ones
    Len<R> Tl[5];        // the same between the solves
    Src<R, C> msrc[4];   // members in post-swap position order: A, X2 (at u), B, Y2 (at v)
    int mbr[4];          // branch of each member
    int bmem[5];         // member of each branch (-1: central)
    double ex5[5][4 * C];
    int warm[5];         // branch b starts from a learned length (its P matrices are recomputed)
    int next, grp;       // work item taken from the counter, its group
    const float* mlo[4]; // members' FP32 residual partials (mixed precision scores), or null
    float Plo[5][C * 16];// residuals of the five P matrices at the final lengths (pairs with Pm)
    NewtonSmem<R, C> ns;
};

// kClus: launched as clusters of CTAs; the CTAs of a cluster work on the same
// item, each on its share of the sites (make_sites; its sum-table in shared
// memory), with the Newton sums and scores reduced over the cluster.
template <typename R, int C, bool kSmemTab, bool kClus>
__global__ void __launch_bounds__(512) k_propose(const PropGroup* __restrict__ groups, const int* __restrict__ gstart,
                                                 int ngroups, int* counter, Cfg cfg, unsigned long long* stats,
                                                 unsigned char* scratch, size_t scratch_per_cta, Geo geo, int lo,
                                                 int hi) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int total = gstart[ngroups];
    if (total <= lo || total > hi) return;  // another launch shape's number of items
    ProposeSmem<R, C>& sm = *reinterpret_cast<ProposeSmem<R, C>*>(smraw);
    unsigned char* const tab_base = kSmemTab ? smraw + ((sizeof(ProposeSmem<R, C>) + 15) & ~size_t(15))
                                             : scratch + (size_t)blockIdx.x * scratch_per_cta;
    const int nb = cfg.propose_mode == 1 ? 1 : 5;
    unsigned long long evals_total = 0, sweeps_total = 0, nonconv = 0;
    Team tm{kClus ? (int)cluster_ctas() : 1, kClus ? (int)cluster_rank() : 0, 0, 0};
    const int rank = tm.rank;
    if (kClus && threadIdx.x == 0) cluster_exchange_init(sm.ns);  // before the first cluster barrier
    if (sizeof(R) == 4) sm.ns.et.init();
    while (true) {
        // previous item done with shared memory (in every CTA of the cluster: rank 0 writes theirs)
        if constexpr (kClus) cooperative_groups::this_cluster().sync();
        else __syncthreads();
        if (threadIdx.x == 0 && rank == 0) {
            const int x = atomicAdd(counter, 1);
            int k = 0;
            while (k + 1 < ngroups && gstart[k + 1] <= x) ++k;
            if constexpr (kClus) {
                cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
                for (int r = 0; r < tm.kp; ++r) {
                    *cl.map_shared_rank(&sm.next, r) = x;
                    *cl.map_shared_rank(&sm.grp, r) = k;
                }
            } else {
                sm.next = x;
                sm.grp = k;
            }
        }
        if constexpr (kClus) cooperative_groups::this_cluster().sync();
        else __syncthreads();
        const int x = sm.next;
        if (x >= total) break;
        const PropGroup& G = groups[sm.grp];
        const int o = x - gstart[sm.grp];
        const Model& M = G.M;
        const int n = G.fr.n, NN = 2 * n - 2, P = G.A.P;
        const Sites sx = make_sites(P, geo, rank, tm.kp);
        STab<R, C> st;
        st.init(tab_base, sx.ld);
        for (int m = 0; m < sx.cnt; ++m) st.w[sx.pl0 + m * sx.pstep] = (R)G.A.w[sx.p0 + m * sx.step];
        const size_t sstride = (size_t)P * 4 * C;
        const Item it = G.items[o];
        const int gi = it.tree - G.first;
        const int32_t* up = G.fr.up + (size_t)it.tree * NN;
        const int32_t* ch = G.fr.ch + (size_t)it.tree * NN * 2;
        const double* len = G.fr.len + (size_t)it.tree * NN;
        const R* clv = reinterpret_cast<const R*>(G.g.clv) + (size_t)gi * G.g.tree_stride;
        const int32_t* scl = G.g.scl + (size_t)gi * G.g.scl_stride;
        const int v = it.v, u = up[v];
        const int sib = ch[2 * u] == v ? ch[2 * u + 1] : ch[2 * u];
        const int c0 = ch[2 * v], c1 = ch[2 * v + 1];
        // branch b's node in the parent (its P matrix is the parent's): central v, A u, B sib, C c0, D c1
        const int bnode[5] = {v, u, sib, c0, c1};
        const R* Psrc = reinterpret_cast<const R*>(G.Pm) + (size_t)gi * NN * C * 16;
        if (threadIdx.x < 16) {
            const int i = threadIdx.x >> 2, k = threadIdx.x & 3;
            sm.Mt[threadIdx.x] = (R)(M.sqpi[i] * M.R[i * 4 + k]);
            if (threadIdx.x < 4) sm.pi[threadIdx.x] = (R)M.pi[threadIdx.x];
        }
        const double* rr = G.rates ? G.rates + (size_t)it.tree * kMaxCat : M.rates;  // the parent's shape
        init_newton_smem<R, C>(M, cfg, sm.ns, rr);
        if (threadIdx.x == 0) {
            const int node[4] = {u, it.swap == 0 ? c0 : c1, sib, it.swap == 0 ? c1 : c0};
            const int brn[4] = {1, it.swap == 0 ? 3 : 4, 2, it.swap == 0 ? 4 : 3};
            sm.bmem[0] = -1;
            const float* clo = reinterpret_cast<const float*>(G.g.clv_lo);  // mixed precision only
            if (clo) clo += (size_t)gi * G.g.tree_stride;
            for (int m = 0; m < 4; ++m) {
                Src<R, C> y;
                int slot = -1;
                if (m == 0) {
                    if (u == n) { y.clv = nullptr; y.scl = nullptr; y.tip = G.A.tips; }
                    else {
                        slot = n - 2 + (u - n - 1);
                        y.clv = clv + (size_t)slot * sstride; y.scl = scl + (size_t)slot * P; y.tip = nullptr;
                    }
                } else if (node[m] < n) {
                    y.clv = nullptr; y.scl = nullptr; y.tip = G.A.tips + (size_t)node[m] * P;
                } else {
                    slot = node[m] - n;
                    y.clv = clv + (size_t)slot * sstride; y.scl = scl + (size_t)slot * P; y.tip = nullptr;
                }
                sm.mlo[m] = (clo && slot >= 0) ? clo + (size_t)slot * sstride : nullptr;
                sm.msrc[m] = y;
                sm.mbr[m] = brn[m];
                sm.bmem[brn[m]] = m;
            }
        }
        for (int z = threadIdx.x; z < 5 * C * 16; z += blockDim.x) {
            const int b = z / (C * 16), q = z % (C * 16);
            sm.Pm[b][q] = Psrc[(size_t)bnode[b] * C * 16 + q];
        }
        if (threadIdx.x < 5) {
            double t0 = len[bnode[threadIdx.x]];
            int warm = 0;
            if (G.init && (nb == 5 || threadIdx.x == 0)) {  // warm start of the optimised branches; NaN = keep
                const double y = G.init[(size_t)o * 5 + threadIdx.x];
                if (y == y) { t0 = y; warm = 1; }
            }
            sm.T[threadIdx.x] = t0;
            sm.Tl[threadIdx.x] = len_of<R>(t0);
            sm.warm[threadIdx.x] = warm;
        }
        __syncthreads();
        if (G.init) {  // P matrices at the learned starting lengths (the others are the parent's)
            for (int z = threadIdx.x; z < 5 * 4 * C; z += blockDim.x) {
                const int b = z / (4 * C), q = z % (4 * C);
                if (sm.warm[b]) sm.ex5[b][q] = exp(M.lam[q / C] * rr[q % C] * sm.T[b]);
            }
            __syncthreads();
            for (int z = threadIdx.x; z < 5 * 16 * C; z += blockDim.x) {
                const int b = z / (16 * C), q = z % (16 * C), r = q % C, ij = q / C;
                if (!sm.warm[b]) continue;
                double acc = 0.0;
#pragma unroll
                for (int k = 0; k < 4; ++k) acc += sm.ns.W[ij * 4 + k] * sm.ex5[b][k * C + r];
                sm.Pm[b][q] = (R)acc;
            }
            __syncthreads();
        }
        int sweeps = 0, item_evals = 0;
        for (int sw = 0; sw < cfg.prop_max_sweeps; ++sw) {
            ++sweeps;
            for (int b = 0; b < nb; ++b) {
                // Central branch: X = P0 a0 * P1 a1 (at u), Y = P2 a2 * P3 a3 (at v).
                // Branch of member mb: X = mb itself; Y = P2 partner * Pcentral (P0 o1 * P1 o2).
                int i0m, i1m, i2m, i3m;
                if (b == 0) { i0m = 0; i1m = 1; i2m = 2; i3m = 3; }
                else {
                    const int mb = sm.bmem[b];
                    i3m = mb; i2m = mb ^ 1; i0m = mb < 2 ? 2 : 0; i1m = i0m + 1;
                }
                const Src<R, C> a0 = sm.msrc[i0m], a1 = sm.msrc[i1m], a2 = sm.msrc[i2m], a3 = sm.msrc[i3m];
                const R* P0 = sm.Pm[sm.mbr[i0m]];
                const R* P1 = sm.Pm[sm.mbr[i1m]];
                const R* P2 = sm.Pm[sm.mbr[i2m]];
                const R* P3 = sm.Pm[sm.mbr[i3m]];
                const Len<R> told = sm.Tl[b], tbeg = newton_begin<C>(told, sm.ns);
                for (int m = 0; m < sx.cnt; ++m) {
                    const int pl = sx.pl0 + m * sx.pstep, p = sx.p0 + m * sx.step;
                    R X[4 * C], Y[4 * C], t0[4 * C], t1[4 * C];
                    int k0, k1, k2, k3;
                    apply_p<R, C>(P0, a0, P, p, p, t0, k0);
                    apply_p<R, C>(P1, a1, P, p, p, t1, k1);
                    mul_vec<R, C>(t0, t1);
                    if (b == 0) {
#pragma unroll
                        for (int q = 0; q < 4 * C; ++q) X[q] = t0[q];
                        apply_p<R, C>(P2, a2, P, p, p, Y, k2);
                        apply_p<R, C>(P3, a3, P, p, p, t1, k3);
                        mul_vec<R, C>(Y, t1);
                    } else {
                        apply_p_reg<R, C>(sm.Pm[0], t0, X);  // X used as scratch for the far side
                        apply_p<R, C>(P2, a2, P, p, p, Y, k2);
                        mul_vec<R, C>(Y, X);
                        load_raw<R, C>(a3, P, p, p, X, k3);
                    }
                    // b > 0: X is the member's stored vector (kept above 2^-kScaleExp by the
                    // rescaling) or a tip, so it needs no normalisation: its scale multiplies
                    // the site's sum-table row by a power of two, exactly, which the Newton
                    // ratios L'/L, L''/L do not see and the row's exponent field records
                    int ex = b == 0 ? normalise<R, C>(X) : 0, ey = normalise<R, C>(Y);
                    R s4[4 * C];
                    sumtable<R, C>(sm.Mt, sm.pi, X, Y, s4);
                    st.put(pl, s4, ex + ey - Prec<R>::kScaleExp * (k0 + k1 + k2 + k3));
                }
                int ev;
                bool conv;
                // new length; the solve leaves P matrices of branch b at it in sm.Pm[b]
                newton_solve<R, C, kClus>(cfg, st, sx, tbeg, told, &sm.Tl[b], sw + 1, sm.ns, ev, conv, sm.Pm[b], tm);
                evals_total += ev;
                item_evals += ev;
                if (!conv) ++nonconv;
            }
            if (sm.ns.moved_at != sw + 1) break;
        }
        if (threadIdx.x < nb) sm.T[threadIdx.x] = len_dbl(sm.Tl[threadIdx.x]);
        __syncthreads();
        // exact lnL at the final lengths: the last sum-table at its new length, or,
        // in mixed precision, the pair form of the four members around the new edge
        double f1;
        if constexpr (sizeof(R) == 4) {
            for (int z = threadIdx.x; z < 5 * 4 * C; z += blockDim.x) {
                const int b = z / (4 * C), q = z % (4 * C);
                sm.ex5[b][q] = exp(sm.ns.lr[q] * sm.T[b]);
            }
            __syncthreads();
            for (int z = threadIdx.x; z < 5 * 16 * C; z += blockDim.x) {
                const int b = z / (16 * C), q = z % (16 * C);
                f2_pmat_entry<C>(sm.ns.W, sm.ex5[b], q, reinterpret_cast<float*>(sm.Pm[b]), sm.Plo[b]);
            }
            __syncthreads();
            Src2<C> mem[4];
#pragma unroll
            for (int m = 0; m < 4; ++m)
                mem[m] = Src2<C>{reinterpret_cast<const float*>(sm.msrc[m].clv), sm.mlo[m], sm.msrc[m].scl,
                                 sm.msrc[m].tip};
            f1 = propose_score_f2<C, kClus>(mem, sm.mbr, reinterpret_cast<const float*>(sm.Pm), &sm.Plo[0][0], M.pi,
                                            G.A.w, P, sx, sm.ns.red, tm);
        } else {
            f1 = eval_lnl<C, kClus>(st, sx, sm.T[nb - 1], sm.ns, tm);
        }
        sweeps_total += sweeps;
        if (threadIdx.x == 0 && rank == 0) {
            if (__double_as_longlong(cfg.prior_rate) != 0) {  // MAP: log prior of the neighbour's lengths
                double sum = 0.0;
                for (int w = 1; w < NN; ++w) sum += len[w];
                for (int b = 0; b < 5; ++b) sum += sm.T[b] - len[bnode[b]];
                f1 += (double)(NN - 1) * cfg.prior_log - cfg.prior_rate * sum;
            }
            G.lnl_out[o] = f1;
            if (G.evals_out) G.evals_out[o] = item_evals;
            for (int b = 0; b < 5; ++b) G.len5_out[(size_t)o * 5 + b] = sm.T[b];
            if (G.cost_out) {  // how far the proposal moved the five lengths: predicts the visit's cost
                float cst = 0.f;
                for (int b = 0; b < 5; ++b) cst += fabsf(logf((float)(sm.T[b] / len[bnode[b]])));
                G.cost_out[o] = cst;
            }
            const int k = f1 >= *G.lmax - G.thr;
            G.kept[o] = k;
            if (G.tab) {  // no table: a hill-climb's neighbourhood scoring
                Slot* sl = &G.tab[it.slot];
                sl->lnl = f1;
                sl->tag = ((unsigned long long)dround(G.round) << 48) | (unsigned long long)(k ? 4 : 1);
            }
        }
    }
    if (threadIdx.x == 0 && rank == 0) {
        atomicAdd(&stats[kStPropEvals], evals_total);
        atomicAdd(&stats[kStPropSweeps], sweeps_total);
        atomicAdd(&stats[kStNonconv], nonconv);
    }
    if (kClus && threadIdx.x == 0 && sm.ns.abort_) atomicAdd(&stats[kStTimeout], 1ull);
    if constexpr (kClus) cooperative_groups::this_cluster().sync();  // no CTA leaves while others may read it
}

// ---------------------------------------------------------------- full optimisation (K7)
// One CTA or cluster per tree (persistent loop).  Bottom-up D pass, then sweeps over the
// schedule: visit edge v = compute U_v (stored for inner v), sum-table of
// (U_v, D_v), Newton on the length; refresh D_v after its subtree.  In FP64
// the lnL at the final lengths follows (with max_sweeps = 0: at the given ones); in
// mixed precision k_score makes it, and a launch has max_sweeps > 0.
template <typename R, int C>
struct FullSmem {
    R Mt[16];
    R pi[4];
    int next, grp;
    alignas(16) R Pst[2][C * 16];         // the current operation's P matrices, when the tree's stay in the slab
    NewtonSmem<R, C> ns;
};
// Shared memory after FullSmem: lengths, the tree (parents and children as
// bytes, the schedule), then the P matrices (p_smem), then the sum-table.
__host__ __device__ inline size_t full_meta_bytes(int nn) {
    const int n = (nn + 2) / 2;
    return (size_t)nn * 8 + (((size_t)3 * nn + 2 * 3 * n + 15) & ~size_t(15));
}
constexpr unsigned short kUpd16 = 0x8000;  // kUpd in a 16-bit schedule entry

// kClus: launched as clusters of CTAs working on the same tree, each on its share
// of the sites (make_sites: partials slab and sum-table of its share), Newton
// sums and scores reduced over the cluster.
//
// A launch is bound by the latency of its 2n - 3 solves per sweep, which follow one
// another; what shortens them: the schedule and the tree in shared memory (they
// were chains of three or four global loads before each operation), the P matrices
// of an operation there too (read through L1 they were evicted by the vectors that
// stream past), and as many lanes and CTAs per tree as the number of trees leaves
// room for (Sites).  8 trees of 27 x 816 patterns took 12.9 ms on one CTA each with
// those chains, now 6.0; 32 of 128 x 6273 289 ms, now 165; 515 of them 526 ms, now 340
// (there a solve's 54 thousand cycles are half sum-table builds, which wait for their
// stored vectors: 2.5 TB/s on average, of 6.8 that a copy reaches, with long scoreboard the
// first stall, so it is the latency of too few bytes in flight and not their rate).
template <typename R, int C, bool kSmemTab, bool kClus>
__global__ void __launch_bounds__(512) k_fullopt(const FullGroup* __restrict__ groups, const int* __restrict__ gstart,
                                                 int ngroups, int* counter, int nn_max, Cfg cfg,
                                                 unsigned long long* stats, unsigned char* scratch,
                                                 size_t scratch_per_cta, unsigned char* slab, size_t slab_per_cta,
                                                 int p_smem, Geo geo, int lo, int hi) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int total = gstart[ngroups];
    if (total <= lo || total > hi) return;  // another launch shape's number of trees
    FullSmem<R, C>& sm = *reinterpret_cast<FullSmem<R, C>*>(smraw);
    size_t off = (sizeof(FullSmem<R, C>) + 15) & ~size_t(15);
    double* len = reinterpret_cast<double*>(smraw + off);         // the lengths before and after the sweeps,
    Len<R>* const lens = reinterpret_cast<Len<R>*>(smraw + off);  // and between the solves
    uint16_t* const sched = reinterpret_cast<uint16_t*>(len + nn_max);
    uint8_t* const up = reinterpret_cast<uint8_t*>(sched + 3 * ((nn_max + 2) / 2));
    uint8_t* const ch = up + nn_max;
    off += full_meta_bytes(nn_max);
    R* const Psm = reinterpret_cast<R*>(smraw + off);  // P matrices here when p_smem
    if (p_smem) off += (size_t)nn_max * C * 16 * sizeof(R);
    unsigned char* const tab_base = kSmemTab ? smraw + off : scratch + (size_t)blockIdx.x * scratch_per_cta;
    unsigned long long evals_total = 0, sweeps_total = 0, nonconv = 0;
    Team tm{kClus ? (int)cluster_ctas() : 1, kClus ? (int)cluster_rank() : 0, 0, 0};
    const int rank = tm.rank;
    if (kClus && threadIdx.x == 0) cluster_exchange_init(sm.ns);  // before the first cluster barrier
    if (sizeof(R) == 4) sm.ns.et.init();
    bool first = true;  // thread 0: this CTA (cluster) has not taken a tree yet
    while (true) {
        // previous tree done with shared memory (in every CTA of the cluster: rank 0 writes theirs)
        if constexpr (kClus) cooperative_groups::this_cluster().sync();
        else __syncthreads();
        if (threadIdx.x == 0 && rank == 0) {
            // Cluster c's first tree is tree c (the costliest trees come first, and clusters
            // in launch order are spread over the SMs), later ones come from the counter
            // after the grid's first trees.  With fewer trees than clusters, taking the
            // first trees from the counter let two CTAs of one SM win trees while other SMs
            // stayed idle (a capacity-sized graph launch).
            const int nclus = (int)gridDim.x / tm.kp;
            const int x = first ? (int)blockIdx.x / tm.kp : nclus + atomicAdd(counter, 1);
            first = false;
            int k = 0;
            while (k + 1 < ngroups && gstart[k + 1] <= x) ++k;
            if constexpr (kClus) {
                cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
                for (int r = 0; r < tm.kp; ++r) {
                    *cl.map_shared_rank(&sm.next, r) = x;
                    *cl.map_shared_rank(&sm.grp, r) = k;
                }
            } else {
                sm.next = x;
                sm.grp = k;
            }
        }
        if constexpr (kClus) cooperative_groups::this_cluster().sync();
        else __syncthreads();
        const int x = sm.next;
        if (x >= total) break;
        const FullGroup& G = groups[sm.grp];
        const int gi = G.order ? G.order[x - gstart[sm.grp]] : x - gstart[sm.grp];
        const Model& M = G.M;
        const Aln& A = G.A;
        const int n = G.ts.n, NN = 2 * n - 2, P = A.P, nsched = 3 * n - 5;
        const Sites sx = make_sites(P, geo, rank, tm.kp);
        const int Ps = sx.ld;
        STab<R, C> st;
        st.init(tab_base, Ps);
        for (int m = 0; m < sx.cnt; ++m) st.w[sx.pl0 + m * sx.pstep] = (R)A.w[sx.p0 + m * sx.step];
        const size_t sstride = (size_t)Ps * 4 * C;
        const int tree = G.first + gi;
        double* glen = G.ts.len + (size_t)tree * NN;
        // this CTA's own slab, reused tree after tree: partials, scalers and the P
        // matrices of every edge; the P matrices move to shared memory when the
        // launch shape leaves it free (p_smem, see full_p_smem), else an operation
        // copies the two it reads
        unsigned char* const b = slab + (size_t)blockIdx.x * slab_per_cta;
        const size_t clv_bytes = ((size_t)(2 * n - 5) * Ps * 4 * C * sizeof(R) + 255) & ~size_t(255);
        const size_t scl_bytes = ((size_t)(2 * n - 5) * Ps * 4 + 255) & ~size_t(255);
        R* const clv = reinterpret_cast<R*>(b);
        int32_t* const scl = reinterpret_cast<int32_t*>(b + clv_bytes);
        R* const Pm = p_smem ? Psm : reinterpret_cast<R*>(b + clv_bytes + scl_bytes);
        if (threadIdx.x < 16) {
            const int i = threadIdx.x >> 2, k = threadIdx.x & 3;
            sm.Mt[threadIdx.x] = (R)(M.sqpi[i] * M.R[i * 4 + k]);
            if (threadIdx.x < 4) sm.pi[threadIdx.x] = (R)M.pi[threadIdx.x];
        }
        // per-tree category rates (a visit that re-optimises the Gamma shape), else the model's
        const double* rr = G.rates ? G.rates + (size_t)gi * kMaxCat : M.rates;
        init_newton_smem<R, C>(M, cfg, sm.ns, rr);
        for (int v = threadIdx.x; v < NN; v += blockDim.x) {
            if (G.max_sweeps > 0) lens[v] = len_of<R>(glen[v]);
            else len[v] = glen[v];
            up[v] = (uint8_t)G.ts.up[(size_t)tree * NN + v];
            ch[2 * v] = (uint8_t)G.ts.ch[((size_t)tree * NN + v) * 2];
            ch[2 * v + 1] = (uint8_t)G.ts.ch[((size_t)tree * NN + v) * 2 + 1];
        }
        for (int k = threadIdx.x; k < nsched; k += blockDim.x) {
            const int op = G.ts.sched[(size_t)tree * 3 * n + k];
            sched[k] = (uint16_t)((op & 0xff) | (op & kUpd ? kUpd16 : 0));
        }
        __syncthreads();
        for (int z = threadIdx.x; z < NN * C * 4; z += blockDim.x) {
            const int v = z / (C * 4), r = (z / 4) % C, i = z & 3;
            if (v > 0) pmat_row<R>(M, glen[v] * rr[r], i, Pm + (size_t)v * C * 16 + i * 4 * C + r, C);
        }
        __syncthreads();
        auto srcD = [&](int v) {
            Src<R, C> y;
            if (v < n) { y.clv = nullptr; y.scl = nullptr; y.tip = A.tips + (size_t)v * P; }
            else { y.clv = clv + (size_t)(v - n) * sstride; y.scl = scl + (size_t)(v - n) * Ps; y.tip = nullptr; }
            return y;
        };
        auto srcU = [&](int v) {  // the vector at up[v] without v's subtree, for inner v != n; leaf 0 for n
            Src<R, C> y;
            const int slot = n - 2 + (v - n - 1);
            y.clv = clv + (size_t)slot * sstride; y.scl = scl + (size_t)slot * Ps; y.tip = nullptr;
            if (v == n) { y.clv = nullptr; y.scl = nullptr; y.tip = A.tips; }
            return y;
        };
        // the P matrices of edges a and b for the operation that follows
        const R *Pa = sm.Pst[0], *Pb = sm.Pst[1];
        auto stage_p = [&](int a, int b) {
            if (p_smem) {
                Pa = Psm + (size_t)a * C * 16;
                Pb = Psm + (size_t)b * C * 16;
                return;
            }
            __syncthreads();  // the operation before is done with the staged pair
            for (int z = threadIdx.x; z < 2 * C * 16; z += blockDim.x)
                (&sm.Pst[0][0])[z] = Pm[(size_t)(z < C * 16 ? a : b) * C * 16 + z % (C * 16)];
            __syncthreads();
        };
        auto refreshD = [&](int v) {
            const int c0 = ch[2 * v], c1 = ch[2 * v + 1];
            stage_p(c0, c1);
            const Src<R, C> s0 = srcD(c0), s1 = srcD(c1);
            for (int m = 0; m < sx.cnt; ++m) {
                const int p = sx.pl0 + m * sx.pstep, pg = sx.p0 + m * sx.step;
                R y0[4 * C], y1[4 * C];
                int k0, k1;
                apply_p<R, C>(Pa, s0, Ps, p, pg, y0, k0);
                apply_p<R, C>(Pb, s1, Ps, p, pg, y1, k1);
                mul_vec<R, C>(y0, y1);
                const int sc = rescale<R, C>(y0);
                store_vec<R, C>(clv + (size_t)(v - n) * sstride, Ps, p, y0);
                scl[(size_t)(v - n) * Ps + p] = k0 + k1 + sc;
            }
        };
        // builds the sum-table of edge (v, up v), storing U_v for inner v
        auto visit_build = [&](int v) {
            const int u = up[v], sib = ch[2 * u] == v ? ch[2 * u + 1] : ch[2 * u];
            if (v != n) stage_p(sib, u);
            const Src<R, C> sv = srcD(v), ss = v == n ? srcU(n) : srcD(sib), su = srcU(v == n ? n : u);
            for (int m = 0; m < sx.cnt; ++m) {
                const int p = sx.pl0 + m * sx.pstep, pg = sx.p0 + m * sx.step;
                R X[4 * C], Y[4 * C];
                int cx, cy;
                // D_v first: its load then overlaps the two below instead of waiting
                // behind the store of U_v (the same array, so it could not be hoisted)
                load_raw<R, C>(sv, Ps, p, pg, Y, cy);
                if (v == n) {
                    load_raw<R, C>(su, Ps, p, pg, X, cx);
                } else {
                    R y1[4 * C];
                    int k0, k1;
                    apply_p<R, C>(Pa, ss, Ps, p, pg, X, k0);
                    apply_p<R, C>(Pb, su, Ps, p, pg, y1, k1);
                    mul_vec<R, C>(X, y1);
                    const int sc = rescale<R, C>(X);
                    cx = k0 + k1 + sc;
                    if (v >= n) {
                        const int slot = n - 2 + (v - n - 1);
                        store_vec<R, C>(clv + (size_t)slot * sstride, Ps, p, X);
                        scl[(size_t)slot * Ps + p] = cx;
                    }
                }
                // Y is D_v as stored (kept above 2^-kScaleExp by the rescaling) or a tip:
                // no normalisation needed (an exact power-of-two scale of the row)
                const int ex = normalise<R, C>(X);
                R s4[4 * C];
                sumtable<R, C>(sm.Mt, sm.pi, X, Y, s4);
                st.put(p, s4, ex - Prec<R>::kScaleExp * (cx + cy));
            }
        };
        // the stored vectors an operation of the schedule reads, requested into L2
        // while the operation before it runs (its Newton iterations touch no HBM): a
        // slot is one run of memory, so one thread asks for it in one instruction
        auto prefetch_op = [&](int op) {
            auto slot = [&](int sl) {
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(clv + (size_t)sl * sstride),
                             "r"((unsigned)(sstride * sizeof(R)))
                             : "memory");
            };
            if (op & kUpd16) {
                const int w = op & 0xff;
                if (ch[2 * w] >= n) slot(ch[2 * w] - n);
                if (ch[2 * w + 1] >= n) slot(ch[2 * w + 1] - n);
                return;
            }
            if (op != n) {
                const int u = up[op];
                const int sib = ch[2 * u] == op ? ch[2 * u + 1] : ch[2 * u];
                if (sib >= n) slot(sib - n);
                if (u != n) slot(n - 2 + (u - n - 1));
            }
            if (op >= n) slot(op - n);
        };
        // bottom-up D pass
        for (int v = NN - 1; v >= n; --v) refreshD(v);
        int sweeps = 0, last = n;
        if (G.max_sweeps == 0) visit_build(n);  // FP64 (mixed precision scores fixed lengths by k_score alone)
        for (int sw = 0; sw < G.max_sweeps; ++sw) {
            ++sweeps;
            for (int k = 0; k < nsched; ++k) {
                const int op = sched[k];
                if (op & kUpd16) {
                    if (threadIdx.x == 0 && k + 1 < nsched) prefetch_op(sched[k + 1]);
                    refreshD(op & 0xff);
                    continue;
                }
                const int v = op;
                const Len<R> told = lens[v], tbeg = newton_begin<C>(told, sm.ns);
                visit_build(v);
                if (threadIdx.x == 0 && k + 1 < nsched) prefetch_op(sched[k + 1]);
                int ev;
                bool conv;
                // the solve leaves the P matrices of edge v at its new length in Pm
                newton_solve<R, C, kClus>(cfg, st, sx, tbeg, told, &lens[v], sw + 1, sm.ns, ev, conv,
                                          Pm + (size_t)v * C * 16, tm);
                evals_total += ev;
                if (!conv) ++nonconv;
                last = v;
            }
            if (sm.ns.moved_at != sw + 1) break;
        }
        __syncthreads();
        if (sweeps > 0)
            for (int v = threadIdx.x; v < NN; v += blockDim.x) len[v] = len_dbl(lens[v]);
        __syncthreads();
        sweeps_total += sweeps;
        // exact lnL at the final lengths: the last visited edge's sum-table (FP64); in
        // mixed precision k_score follows on the lengths written here
        double f1 = 0.0;
        if constexpr (sizeof(R) == 8) f1 = eval_lnl<C, kClus>(st, sx, len[last], sm.ns, tm);
        __syncthreads();
        if (rank == 0)
            for (int v = threadIdx.x; v < NN; v += blockDim.x) glen[v] = len[v];
        if (sizeof(R) == 8 && threadIdx.x == 0 && rank == 0) {
            if (__double_as_longlong(cfg.prior_rate) != 0) {  // MAP: log prior of the lengths
                double sum = 0.0;
                for (int w = 1; w < NN; ++w) sum += len[w];
                f1 += (double)(NN - 1) * cfg.prior_log - cfg.prior_rate * sum;
            }
            G.lnl_out[gi] = f1;
        }
    }
    if (threadIdx.x == 0 && rank == 0) {
        atomicAdd(&stats[kStFullEvals], evals_total);
        atomicAdd(&stats[kStFullSweeps], sweeps_total);
        atomicAdd(&stats[kStNonconv], nonconv);
    }
    if (kClus && threadIdx.x == 0 && sm.ns.abort_) atomicAdd(&stats[kStTimeout], 1ull);
    if constexpr (kClus) cooperative_groups::this_cluster().sync();  // no CTA leaves while others may read it
}

inline int blocks_for(long long n, int t) { return (int)((n + t - 1) / t); }
// 256-thread blocks for a thread per tree and edge (grid-stride past 4096 blocks)
inline int tree_edge_blocks(int n, long long trees) {
    return (int)std::min<long long>((trees * (2 * n - 3) + 255) / 256, 4096);
}

}  // namespace

// ================================================================= launchers
void launch_canon(cudaStream_t s, int n, DCount count, const int32_t* edges, const double* lengths, TreeSet ts,
                  int32_t* err) {
    if (count.cap <= 0) return;
    k_canon<<<blocks_for(count.cap, kCanonWarps), 32 * kCanonWarps, 0, s>>>(n, count, edges, lengths, ts, err);
    ++g_launches;
}
void launch_canon(cudaStream_t s, int n, int count, const int32_t* edges, const double* lengths, TreeSet ts,
                  int32_t* err) {
    launch_canon(s, n, hcount(count), edges, lengths, ts, err);
}

void launch_table_init(cudaStream_t s, Slot* tab, size_t nslots) {
    k_table_init<<<2432, 256, 0, s>>>(tab, nslots);
    ++g_launches;
}

void launch_enum(cudaStream_t s, int n, DCount F, TreeSet fr, uint64_t* nkey, int32_t* cinfo) {
    long long total = (long long)F.cap * 2 * (n - 3);
    if (total <= 0) return;
    k_enum<<<(int)std::min<long long>(blocks_for(total, 256), 65535), 256, 0, s>>>(n, F, fr, nkey, cinfo);
    ++g_launches;
}

void launch_cand_insert(cudaStream_t s, Slot* tab, int log2, DCount ncand, const uint64_t* nkey, const int32_t* cinfo,
                        TreeSet fr, DRound round, int32_t* cslot, int32_t* flag, int32_t* err,
                        unsigned long long* stats) {
    if (ncand.cap <= 0) return;
    k_cand_insert<<<blocks_for(ncand.cap, 256), 256, 0, s>>>(tab, log2, ncand, nkey, cinfo, fr, round, cslot, flag, err,
                                                             stats);
    ++g_launches;
}

void launch_cand_arb(cudaStream_t s, int phase, Slot* tab, DCount ncand, const int32_t* cinfo, TreeSet fr,
                     DRound round, const int32_t* cslot, int32_t* flag) {
    if (ncand.cap <= 0) return;
    k_cand_arb<<<blocks_for(ncand.cap, 256), 256, 0, s>>>(phase, tab, ncand, cinfo, fr, round, cslot, flag);
    ++g_launches;
}

void launch_scan(cudaStream_t s, const int32_t* in, int32_t* out, int N, int32_t* tmp) {
    if (N <= 0) return;
    int nb = blocks_for(N, 1024);
    k_scan_block<<<nb, 1024, 0, s>>>(in, out, N, tmp);
    ++g_launches;
    k_scan_sums<<<1, 1024, 0, s>>>(tmp, nb);
    ++g_launches;
    k_scan_add<<<nb, 1024, 0, s>>>(out, N, tmp);
    ++g_launches;
}

void launch_scan_total(cudaStream_t s, const int32_t* in, const int32_t* out, int N, int32_t* total) {
    k_scan_total<<<1, 32, 0, s>>>(in, out, N, total);
    ++g_launches;
}

void launch_mul_counts(cudaStream_t s, int na, const int* F, const int* m, int* ncand) {
    k_mul_counts<<<1, 32 * ((na + 31) / 32), 0, s>>>(na, F, m, ncand);
    ++g_launches;
}

void launch_prefix_counts(cudaStream_t s, int ng, const int* cnt, const int* perm, int* gstart) {
    k_prefix_counts<<<1, 32, 0, s>>>(ng, cnt, perm, gstart);
    ++g_launches;
}

void launch_make_items(cudaStream_t s, int ncand, const int32_t* flag, const int32_t* pos, const int32_t* cinfo,
                       const int32_t* cslot, const uint64_t* nkey, Item* items, uint64_t* ikey) {
    if (ncand <= 0) return;
    k_make_items<<<blocks_for(ncand, 256), 256, 0, s>>>(ncand, flag, pos, cinfo, cslot, nkey, items, ikey);
    ++g_launches;
}

void launch_compact_idx(cudaStream_t s, int N, const int32_t* flag, const int32_t* pos, int32_t* idx) {
    if (N <= 0) return;
    k_compact_idx<<<blocks_for(N, 256), 256, 0, s>>>(N, flag, pos, idx);
    ++g_launches;
}

void launch_fill_i32(cudaStream_t s, int N, int32_t* a, int32_t va, int32_t* b, int32_t vb) {
    if (N <= 0) return;
    k_fill_i32<<<blocks_for(N, 256), 256, 0, s>>>(N, a, va, b, vb);
    ++g_launches;
}

void launch_climb_best(cudaStream_t s, int F, int m, const double* lnl, const uint64_t* ikey, int32_t* best) {
    if (F <= 0 || m <= 0) return;
    k_climb_best<<<blocks_for(F, 8), 256, 0, s>>>(F, m, lnl, ikey, best);
    ++g_launches;
}

void launch_insert_trees(cudaStream_t s, Slot* tab, int log2, DCount count, TreeSet ts, const double* lnl,
                         const int32_t* status, DRound round, int32_t* winner, int32_t* err) {
    if (count.cap <= 0) return;
    k_insert_trees<<<blocks_for(count.cap, 256), 256, 0, s>>>(tab, log2, count, ts, lnl, status, winner, err);
    ++g_launches;
    k_insert_trees_fin<<<blocks_for(count.cap, 256), 256, 0, s>>>(tab, count, lnl, status, round, winner);
    ++g_launches;
}

void launch_finalize_trees(cudaStream_t s, Slot* tab, DCount count, const int32_t* slot_of, const double* lnl,
                           const double* lmax, double thr, DRound round, int32_t* good, unsigned long long* stats,
                           const double* alpha) {
    if (count.cap <= 0) return;
    k_finalize_trees<<<blocks_for(count.cap, 256), 256, 0, s>>>(tab, count, slot_of, lnl, lmax, thr, round, good,
                                                                stats, alpha);
    ++g_launches;
}

void launch_lmax(cudaStream_t s, DCount count, const double* lnl, const int32_t* mask, double* lmax) {
    if (count.cap <= 0) return;
    k_lmax<<<std::min(blocks_for(count.cap, 256), 1024), 256, 0, s>>>(count, lnl, mask, lmax);
    ++g_launches;
}

void launch_dump(cudaStream_t s, const Slot* tab, size_t nslots, int32_t* flag) {
    k_dump_flag<<<1024, 256, 0, s>>>(tab, nslots, flag);
    ++g_launches;
}

void launch_dump_gather(cudaStream_t s, const Slot* tab, size_t nslots, const int32_t* flag, const int32_t* pos,
                        uint64_t* keys, uint8_t* status, double* lnl) {
    k_dump_gather<<<1024, 256, 0, s>>>(tab, nslots, flag, pos, keys, status, lnl);
    ++g_launches;
}

void launch_materialize(cudaStream_t s, int n, DCount nk, const int32_t* kidx, const Item* items, TreeSet fr,
                        const double* len5, int32_t* edges_out, double* lengths_out, int32_t* slot_of) {
    if (nk.cap <= 0) return;
    k_materialize<<<tree_edge_blocks(n, nk.cap), 256, 0, s>>>(n, nk, kidx, items, fr, len5, edges_out, lengths_out,
                                                          slot_of);
    ++g_launches;
}

void launch_gather_out(cudaStream_t s, int n, DCount count, const int32_t* idx, TreeSet ts, const double* lnl,
                       int32_t* edges_out, double* lengths_out, double* lnl_out, uint64_t* keys_out) {
    if (count.cap <= 0) return;
    k_gather_out<<<tree_edge_blocks(n, count.cap), 256, 0, s>>>(n, count, idx, ts, lnl, edges_out, lengths_out, lnl_out,
                                                             keys_out);
    ++g_launches;
}

void launch_frontier_alpha(cudaStream_t s, TreeSet fr, int count, const Slot* tab, int log2, double base,
                           double* alpha) {
    if (count <= 0) return;
    k_frontier_alpha<<<blocks_for(count, 128), 128, 0, s>>>(fr, count, tab, log2, base, alpha);
    ++g_launches;
}

void launch_cost_order(cudaStream_t s, DCount count, const int32_t* kidx, const float* cost, int32_t* order) {
    if (count.cap <= 0) return;
    k_cost_order<<<1, 1024, 0, s>>>(count, kidx, cost, order);
    ++g_launches;
}

void launch_gamma_rates(cudaStream_t s, int count, int C, const double* alpha, double* rates) {
    if (count <= 0) return;
    k_gamma_rates<<<blocks_for(count, 64), 64, 0, s>>>(count, C, alpha, rates);
    ++g_launches;
}

void launch_split_frequencies(cudaStream_t s, TreeSet ts, int count, const double* lnl, const double* lmax,
                              SplitSlot* tab, int log2, int32_t* err) {
    const size_t nslots = (size_t)1 << log2;
    k_split_init<<<(int)std::min<size_t>((nslots + 255) / 256, 4096), 256, 0, s>>>(tab, nslots);
    ++g_launches;
    const long long work = (long long)count * (ts.n - 3);
    if (work > 0) {
        k_split_add<<<blocks_for(work, 256), 256, 0, s>>>(ts, count, lnl, lmax, tab, log2, err);
        ++g_launches;
    }
}

void launch_split_dump(cudaStream_t s, const SplitSlot* tab, size_t nslots, int32_t* flag, const int32_t* pos,
                       uint64_t* splits, double* w, unsigned long long* trees, bool gather) {
    const int grid = (int)std::min<size_t>((nslots + 255) / 256, 4096);
    if (!gather) k_split_flag<<<grid, 256, 0, s>>>(tab, nslots, flag);
    else k_split_gather<<<grid, 256, 0, s>>>(tab, nslots, flag, pos, splits, w, trees);
    ++g_launches;
}

void launch_len5_inherit(cudaStream_t s, int n, DCount count, const Item* items, TreeSet fr, double* len5) {
    if (count.cap <= 0) return;
    k_len5_inherit<<<blocks_for(count.cap, 128), 128, 0, s>>>(n, count, items, fr, len5);
    ++g_launches;
}

void launch_prop_full_finish(cudaStream_t s, DCount count, const Item* items, const double* lnl, const double* lmax,
                             double thr, DRound round, Slot* tab, int32_t* kept) {
    if (count.cap <= 0) return;
    k_prop_full_finish<<<blocks_for(count.cap, 256), 256, 0, s>>>(count, items, lnl, lmax, thr, round, tab, kept);
    ++g_launches;
}

void launch_gather_i32(cudaStream_t s, DCount count, const int32_t* idx, const int32_t* src, int32_t* dst) {
    if (count.cap <= 0) return;
    k_gather_i32<<<blocks_for(count.cap, 256), 256, 0, s>>>(count, idx, src, dst);
    ++g_launches;
}

void launch_lengths_to_input(cudaStream_t s, int n, int count, TreeSet ts, double* lengths_out) {
    if (count <= 0) return;
    k_lengths_to_input<<<tree_edge_blocks(n, count), 256, 0, s>>>(n, count, ts, lengths_out);
    ++g_launches;
}

// Sum-table of ld local sites: 4C values, the weight and (FP64) the exponent of each, the
// exponent as the 32-bit integer that it is: with 8 bytes for it, the shared memory that
// the launch takes beside the table left room for 1532 patterns of 128 taxa, now for 1576.
size_t sumtable_bytes(int prec, int C, int ld) {
    const size_t pcap = (size_t)((ld + 3) & ~3);
    return prec == 0 ? ((4 * (size_t)C + 1) * 8 + 4) * pcap : (4 * (size_t)C + 1) * 4 * pcap;
}

namespace {
constexpr size_t kSmemPerCta = 227 * 1024, kSmemPerCta2 = 233472 / 2 - 1024;  // one CTA per SM, two CTAs per SM
// Lets a kernel's launches take any amount of dynamic shared memory that a CTA can have
// beside the kernel's own (kOwn bytes at most): the limit belongs to the kernel, so one that
// followed each launch's size could be lowered by another thread before the launch it was for.
template <size_t kOwn = 0, typename K>
cudaError_t allow_smem(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kSmemPerCta - kOwn));
}
template <typename F>
size_t by_kind(int prec, int C, F f) {
    if (prec == 0) return C == 1 ? f(double(), std::integral_constant<int, 1>()) : f(double(), std::integral_constant<int, 4>());
    return C == 1 ? f(float(), std::integral_constant<int, 1>()) : f(float(), std::integral_constant<int, 4>());
}
size_t propose_fixed(int prec, int C) {
    return by_kind(prec, C, [](auto r, auto c) { return (sizeof(ProposeSmem<decltype(r), decltype(c)::value>) + 15) & ~size_t(15); });
}
size_t full_fixed(int prec, int C, int n) {
    return by_kind(prec, C, [](auto r, auto c) { return (sizeof(FullSmem<decltype(r), decltype(c)::value>) + 15) & ~size_t(15); }) +
           full_meta_bytes(2 * n - 2);
}
// Where a full optimisation keeps the P matrices of a tree's edges: in shared
// memory where that does not cost a resident CTA (512 threads take the SM's whole
// register file, smaller CTAs run two to an SM), otherwise in the CTA's slab.
bool full_p_smem(int prec, int C, int n, size_t f, int threads) {
    const size_t pb = (size_t)(2 * n - 2) * C * 16 * (prec == 0 ? 8 : 4);
    return f + pb <= (threads < 512 && f <= kSmemPerCta2 ? kSmemPerCta2 : kSmemPerCta);
}
}  // namespace

size_t propose_smem_bytes(int prec, int C, int ld) {
    return propose_fixed(prec, C) + (ld ? sumtable_bytes(prec, C, ld) : 0);
}
size_t fullopt_smem_bytes(int prec, int C, int n, int ld, int threads) {
    const size_t f = full_fixed(prec, C, n) + (ld ? sumtable_bytes(prec, C, ld) : 0);
    return f + (full_p_smem(prec, C, n, f, threads) ? (size_t)(2 * n - 2) * C * 16 * (prec == 0 ? 8 : 4) : 0);
}

namespace {
template <typename R, int C>
void partials_t(cudaStream_t s, const Model& M, Aln A, TreeSet ts, int first, DCount count, ClvGroup g, bool with_up,
                int threads, R* pm, const double* rates) {
    const int NN = 2 * ts.n - 2;
    long long rows = (long long)count.cap * NN * C * 4;
    // mixed precision: P pairs (residuals after the FP32 matrices of all trees) and pair partials
    float* lo = sizeof(R) == 4 ? reinterpret_cast<float*>(pm) + (size_t)count.cap * NN * C * 16 : nullptr;
    k_pmats<R><<<(int)std::min<long long>(blocks_for(rows, 256), 8192), 256, 0, s>>>(M, ts, first, count, pm, rates,
                                                                                   lo);
    ++g_launches;
    if constexpr (sizeof(R) == 4) {
        const size_t sm2 = (size_t)NN * C * 16 * 8;
        allow_smem(k_partials_f2<C>);
        dim3 grid(count.cap, blocks_for(A.P, threads));
        k_partials_f2<C><<<grid, threads, sm2, s>>>(M, A, ts, first, count, g, reinterpret_cast<float*>(pm), lo,
                                                    with_up ? 1 : 0);
    } else {
        const size_t smem = (size_t)NN * C * 16 * sizeof(R);
        allow_smem(k_partials<R, C>);
        dim3 grid(count.cap, blocks_for(A.P, threads));
        k_partials<R, C><<<grid, threads, smem, s>>>(M, A, ts, first, count, g, pm, with_up ? 1 : 0);
    }
    ++g_launches;
}
}  // namespace

size_t pmat_bytes(int prec, int C, int n, int count) {
    // FP32: the matrices, then their FP32 rounding residuals (pairs for the scores)
    return (size_t)count * (2 * n - 2) * C * 16 * 8;
}

void launch_partials(cudaStream_t s, int prec, const Model& M, Aln A, TreeSet ts, int first, DCount count, ClvGroup g,
                     bool with_up, int threads, void* pm, const double* rates) {
    if (count.cap <= 0) return;
    if (prec == 0) {
        double* q = reinterpret_cast<double*>(pm);
        if (M.C == 1) partials_t<double, 1>(s, M, A, ts, first, count, g, with_up, threads, q, rates);
        else partials_t<double, 4>(s, M, A, ts, first, count, g, with_up, threads, q, rates);
    } else {
        float* q = reinterpret_cast<float*>(pm);
        if (M.C == 1) partials_t<float, 1>(s, M, A, ts, first, count, g, with_up, threads, q, rates);
        else partials_t<float, 4>(s, M, A, ts, first, count, g, with_up, threads, q, rates);
    }
}

namespace {
using PropKernel = void (*)(const PropGroup*, const int*, int, int*, Cfg, unsigned long long*, unsigned char*, size_t,
                            Geo, int, int);
using FullKernel = void (*)(const FullGroup*, const int*, int, int*, int, Cfg, unsigned long long*, unsigned char*,
                            size_t, unsigned char*, size_t, int, Geo, int, int);
// A kernel's form for a launch shape: clusters, one CTA with its table in shared
// memory, or one CTA with its table in global scratch.
template <typename R, int C>
PropKernel prop_kernel(bool clus, bool smem_tab) {
    return clus ? k_propose<R, C, true, true> : smem_tab ? k_propose<R, C, true, false> : k_propose<R, C, false, false>;
}
PropKernel prop_kernel(int prec, int C, bool clus, bool smem_tab) {
    if (prec == 0) return C == 1 ? prop_kernel<double, 1>(clus, smem_tab) : prop_kernel<double, 4>(clus, smem_tab);
    return C == 1 ? prop_kernel<float, 1>(clus, smem_tab) : prop_kernel<float, 4>(clus, smem_tab);
}
template <typename R, int C>
FullKernel full_kernel(bool clus, bool smem_tab) {
    return clus ? k_fullopt<R, C, true, true> : smem_tab ? k_fullopt<R, C, true, false> : k_fullopt<R, C, false, false>;
}
FullKernel full_kernel(int prec, int C, bool clus, bool smem_tab) {
    if (prec == 0) return C == 1 ? full_kernel<double, 1>(clus, smem_tab) : full_kernel<double, 4>(clus, smem_tab);
    return C == 1 ? full_kernel<float, 1>(clus, smem_tab) : full_kernel<float, 4>(clus, smem_tab);
}

// Resident CTAs of a kernel on the whole GPU as clusters of kp (a multiple of kp; 0:
// cannot run), or as single CTAs (kp = 1).
template <typename K>
int resident(K kern, int kp, int threads, size_t smem, int sms) {
    if (smem > kSmemPerCta || kp * ((threads + 31) / 32) > kMaxTeamWarps) return 0;
    int nb = 0;
    cudaError_t e = allow_smem(kern);
    if (e == cudaSuccess && kp == 1) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, threads, smem);
        nb *= sms;
    } else if (e == cudaSuccess) {
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(kp * 1024);
        lc.blockDim = dim3(threads);
        lc.dynamicSmemBytes = smem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kp;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        lc.attrs = at;
        lc.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&nb, kern, &lc);
        nb *= kp;
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

template <typename K, typename... A>
void launch_shape(K kern, cudaStream_t s, int kp, int threads, int grid, size_t smem, A... args) {
    allow_smem(kern);
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid / kp * kp);
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kp;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = kp > 1 ? 1 : 0;
    cudaLaunchKernelEx(&lc, kern, args...);
    ++g_launches;
}
}  // namespace

int propose_resident(int prec, int C, const Shape& h, int maxP, int sms) {
    return resident(prop_kernel(prec, C, h.kp > 1, h.smem_tab), h.kp, h.pt,
                    propose_smem_bytes(prec, C, h.smem_tab ? geo_local(maxP, h.geo, h.pt) : 0), sms);
}
int fullopt_resident(int prec, int C, const Shape& h, int maxN, int maxP, int sms) {
    return resident(full_kernel(prec, C, h.kp > 1, h.smem_tab), h.kp, h.pt,
                    fullopt_smem_bytes(prec, C, maxN, h.smem_tab ? geo_local(maxP, h.geo, h.pt) : 0, h.pt), sms);
}
int geometry_resident(int prec, int C, bool full, int K, int threads, size_t smem, int sms) {
    if (prec != 1 || C != 4) return 0;
    return full ? resident(full_kernel(prec, C, true, true), K, threads, smem, sms)
                : resident(prop_kernel(prec, C, true, true), K, threads, smem, sms);
}

void launch_propose(cudaStream_t s, int prec, int C, const PropGroup* groups, const int* gstart, int ngroups,
                    int* counter, Cfg cfg, unsigned long long* stats, const Shape& h, int grid, void* scratch,
                    size_t scratch_per_cta, int maxP, int lo, int hi) {
    launch_shape(prop_kernel(prec, C, h.kp > 1, h.smem_tab), s, h.kp, h.pt, grid,
                 propose_smem_bytes(prec, C, h.smem_tab ? geo_local(maxP, h.geo, h.pt) : 0), groups, gstart, ngroups,
                 counter, cfg, stats, reinterpret_cast<unsigned char*>(scratch), scratch_per_cta, h.geo, lo, hi);
}

void launch_fullopt(cudaStream_t s, int prec, int C, const FullGroup* groups, const int* gstart, int ngroups,
                    int* counter, int maxN, int maxP, Cfg cfg, unsigned long long* stats, const Shape& h, int grid,
                    void* scratch, size_t scratch_per_cta, void* slab, size_t slab_per_cta, int lo, int hi) {
    const int ld = h.smem_tab ? geo_local(maxP, h.geo, h.pt) : 0;
    const size_t f = full_fixed(prec, C, maxN) + (ld ? sumtable_bytes(prec, C, ld) : 0);
    launch_shape(full_kernel(prec, C, h.kp > 1, h.smem_tab), s, h.kp, h.pt, grid,
                 fullopt_smem_bytes(prec, C, maxN, ld, h.pt), groups, gstart, ngroups, counter, 2 * maxN - 2, cfg,
                 stats, reinterpret_cast<unsigned char*>(scratch), scratch_per_cta,
                 reinterpret_cast<unsigned char*>(slab), slab_per_cta, full_p_smem(prec, C, maxN, f, h.pt) ? 1 : 0,
                 h.geo, lo, hi);
}

int score_units(int P) { return (P + kScoreUnit - 1) / kScoreUnit; }

void launch_score(cudaStream_t s, int C, const FullGroup* groups, const int* gstart, int ngroups, int maxN, int maxP,
                  Cfg cfg, int t0, int t1, double* part, int sms) {
    if (t1 <= t0) return;
    const int units = score_units(maxP), S = C == 1 ? 1 : 2;
    // (in a recorded round, whose count only the device knows, by the capacity t1 - t0)
    // few trees: one unit per CTA; many: 24 warps per SM (80 registers a thread) as three
    // CTAs where their P matrices fit, else as one; two passes per CTA (a pass costs
    // several times the P matrices that each CTA makes)
    const long long tt = (long long)(t1 - t0) * units;
    const size_t smem = score_smem(C, 2 * maxN - 2);
    const int threads = tt <= 4LL * sms ? S * kScoreUnit
                        : 3 * (smem + 2048) <= (size_t)228 * 1024 ? 2 * S * kScoreUnit : 6 * S * kScoreUnit;
    const int passes = (units + threads / (S * kScoreUnit) - 1) / (threads / (S * kScoreUnit));
    const int chunks = tt <= 16LL * sms ? passes : (passes + 1) / 2;
    const bool few = threads == S * kScoreUnit;
    auto kern = C == 1 ? (few ? k_score<1, 256> : k_score<1, 768>) : (few ? k_score<4, 256> : k_score<4, 768>);
    allow_smem<1024>(kern);
    const int grid = (int)std::min<long long>((long long)(t1 - t0) * chunks, 16LL * sms);
    kern<<<grid, threads, smem, s>>>(groups, gstart, ngroups, 2 * maxN - 2, t0, t1, chunks, units, part);
    ++g_launches;
    k_score_sum<<<blocks_for(t1 - t0, 4), 128, 0, s>>>(groups, gstart, ngroups, t0, t1, units, part, cfg.prior_rate,
                                                       cfg.prior_log);
    ++g_launches;
}

size_t fullopt_slab_bytes(int prec, int C, int n, int P) {
    const size_t slots = (size_t)(2 * n - 5), rs = prec == 0 ? 8 : 4;
    return ((slots * P * 4 * C * rs + 255) & ~size_t(255)) + ((slots * P * 4 + 255) & ~size_t(255)) +
           (((size_t)(2 * n - 2) * C * 16 * rs + 255) & ~size_t(255));
}

}  // namespace pt
