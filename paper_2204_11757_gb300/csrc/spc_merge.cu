// S5-S6: the merge loop of Algorithm 1, done in parallel, and the relabelling.
//
// Algorithm 1 walks the edges in ascending (f, eid) order and merges the two super-nodes of
// an edge unless they are already one, until n_c super-nodes remain.  Because the keys
// (f, eid) are all distinct, that loop is Kruskal's algorithm stopped after n - n_c successful
// merges: the merging edges are exactly the n - n_c lightest edges of the (unique) minimum
// spanning forest, and the partition is the components of those edges.  So:
//   1. Boruvka rounds build the minimum spanning forest: every component picks its lightest
//      incident edge by atomicMin on the key (two phases for 64-bit scores: the score bits,
//      then the edge id among the edges that tie), picked edges are forest edges (cut
//      property) and are united in a lock-free union-find whose roots are always the smallest
//      node id of their set; edges inside one component drop out of the work list.  Only a
//      prefix of the score order takes part: Kruskal's first n - n_c merges all lie among the
//      lightest edges, so the rounds run on the edges up to a threshold chosen from a score
//      histogram to hold about 1.5 (n - n_c) edges (on very large graphs the slab's edges are
//      first compacted into the work list); if that prefix's forest has fewer than n - n_c
//      edges, the rounds resume on the next slab, the forest found so far kept.
//   2. For one graph the forest edges are listed as they are picked, an exact radix select on
//      11-bit digits of (score, eid) finds the (n - n_c)-th lightest and every forest edge up to
//      it is united in a second union-find; for batches the forest edges are compacted in eid
//      order, radix-sorted by score and then by graph (stable, so ties stay in eid order) and the
//      first n_b - target_b of each graph are united.
//   3. Relabel: root = smallest member; flag roots, exclusive scan, id = scan[root] (Definition
//      1's super-nodes, numbered by smallest member).
// Small graphs -- one, or a batch of which every graph fits -- take these steps in one CTA each, in
// shared memory (k_select_small).
// Every retry loop is bounded (spin_limit: kSpinLimit unless the context lowered it); giving up
// sets DEV_TIMEOUT in the status word.
#include <algorithm>
#include <atomic>
#include <memory>

#include "spc_scan.cuh"

namespace spc {

namespace {

__device__ __forceinline__ int32_t ld_parent(const int32_t* parent, int32_t x) {
    return __ldcg(parent + x);
}

// find with path halving; parent pointers only ever move to an ancestor, so racing writes are
// benign.  Bounded: the chain of a forest over n nodes is shorter than kSpinLimit.  Giving up
// returns a node of the set (an ancestor of x): every index stays in range.
__device__ __forceinline__ int32_t uf_find(int32_t* parent, int32_t x, uint32_t* status) {
    const uint32_t lim = spin_limit(status);
    for (uint32_t it = 0; it < lim; ++it) {
        int32_t p = ld_parent(parent, x);
        if (p == x) return x;
        int32_t gp = ld_parent(parent, p);
        if (gp == p) return p;
        parent[x] = gp;
        x = gp;
    }
    atomicOr(status, DEV_TIMEOUT);
    return x;
}

// uf_find of several nodes at once (those whose bit of `live` is set): every step's loads are in
// flight together.  kStatic: no set is united while the walks run (a phase or kernel of its
// own), so a parent held by L1 is at worst an older ancestor and the walks read through L1
// (Boruvka's first phase over a further slab, 1 M nodes: 149 -> 48 us).
template <int N, bool kStatic>
__device__ __forceinline__ void uf_find_n(int32_t* parent, int32_t (&x)[N], unsigned live,
                                          uint32_t* status) {
    if (!live) return;
    const uint32_t lim = spin_limit(status);
    for (uint32_t it = 0; it < lim; ++it) {
        int32_t p[N], gp[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            p[i] = x[i];
            if (live >> i & 1u) p[i] = kStatic ? parent[x[i]] : ld_parent(parent, x[i]);
        }
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (p[i] == x[i]) live &= ~(1u << i);
        if (!live) return;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            gp[i] = p[i];
            if (live >> i & 1u) gp[i] = kStatic ? parent[p[i]] : ld_parent(parent, p[i]);
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if (!(live >> i & 1u)) continue;
            if (gp[i] == p[i]) live &= ~(1u << i);
            else parent[x[i]] = gp[i];
            x[i] = gp[i];
        }
        if (!live) return;
    }
    atomicOr(status, DEV_TIMEOUT);
}

// atomicMin of v into a[idx] by every active lane of the warp (all 32 lanes call it).  When
// neighbouring lanes target the same slot -- the edges of a hub component -- the lanes of each
// slot first take their minimum together and one lane issues the atomic.
// `hot` (may be null): one slot, hot->idx, whose minimum the block keeps in shared memory.
struct HotMin {
    int32_t idx;
    unsigned long long v;
};

__device__ __forceinline__ void warp_atomic_min_u64(unsigned long long* a, int32_t idx,
                                                    unsigned long long v, bool act,
                                                    HotMin* hot = nullptr) {
    const int lane = threadIdx.x & 31;
    const int32_t key = act ? idx : -1;
    const int32_t prev = __shfl_up_sync(0xffffffffu, key, 1);
    if (!__any_sync(0xffffffffu, act && lane > 0 && prev == key)) {
        if (act) {
            if (hot && idx == hot->idx) atomicMin(&hot->v, v);
            else atomicMin(a + idx, v);
        }
        return;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    if (!act) return;  // inactive lanes form their own group
    const unsigned hi = (unsigned)(v >> 32), lo = (unsigned)v;
    const unsigned hmin = __reduce_min_sync(peers, hi);
    const unsigned lmin = __reduce_min_sync(peers, hi == hmin ? lo : 0xffffffffu);
    if (lane == __ffs(peers) - 1) {
        const unsigned long long w = ((unsigned long long)hmin << 32) | lmin;
        if (hot && idx == hot->idx) atomicMin(&hot->v, w);
        else atomicMin(a + idx, w);
    }
}

__device__ __forceinline__ void warp_atomic_min_i32(int32_t* a, int32_t idx, int32_t v,
                                                    bool act) {
    const int lane = threadIdx.x & 31;
    const int32_t key = act ? idx : -1;
    const int32_t prev = __shfl_up_sync(0xffffffffu, key, 1);
    if (!__any_sync(0xffffffffu, act && lane > 0 && prev == key)) {
        if (act) atomicMin(a + idx, v);
        return;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    if (!act) return;
    const int32_t vmin = __reduce_min_sync(peers, v);
    if (lane == __ffs(peers) - 1) atomicMin(a + idx, vmin);
}

// unite the sets of a and b; the larger root is hooked below the smaller one with a CAS, so a
// root is always the smallest node id of its set.  Returns true if the sets were distinct.
__device__ __forceinline__ bool uf_unite(int32_t* parent, int32_t a, int32_t b,
                                         uint32_t* status) {
    const uint32_t lim = spin_limit(status);
    int32_t x[2] = {a, b};
    for (uint32_t it = 0; it < lim; ++it) {
        uf_find_n<2, false>(parent, x, 3u, status);
        if (x[0] == x[1]) return false;
        if (x[0] > x[1]) { int32_t t = x[0]; x[0] = x[1]; x[1] = t; }
        int32_t old = atomicCAS(parent + x[1], x[1], x[0]);
        if (old == x[1]) return true;
    }
    atomicOr(status, DEV_TIMEOUT);
    return false;
}

__global__ void k_iota(int32_t* a, int64_t n) {
    spc::pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        a[i] = (int32_t)i;
}

// Start state of the spanning-forest rounds in one launch: parent[i] = i, both parities'
// best-key slots "none", best-edge slots "none" (64-bit scores), forest flags and merge marks
// cleared, the two work-list counts zero.
__global__ void k_bv_init(int64_t n, int64_t m, int32_t* __restrict__ parent,
                          unsigned long long* __restrict__ bk0, unsigned long long* __restrict__ bk1,
                          int32_t* __restrict__ be0, int32_t* __restrict__ be1,
                          uint8_t* __restrict__ msf, uint8_t* __restrict__ merged,
                          int32_t* __restrict__ counts) {
    spc::pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = t0; i < n; i += stride) {
        parent[i] = (int32_t)i;
        bk0[i] = ~0ull;
        bk1[i] = ~0ull;
        if (be0) {
            be0[i] = INT32_MAX;
            be1[i] = INT32_MAX;
        }
    }
    for (int64_t e = t0; e <= m; e += stride) {
        msf[e] = 0;
        if (merged && e < m) merged[e] = 0;
    }
    if (t0 < 2) counts[t0] = 0;
}

template <class KT> struct MinKey;
// 64-bit scores: best_k holds the score bits, best_e the smallest edge id among the ties
template <> struct MinKey<unsigned long long> {
    static constexpr bool two_phase = true;
    __device__ static unsigned long long pack(unsigned long long k, int32_t) { return k; }
};
// 32-bit scores: one atomicMin on (score bits << 32 | edge id)
template <> struct MinKey<unsigned int> {
    static constexpr bool two_phase = false;
    __device__ static unsigned long long pack(unsigned int k, int32_t e) {
        return ((unsigned long long)k << 32) | (uint32_t)e;
    }
};

// Boruvka phase A: current roots of both ends; keep inter-component edges; lower the
// component minima.  The first Boruvka pass reads every edge directly and keeps only the
// score prefix.  Each thread takes kMkItems edges per pass (their loads overlap), and the
// survivors are appended with one global atomic per block and pass.
constexpr int kMkItems = 2;
constexpr uint32_t kNoSlab = 0xffffffffu;  // no lower bound on the score slab

// Per-graph score slabs of a batch: the first Boruvka pass keeps an edge of graph g when its
// key lies in (lo[g], tau[g]] (lo[g] all ones: no lower bound).  node_graph null: no slabs.
template <class KT>
struct GraphSlab {
    const int32_t* node_graph;
    const KT* tau;
    const KT* lo;
    __device__ __forceinline__ bool outside(int32_t u, KT k) const {
        const int32_t g = node_graph[u];
        const KT l = lo[g];
        return k > tau[g] || (l != ~KT(0) && k <= l);
    }
};

// The start of a further slab: the forest found so far (parent, forest flags) stays; the
// best-edge slots of both parities and the work-list counts are reset.
__global__ void k_bv_reinit(int64_t n, unsigned long long* __restrict__ bk0,
                            unsigned long long* __restrict__ bk1, int32_t* __restrict__ be0,
                            int32_t* __restrict__ be1, int32_t* __restrict__ counts) {
    spc::pdl_wait();
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = t0; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        bk0[i] = ~0ull;
        bk1[i] = ~0ull;
        if (be0) {
            be0[i] = INT32_MAX;
            be1[i] = INT32_MAX;
        }
    }
    if (t0 < 2) counts[t0] = 0;
}

constexpr int kSlItems = 16;  // consecutive edges a thread takes when it lists a slab's edges
constexpr int64_t kSlabListMin = int64_t{1} << 25;

template <class KT>
__global__ void __launch_bounds__(kThreads)
k_bv_minkey(int round0, int direct, int64_t m, const int32_t* __restrict__ in_count,
            const int32_t* __restrict__ wi_e, const int32_t* __restrict__ wi_u,
            const int32_t* __restrict__ wi_v, const int32_t* __restrict__ eu,
            const int32_t* __restrict__ ev, const KT* __restrict__ key, GraphSlab<KT> gs,
            int32_t* parent, unsigned long long* best_k, int32_t* wo_e, int32_t* wo_u,
            int32_t* wo_v, int32_t* out_count, uint32_t* status) {
    spc::pdl_wait();
    __shared__ int32_t sh_wsum[kThreads / 32];
    __shared__ int32_t sh_base;
    const int64_t cnt = round0 ? m : (int64_t)*in_count;
    const int64_t per = (int64_t)blockDim.x * kMkItems;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t base = (int64_t)blockIdx.x * per; base < cnt; base += (int64_t)gridDim.x * per) {
        int32_t e[kMkItems], u[kMkItems], v[kMkItems];
        bool in[kMkItems];
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            const int64_t i = base + (int64_t)it * blockDim.x + threadIdx.x;
            in[it] = i < cnt;
            e[it] = 0; u[it] = 0; v[it] = 0;
            if (in[it]) {
                if (round0) { e[it] = (int32_t)i; u[it] = eu[i]; v[it] = ev[i]; }
                else { e[it] = wi_e[i]; u[it] = wi_u[i]; v[it] = wi_v[i]; }
            }
        }
        KT k[kMkItems];
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            k[it] = in[it] ? key[e[it]] : KT(0);
            if (round0 && in[it] && gs.node_graph && gs.outside(u[it], k[it])) in[it] = false;
        }
        int32_t ru[kMkItems], rv[kMkItems];
        int32_t nkeep = 0;
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            // direct: the selection's first round, every node still its own component (four walks
            // together cost registers: 1.56 -> 2.13 ms over the launches of 2,500 meshes)
            ru[it] = in[it] ? (direct ? u[it] : uf_find(parent, u[it], status)) : 0;
            rv[it] = in[it] ? (direct ? v[it] : uf_find(parent, v[it], status)) : 0;
            in[it] = in[it] && ru[it] != rv[it];
            const unsigned long long pk = MinKey<KT>::pack(k[it], e[it]);
            warp_atomic_min_u64(best_k, ru[it], pk, in[it]);
            warp_atomic_min_u64(best_k, rv[it], pk, in[it]);
            nkeep += in[it] ? 1 : 0;
        }
        // block-wide exclusive prefix of the survivors, one global atomic per block and pass
        int32_t incl = nkeep;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) sh_wsum[warp] = incl;
        __syncthreads();
        if (threadIdx.x == 0) {
            int32_t tot = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
                const int32_t t = sh_wsum[w];
                sh_wsum[w] = tot;
                tot += t;
            }
            sh_base = tot ? atomicAdd(out_count, tot) : 0;
        }
        __syncthreads();
        int32_t slot = sh_base + sh_wsum[warp] + incl - nkeep;
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            if (in[it]) {
                wo_e[slot] = e[it];
                wo_u[slot] = ru[it];
                wo_v[slot] = rv[it];
                ++slot;
            }
        }
        __syncthreads();
    }
}


// The last Boruvka rounds in one CTA.  Once the work list holds at most kFinishMax items (the
// last rounds of a large level; every round of a small one) a round is a few microseconds of
// work and three launches; here one CTA of kFinishThreads runs every remaining round, its
// phases separated by block barriers: the lowering of the component minima (as k_bv_minkey,
// the survivors compacted into the other list through a shared-memory counter), the tie-break
// by edge id for 64-bit scores (as k_bv_tiebreak), the hook (as k_bv_hook).  Each component's
// lightest edge is unique, so the forest does not depend on the order of the lists.
// round0: the first round reads the edges directly (e = i, u = eu[i], v = ev[i]) with the
// score-prefix filter, like k_bv_minkey's first round.
constexpr int kFinishMax = 16384;
constexpr int kFinishThreads = 1024;

template <class KT>
__global__ void __launch_bounds__(kFinishThreads, 1)
k_bv_finish(int round0, int par0, int64_t m, int32_t* count_in, int32_t* li_e, int32_t* li_u,
            int32_t* li_v, int32_t* lo_e, int32_t* lo_u, int32_t* lo_v,
            const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
            const KT* __restrict__ key, GraphSlab<KT> gs, int32_t* parent,
            unsigned long long* bk0, unsigned long long* bk1, int32_t* be0, int32_t* be1,
            uint8_t* msf, uint32_t* status) {
    spc::pdl_wait();
    __shared__ int32_t sh_cnt[2];
    int64_t cnt = round0 ? m : (int64_t)*count_in;
    int par = par0;
    int32_t *ie = li_e, *iu = li_u, *iv = li_v, *oe = lo_e, *ou = lo_u, *ov = lo_v;
    for (int r = 0; cnt > 0; ++r) {
        if (r >= 64) {  // every round at least halves the components that still have edges
            if (threadIdx.x == 0) atomicOr(status, DEV_TIMEOUT);
            break;
        }
        unsigned long long* bk = par ? bk1 : bk0;
        unsigned long long* bk_next = par ? bk0 : bk1;
        int32_t* be = par ? be1 : be0;
        int32_t* be_next = par ? be0 : be1;
        if (threadIdx.x == 0) sh_cnt[0] = 0;
        __syncthreads();
        // lower the component minima; keep the edges between two components
        for (int64_t i = threadIdx.x; i < cnt; i += kFinishThreads) {
            int32_t e, u, v;
            if (round0 && r == 0) { e = (int32_t)i; u = eu[i]; v = ev[i]; }
            else { e = ie[i]; u = iu[i]; v = iv[i]; }
            const KT k = key[e];
            if (round0 && r == 0 && gs.node_graph && gs.outside(u, k)) continue;
            const int32_t ru = uf_find(parent, u, status), rv = uf_find(parent, v, status);
            if (ru == rv) continue;
            const unsigned long long pk = MinKey<KT>::pack(k, e);
            atomicMin(bk + ru, pk);
            atomicMin(bk + rv, pk);
            const int32_t slot = atomicAdd(&sh_cnt[0], 1);
            oe[slot] = e;
            ou[slot] = ru;
            ov[slot] = rv;
        }
        __syncthreads();
        const int32_t kept = sh_cnt[0];
        if (MinKey<KT>::two_phase) {  // among equal scores, the smallest edge id
            for (int32_t i = threadIdx.x; i < kept; i += kFinishThreads) {
                const int32_t e = oe[i], ru = ou[i], rv = ov[i];
                const unsigned long long k = (unsigned long long)key[e];
                if (k == bk[ru]) atomicMin(be + ru, e);
                if (k == bk[rv]) atomicMin(be + rv, e);
            }
            __syncthreads();
        }
        // hook the picked edges; clear the next round's slots of these components
        for (int32_t i = threadIdx.x; i < kept; i += kFinishThreads) {
            const int32_t e = oe[i], ru = ou[i], rv = ov[i];
            bool picked;
            if (MinKey<KT>::two_phase) {
                picked = be[ru] == e || be[rv] == e;
                be_next[ru] = INT32_MAX;
                be_next[rv] = INT32_MAX;
            } else {
                picked = (int32_t)(uint32_t)bk[ru] == e || (int32_t)(uint32_t)bk[rv] == e;
            }
            bk_next[ru] = ~0ull;
            bk_next[rv] = ~0ull;
            if (picked) {
                msf[e] = 1;
                uf_unite(parent, ru, rv, status);
            }
        }
        __syncthreads();
        cnt = kept;
        par ^= 1;
        int32_t* t;
        t = ie; ie = oe; oe = t;
        t = iu; iu = ou; ou = t;
        t = iv; iv = ov; ov = t;
    }
}

// The score prefix's bins: 512 to a binade, 64 binades up to 2, the largest score there is (smaller
// scores share bin 0, larger ones -- a caller's own -- the last bin).  The 15 highest bits of a
// binary64 score gave 16 bins to a binade, and a level's scores lie within one or two: the first
// prefix of the 129^3 mesh held 5.5 M edges instead of the 1.6 M asked for, its selection took 2.1
// ms instead of 0.8 and the seven levels 19.8 instead of 18.4.
constexpr int kTauBins = 32768;

template <class KT>
__device__ __forceinline__ uint32_t tau_bin(KT k) {
    constexpr int kShift = sizeof(KT) == 8 ? 43 : 14;
    constexpr KT kTwo = sizeof(KT) == 8 ? (KT)0x4000000000000000ull : (KT)0x40000000u;
    constexpr KT kBase = (kTwo >> kShift) - (kTauBins - 1);
    const KT b = k >> kShift;
    return b <= kBase ? 0u : b - kBase >= (KT)kTauBins ? kTauBins - 1 : (uint32_t)(b - kBase);
}

// histogram of the scores' bins, per block in shared memory, over a sample of the keys: one chunk
// of kHistChunk consecutive keys in every 2^samp (samp 0: every key).  The threshold it gives only
// sizes the score prefix, never changes a result.
constexpr int kHistChunk = 256;

template <class KT>
__global__ void __launch_bounds__(1024)
k_key_hist(int64_t m, const KT* __restrict__ key, int samp,
           uint32_t* __restrict__ hist) {
    spc::pdl_wait();
    extern __shared__ uint32_t sh_hist[];
    for (int b = threadIdx.x; b < kTauBins; b += blockDim.x) sh_hist[b] = 0;
    __syncthreads();
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = ((v / kHistChunk) << samp) * kHistChunk + v % kHistChunk;
        if (i >= m) break;  // i grows with v
        const uint32_t b = tau_bin(key[i]);
        const unsigned peers = __match_any_sync(__activemask(), b);
        if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&sh_hist[b], __popc(peers));
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kTauBins; b += blockDim.x)
        if (sh_hist[b]) atomicAdd(hist + b, sh_hist[b]);
}

// inclusive scan of x over the block (blockDim.x a multiple of 32, at most 1024), by warp
// shuffles and one pass over the warp totals; ws: 32 words of shared memory.  All threads call
// it; ws may be reused after it returns.
__device__ __forceinline__ unsigned long long block_incl_scan(unsigned long long x,
                                                               unsigned long long* ws) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
        unsigned long long y = lane < nw ? ws[lane] : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long z = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += z;
        }
        ws[lane] = y;
    }
    __syncthreads();
    const unsigned long long r = x + (w ? ws[w - 1] : 0ull);
    __syncthreads();
    return r;
}

// Boruvka phase B (64-bit scores only): among the edges whose score equals the component
// minimum, keep the smallest edge id.
__global__ void __launch_bounds__(kThreads)
k_bv_tiebreak(const int32_t* __restrict__ count, const int32_t* __restrict__ wl_e,
              const int32_t* __restrict__ wl_u, const int32_t* __restrict__ wl_v,
              const unsigned long long* __restrict__ key, const unsigned long long* best_k,
              int32_t* best_e) {
    spc::pdl_wait();
    const int64_t cnt = *count;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x; i0 < cnt;
         i0 += (int64_t)gridDim.x * blockDim.x) {  // uniform per warp: the helpers need it
        const int64_t i = i0 + threadIdx.x;
        const bool act = i < cnt;
        int32_t e = 0, ru = 0, rv = 0;
        unsigned long long k = 0;
        if (act) {
            e = wl_e[i]; ru = wl_u[i]; rv = wl_v[i];
            k = key[e];
        }
        warp_atomic_min_i32(best_e, ru, e, act && k == best_k[ru]);
        warp_atomic_min_i32(best_e, rv, e, act && k == best_k[rv]);
    }
}

// Boruvka phase C: an edge picked by either end is a forest edge; unite.  Also clears the
// other parity's minima at both ends, ready for the next round (the roots that next round
// touches are all ends of this round's work list).
template <class KT>
__global__ void __launch_bounds__(kThreads)
k_bv_hook(const int32_t* __restrict__ count, const int32_t* __restrict__ wl_e,
          const int32_t* __restrict__ wl_u, const int32_t* __restrict__ wl_v,
          const unsigned long long* __restrict__ best_k, const int32_t* __restrict__ best_e,
          unsigned long long* other_k, int32_t* other_e, int32_t* parent, uint8_t* msf,
          int32_t* spent_count, uint32_t* status) {
    spc::pdl_wait();
    // this round's input count is read by nobody after phase A: zero it here, it is the
    // next round's output count
    if (blockIdx.x == 0 && threadIdx.x == 0) *spent_count = 0;
    const int64_t cnt = *count;
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x; i0 < cnt;
         i0 += (int64_t)gridDim.x * blockDim.x) {  // uniform per warp
        const int64_t i = i0 + threadIdx.x;
        const bool act = i < cnt;
        int32_t e = 0, ru = -1, rv = -1;
        if (act) { e = wl_e[i]; ru = wl_u[i]; rv = wl_v[i]; }
        // a slot shared with the previous lane (a hub component) is cleared by that lane
        const int32_t pu = __shfl_up_sync(0xffffffffu, ru, 1);
        const int32_t pv = __shfl_up_sync(0xffffffffu, rv, 1);
        if (!act) continue;
        const bool clr_u = lane == 0 || pu != ru, clr_v = lane == 0 || pv != rv;
        bool picked;
        if (MinKey<KT>::two_phase) {
            picked = best_e[ru] == e || best_e[rv] == e;
            if (clr_u) other_e[ru] = INT32_MAX;
            if (clr_v) other_e[rv] = INT32_MAX;
        } else {
            picked = (int32_t)(uint32_t)best_k[ru] == e || (int32_t)(uint32_t)best_k[rv] == e;
        }
        if (clr_u) other_k[ru] = ~0ull;
        if (clr_v) other_k[rv] = ~0ull;
        if (picked) {
            msf[e] = 1;
            uf_unite(parent, ru, rv, status);
        }
    }
}

// forest edges -> (score key, eid) list in eid order
template <class KT>
__global__ void __launch_bounds__(kThreads)
k_compact_msf(int64_t m, const uint8_t* __restrict__ msf, const int32_t* __restrict__ pos,
              const KT* __restrict__ key, KT* __restrict__ out_k, uint32_t* __restrict__ out_v) {
    spc::pdl_wait();
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        if (msf[e]) {
            const int32_t q = pos[e];
            out_k[q] = key[e];
            out_v[q] = (uint32_t)e;
        }
    }
}

// graph id of every node of a block-diagonal batch
__global__ void k_node_graph(int64_t n, int64_t B, const int64_t* __restrict__ graph_ptr,
                             int32_t* __restrict__ node_graph) {
    spc::pdl_wait();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = B;  // largest b with graph_ptr[b] <= x
        while (hi - lo > 1) {
            int64_t mid = (lo + hi) >> 1;
            if (graph_ptr[mid] <= x) lo = mid; else hi = mid;
        }
        node_graph[x] = (int32_t)lo;
    }
}

// second sort key for batches: graph of the edge's smaller end point
__global__ void k_graph_keys(const int32_t* __restrict__ count, const uint32_t* __restrict__ eids,
                             const int32_t* __restrict__ eu, const int32_t* __restrict__ node_graph,
                             uint32_t* __restrict__ gkey) {
    spc::pdl_wait();
    const int64_t cnt = *count;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (int64_t)gridDim.x * blockDim.x)
        gkey[i] = (uint32_t)node_graph[eu[eids[i]]];
}

// ---- per-graph score prefixes of a batch ------------------------------------------------
// Graphs of a batch are disjoint, so each one's Kruskal merges are the lightest forest edges
// of any prefix of its own scores whose forest holds them (the argument of the single-graph
// prefix, graph by graph).  Each graph's first slab is its lightest 1.5 (n_b - n_c,b) keys;
// a graph whose forest falls short takes the next slab of twice as many keys.  One CTA per
// graph finds the threshold with two histogram passes over its keys (2048 bins each: the 11
// highest value bits, then the next 11 among the keys of the chosen bin), so the slab's top
// is exact up to its low bits (they are all included).
constexpr int kGpThreads = 256;
constexpr int kGpBins = 2048;
template <class KT> struct GpShift;
template <> struct GpShift<unsigned int> { static constexpr int s1 = 20, s2 = 9; };
template <> struct GpShift<unsigned long long> { static constexpr int s1 = 52, s2 = 41; };

// the first bin whose running count over hist reaches `need` (1 <= need <= total); also the
// count before it.  Every thread of the block calls it.
__device__ void cta_find_bin(const uint32_t* hist, int64_t need, int* bin_out,
                             int64_t* before_out) {
    __shared__ unsigned long long s_part[32];
    __shared__ int s_bin;
    __shared__ long long s_before;
    const int kPer = kGpBins / (int)blockDim.x;  // blocks of 256, 512 or 1024 threads
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    unsigned long long loc = 0;
    for (int j = 0; j < kPer; ++j) loc += hist[t * kPer + j];
    unsigned long long incl = loc;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_part[w] = incl;
    if (t == 0) s_bin = kGpBins - 1;
    __syncthreads();
    // (the counts of one graph's edges: below 2^31)
    const unsigned base = __reduce_add_sync(0xffffffffu, lane < w ? (unsigned)s_part[lane] : 0u);
    unsigned long long run = base + incl - loc;  // count before this thread's bins
    if (run < (unsigned long long)need && run + loc >= (unsigned long long)need) {
        for (int j = 0; j < kPer; ++j) {
            const uint32_t c = hist[t * kPer + j];
            if (run + c >= (unsigned long long)need) {
                s_bin = t * kPer + j;
                s_before = (long long)run;
                break;
            }
            run += c;
        }
    }
    __syncthreads();
    *bin_out = s_bin;
    *before_out = s_before;
    __syncthreads();
}

// the smallest threshold t (its low s2 bits all set) with at least `need` keys of key[e0, e1)
// at or below it, and (unless null) their number; 1 <= need <= e1 - e0.  Every thread of the block
// calls it.
template <class KT>
__device__ KT cta_select_key(const KT* __restrict__ key, int64_t e0, int64_t e1, int64_t need,
                             uint32_t* hist, int64_t* below = nullptr) {
    constexpr int S1 = GpShift<KT>::s1, S2 = GpShift<KT>::s2;
    constexpr int kB = 8;  // keys per thread in flight (one CTA may walk a large graph)
    const int64_t step = (int64_t)blockDim.x * kB;
    for (int i = threadIdx.x; i < kGpBins; i += blockDim.x) hist[i] = 0u;
    __syncthreads();
    for (int64_t b0 = e0 + threadIdx.x; b0 < e1; b0 += step) {
        KT k[kB];
#pragma unroll
        for (int q = 0; q < kB; ++q) {
            const int64_t e = b0 + (int64_t)q * blockDim.x;
            k[q] = e < e1 ? key[e] : KT(0);
        }
#pragma unroll
        for (int q = 0; q < kB; ++q)
            if (b0 + (int64_t)q * blockDim.x < e1)
                atomicAdd(&hist[(uint32_t)(k[q] >> S1) & (kGpBins - 1)], 1u);
    }
    __syncthreads();
    int c1;
    int64_t before;
    cta_find_bin(hist, need, &c1, &before);
    for (int i = threadIdx.x; i < kGpBins; i += blockDim.x) hist[i] = 0u;
    __syncthreads();
    for (int64_t b0 = e0 + threadIdx.x; b0 < e1; b0 += step) {
        KT k[kB];
#pragma unroll
        for (int q = 0; q < kB; ++q) {
            const int64_t e = b0 + (int64_t)q * blockDim.x;
            k[q] = e < e1 ? key[e] : KT(0);
        }
#pragma unroll
        for (int q = 0; q < kB; ++q)
            if (b0 + (int64_t)q * blockDim.x < e1 && (int)(k[q] >> S1) == c1)
                atomicAdd(&hist[(uint32_t)(k[q] >> S2) & (kGpBins - 1)], 1u);
    }
    __syncthreads();
    int c2;
    int64_t before2;
    cta_find_bin(hist, need - before, &c2, &before2);
    if (below) *below = before + before2 + hist[c2];
    return ((KT)c1 << S1) | ((KT)c2 << S2) | (((KT)1 << S2) - 1);
}

// attempt 0: every graph's first slab [0, tau]; later attempts: a graph whose forest (the
// forest flags of its edge range) holds fewer than its n_b - n_c,b merges, and whose slab does
// not yet reach its last key, takes the next slab (old tau, new tau] of twice the keys (and
// counts into *n_short); every other graph an empty slab.
template <class KT>
__global__ void __launch_bounds__(kGpThreads)
k_graph_prefix(int64_t B, int attempt, const int64_t* __restrict__ graph_ptr,
               const int32_t* __restrict__ up_ptr, const int64_t* __restrict__ targets,
               const KT* __restrict__ key, const uint8_t* __restrict__ msf,
               int64_t* __restrict__ need, KT* __restrict__ tau, KT* __restrict__ lo,
               int32_t* n_short) {
    spc::pdl_wait();
    __shared__ uint32_t hist[kGpBins];
    __shared__ int s_short;
    __shared__ unsigned long long s_sum[kGpThreads / 32];
    constexpr KT kAll = ~KT(0);
    for (int64_t b = blockIdx.x; b < B; b += gridDim.x) {
        const int64_t n0 = graph_ptr[b], n1 = graph_ptr[b + 1];
        const int64_t e0 = up_ptr[n0], e1 = up_ptr[n1], mb = e1 - e0;
        const int64_t k_b = (n1 - n0) - targets[b] > 0 ? (n1 - n0) - targets[b] : 0;
        int64_t nd;
        if (attempt == 0) {
            nd = k_b + k_b / 2;
            if (threadIdx.x == 0) lo[b] = k_b == 0 ? KT(0) : kAll;
        } else {
            // the forest edges of this graph so far
            unsigned long long f = 0;
            for (int64_t b0 = e0 + threadIdx.x; b0 < e1; b0 += (int64_t)blockDim.x * 8) {
                uint8_t fl[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int64_t e = b0 + (int64_t)q * blockDim.x;
                    fl[q] = e < e1 ? msf[e] : 0;
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) f += fl[q] ? 1 : 0;
            }
            for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
            if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = f;
            __syncthreads();
            if (threadIdx.x == 0) {
                unsigned long long tot = 0;
                for (int i = 0; i < kGpThreads / 32; ++i) tot += s_sum[i];
                s_short = ((int64_t)tot < k_b && need[b] < mb) ? 1 : 0;
                lo[b] = tau[b];  // done up to the old top: the next slab starts above it
            }
            __syncthreads();
            if (!s_short) continue;  // empty slab (tau, tau]
            nd = 2 * need[b];
            if (threadIdx.x == 0) atomicAdd(n_short, 1);
        }
        if (k_b == 0) {
            if (threadIdx.x == 0) { tau[b] = KT(0); need[b] = 0; }  // empty slab (0, 0]
        } else if (nd >= mb) {
            if (threadIdx.x == 0) { tau[b] = kAll; need[b] = mb; }   // every key
        } else {
            const KT t = cta_select_key<KT>(key, e0, e1, nd, hist);
            if (threadIdx.x == 0) { tau[b] = t; need[b] = nd; }
        }
        __syncthreads();
    }
}


// per graph: first forest edge position and the number of merges k_b = n_b - target_b
__global__ void k_graph_segments(int64_t B, const int64_t* __restrict__ graph_ptr,
                                 const int64_t* __restrict__ targets,
                                 const int32_t* __restrict__ up_ptr,
                                 const int32_t* __restrict__ msf_pos, int32_t* __restrict__ seg_start,
                                 int32_t* __restrict__ k_graph) {
    spc::pdl_wait();
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < B;
         b += (int64_t)gridDim.x * blockDim.x) {
        seg_start[b] = msf_pos[up_ptr[graph_ptr[b]]];
        const int64_t nb = graph_ptr[b + 1] - graph_ptr[b];
        int64_t k = nb - targets[b];
        k_graph[b] = (int32_t)(k < 0 ? 0 : k);
    }
}

// unite the ends of the first k forest edges of every graph (sorted by score)
__global__ void __launch_bounds__(kThreads)
k_select_unite(const int32_t* __restrict__ count, const uint32_t* __restrict__ eids,
               const uint32_t* __restrict__ gkey, const int32_t* __restrict__ seg_start,
               const int32_t* __restrict__ k_graph, const int32_t* __restrict__ eu,
               const int32_t* __restrict__ ev, int32_t* parent,
               uint8_t* merged, uint32_t* status) {
    spc::pdl_wait();
    const int64_t cnt = *count;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t b = gkey[i];
        if (i - seg_start[b] < k_graph[b]) {
            const int32_t e = (int32_t)eids[i];
            uf_unite(parent, eu[e], ev[e], status);
            if (merged) merged[e] = 1;
        }
    }
}

// ---- exact selection of the k lightest forest edges (single graph) ------------------------------
// Composite key (score bits, eid) is unique.  Round r histograms an 11-bit digit (most
// significant first: the score's digits, then the eid's) over the items whose earlier digits
// match the ones picked so far.  The last block of a round to finish (ticket counter after a
// fence) picks that round's digit -- the bin holding the remaining rank -- and stores it with
// the rank left inside the bin, for the next round.
constexpr int kSelBits = 11;
constexpr int kSelBins = 1 << kSelBits;

template <class KT> struct SelBits {
    static constexpr int kKeyBits = sizeof(KT) == 8 ? 63 : 31;  // sign bit always clear
    static constexpr int kHiRounds = (kKeyBits + kSelBits - 1) / kSelBits;
    static constexpr int kRounds = kHiRounds + 3;                 // eid: 32 bits = 11 + 11 + 10
};

// digit r of (hi, lo) and its width
template <class KT>
__device__ __forceinline__ uint32_t sel_digit(KT hi, uint32_t lo, int r) {
    constexpr int H = SelBits<KT>::kHiRounds, KB = SelBits<KT>::kKeyBits;
    if (r < H) {
        const int top = KB - kSelBits * r;                 // exclusive upper bit of digit r
        const int lowb = top - kSelBits > 0 ? top - kSelBits : 0;
        return (uint32_t)(hi >> lowb) & ((1u << (top - lowb)) - 1u);
    }
    const int q = r - H;
    const int top = 32 - kSelBits * q;
    const int lowb = top - kSelBits > 0 ? top - kSelBits : 0;
    return (lo >> lowb) & ((1u << (top - lowb)) - 1u);
}

// ---- the merge selection of small graphs, one CTA per graph --------------------------------------
// The whole selection of one graph -- score slabs, spanning-forest rounds, the k lightest forest
// edges, the second union-find and the numbering inside the graph -- with the union-find and the
// components' best edges in shared memory.  A graph of a few thousand nodes has too little work per
// round for the whole GPU: every grid barrier or launch costs more than the round's work, while a
// batch keeps an SM per graph busy.  Shared memory bounds it (random 8-byte slots, compare-and-swap
// on them, walks).  2,500 graphs of 200 to 19,881 nodes, binary32, a call of three levels: 19.7 ms
// with the launches of select_batch over all graphs at once, 17.0 so; one graph of 4,096 nodes and
// 12,033 edges down to a half (a sixteenth): 129 (144) us in k_select_coop, 52 (91) here.
template <class KT>
struct SmallArgs {
    int64_t n, m, target;         // one graph: graph_ptr null
    const int64_t* graph_ptr;     // a batch: block b takes graph b when n_min < its nodes <= n_max
    const int64_t* targets;
    const int32_t* up_ptr;
    int32_t n_min, n_max;
    int32_t bytes;                // dynamic shared memory
    const int32_t* eu;
    const int32_t* ev;
    const KT* key;
    unsigned long long* lk;       // scratch for live edges that do not fit into shared memory: keys
    int32_t* le;                  // (32-bit ones with the edge's place below), places (64-bit keys)
    uint32_t* lp;                 // and two 16-bit ends
    KT* fk;                       // scratch: the forest edges' keys and ids
    uint32_t* fe;
    int32_t* lift;                // super-node of every node, counted from 0 in its graph
    uint8_t* merged;
    int32_t* n_c;                 // super-nodes of every graph
    uint32_t* status;
};

// One CTA's limits: edges that one SM reads in a few tens of us, and nodes that fit into 203 KB of
// shared memory (the rest is L1's); 1,024 threads on an SM whatever the class: four CTAs of 256,
// two of 512, one of 1,024.  What the nodes leave of a CTA's shared memory holds the live edges.
// One graph alone leaves the other SMs idle here, and comes only while its work is small: up to
// kSmallOne nodes, and at most kSmallWork of nodes and edges, where an edge counts up to four times
// for every merge wanted (the slabs stop there), or halved at best and at most kSmallHalved edges
// (one slab of few rounds).  64-bit scores cost a pass more per round.  Whole replayed calls here /
// in k_select_coop, binary32: 2,100 nodes and 6,300 edges to a sixteenth 258 / 306 us; 8,192 nodes
// and 24,576 edges to a half 304 / 409, to a sixteenth 450 / 455; binary64, 8,192 nodes and 32,768
// edges to a sixteenth 698 / 501.  Over 948 calls of 800 to 8,192 nodes, 4 to 60 entries a row, three
// weight types, targets from a half to one super-node, this choice loses 1.1 % to the better way of
// each; all of them here would lose 5.8 %, none of them 11.8 %.
constexpr int64_t kSmallOne = 8192;
template <class KT>
constexpr int64_t kSmallWork = MinKey<KT>::two_phase ? 14000 : 20000;
constexpr int64_t kSmallHalved = 30000;
constexpr int kSmallEdgeBits = 17;
constexpr int64_t kSmallEdges = int64_t{1} << kSmallEdgeBits;
constexpr int kSmallBytes[3] = {54 * 1024, 110 * 1024, 203 * 1024};
// A batch's graphs of up to kTinyNodes nodes, when at least kTinyMin of them make up for the launch,
// take CTAs of two warps, 16 on an SM (with four CTAs of 256 threads a graph of a few nodes held a
// quarter of an SM for 8 us).  Whole replayed calls, the launches over all graphs at once / CTAs of 256 /
// these: 10^5 graphs of 20 to 50 nodes, one level, binary32, 3.43 / 3.66 / 2.28 ms; 10^5 of 3 to 11
// 1.53 / 2.02 / 1.14; up to 128 nodes here, 4 10^4 graphs of 50 to 119 2.80 / 2.64 / 3.34 (2.55 with 64).
constexpr int kTinyNodes = 64;
constexpr int kTinyBytes = 12 * 1024;
constexpr int64_t kTinyMin = 1000;
template <class KT>
struct SmallMem {
    // best slot, 16-bit parent and (64-bit scores) best edge of every node
    static constexpr int kNode = 8 + 2 + (MinKey<KT>::two_phase ? 4 : 0);
    static constexpr int kItem = 8 + 4 + (MinKey<KT>::two_phase ? 4 : 0);  // of a live edge
    static constexpr int kFixed = kGpBins * 4;
    static constexpr int nodes(int bytes) { return (bytes - kFixed) / kNode / 4 * 4; }
    static constexpr int kMaxNodes = nodes(kSmallBytes[2]);
};
static_assert(SmallMem<unsigned int>::kMaxNodes < 65536 &&
                  SmallMem<unsigned long long>::kMaxNodes >= kSmallOne,
              "16-bit ends and parents; one graph fits");

// union-find in shared memory, as uf_find_n and uf_unite above (bounded; giving up returns a node
// of the set)
template <int N>
__device__ __forceinline__ void sm_find_n(volatile uint16_t* par, int32_t (&x)[N], unsigned live,
                                          uint32_t lim, uint32_t* status) {
    for (uint32_t it = 0; it < lim; ++it) {
        int32_t p[N];
#pragma unroll
        for (int i = 0; i < N; ++i) p[i] = (live >> i & 1u) ? (int32_t)par[x[i]] : x[i];
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (p[i] == x[i]) live &= ~(1u << i);
        if (!live) return;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if (!(live >> i & 1u)) continue;
            const int32_t gp = par[p[i]];
            if (gp == p[i]) live &= ~(1u << i);
            else par[x[i]] = (uint16_t)gp;
            x[i] = gp;
        }
        if (!live) return;
    }
    atomicOr(status, DEV_TIMEOUT);
}

__device__ __forceinline__ bool sm_unite(uint16_t* par, int32_t a, int32_t b, uint32_t lim,
                                         uint32_t* status) {
    int32_t x[2] = {a, b};
    for (uint32_t it = 0; it < lim; ++it) {
        sm_find_n<2>(par, x, 3u, lim, status);
        if (x[0] == x[1]) return false;
        if (x[0] > x[1]) {
            const int32_t t = x[0];
            x[0] = x[1];
            x[1] = t;
        }
        if (atomicCAS(par + x[1], (uint16_t)x[1], (uint16_t)x[0]) == x[1]) return true;
    }
    atomicOr(status, DEV_TIMEOUT);
    return false;
}

// atomicMin that first looks (the slot of a component with many edges is rarely lowered)
__device__ __forceinline__ void sm_min(unsigned long long* a, unsigned long long v) {
    if (v < *reinterpret_cast<volatile unsigned long long*>(a)) atomicMin(a, v);
}

constexpr int kSmallFlight = 4;  // live edges of a thread in flight
// Up to kSmallAll edges a graph's first slab is all of them (the two histogram passes of a threshold
// cost more), and up to kSmallRank forest edges the k lightest are found by comparing each with all:
// 2 10^4 graphs of 20 to 50 nodes, one level, binary32, replayed: 1,343 -> 875 us, 8,000 of 50 to 119
// 855 -> 692.
constexpr int kSmallAll = 512;
constexpr int kSmallRank = 256;

template <class KT, int T>
__global__ void __launch_bounds__(T, 1024 / T) k_select_small(SmallArgs<KT> a) {
    spc::pdl_wait();
    constexpr bool two = MinKey<KT>::two_phase;
    constexpr int H = SelBits<KT>::kHiRounds, P = kSmallFlight;
    extern __shared__ unsigned long long sm_raw[];
    __shared__ int32_t s_forest, s_live;
    __shared__ int32_t s_max[2];
    __shared__ int32_t s_sum[T / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lim = spin_limit(a.status);
    const int64_t b = blockIdx.x;
    const int64_t n0 = a.graph_ptr ? a.graph_ptr[b] : 0;
    const int64_t n1 = a.graph_ptr ? a.graph_ptr[b + 1] : a.n;
    const int32_t nb = (int32_t)(n1 - n0), first = (int32_t)n0;
    if (nb <= a.n_min || nb > a.n_max) return;  // another class's graph
    const int64_t e0 = a.graph_ptr ? a.up_ptr[n0] : 0, e1 = a.graph_ptr ? a.up_ptr[n1] : a.m;
    const int32_t mb = (int32_t)(e1 - e0);
    const int64_t k_b = nb - (a.graph_ptr ? a.targets[b] : a.target);
    const int32_t k = k_b > 0 ? (int32_t)k_b : 0;
    const int32_t nm = (nb + 3) / 4 * 4;
    const int32_t cap = (a.bytes - SmallMem<KT>::kFixed - nm * SmallMem<KT>::kNode) /
                        SmallMem<KT>::kItem;
    unsigned long long* best = sm_raw;                               // [nm] best slots
    unsigned long long* sk = best + nm;                              // [cap] live edges: lk, lp, le
    uint32_t* hist = reinterpret_cast<uint32_t*>(sk + cap);          // [kGpBins]
    uint32_t* sp = hist + kGpBins;                                   // [cap]
    int32_t* se = reinterpret_cast<int32_t*>(sp + cap);              // [cap] when two
    int32_t* beste = se + (two ? cap : 0);                           // [nm] when two
    uint16_t* par = reinterpret_cast<uint16_t*>(beste + (two ? nm : 0));  // [nm]
    const KT* __restrict__ key = a.key + e0;
    const int32_t* __restrict__ eu = a.eu + e0;
    const int32_t* __restrict__ ev = a.ev + e0;
    KT* fk = a.fk + e0;
    uint32_t* fe = a.fe + e0;
    for (int32_t x = tid; x < nb; x += T) {
        par[x] = (uint16_t)x;
        best[x] = ~0ull;
        if (two) beste[x] = INT32_MAX;
    }
    if (a.merged)
        for (int32_t e = tid; e < mb; e += T) a.merged[e0 + e] = 0;
    if (tid == 0) {
        s_forest = 0;
        s_live = 0;
        s_max[0] = 0;
        s_max[1] = 0;
    }
    __syncthreads();
    // ---- forest: slabs of 1.5 k keys, then twice as many, until the forest holds k edges
    int32_t forest = 0;
    int64_t need = (int64_t)k + k / 2, taken = 0;  // taken: keys at or below lo
    KT lo = 0;
    bool above = false;  // the slab starts above lo
    // 32-bit keys: every round's entries of the best slots lie below the earlier rounds', so the
    // slots need no reset (15 bits of round, 32 of key, 17 of the edge's place in its graph)
    constexpr int kTagShift = 32 + kSmallEdgeBits;
    unsigned tag = 0x7fffu;
    while (k > 0) {
        const bool all = need >= mb || mb <= kSmallAll;
        int64_t upto = mb;
        const KT tau = all ? ~KT(0) : cta_select_key<KT>(key, 0, mb, need, hist, &upto);
        // the slab's edges, listed densely: thread t takes the places t, t + T, ...
        bool shared = upto - taken <= cap;
        unsigned long long* lk = shared ? sk : a.lk + e0;
        uint32_t* lp = shared ? sp : a.lp + e0;
        int32_t* le = shared ? se : a.le + e0;
        for (int32_t w0 = warp * 32; w0 < mb; w0 += 2 * P * T) {  // warp-uniform
            KT kk[2 * P];
            unsigned in = 0;
#pragma unroll
            for (int q = 0; q < 2 * P; ++q) {
                const int32_t e = w0 + q * T + lane;
                kk[q] = e < mb ? key[e] : KT(0);
                if (e < mb && kk[q] <= tau && (!above || kk[q] > lo)) in |= 1u << q;
            }
            // the ends of every taken edge in flight: no branch between the loads
            int32_t u[2 * P], v[2 * P];
#pragma unroll
            for (int q = 0; q < 2 * P; ++q) {
                const int32_t e = in >> q & 1u ? w0 + q * T + lane : 0;
                u[q] = eu[e];
                v[q] = ev[e];
            }
            const int32_t mine = __reduce_add_sync(0xffffffffu, __popc(in));
            int32_t at = 0;
            if (lane == 0 && mine > 0) at = atomicAdd(&s_live, mine);
            at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
            for (int q = 0; q < 2 * P; ++q) {
                const bool take = in >> q & 1u;
                const unsigned lanes = __ballot_sync(0xffffffffu, take);
                const int32_t to = at + __popc(lanes & ((1u << lane) - 1u));
                at += __popc(lanes);
                if (!take) continue;
                const int32_t e = w0 + q * T + lane;
                if constexpr (two) {
                    lk[to] = kk[q];
                    le[to] = e;
                } else {
                    lk[to] = ((unsigned long long)kk[q] << kSmallEdgeBits) | (uint32_t)e;
                }
                lp[to] = (uint32_t)(u[q] - first) | ((uint32_t)(v[q] - first) << 16);
            }
        }
        __syncthreads();
        const int32_t live0 = s_live;
        int32_t cnt = (live0 - tid + T - 1) / T;
        int32_t most = (live0 + T - 1) / T;  // the longest column
        for (int round = 0;; ++round) {
            // the live edges between components lower both components' best slots
            --tag;
            const bool move = !shared && (int64_t)most * T <= cap;  // into shared memory
            unsigned long long* dk = move ? sk : lk;
            uint32_t* dp = move ? sp : lp;
            int32_t* de = move ? se : le;
            int32_t keep = 0;
            for (int32_t j0 = 0; j0 < cnt; j0 += P) {
                unsigned long long pk[P];
                int32_t e[P], x[2 * P];
                unsigned live = 0;
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const int32_t at = (j0 + q) * T + tid;
                    const bool in = j0 + q < cnt;
                    pk[q] = in ? lk[at] : 0ull;
                    e[q] = two && in ? le[at] : 0;
                    const uint32_t uv = in ? lp[at] : 0u;
                    x[2 * q] = (int32_t)(uv & 0xffffu);
                    x[2 * q + 1] = (int32_t)(uv >> 16);
                    if (in) live |= 3u << (2 * q);
                }
                // round 0 of the first slab: every node is its own component
                if (round > 0 || above) sm_find_n<2 * P>(par, x, live, lim, a.status);
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const int32_t u = x[2 * q], v = x[2 * q + 1];
                    if (u == v) continue;  // (both 0 past the end)
                    const unsigned long long t =
                        two ? pk[q] : pk[q] | (unsigned long long)tag << kTagShift;
                    sm_min(best + u, t);
                    sm_min(best + v, t);
                    const int32_t to = keep * T + tid;
                    dk[to] = pk[q];
                    if (two) de[to] = e[q];
                    dp[to] = (uint32_t)u | ((uint32_t)v << 16);
                    ++keep;
                }
            }
            cnt = keep;
            if (move) {
                shared = true;
                lk = sk;
                lp = sp;
                le = se;
            }
            const int32_t wmax = __reduce_max_sync(0xffffffffu, cnt);
            if (lane == 0 && wmax > 0) atomicMax(&s_max[round & 1], wmax);
            __syncthreads();
            most = s_max[round & 1];
            if (tid == 0) s_max[(round & 1) ^ 1] = 0;
            if (most == 0) break;
            if (round > 64) {  // every round at least halves the components that still have edges
                if (tid == 0) atomicOr(a.status, DEV_TIMEOUT);
                break;
            }
            if constexpr (two) {  // the smallest edge id among the ties
                for (int32_t j = 0; j < cnt; ++j) {
                    const int32_t at = j * T + tid;
                    const uint32_t uv = lp[at];
                    const int32_t e = le[at], u = (int32_t)(uv & 0xffffu), v = (int32_t)(uv >> 16);
                    const unsigned long long pk = lk[at];
                    if (best[u] == pk) atomicMin(beste + u, e);
                    if (best[v] == pk) atomicMin(beste + v, e);
                }
                __syncthreads();
            }
            // the chosen edges are forest edges
            for (int32_t j0 = 0; j0 < cnt; j0 += P) {
                unsigned long long pk[P];
                int32_t e[P];
                uint32_t uv[P];
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const int32_t at = (j0 + q) * T + tid;
                    const bool in = j0 + q < cnt;
                    pk[q] = in ? lk[at] : 0ull;
                    e[q] = two && in ? le[at] : (int32_t)(pk[q] & (kSmallEdges - 1));
                    uv[q] = in ? lp[at] : 0u;
                }
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    if (uv[q] == 0u) continue;  // two components: not both 0
                    const int32_t u = (int32_t)(uv[q] & 0xffffu), v = (int32_t)(uv[q] >> 16);
                    bool pick;
                    if constexpr (two) {
                        pick = (best[u] == pk[q] && beste[u] == e[q]) ||
                               (best[v] == pk[q] && beste[v] == e[q]);
                    } else {
                        const unsigned long long t = pk[q] | (unsigned long long)tag << kTagShift;
                        pick = best[u] == t || best[v] == t;
                    }
                    if (pick && sm_unite(par, u, v, lim, a.status)) {
                        const int32_t at_f = atomicAdd(&s_forest, 1);
                        fk[at_f] = two ? (KT)pk[q] : (KT)(pk[q] >> kSmallEdgeBits);
                        fe[at_f] = (uint32_t)e[q];
                    }
                }
            }
            __syncthreads();
            if constexpr (two) {
                for (int32_t j = 0; j < cnt; ++j) {
                    const uint32_t uv = lp[j * T + tid];
                    const int32_t u = (int32_t)(uv & 0xffffu), v = (int32_t)(uv >> 16);
                    best[u] = ~0ull;
                    best[v] = ~0ull;
                    beste[u] = INT32_MAX;
                    beste[v] = INT32_MAX;
                }
                __syncthreads();
            }
        }
        forest = s_forest;
        if (forest >= k || all) break;
        lo = tau;
        taken = upto;
        above = true;
        need *= 2;
        __syncthreads();  // every thread has read s_forest and s_max
        if (tid == 0) {
            s_live = 0;
            s_max[0] = 0;
            s_max[1] = 0;
        }
        __syncthreads();
    }
    __syncthreads();
    if (forest > k && forest <= (T < kSmallRank ? T : kSmallRank)) {
        // ---- the k lightest of few: every forest edge's rank by comparison
        KT* rk = reinterpret_cast<KT*>(hist);
        uint32_t* re = hist + kSmallRank * (sizeof(KT) / 4);
        if (tid < forest) {
            rk[tid] = fk[tid];
            re[tid] = fe[tid];
        }
        for (int32_t x = tid; x < nb; x += T) par[x] = (uint16_t)x;
        __syncthreads();
        if (tid < forest) {
            const KT x = rk[tid];
            const uint32_t y = re[tid];
            int32_t rank = 0;
#pragma unroll 4
            for (int32_t i = 0; i < forest; ++i)
                rank += rk[i] < x || (rk[i] == x && re[i] < y) ? 1 : 0;
            if (rank < k) {
                sm_unite(par, eu[y] - first, ev[y] - first, lim, a.status);
                if (a.merged) a.merged[e0 + y] = 1;
            }
        }
    } else if (forest > k) {
        // ---- the k lightest: the key digits of the k-th, most significant first, until all items
        // that share them are wanted
        KT hi = 0;
        uint32_t low = 0;
        int64_t rest = k;
        int r = 0;
        for (;; ++r) {
            for (int i = tid; i < kSelBins; i += T) hist[i] = 0u;
            __syncthreads();
            const int top = r < H ? SelBits<KT>::kKeyBits - kSelBits * r : 32 - kSelBits * (r - H);
            const int lowb = top - kSelBits > 0 ? top - kSelBits : 0;
#pragma unroll 4
            for (int32_t i = tid; i < forest; i += T) {
                const KT x = fk[i];
                const uint32_t y = fe[i];
                const bool same = r < H ? (r == 0 || (x >> top) == hi)
                                        : x == hi && (r == H || (y >> top) == low);
                if (same) atomicAdd(hist + sel_digit<KT>(x, y, r), 1u);
            }
            __syncthreads();
            int bin;
            int64_t before;
            cta_find_bin(hist, rest, &bin, &before);
            rest -= before;
            const bool whole = (int64_t)hist[bin] == rest;
            if (r < H) hi = (KT)((hi << (top - lowb)) | (KT)bin);
            else low = (low << (top - lowb)) | (uint32_t)bin;
            __syncthreads();
            if (whole || r == SelBits<KT>::kRounds - 1) break;
        }
        for (int32_t x = tid; x < nb; x += T) par[x] = (uint16_t)x;
        __syncthreads();
        const int top = r < H ? SelBits<KT>::kKeyBits - kSelBits * r : 32 - kSelBits * (r - H);
        const int lowb = top - kSelBits > 0 ? top - kSelBits : 0;
        for (int32_t i0 = tid; i0 < forest; i0 += P * T) {
            KT x[P];
            uint32_t y[P];
            int32_t u[P], v[P];
            bool in[P];
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int32_t i = i0 + q * T < forest ? i0 + q * T : 0;
                x[q] = fk[i];
                y[q] = fe[i];
            }
#pragma unroll
            for (int q = 0; q < P; ++q) {
                in[q] = i0 + q * T < forest &&
                        (r < H ? (x[q] >> lowb) <= hi
                               : x[q] < hi || (x[q] == hi && (y[q] >> lowb) <= low));
                u[q] = eu[y[q]];
                v[q] = ev[y[q]];
                if (in[q] && a.merged) a.merged[e0 + y[q]] = 1;
            }
#pragma unroll
            for (int q = 0; q < P; ++q)
                if (in[q]) sm_unite(par, u[q] - first, v[q] - first, lim, a.status);
        }
    } else if (a.merged) {
        for (int32_t i = tid; i < forest; i += T) a.merged[e0 + fe[i]] = 1;
    }
    __syncthreads();
    // ---- numbering by smallest member: roots are their sets' smallest nodes
    int32_t* ids = reinterpret_cast<int32_t*>(best);  // [nb]
    const int32_t per = (nb + T - 1) / T;
    const int32_t x0 = tid * per < nb ? tid * per : nb, x1 = x0 + per < nb ? x0 + per : nb;
    int32_t roots = 0;
    for (int32_t x = x0; x < x1; ++x) roots += par[x] == x ? 1 : 0;
    const int32_t incl = scanf::warp_incl_scan(roots);
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int32_t t = scanf::warp_incl_scan(lane < T / 32 ? s_sum[lane] : 0);
        if (lane < T / 32) s_sum[lane] = t;
    }
    __syncthreads();
    int32_t id = (warp > 0 ? s_sum[warp - 1] : 0) + incl - roots;
    for (int32_t x = x0; x < x1; ++x) {
        const bool root = par[x] == x;
        ids[x] = root ? id : 0;
        id += root ? 1 : 0;
    }
    __syncthreads();
    for (int32_t y0 = tid; y0 < nb; y0 += P * T) {
        int32_t x[P];
        unsigned live = 0;
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const bool in = y0 + q * T < nb;
            x[q] = in ? y0 + q * T : 0;
            if (in) live |= 1u << q;
        }
        sm_find_n<P>(par, x, live, lim, a.status);
#pragma unroll
        for (int q = 0; q < P; ++q)
            if (y0 + q * T < nb) a.lift[n0 + y0 + q * T] = ids[x[q]];
    }
    if (tid == 0) a.n_c[b] = s_sum[T / 32 - 1];
}

// A pass over a batch's graphs, each with `size(b)` items (nodes, edges): one(b, i0, step) for
// i0 = the thread's first item.  A block takes one graph at a time or, of very many graphs, eight:
// a warp for each of at most kWarpGraph items, then the block for the others (5 10^5 graphs of three
// nodes, block by block, waited 0.7 and 0.3 ms in the two kernels below).  Every thread calls it.
constexpr int32_t kWarpGraph = 1024;
constexpr int64_t kGraphGroup = kThreads / 32;

template <class Size, class One>
__device__ __forceinline__ void for_graphs(int64_t B, const Size& size, const One& one) {
    __shared__ int64_t s_list[kGraphGroup];
    __shared__ int s_count;
    if (B < kGraphGroup * gridDim.x) {
        for (int64_t b = blockIdx.x; b < B; b += gridDim.x) one(b, (int32_t)threadIdx.x, kThreads);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t b0 = blockIdx.x * kGraphGroup; b0 < B; b0 += gridDim.x * kGraphGroup) {
        if (threadIdx.x == 0) s_count = 0;
        __syncthreads();
        const int64_t b = b0 + warp;
        if (b < B) {
            if (size(b) <= kWarpGraph) one(b, lane, 32);
            else if (lane == 0) s_list[atomicAdd(&s_count, 1)] = b;
        }
        __syncthreads();
        for (int i = 0; i < s_count; ++i) one(s_list[i], (int32_t)threadIdx.x, kThreads);
        __syncthreads();
    }
}

// a batch's numbering: every graph's super-nodes after those of the graphs before it
__global__ void __launch_bounds__(kThreads)
k_small_shift(int64_t B, const int64_t* __restrict__ graph_ptr, const int32_t* __restrict__ off,
              const int64_t* __restrict__ targets, int32_t* __restrict__ lift,
              int64_t* __restrict__ graph_ptr_c, int32_t* __restrict__ warn) {
    spc::pdl_wait();
    for_graphs(
        B, [&](int64_t b) { return graph_ptr[b + 1] - graph_ptr[b]; },
        [&](int64_t b, int32_t i0, int step) {
            const int32_t o = off[b];
            const int64_t n1 = graph_ptr[b + 1];
            for (int64_t x = graph_ptr[b] + i0; x < n1; x += step) lift[x] += o;
            if (i0 == 0) {
                graph_ptr_c[b] = o;
                if (b == B - 1) graph_ptr_c[B] = off[B];
                if ((int64_t)off[b + 1] - o > targets[b]) atomicOr(warn, 1);
            }
        });
}

// The shape of a batch (out zeroed before): out[0] = the most nodes, out[1] = the most edges of a
// graph, out[3] = the graphs of at most kTinyNodes nodes, out[2] != 0 when the graphs do not take
// the nodes in turn or an edge leaves its graph (such a batch is merged by the general path, which
// indexes by the whole batch's nodes).
__global__ void __launch_bounds__(kThreads)
k_batch_shape(int64_t B, int64_t n, const int64_t* __restrict__ graph_ptr,
              const int32_t* __restrict__ up_ptr, const int32_t* __restrict__ ev,
              int32_t* __restrict__ out) {
    spc::pdl_wait();
    int32_t nodes = 0, edges = 0, tiny = 0;  // of the graphs whose first item this thread takes
    bool bad = false;
    const auto in_turn = [&](int64_t b) {
        const int64_t n0 = graph_ptr[b], n1 = graph_ptr[b + 1];
        return n0 >= 0 && n1 >= n0 && n1 <= n && (b != 0 || n0 == 0) && (b != B - 1 || n1 == n);
    };
    for_graphs(
        B,
        [&](int64_t b) -> int64_t {
            return in_turn(b) ? up_ptr[graph_ptr[b + 1]] - up_ptr[graph_ptr[b]] : 0;
        },
        [&](int64_t b, int32_t first, int step) {
            if (!in_turn(b)) {
                bad = true;
                return;
            }
            const int64_t n0 = graph_ptr[b], n1 = graph_ptr[b + 1];
            const int32_t e0 = up_ptr[n0], e1 = up_ptr[n1];
            for (int64_t i0 = (int64_t)e0 + first; i0 < e1; i0 += 4 * step) {
                int32_t v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    v[q] = i0 + q * step < e1 ? ev[i0 + q * step] : (int32_t)n0;
#pragma unroll
                for (int q = 0; q < 4; ++q) bad = bad || v[q] < n0 || v[q] >= n1;
            }
            if (first == 0) {
                nodes = max(nodes, (int32_t)(n1 - n0));
                edges = max(edges, e1 - e0);
                tiny += n1 - n0 <= kTinyNodes ? 1 : 0;
            }
        });
    if (bad) out[2] = 1;
    nodes = __reduce_max_sync(0xffffffffu, nodes);
    edges = __reduce_max_sync(0xffffffffu, edges);
    tiny = __reduce_add_sync(0xffffffffu, tiny);
    if ((threadIdx.x & 31) == 0 && nodes > 0) {
        atomicMax(out, nodes);
        atomicMax(out + 1, edges);
        if (tiny) atomicAdd(out + 3, tiny);
    }
}

// k_select_small over B graphs of at most n_max nodes (tiny: of at most kTinyNodes), by classes of sizes
template <class KT, int T>
spc_status launch_small_class(spc_context* ctx, SmallArgs<KT>& a, int64_t B, int bytes) {
    a.n_max = T == 64 ? kTinyNodes : SmallMem<KT>::nodes(bytes);
    a.bytes = bytes;
    static std::atomic<unsigned long long> attr_devs{0};  // devices already set up
    const unsigned long long bit = 1ull << (ctx->device & 63);
    if (!(attr_devs.load() & bit)) {
        SPC_CUDA(cudaFuncSetAttribute(k_select_small<KT, T>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
        attr_devs.fetch_or(bit);
    }
    SPC_LAUNCH(ctx, (k_select_small<KT, T>), (unsigned)B, T, bytes, a);
    a.n_min = a.n_max;
    return SPC_OK;
}

template <class KT>
spc_status launch_small(spc_context* ctx, const GraphView& g, const KT* key, const SelectArgs& sa,
                        int64_t B, int64_t n_max, int64_t tiny, int32_t* lift, uint8_t* merged,
                        int32_t* n_c) {
    Work& W = ctx->work;
    SmallArgs<KT> a{};
    a.n = g.n;
    a.m = g.m;
    a.target = sa.target;
    a.graph_ptr = sa.d_graph_ptr;
    a.targets = sa.d_targets;
    a.up_ptr = W.up_ptr.as<int32_t>();
    a.n_min = -1;
    a.eu = W.eu.as<int32_t>();
    a.ev = W.ev.as<int32_t>();
    a.key = key;
    a.lk = W.sel_key2.as<unsigned long long>();
    a.le = W.wl_e[0].as<int32_t>();
    a.lp = W.wl_u[0].as<uint32_t>();
    a.fk = W.sel_key.as<KT>();
    a.fe = W.sel_val.as<uint32_t>();
    a.lift = lift;
    a.merged = merged;
    a.n_c = n_c;
    a.status = ctx->d_status;
    // every key read, the lift written (on the first class's launch for all of them)
    note_bytes(ctx, (double)g.m * sizeof(KT) + 4.0 * g.n);
    if (B <= ctx->num_sms)  // a graph per SM or less takes the most threads
        return launch_small_class<KT, 1024>(ctx, a, B, kSmallBytes[2]);
    const bool few = tiny < kTinyMin;  // too few tiny graphs for a launch of their own
    if (n_max <= kTinyNodes && !few) return launch_small_class<KT, 64>(ctx, a, B, kTinyBytes);
    if (!few && n_max <= SmallMem<KT>::nodes(kSmallBytes[0]))
        SPC_TRY((launch_small_class<KT, 64>(ctx, a, B, kTinyBytes)));
    if (n_max <= SmallMem<KT>::nodes(kSmallBytes[0]))
        return launch_small_class<KT, 256>(ctx, a, B, kSmallBytes[0]);
    // The smaller classes on the second stream: their CTAs fill the SMs that the largest leaves at
    // its end (2,500 graphs, the whole call: 16.77 ms one class after the other, 16.22 so).  A
    // graph's lists lie in its own edges' range, so the classes share no scratch.
    std::unique_ptr<SideBranch> side(new SideBranch(ctx));
    SPC_TRY(side->status());
    const bool three = n_max > SmallMem<KT>::nodes(kSmallBytes[1]);
    SmallArgs<KT> last = a;
    if (!few) SPC_TRY((launch_small_class<KT, 64>(ctx, a, B, kTinyBytes)));
    SPC_TRY((launch_small_class<KT, 256>(ctx, a, B, kSmallBytes[0])));
    if (three) SPC_TRY((launch_small_class<KT, 512>(ctx, a, B, kSmallBytes[1])));
    side->leave();
    last.n_min = a.n_min;
    if (three) return launch_small_class<KT, 1024>(ctx, last, B, kSmallBytes[2]);
    return launch_small_class<KT, 512>(ctx, last, B, kSmallBytes[1]);
}

// root flags (a root is its set's smallest member and its own parent)
__global__ void __launch_bounds__(kThreads)
k_roots(int64_t n, const int32_t* __restrict__ parent, int32_t* __restrict__ flag,
        int32_t* __restrict__ warn) {
    spc::pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) *warn = 0;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x)
        flag[x] = parent[x] == (int32_t)x ? 1 : 0;
}

__global__ void __launch_bounds__(kThreads)
k_lift(int64_t n, int32_t* parent, const int32_t* __restrict__ ids, int32_t* __restrict__ lift,
       uint32_t* status) {
    spc::pdl_wait();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x)
        lift[x] = ids[uf_find(parent, (int32_t)x, status)];
}

__global__ void k_graph_ptr_c(int64_t B, const int64_t* __restrict__ graph_ptr,
                              const int32_t* __restrict__ ids, const int64_t* __restrict__ targets,
                              int64_t* __restrict__ graph_ptr_c, int32_t* __restrict__ warn) {
    spc::pdl_wait();
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b <= B;
         b += (int64_t)gridDim.x * blockDim.x) {
        graph_ptr_c[b] = ids[graph_ptr[b]];
        if (b < B) {
            const int64_t nc = (int64_t)ids[graph_ptr[b + 1]] - ids[graph_ptr[b]];
            if (nc > targets[b]) atomicOr(warn, 1);
        }
    }
}

// relabel (S6) from the second union-find in W.parent2, plus per-graph offsets and the status
spc_status finish_batch(spc_context* ctx, const GraphView& g, const SelectArgs& sa, int32_t* lift,
                        int64_t* n_c_out, int64_t* graph_ptr_c, int32_t* status_out) {
    Work& W = ctx->work;
    const int64_t n = g.n;
    const int maxb = ctx->num_sms * 8;
    uint32_t* status = ctx->d_status;
    int32_t* counters = W.counters.as<int32_t>();
    int32_t* parent2 = W.parent2.as<int32_t>();
    // ---- 3. relabel ------------------------------------------------------------------
    int32_t* flag = W.flag.as<int32_t>();
    int32_t* ids = W.ids.as<int32_t>();
    int32_t* warn = counters + 2;
    SPC_LAUNCH(ctx, k_roots, grid_for(n, kThreads, maxb), kThreads, 0, n, parent2, flag, warn);
    SPC_TRY(scan_i32(ctx, flag, ids, n));
    SPC_LAUNCH(ctx, k_lift, grid_for(n, kThreads, maxb), kThreads, 0, n, parent2, ids, lift,
               status);
    SPC_LAUNCH(ctx, k_graph_ptr_c, grid_for(sa.B + 1, kThreads, maxb), kThreads, 0, sa.B,
               sa.d_graph_ptr, ids, sa.d_targets, graph_ptr_c, warn);
    int64_t vals[3];
    {
        // a walk that gave up can leave n_c in the lift: nothing may index with it
        const void* ptrs[3] = {ids + n, warn, status};
        const int bytes[3] = {4, 4, 4};
        SPC_TRY(read_vals(ctx, 3, ptrs, bytes, vals));
        const spc_status st = status_from_bits((uint32_t)vals[2]);
        if (st < 0) return st;
    }
    const int64_t n_c = vals[0];
    const int32_t warn_b = (int32_t)vals[1];
    *n_c_out = n_c;
    *status_out = warn_b != 0 ? SPC_WARN_TARGET_NOT_REACHED : SPC_OK;
    return SPC_OK;
}

// key_hist: the score-prefix histogram (kTauBins words, zero between selections), then the radix
// select's histograms of every round (zeroed by the selection); zeroed once on allocation
constexpr size_t kKeyHistBytes = (size_t)(kTauBins + SelBits<uint64_t>::kRounds * kSelBins) * 4;
static spc_status ensure_key_hist(spc_context* ctx) {
    return ensure_zeroed(ctx, ctx->work.key_hist, kKeyHistBytes);
}

// ---- the merge selection of one graph in one cooperative kernel --------------------------------
// Every phase of the selection -- Boruvka rounds on the score prefix, the prefix's extensions, the
// select of the n - n_c lightest forest edges, their union, the relabelling -- reads what the phase
// before it wrote, and most are a few microseconds of work.  As separate launches a level took
// about 35 of them and eight to twelve sizes read back by the host (10-15 us of idle GPU each).
// Here the phases are separated by grid barriers of one resident grid (a cooperative launch; every
// barrier wait is bounded), the sizes stay on the device, and the host reads the super-node count
// alone.  Forest edges are appended to a list as they are picked, so no flag per edge is kept,
// scanned or compacted; the select is order-free, because every (score, eid) is distinct.
//
// What bounds it: random accesses to parents and best slots (latency: the grid holds
// kCoopBlocks * kCoopThreads threads per SM) on large levels; on small ones chains of dependent
// L2 reads (a phase of a few hundred items takes 5-9 us) and the barriers (1.4 us each on 152 CTAs
// and more, 3-5 with the wait for the slowest).  The rounds whose work list has at most
// kCoopTail items run in one CTA, with block barriers, while the others wait.
// Against the separate launches, whole calls: 64x64 mesh 0.77 -> 0.65 ms, 257x250 mesh (6 levels)
// 3.68 -> 3.22, 129^3 mesh 22.6 -> 21.8, 2^23-point random geometric graph 23.4 -> 21.9, 10^6
// points in one level 3.89 -> 3.36; a replayed 2048^2 mesh, which reads nothing back, 9.04 -> 9.05.
// Device time of the kernel, all levels of the 2048^2 mesh, at threads x CTAs per SM: 512 x 3 2.43
// ms, 512 x 4 2.51, 512 x 2 2.64, 1024 x 1 2.66, 256 x 6 2.75.
constexpr int kCoopThreads = 512;
constexpr int kCoopBlocks = 3;           // per SM
constexpr int kCoopTail = 2 * kCoopThreads;
constexpr int kRestMax = 4096;           // candidates every CTA selects among by itself

// counters of a call, zero before it: the last CTA to leave zeroes them (and the grid the score
// histogram) for the next call, so no memset comes between the launches; kCtNc is the result
enum { kCtList0 = 0, kCtList1 = 1, kCtForest = 2, kCtCand = 3, kCtBar = 4, kCtTau = 5,
       kCtDone = 6, kCtZeroed = 7, kCtNc = 7, kCtCount = 8 };
constexpr int kCtFirst = 16;  // their place among the context's counters

template <class KT>
struct CoopArgs {
    int64_t n, m, need, k_need;  // need: edges of the first prefix; k_need = n - n_c >= 0
    const int32_t* eu;
    const int32_t* ev;
    const KT* key;
    uint32_t* hist;              // score histogram of the prefix (null: no prefix)
    int hist_samp, slab_list;
    int32_t* parent;
    int32_t* parent2;
    unsigned long long* bk[2];
    int32_t* be[2];
    int32_t* wl[2][3];           // work lists: edge, root, root
    KT* fk;                      // forest edges: key, eid
    uint32_t* fe;
    KT* ck;                      // select candidates
    uint32_t* cv;
    uint32_t* rhist;             // one histogram per select round
    int32_t* blk;                // roots per CTA
    int32_t* ids;
    int32_t* lift;
    uint8_t* merged;             // may be null
    int32_t* ct;
    uint32_t* status;
};

// every CTA of the grid waits for every other; false when the wait was given up (then every CTA
// leaves).  *bar counts arrivals, zero at launch.
__device__ bool grid_sync(uint32_t* bar, uint32_t* status) {
    __shared__ bool sh_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        bool good = true;
        if (gridDim.x > 1) {
            __threadfence();
            const uint32_t goal = (atomicAdd(bar, 1u) / gridDim.x + 1u) * gridDim.x;
            const uint32_t lim = spin_limit(status);
            uint32_t spins = 0, seen;
            do {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];"
                             : "=r"(seen)
                             : "l"(bar)
                             : "memory");
                if (seen < goal && ++spins > lim) {
                    atomicOr(status, DEV_TIMEOUT);
                    good = false;
                    break;
                }
            } while (seen < goal);
            __threadfence();
        }
        sh_ok = good;
    }
    __syncthreads();
    return sh_ok;
}

// positions for `mine` items of every thread of the block, one global atomic for the block; every
// thread calls it
__device__ __forceinline__ int32_t block_append(int32_t mine, int32_t* count) {
    __shared__ int32_t sh_w[kCoopThreads / 32];
    __shared__ int32_t sh_base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    __syncthreads();  // sh_w and sh_base of the call before have been read
    if (lane == 31) sh_w[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int32_t s = lane < kCoopThreads / 32 ? sh_w[lane] : 0;
        int32_t si = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(0xffffffffu, si, o);
            if (lane >= o) si += t;
        }
        if (lane < kCoopThreads / 32) sh_w[lane] = si - s;
        if (lane == 31) sh_base = si ? atomicAdd(count, si) : 0;
    }
    __syncthreads();
    return sh_base + sh_w[warp] + incl - mine;
}

// smallest of the 32768 bins whose cumulative count reaches `need` (the last bin when none does);
// one CTA
__device__ void coop_pick_tau(const uint32_t* hist, int64_t need, int32_t* tau) {
    constexpr int kPer = 32768 / kCoopThreads;
    __shared__ unsigned long long sh_ws[32];
    const uint4* h4 = reinterpret_cast<const uint4*>(hist) + (int64_t)threadIdx.x * (kPer / 4);
    unsigned long long loc = 0;
#pragma unroll 4
    for (int j = 0; j < kPer / 4; ++j) {
        const uint4 q = __ldcg(h4 + j);
        loc += (unsigned long long)q.x + q.y + q.z + q.w;
    }
    const unsigned long long incl = block_incl_scan(loc, sh_ws);
    unsigned long long run = incl - loc;
    if (threadIdx.x == kCoopThreads - 1 && incl < (unsigned long long)need) *tau = 32767;
    if (run < (unsigned long long)need && incl >= (unsigned long long)need) {
        for (int j = 0; j < kPer; ++j) {
            run += __ldcg(hist + (int64_t)threadIdx.x * kPer + j);
            if (run >= (unsigned long long)need) {
                *tau = threadIdx.x * kPer + j;
                break;
            }
        }
    }
}

// Boruvka phase A over the work list (kEdges: over every edge of the slab (lo, top]): current roots
// of both ends; edges between two components go to the out list and lower both minima
template <class KT, bool kEdges>
__device__ __forceinline__ void coop_minkey(const CoopArgs<KT>& a, int64_t cnt, int in, int out,
                                            bool direct, uint32_t top, uint32_t lo, int64_t bid,
                                            int64_t nblk) {
    unsigned long long* best = a.bk[in];
    int32_t* const oe = a.wl[out][0];
    int32_t* const ou = a.wl[out][1];
    int32_t* const ov = a.wl[out][2];
    // The atomics of one address serialise, and most edges of a late slab end in one giant
    // component.  Each CTA keeps the minimum of one component -- that of its first edge, most
    // likely the giant -- in shared memory and lowers the slot once.
    __shared__ HotMin sh_hot;
    __syncthreads();
    if (threadIdx.x == 0) {
        sh_hot.idx = -2;
        sh_hot.v = ~0ull;
    }
    __syncthreads();
    const int64_t per = (int64_t)kCoopThreads * kMkItems;
    for (int64_t base = bid * per; base < cnt; base += nblk * per) {
        int32_t e[kMkItems], u[kMkItems], v[kMkItems];
        bool act[kMkItems];
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            const int64_t i = base + (int64_t)it * kCoopThreads + threadIdx.x;
            act[it] = i < cnt;
            e[it] = u[it] = v[it] = 0;
            if (act[it]) {
                if (kEdges) {
                    e[it] = (int32_t)i;
                    u[it] = a.eu[i];
                    v[it] = a.ev[i];
                } else {
                    e[it] = a.wl[in][0][i];
                    u[it] = a.wl[in][1][i];
                    v[it] = a.wl[in][2][i];
                }
            }
        }
        int32_t nkeep = 0;
        KT k[kMkItems];
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) k[it] = act[it] ? a.key[e[it]] : KT(0);
        int32_t rt[2 * kMkItems];
        unsigned live = 0;
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            if (kEdges && act[it]) {
                const uint32_t bin = tau_bin(k[it]);
                act[it] = bin <= top && (lo == kNoSlab || bin > lo);
            }
            rt[2 * it] = u[it];
            rt[2 * it + 1] = v[it];
            if (act[it]) live |= 3u << (2 * it);
        }
        // direct: the first round of the selection, every node its own component
        if (!direct) uf_find_n<2 * kMkItems, true>(a.parent, rt, live, a.status);
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            u[it] = rt[2 * it];
            v[it] = rt[2 * it + 1];
            act[it] = act[it] && u[it] != v[it];
            const unsigned long long pk = MinKey<KT>::pack(k[it], e[it]);
            warp_atomic_min_u64(best, u[it], pk, act[it], &sh_hot);
            warp_atomic_min_u64(best, v[it], pk, act[it], &sh_hot);
            nkeep += act[it] ? 1 : 0;
        }
        int32_t slot = block_append(nkeep, a.ct + kCtList0 + out);
        if (threadIdx.x == 0 && sh_hot.idx < 0 && act[0]) sh_hot.idx = u[0];  // from the next pass
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            if (act[it]) {
                oe[slot] = e[it];
                ou[slot] = u[it];
                ov[slot] = v[it];
                ++slot;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh_hot.v != ~0ull) atomicMin(best + sh_hot.idx, sh_hot.v);
}

// the slab's edges as the first work list (very large selections): keys streamed, ends read only
// for the slab's edges
template <class KT>
__device__ __forceinline__ void coop_slab_list(const CoopArgs<KT>& a, uint32_t top, uint32_t lo) {
    constexpr int kVec = (int)(kSlItems * sizeof(KT) / 16);
    const int64_t per = (int64_t)kCoopThreads * kSlItems;
    for (int64_t base = (int64_t)blockIdx.x * per; base < a.m; base += (int64_t)gridDim.x * per) {
        const int64_t i0 = base + (int64_t)threadIdx.x * kSlItems;
        unsigned keep = 0;  // bit it: edge i0 + it lies in the slab
        if (i0 + kSlItems <= a.m) {
            const uint4* p = reinterpret_cast<const uint4*>(a.key + i0);
#pragma unroll
            for (int j = 0; j < kVec; ++j) {
                const uint4 q = p[j];
                KT k[16 / sizeof(KT)];
                memcpy(k, &q, 16);
#pragma unroll
                for (int t = 0; t < (int)(16 / sizeof(KT)); ++t) {
                    const uint32_t bin = tau_bin(k[t]);
                    if (bin <= top && (lo == kNoSlab || bin > lo))
                        keep |= 1u << (j * (int)(16 / sizeof(KT)) + t);
                }
            }
        } else {
            for (int it = 0; it < kSlItems && i0 + it < a.m; ++it) {
                const uint32_t bin = tau_bin(a.key[i0 + it]);
                if (bin <= top && (lo == kNoSlab || bin > lo)) keep |= 1u << it;
            }
        }
        int32_t slot = block_append(__popc(keep), a.ct + kCtList0);
        while (keep) {
            const int64_t i = i0 + __ffs(keep) - 1;
            keep &= keep - 1;
            a.wl[0][0][slot] = (int32_t)i;
            a.wl[0][1][slot] = a.eu[i];
            a.wl[0][2][slot] = a.ev[i];
            ++slot;
        }
    }
}

// phase B (64-bit scores): among the edges whose score equals the component's minimum, the
// smallest edge id
template <class KT>
__device__ __forceinline__ void coop_tiebreak(const CoopArgs<KT>& a, int64_t cnt, int par, int list,
                                              int64_t bid, int64_t nblk) {
    const int64_t stride = nblk * kCoopThreads;
    for (int64_t i0 = bid * kCoopThreads; i0 < cnt; i0 += stride) {  // uniform per warp
        const int64_t i = i0 + threadIdx.x;
        const bool act = i < cnt;
        int32_t e = 0, u = 0, v = 0;
        unsigned long long k = 0;
        if (act) {
            e = a.wl[list][0][i];
            u = a.wl[list][1][i];
            v = a.wl[list][2][i];
            k = (unsigned long long)a.key[e];
        }
        warp_atomic_min_i32(a.be[par], u, e, act && k == __ldcg(a.bk[par] + u));
        warp_atomic_min_i32(a.be[par], v, e, act && k == __ldcg(a.bk[par] + v));
    }
}

// phase C: an edge picked by either end is a forest edge: united and appended to the forest; the
// other parity's slots of both ends are cleared for the next round
template <class KT>
__device__ __forceinline__ void coop_hook(const CoopArgs<KT>& a, int64_t cnt, int par, int list,
                                          int64_t bid, int64_t nblk) {
    const int lane = threadIdx.x & 31;
    const int64_t per = (int64_t)kCoopThreads * kMkItems;
    for (int64_t base = bid * per; base < cnt; base += nblk * per) {  // uniform per block
        int32_t e[kMkItems], u[kMkItems], v[kMkItems];
        bool picked[kMkItems];
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            const int64_t i = base + (int64_t)it * kCoopThreads + threadIdx.x;
            e[it] = u[it] = v[it] = -1;
            if (i < cnt) {
                e[it] = a.wl[list][0][i];
                u[it] = a.wl[list][1][i];
                v[it] = a.wl[list][2][i];
            }
        }
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            // a slot shared with the previous lane (a hub component) is cleared by that lane
            const int32_t pu = __shfl_up_sync(0xffffffffu, u[it], 1);
            const int32_t pv = __shfl_up_sync(0xffffffffu, v[it], 1);
            picked[it] = false;
            if (e[it] < 0) continue;
            const bool clr_u = lane == 0 || pu != u[it], clr_v = lane == 0 || pv != v[it];
            if (MinKey<KT>::two_phase) {
                const int32_t bu = __ldcg(a.be[par] + u[it]), bv = __ldcg(a.be[par] + v[it]);
                picked[it] = bu == e[it] || bv == e[it];
                if (clr_u) a.be[par ^ 1][u[it]] = INT32_MAX;
                if (clr_v) a.be[par ^ 1][v[it]] = INT32_MAX;
            } else {
                const unsigned long long bu = __ldcg(a.bk[par] + u[it]),
                                         bv = __ldcg(a.bk[par] + v[it]);
                picked[it] = (int32_t)(uint32_t)bu == e[it] || (int32_t)(uint32_t)bv == e[it];
            }
            if (clr_u) a.bk[par ^ 1][u[it]] = ~0ull;
            if (clr_v) a.bk[par ^ 1][v[it]] = ~0ull;
        }
        int32_t npick = 0;
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            if (picked[it]) uf_unite(a.parent, u[it], v[it], a.status);
            npick += picked[it] ? 1 : 0;
        }
        int32_t slot = block_append(npick, a.ct + kCtForest);
        // a forest has fewer than m edges unless a union-find walk gave up (reported)
#pragma unroll
        for (int it = 0; it < kMkItems; ++it) {
            if (picked[it] && (int64_t)slot < a.m) {
                a.fk[slot] = a.key[e[it]];
                a.fe[slot] = (uint32_t)e[it];
                ++slot;
            }
        }
    }
}

// Every node's parent its root, between phases.  On graphs without locality the trees of a round's
// unions are deep, and all walks of the next phase run down them at once, before any has shortened
// the way for the others; one walk per node first leaves the phase walks of one step.  Before a
// further slab it costs no barrier (the slots are reset then); between the rounds of a slab one, so
// there only while the round's edges outnumber half the nodes, and up to kFlattenNodes nodes (a
// random graph of 10^6 nodes gains nothing).  The kernel, without / with, binary32: random graphs of
// 10^5 nodes and 6 10^5 edges to n/2 752 -> 505 us, to n/16 1,546 -> 830, to n/256 1,561 -> 763; 3 10^4
// nodes to n/16 450 -> 311; 10^5 points to n/16 754 -> 606; meshes and halved point sets unchanged.
constexpr int64_t kFlattenNodes = int64_t{1} << 18;

template <class KT>
__device__ __forceinline__ void coop_flatten(const CoopArgs<KT>& a, int64_t t0, int64_t stride) {
    for (int64_t i = t0; i < a.n; i += stride)
        a.parent[i] = uf_find(a.parent, (int32_t)i, a.status);
}

// histogram of digit r over the items whose digits 0 .. r-1 are dig[0 .. r-1], into sh_h
template <class KT>
__device__ __forceinline__ void coop_digit_hist(int r, int64_t n, const KT* keys,
                                                const uint32_t* vals, const uint32_t* dig,
                                                uint32_t* sh_h, int64_t bid, int64_t nblk) {
    for (int b = threadIdx.x; b < kSelBins; b += kCoopThreads) sh_h[b] = 0;
    __syncthreads();
    for (int64_t i0 = bid * kCoopThreads; i0 < n; i0 += nblk * kCoopThreads) {
        const int64_t i = i0 + threadIdx.x;
        bool match = i < n;
        uint32_t d = 0;
        if (match) {
            const KT hi = keys[i];
            const uint32_t lo = vals[i];
            for (int q = 0; q < r; ++q) match = match && sel_digit<KT>(hi, lo, q) == dig[q];
            d = sel_digit<KT>(hi, lo, r);
        }
        // candidates often share their digits (exactly equal scores)
        const unsigned peers = __match_any_sync(0xffffffffu, match ? d : 0xffffffffu);
        if (match && (int)(threadIdx.x & 31) == __ffs(peers) - 1)
            atomicAdd(&sh_h[d], (uint32_t)__popc(peers));
    }
    __syncthreads();
}

// the bin of h that holds rank *need (1-based): dig = the bin, *need = the rank inside it.  Every
// thread of the CTA calls it; h is shared or global memory.
__device__ __forceinline__ void coop_pick_bin(const uint32_t* h, uint32_t* dig,
                                              unsigned long long* need) {
    constexpr int kPer = kSelBins / kCoopThreads;
    __shared__ unsigned long long sh_ws[32];
    uint32_t c[kPer];
    unsigned long long loc = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        c[j] = *(const volatile uint32_t*)(h + threadIdx.x * kPer + j);
        loc += c[j];
    }
    const unsigned long long incl = block_incl_scan(loc, sh_ws);
    const unsigned long long want = *need;
    unsigned long long run = incl - loc;
    __syncthreads();  // every thread has read *need
    if (run < want && incl >= want) {
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            if (run < want && run + c[j] >= want) {
                *dig = (uint32_t)(threadIdx.x * kPer + j);
                *need = want - run;
                run = want;  // picked
            } else {
                run += c[j];
            }
        }
    }
    __syncthreads();
}

template <class KT>
__global__ void __launch_bounds__(kCoopThreads, kCoopBlocks)
k_select_coop(const __grid_constant__ CoopArgs<KT> a) {
    spc::pdl_wait();
    __shared__ uint32_t sh_h[kSelBins];
    __shared__ uint32_t sh_dig[16];
    __shared__ unsigned long long sh_need;
    const int64_t nblk = gridDim.x, bid = blockIdx.x;
    const int64_t t0 = bid * kCoopThreads + threadIdx.x, stride = nblk * kCoopThreads;
    uint32_t* const bar = reinterpret_cast<uint32_t*>(a.ct + kCtBar);
    const bool two = MinKey<KT>::two_phase;
    // ---- start state; the first prefix's threshold ------------------------------------------
    const bool forest = a.k_need > 0;  // else nothing merges
    for (int64_t i = t0; i < a.n; i += stride) {
        a.parent2[i] = (int32_t)i;
        if (forest) {
            a.parent[i] = (int32_t)i;
            a.bk[0][i] = ~0ull;
            a.bk[1][i] = ~0ull;
            if (two) {
                a.be[0][i] = INT32_MAX;
                a.be[1][i] = INT32_MAX;
            }
        }
    }
    if (a.merged)
        for (int64_t e = t0; e < a.m; e += stride) a.merged[e] = 0;
    for (int64_t i = t0; i < SelBits<KT>::kRounds * kSelBins; i += stride) a.rhist[i] = 0;
    bool prefix = a.hist != nullptr;
    int64_t need = a.need;
    if (forest && prefix && bid == nblk - 1)
        coop_pick_tau(a.hist, (need + (int64_t{1} << a.hist_samp) - 1) >> a.hist_samp,
                      a.ct + kCtTau);
    if (!grid_sync(bar, a.status)) return;
    int64_t n_msf = 0;
    if (forest) {
        uint32_t lo = kNoSlab;
        for (int attempt = 0; attempt < 64; ++attempt) {
            const uint32_t top = prefix ? (uint32_t)__ldcg(a.ct + kCtTau) : 0xffffffffu;
            // ---- Boruvka rounds on the slab (lo, top] -------------------------------------
            bool edges = true;
            if (a.slab_list && (prefix || lo != kNoSlab)) {
                coop_slab_list(a, top, lo);
                if (!grid_sync(bar, a.status)) return;
                edges = false;
            }
            int in = 0;
            for (int round = 0; round < 64; ++round) {
                const int out = in ^ 1;
                if (edges && round == 0)
                    coop_minkey<KT, true>(a, a.m, in, out, attempt == 0, top, lo, bid, nblk);
                else
                    coop_minkey<KT, false>(a, __ldcg(a.ct + in), in, out,
                                           attempt == 0 && round == 0, top, lo, bid, nblk);
                if (!grid_sync(bar, a.status)) return;
                int64_t cnt = __ldcg(a.ct + out);
                if (cnt == 0) break;
                if (two) {
                    coop_tiebreak(a, cnt, in, out, bid, nblk);
                    if (!grid_sync(bar, a.status)) return;
                }
                coop_hook(a, cnt, in, out, bid, nblk);
                if (t0 == 0) a.ct[in] = 0;  // the next round's out list
                if (cnt <= kCoopTail) {
                    // the remaining rounds in the first CTA
                    if (!grid_sync(bar, a.status)) return;
                    if (bid == 0) {
                        int ti = out;
                        for (int tr = 0; tr < 64; ++tr) {
                            const int to = ti ^ 1;
                            coop_minkey<KT, false>(a, cnt, ti, to, false, top, lo, 0, 1);
                            __threadfence_block();
                            __syncthreads();
                            cnt = __ldcg(a.ct + to);
                            if (cnt == 0) break;
                            if (two) {
                                coop_tiebreak(a, cnt, ti, to, 0, 1);
                                __syncthreads();
                            }
                            coop_hook(a, cnt, ti, to, 0, 1);
                            __syncthreads();
                            if (threadIdx.x == 0) a.ct[ti] = 0;
                            __threadfence_block();
                            __syncthreads();
                            ti = to;
                        }
                    }
                    break;
                }
                if (!grid_sync(bar, a.status)) return;
                if (a.n <= kFlattenNodes && cnt * 2 > a.n) {
                    coop_flatten(a, t0, stride);
                    if (!grid_sync(bar, a.status)) return;
                }
                in = out;
            }
            if (!grid_sync(bar, a.status)) return;
            // the prefix's forest holds Kruskal's first n_msf merges: enough at n - n_c
            n_msf = __ldcg(a.ct + kCtForest);
            if (n_msf > a.m) n_msf = a.m;
            if (!prefix || n_msf >= a.k_need) break;
            // the next slab: twice the edges, or, when the forest came within 15 % of n - n_c,
            // the prefix its yield so far extrapolates to, and a quarter more
            int64_t next = need * 2;
            if (n_msf * 20 >= a.k_need * 17) {
                const int64_t est =
                    (int64_t)((double)need * (double)a.k_need / (double)n_msf * 1.25);
                const int64_t least = est > need + need / 8 ? est : need + need / 8;
                next = least < next ? least : next;
            }
            need = next;
            if (need >= a.m) prefix = false;  // the last slab: every remaining score
            lo = top;
            for (int64_t i = t0; i < a.n; i += stride) {
                a.parent[i] = uf_find(a.parent, (int32_t)i, a.status);  // (coop_flatten)
                a.bk[0][i] = ~0ull;
                a.bk[1][i] = ~0ull;
                if (two) {
                    a.be[0][i] = INT32_MAX;
                    a.be[1][i] = INT32_MAX;
                }
            }
            if (t0 == 0) {
                a.ct[kCtList0] = 0;
                a.ct[kCtList1] = 0;
            }
            if (prefix && bid == nblk - 1)
                coop_pick_tau(a.hist, (need + (int64_t{1} << a.hist_samp) - 1) >> a.hist_samp,
                              a.ct + kCtTau);
            if (!grid_sync(bar, a.status)) return;
        }
        // ---- the (n - n_c)-th smallest (score, eid) of the forest, by 11-bit digits -----------
        constexpr int R = SelBits<KT>::kRounds, H = SelBits<KT>::kHiRounds,
                      KB = SelBits<KT>::kKeyBits;
        const bool all = a.k_need >= n_msf;
        if (!all) {
            // rounds over the whole forest: 22 bits of a binary32 score, 33 of a binary64 one
            // leave few candidates
            constexpr int kFull = sizeof(KT) == 8 ? 3 : 2;
            if (threadIdx.x < 16) sh_dig[threadIdx.x] = 0;
            if (threadIdx.x == 0) sh_need = (unsigned long long)a.k_need;
            __syncthreads();
            const KT* keys = a.fk;
            const uint32_t* vals = a.fe;
            int64_t items = n_msf;
            for (int r = 0; r < R; ++r) {
                if (r == kFull) {
                    // the items still matching
                    for (int64_t i0 = bid * kCoopThreads; i0 < n_msf; i0 += stride) {
                        const int64_t i = i0 + threadIdx.x;
                        KT hi = 0;
                        uint32_t lw = 0;
                        bool keep = i < n_msf;
                        if (keep) {
                            hi = a.fk[i];
                            lw = a.fe[i];
                            for (int q = 0; q < kFull; ++q)
                                keep = keep && sel_digit<KT>(hi, lw, q) == sh_dig[q];
                        }
                        const int32_t slot = block_append(keep ? 1 : 0, a.ct + kCtCand);
                        if (keep) {
                            a.ck[slot] = hi;
                            a.cv[slot] = lw;
                        }
                    }
                    if (!grid_sync(bar, a.status)) return;
                    keys = a.ck;
                    vals = a.cv;
                    items = __ldcg(a.ct + kCtCand);
                }
                if (r >= kFull && items <= kRestMax) {  // every CTA by itself
                    coop_digit_hist(r, items, keys, vals, sh_dig, sh_h, 0, 1);
                    coop_pick_bin(sh_h, sh_dig + r, &sh_need);
                } else {
                    coop_digit_hist(r, items, keys, vals, sh_dig, sh_h, bid, nblk);
                    uint32_t* const gh = a.rhist + r * kSelBins;
                    for (int b = threadIdx.x; b < kSelBins; b += kCoopThreads)
                        if (sh_h[b]) atomicAdd(gh + b, sh_h[b]);
                    if (!grid_sync(bar, a.status)) return;
                    coop_pick_bin(gh, sh_dig + r, &sh_need);
                }
            }
        }
        KT thi = ~KT(0);
        uint32_t tlo = ~0u;
        if (!all) {
            thi = 0;
            tlo = 0;
            for (int q = 0; q < H; ++q) {
                const int hb = KB - kSelBits * q;
                thi |= (KT)sh_dig[q] << (hb - kSelBits > 0 ? hb - kSelBits : 0);
            }
            for (int q = 0; q < 3; ++q) {
                const int hb = 32 - kSelBits * q;
                tlo |= sh_dig[H + q] << (hb - kSelBits > 0 ? hb - kSelBits : 0);
            }
        }
        for (int64_t i = t0; i < n_msf; i += stride) {
            const KT hi = a.fk[i];
            const uint32_t lw = a.fe[i];
            if (hi < thi || (hi == thi && lw <= tlo)) {
                uf_unite(a.parent2, a.eu[lw], a.ev[lw], a.status);
                if (a.merged) a.merged[lw] = 1;
            }
        }
        if (!grid_sync(bar, a.status)) return;
    }
    // ---- relabel: each CTA a contiguous range of nodes ------------------------------------------
    const int64_t span = (a.n + nblk - 1) / nblk;
    const int64_t x0 = bid * span < a.n ? bid * span : a.n;
    const int64_t x1 = x0 + span < a.n ? x0 + span : a.n;
    int32_t roots = 0;
    for (int64_t x = x0 + threadIdx.x; x < x1; x += kCoopThreads)
        roots += __ldcg(a.parent2 + x) == (int32_t)x ? 1 : 0;
    roots = __reduce_add_sync(0xffffffffu, roots);
    if (threadIdx.x == 0) sh_dig[0] = 0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && roots) atomicAdd(&sh_dig[0], (uint32_t)roots);
    __syncthreads();
    if (threadIdx.x == 0) a.blk[bid] = (int32_t)sh_dig[0];
    if (!grid_sync(bar, a.status)) return;
    int32_t before = 0;
    for (int64_t c = threadIdx.x; c < bid; c += kCoopThreads) before += __ldcg(a.blk + c);
    before = __reduce_add_sync(0xffffffffu, before);
    if (threadIdx.x == 0) sh_dig[0] = 0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && before) atomicAdd(&sh_dig[0], (uint32_t)before);
    __syncthreads();
    __shared__ unsigned long long sh_ws[32];
    unsigned long long run = sh_dig[0];
    for (int64_t b = x0; b < x1; b += kCoopThreads) {
        const int64_t x = b + threadIdx.x;
        const bool root = x < x1 && __ldcg(a.parent2 + x) == (int32_t)x;
        const unsigned long long incl = block_incl_scan(root ? 1ull : 0ull, sh_ws);
        if (root) a.ids[x] = (int32_t)(run + incl - 1);
        if (threadIdx.x == kCoopThreads - 1) sh_need = incl;
        __syncthreads();
        run += sh_need;
        __syncthreads();
    }
    if (bid == nblk - 1 && threadIdx.x == 0) a.ct[kCtNc] = (int32_t)run;
    if (!grid_sync(bar, a.status)) return;
    // Shallow trees (a target of n / 8 or more): four walks of a thread together (4 M nodes halved:
    // 29 -> 17 us).  A small target leaves deep trees under giant components: one walk at a time,
    // past L1, each shortened by the walks before it (1 M nodes to n / 256: 128 us; four together
    // 200, and through L1, where nobody sees another SM's shortening, 270-560).
    if ((a.n - a.k_need) * 8 < a.n) {
        for (int64_t x = t0; x < a.n; x += stride)
            a.lift[x] = __ldcg(a.ids + uf_find(a.parent2, (int32_t)x, a.status));
    } else {
        for (int64_t x = t0; x < a.n; x += 4 * stride) {
            int32_t r[4];
            unsigned live = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                r[i] = (int32_t)(x + i * stride);
                if (x + i * stride < a.n) live |= 1u << i;
            }
            uf_find_n<4, true>(a.parent2, r, live, a.status);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (x + i * stride < a.n) a.lift[x + i * stride] = __ldcg(a.ids + r[i]);
        }
    }
    if (a.hist)
        for (int64_t i = t0; i < kTauBins; i += stride) a.hist[i] = 0u;
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(a.ct + kCtDone, 1) == (int32_t)nblk - 1)
        for (int i = 0; i < kCtZeroed; ++i) a.ct[i] = 0;  // every other CTA has left its barriers
}

// whether one graph of n nodes and m edges that wants k merges is selected in one CTA
template <class KT>
bool one_cta(int64_t n, int64_t m, int64_t k) {
    if (n > kSmallOne || m > kSmallEdges) return false;
    return std::min(m, 4 * k) + n <= kSmallWork<KT> || (2 * k <= n + 1 && m <= kSmallHalved);
}

// one cooperative grid that the device holds at once, at most one CTA per kCoopThreads * 2 items
template <class KT>
spc_status select_single(spc_context* ctx, const GraphView& g, const KT* key, int64_t target,
                         int32_t* lift, uint8_t* merged, int64_t* n_c_out, int32_t* status_out) {
    Work& W = ctx->work;
    const int64_t n = g.n, m = g.m;
    const int64_t k_need = n - target > 0 ? n - target : 0;
    if (one_cta<KT>(n, m, k_need)) {
        SelectArgs sa;
        sa.target = target;
        int32_t* nc = W.counters.as<int32_t>() + 4;
        SPC_TRY(launch_small<KT>(ctx, g, key, sa, 1, n, 0, lift, merged, nc));
        int64_t vals[2];
        const void* ptrs[2] = {nc, ctx->d_status};
        const int bytes[2] = {4, 4};
        SPC_TRY(read_vals(ctx, 2, ptrs, bytes, vals));
        const spc_status st = status_from_bits((uint32_t)vals[1]);
        if (st < 0) return st;
        *n_c_out = vals[0];
        *status_out = vals[0] > target ? SPC_WARN_TARGET_NOT_REACHED : SPC_OK;
        return SPC_OK;
    }
    CoopArgs<KT> a{};
    a.n = n;
    a.m = m;
    a.k_need = k_need;
    a.need = a.k_need + a.k_need / 2;
    a.eu = W.eu.as<int32_t>();
    a.ev = W.ev.as<int32_t>();
    a.key = key;
    // the threshold's histogram samples one key chunk in eight on large selections
    a.hist_samp = m >= (int64_t{1} << 22) ? 3 : 0;
    a.slab_list = m >= kSlabListMin && (reinterpret_cast<uintptr_t>(key) & 15) == 0 ? 1 : 0;
    a.parent = W.parent.as<int32_t>();
    a.parent2 = W.parent2.as<int32_t>();
    for (int i = 0; i < 2; ++i) {
        a.bk[i] = W.best_k[i].as<unsigned long long>();
        a.be[i] = W.best_e[i].as<int32_t>();
        a.wl[i][0] = W.wl_e[i].as<int32_t>();
        a.wl[i][1] = W.wl_u[i].as<int32_t>();
        a.wl[i][2] = W.wl_v[i].as<int32_t>();
    }
    a.fk = W.sel_key.as<KT>();
    a.fe = W.sel_val.as<uint32_t>();
    a.ck = W.sel_key2.as<KT>();
    a.cv = W.sel_val2.as<uint32_t>();
    a.ids = W.ids.as<int32_t>();
    a.lift = lift;
    a.merged = merged;
    a.ct = W.counters.as<int32_t>() + kCtFirst;
    a.status = ctx->d_status;
    SPC_TRY(ensure_key_hist(ctx));
    a.rhist = W.key_hist.as<uint32_t>() + kTauBins;
    static std::atomic<int> per_sm[64];  // resident CTAs per SM, by device (0: not asked yet)
    std::atomic<int>& occ = per_sm[ctx->device & 63];
    int bps = occ.load();
    if (bps == 0) {
        SPC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_select_coop<KT>,
                                                               kCoopThreads, 0));
        SPC_CUDA(cudaFuncSetAttribute(k_key_hist<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      kTauBins * 4));
        if (bps < 1) return SPC_ERR_CUDA;
        occ.store(bps);
    }
    const int64_t big = n > m ? n : m;
    const int grid = grid_for(big, kCoopThreads * 2, ctx->num_sms * bps);
    SPC_TRY(ensure(ctx, W.sel_blk, (size_t)(ctx->num_sms * bps) * 4));
    a.blk = W.sel_blk.as<int32_t>();
    SPC_TRY(clean_selection(ctx));
    W.sel_dirty = true;
    if (m > 65536 && a.k_need > 0 && a.need < m) {
        a.hist = W.key_hist.as<uint32_t>();
        note_bytes(ctx, (double)m * sizeof(KT) / (double)(1 << a.hist_samp));
        SPC_LAUNCH(ctx, k_key_hist<KT>, ctx->num_sms, 1024, kTauBins * 4, m, key, a.hist_samp,
                   W.key_hist.as<uint32_t>());
    }
    // every key read, the first slab's ends read, parents and lift written
    note_bytes(ctx, (double)m * sizeof(KT) + 8.0 * (double)(a.need < m ? a.need : m) + 8.0 * n);
    SPC_LAUNCH_COOP(ctx, k_select_coop<KT>, grid, kCoopThreads, a);
    int64_t vals[2];
    {
        // a barrier wait that was given up leaves the lift unwritten: nothing may index with it
        const void* ptrs[2] = {a.ct + kCtNc, ctx->d_status};
        const int bytes[2] = {4, 4};
        SPC_TRY(read_vals(ctx, 2, ptrs, bytes, vals));
        const spc_status st = status_from_bits((uint32_t)vals[1]);
        if (st < 0) return st;
    }
    W.sel_dirty = false;
    *n_c_out = vals[0];
    *status_out = vals[0] > target ? SPC_WARN_TARGET_NOT_REACHED : SPC_OK;
    return SPC_OK;
}

// A batch: every graph its own score prefix and target; the spanning-forest rounds run over the
// whole batch, one set of launches per round.
template <class KT>
spc_status select_batch(spc_context* ctx, const GraphView& g, const KT* key, const SelectArgs& sa,
                        int32_t* lift, uint8_t* merged, int64_t* n_c_out, int64_t* graph_ptr_c,
                        int32_t* status_out) {
    Work& W = ctx->work;
    const int64_t n = g.n, m = g.m;
    const int maxb = ctx->num_sms * 8;
    uint32_t* status = ctx->d_status;
    int32_t* parent = W.parent.as<int32_t>();
    int32_t* counters = W.counters.as<int32_t>();  // [0..1] work-list counts, [2] warn flag
    constexpr bool two = MinKey<KT>::two_phase;
    // Every graph small: one CTA each, and no slabs or sorts over all of them.  Whole calls below /
    // here, binary32 (binary64): 4 meshes of three levels 1.22 / 0.76 ms (1.36 / 0.78), 400 meshes
    // 4.39 / 4.00 (5.18 / 4.64), 400 to a sixteenth at once 2.86 / 2.69 (2.93 / 2.83), two random
    // geometric graphs of 12,000 nodes 1.56 / 0.96 (1.76 / 1.11).
    {
        int32_t* shape = counters + 24;  // [5]: k_batch_shape's four, the warn flag
        SPC_CUDA(cudaMemsetAsync(shape, 0, 5 * sizeof(int32_t), ctx->stream));
        SPC_LAUNCH(ctx, k_batch_shape, grid_for(sa.B, 1, maxb), kThreads, 0, sa.B, n,
                   sa.d_graph_ptr, W.up_ptr.as<int32_t>(), W.ev.as<int32_t>(), shape);
        int64_t big[4];
        const void* ptrs[4] = {shape, shape + 1, shape + 2, shape + 3};
        const int bytes[4] = {4, 4, 4, 4};
        SPC_TRY(read_vals(ctx, 4, ptrs, bytes, big));
        if (big[0] <= SmallMem<KT>::kMaxNodes && big[1] <= kSmallEdges && big[2] == 0) {
            int32_t* n_c = W.k_graph.as<int32_t>();
            int32_t* off = W.seg_start.as<int32_t>();
            SPC_TRY(launch_small<KT>(ctx, g, key, sa, sa.B, big[0], big[3], lift, merged, n_c));
            SPC_TRY(scan_i32(ctx, n_c, off, sa.B));
            SPC_LAUNCH(ctx, k_small_shift, grid_for(sa.B, 1, maxb), kThreads, 0, sa.B,
                       sa.d_graph_ptr, off, sa.d_targets, lift, graph_ptr_c, shape + 4);
            int64_t vals[3];
            const void* vp[3] = {off + sa.B, shape + 4, status};
            const int vb[3] = {4, 4, 4};
            SPC_TRY(read_vals(ctx, 3, vp, vb, vals));
            const spc_status st = status_from_bits((uint32_t)vals[2]);
            if (st < 0) return st;
            *n_c_out = vals[0];
            *status_out = vals[1] != 0 ? SPC_WARN_TARGET_NOT_REACHED : SPC_OK;
            return SPC_OK;
        }
    }
    int32_t* pos = W.c_pos.as<int32_t>();
    int64_t n_msf = 0;
    int32_t* node_graph = W.node_graph.as<int32_t>();
    SPC_LAUNCH(ctx, k_node_graph, grid_for(n, kThreads, maxb), kThreads, 0, n, sa.B,
               sa.d_graph_ptr, node_graph);
    const bool use_gprefix = m > 65536 && sa.d_graph_ptr && sa.d_targets;
    GraphSlab<KT> gs{nullptr, nullptr, nullptr};
    int64_t* g_need = nullptr;
    KT* g_tau = nullptr;
    KT* g_lo = nullptr;
    int32_t* g_short = nullptr;
    const int g_grid = (int)std::min<int64_t>(sa.B, (int64_t)ctx->num_sms * 8);
    if (use_gprefix) {
        SPC_TRY(ensure(ctx, W.g_need, (size_t)(sa.B + 1) * 8));
        SPC_TRY(ensure(ctx, W.g_tau, (size_t)(sa.B + 1) * sizeof(KT)));
        SPC_TRY(ensure(ctx, W.g_lo, (size_t)(sa.B + 1) * sizeof(KT)));
        SPC_TRY(ensure(ctx, W.g_short, 16));
        g_need = W.g_need.as<int64_t>();
        g_tau = W.g_tau.as<KT>();
        g_lo = W.g_lo.as<KT>();
        g_short = W.g_short.as<int32_t>();
        gs = GraphSlab<KT>{node_graph, g_tau, g_lo};
    }
    for (int attempt = 0;; ++attempt) {
        if (use_gprefix && attempt == 0)
            SPC_LAUNCH(ctx, k_graph_prefix<KT>, g_grid, kGpThreads, 0, sa.B, 0, sa.d_graph_ptr,
                       W.up_ptr.as<int32_t>(), sa.d_targets, key, W.msf.as<uint8_t>(), g_need,
                       g_tau, g_lo, g_short);
        if (attempt == 0) {
            SPC_LAUNCH(ctx, k_bv_init, grid_for(n > m ? n : m + 1, kThreads, maxb), kThreads, 0,
                       n, m, parent, W.best_k[0].as<unsigned long long>(),
                       W.best_k[1].as<unsigned long long>(),
                       two ? W.best_e[0].as<int32_t>() : nullptr,
                       two ? W.best_e[1].as<int32_t>() : nullptr, W.msf.as<uint8_t>(), merged,
                       counters);
        } else {
            SPC_LAUNCH(ctx, k_bv_reinit, grid_for(n, kThreads, maxb), kThreads, 0, n,
                       W.best_k[0].as<unsigned long long>(),
                       W.best_k[1].as<unsigned long long>(),
                       two ? W.best_e[0].as<int32_t>() : nullptr,
                       two ? W.best_e[1].as<int32_t>() : nullptr, counters);
        }
        // ---- 1. Boruvka minimum spanning forest (of the prefixes) ------------------------
        int64_t cur = m;
        for (int round = 0; cur > 0; ++round) {
            const int in = round & 1, out = in ^ 1;
            const int par = round & 1;
            const int first = round == 0 ? 1 : 0;  // reads the edges themselves
            const int direct = (round == 0 && attempt == 0) ? 1 : 0;
            if (cur <= kFinishMax) {  // the remaining rounds in one CTA
                note_bytes(ctx, first ? (double)m * (8 + sizeof(KT))
                                      : (double)cur * (12 + sizeof(KT) + 8 + 32 + 12));
                SPC_LAUNCH(ctx, k_bv_finish<KT>, 1, kFinishThreads, 0, first, par,
                           m, counters + in, W.wl_e[in].as<int32_t>(), W.wl_u[in].as<int32_t>(),
                           W.wl_v[in].as<int32_t>(), W.wl_e[out].as<int32_t>(),
                           W.wl_u[out].as<int32_t>(), W.wl_v[out].as<int32_t>(),
                           W.eu.as<int32_t>(), W.ev.as<int32_t>(), key, gs, parent,
                           W.best_k[0].as<unsigned long long>(),
                           W.best_k[1].as<unsigned long long>(),
                           two ? W.best_e[0].as<int32_t>() : nullptr,
                           two ? W.best_e[1].as<int32_t>() : nullptr, W.msf.as<uint8_t>(),
                           status);
                break;
            }
            // algorithmic bytes: the first round reads every edge's ends and key; a later one
            // reads each work-list item (e, u, v) and key, walks two parents, lowers two best
            // slots (read and write) and writes the item back
            note_bytes(ctx, first ? (double)m * (8 + sizeof(KT))
                                  : (double)cur * (12 + sizeof(KT) + 8 + 32 + 12));
            SPC_LAUNCH(ctx, k_bv_minkey<KT>,
                       grid_for(cur, kThreads * kMkItems, maxb), kThreads, 0,
                       first, direct, m, counters + in,
                       W.wl_e[in].as<int32_t>(), W.wl_u[in].as<int32_t>(),
                       W.wl_v[in].as<int32_t>(), W.eu.as<int32_t>(), W.ev.as<int32_t>(), key, gs,
                       parent, W.best_k[par].as<unsigned long long>(), W.wl_e[out].as<int32_t>(),
                       W.wl_u[out].as<int32_t>(), W.wl_v[out].as<int32_t>(), counters + out,
                       status);
            if (two) {
                note_bytes(ctx, (double)cur * (12 + 8 + 16 + 8));
                SPC_LAUNCH(ctx, k_bv_tiebreak, grid_for(cur, kThreads, maxb), kThreads, 0,
                           counters + out, W.wl_e[out].as<int32_t>(), W.wl_u[out].as<int32_t>(),
                           W.wl_v[out].as<int32_t>(),
                           reinterpret_cast<const unsigned long long*>(key),
                           W.best_k[par].as<unsigned long long>(), W.best_e[par].as<int32_t>());
            }
            // each item and the two best slots read, the forest flag written, one parent swap
            note_bytes(ctx, (double)cur * (12 + 24 + 1 + 8));
            SPC_LAUNCH(ctx, k_bv_hook<KT>, grid_for(cur, kThreads, maxb), kThreads, 0,
                       counters + out, W.wl_e[out].as<int32_t>(), W.wl_u[out].as<int32_t>(),
                       W.wl_v[out].as<int32_t>(), W.best_k[par].as<unsigned long long>(),
                       W.best_e[par].as<int32_t>(), W.best_k[par ^ 1].as<unsigned long long>(),
                       W.best_e[par ^ 1].as<int32_t>(), parent, W.msf.as<uint8_t>(),
                       counters + in, status);
            // next work-list size (a capture replays the recorded round count)
            SPC_TRY(read_loop_count(ctx, counters + out, &cur));
            // every round at least halves the components that still have edges
            if (round > 64) return SPC_ERR_TIMEOUT;
            // slot `out` (list and count) is the next round's input
        }
        SPC_TRY(scan_flags_u8(ctx, W.msf.as<uint8_t>(), pos, m));
        SPC_TRY(read_i32(ctx, pos + m, &n_msf));
        if (!use_gprefix) break;
        // graphs whose forest falls short take their next slab; done when none does
        SPC_CUDA(cudaMemsetAsync(g_short, 0, sizeof(int32_t), ctx->stream));
        SPC_LAUNCH(ctx, k_graph_prefix<KT>, g_grid, kGpThreads, 0, sa.B, attempt + 1,
                   sa.d_graph_ptr, W.up_ptr.as<int32_t>(), sa.d_targets, key,
                   W.msf.as<uint8_t>(), g_need, g_tau, g_lo, g_short);
        int64_t n_short = 0;
        SPC_TRY(read_i32(ctx, g_short, &n_short));
        if (n_short == 0) break;
        if (attempt > 64) return SPC_ERR_TIMEOUT;  // each slab doubles: never reached
    }
    // ---- 2. lightest forest edges per graph ---------------------------------------------
    KT* sk = W.sel_key.as<KT>();
    uint32_t* sv = W.sel_val.as<uint32_t>();
    SPC_LAUNCH(ctx, k_compact_msf<KT>, grid_for(m, kThreads, maxb), kThreads, 0, m,
               W.msf.as<uint8_t>(), pos, key, sk, sv);
    const int key_bits = sizeof(KT) == 8 ? 63 : 31;  // scores are >= +0: sign bit clear
    if (sizeof(KT) == 8) {
        SPC_TRY(radix_sort_u64(ctx, reinterpret_cast<uint64_t*>(sk), sv,
                               W.sel_key2.as<uint64_t>(), W.sel_val2.as<uint32_t>(), n_msf,
                               key_bits));
    } else {
        SPC_TRY(radix_sort_u32(ctx, reinterpret_cast<uint32_t*>(sk), sv,
                               W.sel_key2.as<uint32_t>(), W.sel_val2.as<uint32_t>(), n_msf,
                               key_bits));
    }
    int32_t* cnt_dev = counters + 3;
    SPC_CUDA(cudaMemcpyAsync(cnt_dev, pos + m, sizeof(int32_t), cudaMemcpyDeviceToDevice,
                             ctx->stream));
    uint32_t* gkey = W.sel_key2.as<uint32_t>();  // reuse: free after the score sort
    SPC_LAUNCH(ctx, k_graph_keys, grid_for(n_msf, kThreads, maxb), kThreads, 0, cnt_dev, sv,
               W.eu.as<int32_t>(), node_graph, gkey);
    int gbits = 1;
    while ((1ll << gbits) < sa.B) ++gbits;
    // stable sort by graph id keeps the score order inside every graph
    SPC_TRY(radix_sort_u32(ctx, gkey, sv, W.t_key.as<uint32_t>(), W.t_val.as<uint32_t>(), n_msf,
                           gbits));
    int32_t* seg_start = W.seg_start.as<int32_t>();
    int32_t* k_graph = W.k_graph.as<int32_t>();
    SPC_LAUNCH(ctx, k_graph_segments, grid_for(sa.B, kThreads, maxb), kThreads, 0, sa.B,
               sa.d_graph_ptr, sa.d_targets, W.up_ptr.as<int32_t>(), pos, seg_start, k_graph);
    int32_t* parent2 = W.parent2.as<int32_t>();
    SPC_LAUNCH(ctx, k_iota, grid_for(n, kThreads, maxb), kThreads, 0, parent2, n);
    if (n_msf > 0) {
        SPC_LAUNCH(ctx, k_select_unite, grid_for(n_msf, kThreads, maxb), kThreads, 0, cnt_dev, sv,
                   gkey, seg_start, k_graph, W.eu.as<int32_t>(), W.ev.as<int32_t>(), parent2,
                   merged, status);
    }
    return finish_batch(ctx, g, sa, lift, n_c_out, graph_ptr_c, status_out);
}

}  // namespace

spc_status clean_selection(spc_context* ctx) {
    Work& W = ctx->work;
    if (!W.sel_dirty || !W.counters.p || !W.key_hist.p) return SPC_OK;
    SPC_CUDA(cudaMemsetAsync(W.counters.as<int32_t>() + kCtFirst, 0, kCtCount * 4, ctx->stream));
    SPC_CUDA(cudaMemsetAsync(W.key_hist.p, 0, (size_t)kTauBins * 4, ctx->stream));
    W.sel_dirty = false;
    return SPC_OK;
}

template <class KT>
static spc_status select_any(spc_context* ctx, const GraphView& g, const void* score,
                             const SelectArgs& sa, int32_t* lift, uint8_t* merged, int64_t* n_c,
                             int64_t* graph_ptr_c, int32_t* status) {
    const KT* key = static_cast<const KT*>(score);
    if (sa.B > 1 || sa.d_graph_ptr != nullptr)
        return select_batch<KT>(ctx, g, key, sa, lift, merged, n_c, graph_ptr_c, status);
    return select_single<KT>(ctx, g, key, sa.target, lift, merged, n_c, status);
}

spc_status run_select(spc_context* ctx, const GraphView& g, const void* score,
                      const SelectArgs& sa, int32_t* lift, uint8_t* merged, int64_t* n_c,
                      int64_t* graph_ptr_c, int32_t* status) {
    if (score_is_f32(g.wtype))
        return select_any<unsigned int>(ctx, g, score, sa, lift, merged, n_c, graph_ptr_c, status);
    return select_any<unsigned long long>(ctx, g, score, sa, lift, merged, n_c, graph_ptr_c,
                                          status);
}

}  // namespace spc
