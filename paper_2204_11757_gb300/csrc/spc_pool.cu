// Node-feature pooling onto the super-nodes, and its gradient: the graph-pooling layer built on
// the coarsening (the assignment held fixed).
//
// Definition 2's lift averages over the member pairs of two super-nodes (it divides by
// |u_c| |v_c|).  Its node counterpart is the mean over a super-node's members:
//   xc[U][f] = S(x[v][f] for the members v of U in ascending v) / |U|,
// with one IEEE division.  The paper has no node features, so the summation order S is this
// library's: a 256-ary tree -- a list of at most kPoolChunk items is summed left to right
// from 0 in the feature type; a longer list is replaced by the sums of its consecutive chunks
// of kPoolChunk, recursively.  Gradient: grad_x[v][f] = grad_xc[c(v)][f] / |c(v)|.
//
// The members of every super-node are listed by a stable radix sort of the node ids by their
// super-node (stable, so ascending id inside each super-node).  Each tree level is one pass:
// chunk counts and offsets (scan), the owner of every chunk, and one chunk sum per (chunk,
// feature).  Chunking a list of one item gives that item back (0 + t = t: a sum started at +0
// is never -0), so every super-node runs through the same number of levels, enough for the
// largest list of the call.  Blocks are 32 features x 8 units: a warp reads 32 consecutive
// features of one row, so member rows are read with coalesced loads.
//
// Most lifts have no super-node of more than kPoolChunk members.  Then the tree has one level,
// and one kernel reads every member row once and writes the means (k_pool_gather); the member
// lists need no sort either: each node takes a slot of its super-node as it is counted, and is
// ranked among the super-node's members.  2^22 nodes, 64 binary32 features, about 8 members
// each: the forward's kernels 1.20 -> 0.38 ms; its bytes at the copy rate are 0.18 ms.
#include "spc_scan.cuh"

namespace spc {

namespace {

template <class T> struct PoolOps;
template <> struct PoolOps<float> {
    __device__ static float add(float a, float b) { return __fadd_rn(a, b); }
    __device__ static float div(float a, int64_t c) { return __fdiv_rn(a, __ll2float_rn(c)); }
};
template <> struct PoolOps<double> {
    __device__ static double add(double a, double b) { return __dadd_rn(a, b); }
    __device__ static double div(double a, int64_t c) { return __ddiv_rn(a, __ll2double_rn(c)); }
};

constexpr int64_t kPoolChunk = 256;
constexpr int kPoolRows = 8;  // units (rows, chunks, super-nodes) per block; 32 features each

// member counts; lift values outside [0, n_c) are reported and left out.  Runs of one
// super-node (a hub holds most nodes of a deep coarsening) are counted with one atomic per
// block or per warp.  `slot` (may be null): every node's place among its super-node's members,
// in the order of the atomics.
__global__ void __launch_bounds__(kThreads)
k_pool_counts(int64_t n, const int32_t* __restrict__ lift, int64_t n_c,
              int32_t* __restrict__ cnt, int32_t* __restrict__ slot,
              uint32_t* __restrict__ status) {
    spc::pdl_wait();
    __shared__ int32_t sh_first, sh_base;
    const int lane = threadIdx.x & 31;
    for (int64_t b0 = (int64_t)blockIdx.x * blockDim.x; b0 < n;
         b0 += (int64_t)gridDim.x * blockDim.x) {  // uniform per block
        const int64_t v = b0 + threadIdx.x;
        int32_t u = v < n ? lift[v] : -1;
        if (v < n && (u < 0 || (int64_t)u >= n_c)) {
            atomicOr(status, DEV_BAD_ARG);
            u = -1;
        }
        if (threadIdx.x == 0) sh_first = u;
        __syncthreads();
        const int32_t first = sh_first;
        const bool all_same = __syncthreads_and(u == first || v >= n) != 0;
        if (all_same) {
            if (threadIdx.x == 0 && first >= 0) {
                const int64_t k = n - b0 < (int64_t)blockDim.x ? n - b0 : blockDim.x;
                sh_base = atomicAdd(cnt + first, (int32_t)k);
            }
            if (slot) {
                __syncthreads();
                if (v < n && first >= 0) slot[v] = sh_base + (int32_t)threadIdx.x;
            }
        } else {
            const unsigned peers = __match_any_sync(0xffffffffu, u);
            const int leader = __ffs(peers) - 1;
            int32_t old = 0;
            if (u >= 0 && lane == leader) old = atomicAdd(cnt + u, __popc(peers));
            if (slot) {
                old = __shfl_sync(0xffffffffu, old, leader);
                if (u >= 0) slot[v] = old + __popc(peers & ((1u << lane) - 1u));
            }
        }
        __syncthreads();
    }
}

// scan storer of the member counts: offsets, and stats[0] = the largest count, stats[1] = the sum
// of squared counts
struct PoolOffSt {
    int32_t* off;
    int64_t n;
    unsigned long long* stats;
    struct Local {
        unsigned long long mx, sq;
    };
    __device__ Local begin() const { return Local{0ull, 0ull}; }
    __device__ void operator()(Local& L, int64_t g, bool valid, int32_t excl, int32_t val) const {
        if (!valid) return;
        off[g] = excl;
        const unsigned long long c = (unsigned long long)val;
        L.mx = c > L.mx ? c : L.mx;
        L.sq += c * c;
    }
    __device__ void finish(Local& L) const {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long m = __shfl_xor_sync(0xffffffffu, L.mx, o);
            L.mx = m > L.mx ? m : L.mx;
            L.sq += __shfl_xor_sync(0xffffffffu, L.sq, o);
        }
        if ((threadIdx.x & 31) == 0 && L.mx) {
            atomicMax(stats, L.mx);
            atomicAdd(stats + 1, L.sq);
        }
    }
    __device__ void total(int32_t tot) const { off[n] = tot; }
};

// every node into its slot of its super-node's member range
__global__ void __launch_bounds__(kThreads)
k_pool_place(int64_t n, const int32_t* __restrict__ lift, const int32_t* __restrict__ off,
             const int32_t* __restrict__ slot, uint32_t* __restrict__ items) {
    spc::pdl_wait();
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        items[off[lift[v]] + slot[v]] = (uint32_t)v;
}

// every member to its rank (ascending id) among its super-node's members
__global__ void __launch_bounds__(kThreads)
k_pool_rank(int64_t n, const int32_t* __restrict__ lift, const int32_t* __restrict__ off,
            const uint32_t* __restrict__ items, uint32_t* __restrict__ members) {
    spc::pdl_wait();
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t v = items[p];
        const int32_t u = lift[v], lo = off[u], hi = off[u + 1];
        int32_t r = 0;
#pragma unroll 4
        for (int32_t j = lo; j < hi; ++j) r += items[j] < v ? 1 : 0;
        members[lo + r] = v;
    }
}

// V consecutive features, one aligned load or store of V * sizeof(T) bytes
template <class T, int V>
struct alignas(sizeof(T) * V) PoolVec {
    T x[V];
};

// rows that are read or written once: evict-first accesses, so the coarse rows stay in L2
template <class Vec>
__device__ __forceinline__ Vec pool_ld_once(const Vec* p) {
    if constexpr (sizeof(Vec) == 16) {
        const uint4 z = __ldcs(reinterpret_cast<const uint4*>(p));
        return *reinterpret_cast<const Vec*>(&z);
    } else {
        return *p;
    }
}
template <class Vec>
__device__ __forceinline__ void pool_st_once(Vec* p, const Vec& v) {
    if constexpr (sizeof(Vec) == 16)
        __stcs(reinterpret_cast<uint4*>(p), *reinterpret_cast<const uint4*>(&v));
    else
        *p = v;
}

// sub-warps of lp lanes (a power of two), lane k on the features [kV, kV + V), then + lp V
__device__ __forceinline__ int pool_lane(int lp) { return (int)threadIdx.x & (lp - 1); }

// The means of super-nodes of at most kPoolChunk members: a sub-warp per super-node adds up its
// member rows left to right from 0, kPoolFlight rows in flight, and divides.  Bound by the random
// row reads; 16-byte loads where rows and base are aligned for them.  2^22 rows of 64 binary32
// features: 0.230 ms, 5.3 TB/s of its bytes (8 rows in flight a thread: fewer threads, 0.273).
constexpr int kPoolFlight = 4;

template <class T, int V>
__global__ void __launch_bounds__(kThreads)
k_pool_gather(int64_t n_c, int64_t F, int lp, const int32_t* __restrict__ off,
              const uint32_t* __restrict__ members, const T* __restrict__ x, T* __restrict__ xc) {
    spc::pdl_wait();
    using Vec = PoolVec<T, V>;
    const int64_t units = F / V;
    const int subs = kThreads / lp, k0 = pool_lane(lp);
    const Vec* xv = reinterpret_cast<const Vec*>(x);
    Vec* out = reinterpret_cast<Vec*>(xc);
    for (int64_t u = (int64_t)blockIdx.x * subs + threadIdx.x / lp; u < n_c;
         u += (int64_t)gridDim.x * subs) {
        const int32_t j0 = off[u], j1 = off[u + 1];
        for (int64_t k = k0; k < units; k += lp) {
            Vec acc;
#pragma unroll
            for (int i = 0; i < V; ++i) acc.x[i] = T(0);
            for (int32_t j = j0; j < j1; j += kPoolFlight) {
                Vec t[kPoolFlight];
#pragma unroll
                for (int q = 0; q < kPoolFlight; ++q)
                    if (j + q < j1)
                        t[q] = pool_ld_once(xv + (int64_t)members[j + q] * units + k);
#pragma unroll
                for (int q = 0; q < kPoolFlight; ++q)
                    if (j + q < j1) {
#pragma unroll
                        for (int i = 0; i < V; ++i) acc.x[i] = PoolOps<T>::add(acc.x[i], t[q].x[i]);
                    }
            }
#pragma unroll
            for (int i = 0; i < V; ++i)
                acc.x[i] = j1 > j0 ? PoolOps<T>::div(acc.x[i], j1 - j0) : T(0);
            out[u * units + k] = acc;
        }
    }
}

// sort input: key = super-node, value = node id (in ascending order, so the stable sort keeps
// ascending ids inside every super-node)
__global__ void k_pool_keys(int64_t n, const int32_t* __restrict__ lift,
                            uint32_t* __restrict__ key, uint32_t* __restrict__ val) {
    spc::pdl_wait();
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        key[v] = (uint32_t)lift[v];
        val[v] = (uint32_t)v;
    }
}

// chunks of every super-node's list at the next tree level
__global__ void k_pool_nchunks(int64_t n_c, const int32_t* __restrict__ items,
                               int32_t* __restrict__ nch) {
    spc::pdl_wait();
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n_c;
         u += (int64_t)gridDim.x * blockDim.x)
        nch[u] = (int32_t)((items[u] + kPoolChunk - 1) / kPoolChunk);
}

__global__ void k_pool_owner(int64_t n_c, const int32_t* __restrict__ choff,
                             int32_t* __restrict__ owner) {
    spc::pdl_wait();
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n_c;
         u += (int64_t)gridDim.x * blockDim.x)
        for (int32_t c = choff[u]; c < choff[u + 1]; ++c) owner[c] = (int32_t)u;
}

// One tree level: the sum of every chunk of kPoolChunk consecutive items of a super-node's
// list, left to right from 0.  Level 0 items are member rows of x (members[k]), later levels
// the previous level's sums (prev[k]).
template <class T>
__global__ void __launch_bounds__(32 * kPoolRows)
k_pool_level(int64_t n_c, int64_t F, const int32_t* __restrict__ ioff,
             const int32_t* __restrict__ icnt, const int32_t* __restrict__ choff,
             const int32_t* __restrict__ owner, const uint32_t* __restrict__ members,
             const T* __restrict__ x, const T* __restrict__ prev, T* __restrict__ part,
             const uint32_t* status) {
    spc::pdl_wait();
    if (*status) return;
    const int64_t nchunks = choff[n_c];
    for (int64_t c = (int64_t)blockIdx.x * kPoolRows + threadIdx.y; c < nchunks;
         c += (int64_t)gridDim.x * kPoolRows) {
        const int32_t u = owner[c];
        const int64_t k0 = ioff[u] + (c - choff[u]) * kPoolChunk;
        const int64_t iend = (int64_t)ioff[u] + icnt[u];
        const int64_t k1 = k0 + kPoolChunk < iend ? k0 + kPoolChunk : iend;
        for (int64_t f = threadIdx.x; f < F; f += 32) {
            T acc = T(0);
            int64_t k = k0;
            if (members) {
                for (; k + 4 <= k1; k += 4) {  // four rows in flight, additions in order
                    const T a0 = x[(int64_t)members[k] * F + f];
                    const T a1 = x[(int64_t)members[k + 1] * F + f];
                    const T a2 = x[(int64_t)members[k + 2] * F + f];
                    const T a3 = x[(int64_t)members[k + 3] * F + f];
                    acc = PoolOps<T>::add(acc, a0);
                    acc = PoolOps<T>::add(acc, a1);
                    acc = PoolOps<T>::add(acc, a2);
                    acc = PoolOps<T>::add(acc, a3);
                }
                for (; k < k1; ++k) acc = PoolOps<T>::add(acc, x[(int64_t)members[k] * F + f]);
            } else {
                for (; k < k1; ++k) acc = PoolOps<T>::add(acc, prev[k * F + f]);
            }
            part[c * F + f] = acc;
        }
    }
}

// the mean: the single sum left after the last level, divided by the member count
template <class T>
__global__ void __launch_bounds__(32 * kPoolRows)
k_pool_mean(int64_t n_c, int64_t F, const int32_t* __restrict__ cnt,
            const int32_t* __restrict__ off, const T* __restrict__ part, T* __restrict__ xc,
            const uint32_t* status) {
    spc::pdl_wait();
    if (*status) return;
    for (int64_t u = (int64_t)blockIdx.x * kPoolRows + threadIdx.y; u < n_c;
         u += (int64_t)gridDim.x * kPoolRows) {
        const int32_t c = cnt[u];
        for (int64_t f = threadIdx.x; f < F; f += 32)
            xc[u * F + f] = c > 0 ? PoolOps<T>::div(part[(int64_t)off[u] * F + f], c) : T(0);
    }
}

// grad_x[v] = grad_xc[lift[v]] / members: a sub-warp per row, kBackRows rows of a sub-warp in
// flight (lift, count and gradient reads are dependent), 16-byte accesses where they are
// aligned.  Bound by memory: 2^22 rows of 64 binary32 features write 1.07 GB and gather as much
// from 134 MB of coarse gradients, 0.565 -> 0.297 ms (8 rows in flight 0.416; a multiplication
// in the division's place 0.287).  Binary64 quotients go by one reciprocal per row (div_row) where a
// lane has two of a row or more: the IEEE divisions filled the FP64 pipe (2^18 rows of 256 features,
// the call 1,039 us, 500 so).
constexpr int kBackRows = 4;

__device__ __forceinline__ float back_rcp(float, int32_t) { return 0.f; }
__device__ __forceinline__ double back_rcp(double, int32_t c) { return __drcp_rn((double)c); }
__device__ __forceinline__ float back_div(float g, int32_t c, float) {
    return PoolOps<float>::div(g, c);
}
__device__ __forceinline__ double back_div(double g, int32_t c, double rcp) {
    return div_row(g, (double)c, rcp, __double2hiint(rcp) != 0);
}

template <class T, int V>
__global__ void __launch_bounds__(kThreads)
k_pool_backward(int64_t n, int64_t F, int lp, const int32_t* __restrict__ lift,
                const int32_t* __restrict__ cnt, const T* __restrict__ grad_xc,
                T* __restrict__ grad_x, const uint32_t* status) {
    spc::pdl_wait();
    if (*status) return;
    using Vec = PoolVec<T, V>;
    const int64_t units = F / V;
    const int subs = kThreads / lp, k0 = pool_lane(lp);
    const Vec* g = reinterpret_cast<const Vec*>(grad_xc);
    Vec* out = reinterpret_cast<Vec*>(grad_x);
    const int64_t per = (int64_t)subs * kBackRows;
    for (int64_t b = (int64_t)blockIdx.x * per; b < n; b += (int64_t)gridDim.x * per) {
        const int64_t v0 = b + threadIdx.x / lp;
        int32_t u[kBackRows], c[kBackRows];
#pragma unroll
        for (int q = 0; q < kBackRows; ++q) {
            const int64_t v = v0 + (int64_t)q * subs;
            u[q] = v < n ? lift[v] : 0;
        }
#pragma unroll
        for (int q = 0; q < kBackRows; ++q) c[q] = cnt[u[q]];
        T rcp[kBackRows];
#pragma unroll
        for (int q = 0; q < kBackRows; ++q)
            rcp[q] = V > 1 || units > lp ? back_rcp(T(0), c[q]) : T(0);
        for (int64_t k = k0; k < units; k += lp) {
            Vec t[kBackRows];
#pragma unroll
            for (int q = 0; q < kBackRows; ++q) t[q] = g[(int64_t)u[q] * units + k];
#pragma unroll
            for (int q = 0; q < kBackRows; ++q) {
                const int64_t v = v0 + (int64_t)q * subs;
                if (v < n) {
#pragma unroll
                    for (int i = 0; i < V; ++i) t[q].x[i] = back_div(t[q].x[i], c[q], rcp[q]);
                    pool_st_once(out + v * units + k, t[q]);
                }
            }
        }
    }
}

// member counts of every super-node (slot as in k_pool_counts); values outside [0, n_c) set the
// status word, and later kernels return when it is set
spc_status pool_counts(spc_context* ctx, int64_t n, const int32_t* lift, int64_t n_c,
                       int32_t* slot) {
    Work& W = ctx->work;
    SPC_TRY(ensure(ctx, W.pool_cnt, (size_t)(n_c + 1) * 4));
    SPC_CUDA(cudaMemsetAsync(W.pool_cnt.p, 0, (size_t)(n_c + 1) * 4, ctx->stream));
    if (n > 0) {
        SPC_LAUNCH(ctx, k_pool_counts, grid_for(n, kThreads, ctx->num_sms * 8), kThreads, 0, n,
                   lift, n_c, W.pool_cnt.as<int32_t>(), slot, ctx->d_status);
    }
    return SPC_OK;
}

// features per access (16 bytes where rows and bases allow) and lanes per row
template <class T>
int pool_vec(int64_t F, const void* a, const void* b) {
    constexpr int V = 16 / (int)sizeof(T);
    const uintptr_t bits = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b);
    return F % V == 0 && (bits & 15) == 0 ? V : 1;
}

int pool_lanes(int64_t units) {
    int lp = 1;
    while (lp < 32 && lp < units) lp <<= 1;
    return lp;
}

int pool_grid(int64_t units, int num_sms) {
    return grid_for(units, kPoolRows, num_sms * 16);
}

// Member lists by slots and ranks while no super-node has more than kPoolChunk members and the
// ranking compares at most kPoolRankWork members per node (a sort of the ids is 0.21 ms at 2^22
// nodes, the slots, placing and ranking at about 16 comparisons per node 0.07 ms).
constexpr unsigned long long kPoolRankWork = 64;

template <class T, int V>
spc_status launch_gather(spc_context* ctx, int64_t n_c, int64_t F, const T* x, T* xc) {
    const int lp = pool_lanes(F / V);
    SPC_LAUNCH(ctx, (k_pool_gather<T, V>), grid_for(n_c, kThreads / lp, ctx->num_sms * 64),
               kThreads, 0, n_c, F, lp, ctx->work.pool_off.as<int32_t>(),
               ctx->work.pool_val.as<uint32_t>(), x, xc);
    return SPC_OK;
}

template <class T>
spc_status pool_forward_typed(spc_context* ctx, int64_t n, const int32_t* lift, int64_t n_c,
                              int64_t F, const T* x, T* xc) {
    Work& W = ctx->work;
    const size_t nb = (size_t)(n > 0 ? n : 1) * 4;
    SPC_TRY(ensure(ctx, W.pool_off, (size_t)(n_c + 1) * 4));
    SPC_TRY(ensure(ctx, W.pool_key, nb));
    SPC_TRY(ensure(ctx, W.pool_val, nb));
    SPC_TRY(ensure(ctx, W.pool_key2, nb));
    SPC_TRY(ensure(ctx, W.pool_stats, 16));
    int32_t* slot = W.pool_key.as<int32_t>();
    SPC_TRY(pool_counts(ctx, n, lift, n_c, slot));
    int32_t* cnt = W.pool_cnt.as<int32_t>();
    int32_t* off = W.pool_off.as<int32_t>();
    unsigned long long* stats = W.pool_stats.as<unsigned long long>();
    SPC_CUDA(cudaMemsetAsync(stats, 0, 16, ctx->stream));
    SPC_TRY(scan_fused<int32_t>(ctx, n_c, ArrayLd<int32_t, int32_t>{cnt},
                                PoolOffSt{off, n_c, stats}, 8.0 * n_c));
    // the verdict on the lift (the later kernels index with it) and the largest super-node
    int64_t info[3];
    {
        const void* ptrs[3] = {ctx->d_status, stats, stats + 1};
        const int bytes[3] = {4, 8, 8};
        SPC_TRY(read_vals(ctx, 3, ptrs, bytes, info));
        const spc_status st = status_from_bits((uint32_t)info[0]);
        if (st < 0) return st;
    }
    if (info[1] <= kPoolChunk && (unsigned long long)info[2] <= kPoolRankWork * (uint64_t)n) {
        if (n > 0) {
            const int gn = grid_for(n, kThreads, ctx->num_sms * 8);
            uint32_t* items = W.pool_key2.as<uint32_t>();
            SPC_LAUNCH(ctx, k_pool_place, gn, kThreads, 0, n, lift, off, slot, items);
            SPC_LAUNCH(ctx, k_pool_rank, gn, kThreads, 0, n, lift, off, items,
                       W.pool_val.as<uint32_t>());
        }
        // every member row and the member list read once, the means written once
        note_bytes(ctx, (double)n * F * sizeof(T) + 4.0 * n + (double)n_c * F * sizeof(T));
        if (pool_vec<T>(F, x, xc) > 1)
            return launch_gather<T, 16 / (int)sizeof(T)>(ctx, n_c, F, x, xc);
        return launch_gather<T, 1>(ctx, n_c, F, x, xc);
    }
    SPC_TRY(ensure(ctx, W.pool_val2, nb));
    // tree levels enough for the largest list; chunk buffers at the level-0 bound
    int levels = 1;
    for (int64_t cap = kPoolChunk; cap < info[1]; cap *= kPoolChunk) ++levels;
    const int64_t max_chunks = n_c + n / kPoolChunk + 1;
    SPC_TRY(ensure(ctx, W.pool_nch, (size_t)(n_c + 1) * 4 * 2));
    SPC_TRY(ensure(ctx, W.pool_choff, (size_t)(n_c + 1) * 4 * 2));
    SPC_TRY(ensure(ctx, W.pool_owner, (size_t)max_chunks * 4));
    SPC_TRY(ensure(ctx, W.pool_part, (size_t)max_chunks * F * sizeof(T) * 2));
    int bits = 1;
    while ((1ll << bits) < n_c) ++bits;
    if (n > 0) {
        SPC_LAUNCH(ctx, k_pool_keys, grid_for(n, kThreads, ctx->num_sms * 8), kThreads, 0, n,
                   lift, W.pool_key.as<uint32_t>(), W.pool_val.as<uint32_t>());
        SPC_TRY(radix_sort_u32(ctx, W.pool_key.as<uint32_t>(), W.pool_val.as<uint32_t>(),
                               W.pool_key2.as<uint32_t>(), W.pool_val2.as<uint32_t>(), n, bits));
    }
    const int gu = grid_for(n_c, kThreads, ctx->num_sms * 8);
    const dim3 blk(32, kPoolRows);
    const int32_t* icnt = cnt;   // items per super-node at this level
    const int32_t* ioff = off;   // their offsets
    const T* prev = nullptr;
    T* part = W.pool_part.as<T>();
    for (int l = 0; l < levels; ++l) {
        int32_t* nch = W.pool_nch.as<int32_t>() + (l & 1) * (n_c + 1);
        int32_t* choff = W.pool_choff.as<int32_t>() + (l & 1) * (n_c + 1);
        T* out = part + (size_t)(l & 1) * max_chunks * F;
        SPC_LAUNCH(ctx, k_pool_nchunks, gu, kThreads, 0, n_c, icnt, nch);
        SPC_TRY(scan_i32(ctx, nch, choff, n_c));
        SPC_LAUNCH(ctx, k_pool_owner, gu, kThreads, 0, n_c, choff, W.pool_owner.as<int32_t>());
        // level 0: every feature of every member read once, the member list read once,
        // one sum per chunk and feature written
        if (l == 0)
            note_bytes(ctx, (double)n * F * sizeof(T) + 4.0 * n +
                                (double)max_chunks * F * sizeof(T));
        SPC_LAUNCH(ctx, k_pool_level<T>, pool_grid(max_chunks, ctx->num_sms), blk, 0, n_c, F,
                   ioff, icnt, choff, W.pool_owner.as<int32_t>(),
                   l == 0 ? W.pool_val.as<uint32_t>() : nullptr, x, prev, out, ctx->d_status);
        icnt = nch;
        ioff = choff;
        prev = out;
    }
    SPC_LAUNCH(ctx, k_pool_mean<T>, pool_grid(n_c, ctx->num_sms), blk, 0, n_c, F, cnt, ioff,
               prev, xc, ctx->d_status);
    return SPC_OK;
}

template <class T, int V>
spc_status launch_backward(spc_context* ctx, int64_t n, const int32_t* lift, int64_t F,
                           const T* grad_xc, T* grad_x) {
    const int lp = pool_lanes(F / V);
    SPC_LAUNCH(ctx, (k_pool_backward<T, V>),
               grid_for(n, kThreads / lp * kBackRows, ctx->num_sms * 16), kThreads, 0, n, F, lp,
               lift, ctx->work.pool_cnt.as<int32_t>(), grad_xc, grad_x, ctx->d_status);
    return SPC_OK;
}

template <class T>
spc_status pool_backward_typed(spc_context* ctx, int64_t n, const int32_t* lift, int64_t n_c,
                               int64_t F, const T* grad_xc, T* grad_x) {
    SPC_TRY(pool_counts(ctx, n, lift, n_c, nullptr));
    if (n == 0) return SPC_OK;
    // lift and counts, every coarse gradient once, every fine gradient written once
    note_bytes(ctx, 4.0 * n + 4.0 * n_c + (double)n_c * F * sizeof(T) +
                        (double)n * F * sizeof(T));
    if (pool_vec<T>(F, grad_xc, grad_x) > 1)
        return launch_backward<T, 16 / (int)sizeof(T)>(ctx, n, lift, F, grad_xc, grad_x);
    return launch_backward<T, 1>(ctx, n, lift, F, grad_xc, grad_x);
}

}  // namespace

spc_status run_pool_forward(spc_context* ctx, int64_t n, const int32_t* lift, int64_t n_c,
                            int64_t F, spc_dtype dt, const void* x, void* xc) {
    if (dt == SPC_F32)
        return pool_forward_typed<float>(ctx, n, lift, n_c, F, static_cast<const float*>(x),
                                         static_cast<float*>(xc));
    if (dt == SPC_F64)
        return pool_forward_typed<double>(ctx, n, lift, n_c, F, static_cast<const double*>(x),
                                          static_cast<double*>(xc));
    return SPC_ERR_INVALID_ARG;
}

spc_status run_pool_backward(spc_context* ctx, int64_t n, const int32_t* lift, int64_t n_c,
                             int64_t F, spc_dtype dt, const void* grad_xc, void* grad_x) {
    if (dt == SPC_F32)
        return pool_backward_typed<float>(ctx, n, lift, n_c, F,
                                          static_cast<const float*>(grad_xc),
                                          static_cast<float*>(grad_x));
    if (dt == SPC_F64)
        return pool_backward_typed<double>(ctx, n, lift, n_c, F,
                                           static_cast<const double*>(grad_xc),
                                           static_cast<double*>(grad_x));
    return SPC_ERR_INVALID_ARG;
}

}  // namespace spc
