// Selection, emission and small elementwise kernels of the DARTree path.
//
//   merge_select  (Algorithm 1, scoring + "retain the global top-W"):
//       one cluster of blocks per sequence merges the LM-head kernel's
//       per-CTA partials into every node's log-sum-exp and top-k children,
//       log q~ = min(z - lse, 0), scores them with Eq. 5, and its block 0
//       keeps the top-W as S_d.
//   prune_emit    (Algorithm 1 final step + Lemma 1, Sec. 3.3 flattening):
//       one block per sequence: global top-B by (score desc, node id asc),
//       compaction in id order, parent remap, depths, position ids and the
//       ancestor bit mask.
//   prep / gather / silu / gather_silu / residual_norm: the elementwise parts
//       of the fallback correction head around the two GEMMs (gather_silu
//       adds the per-token row of the split first layer's table).
#include <algorithm>
#include <cstdlib>

#include "dart_device.cuh"
#include "dart_emit.cuh"
#include "dart_kernels.h"

namespace dart {

namespace {

constexpr int kSelThreads = 512;
constexpr int kEmitThreads = 1024;

// merge_select: one cluster of blocks per sequence; a block merges the
// LM-head's partials of several nodes at once, kPer threads each (a thread
// per vocabulary range), and the frontier's candidates are handed to block 0
// of the cluster through distributed shared memory.  The kernel is on every
// depth's serial chain and bound by latency: dependent round trips, barriers,
// and the fetch of its own instructions, which are cold at every depth (the
// LM-head between two launches is larger than the instruction caches), so the
// code is kept small: loops are not unrolled, only the first four keys of
// every (sorted) list are read at once and more only from lists whose fourth
// key is still a candidate, a threshold from group maxima (k <= 16) replaces
// ranked list heads, and up to 16 parents' candidates are ranked by binary
// searches in their sorted lists.
// Measured on GB300 against one block per node that read every list whole and
// handed over through global memory and an atomic ticket (µs per round, same
// box): 8 nodes, k = 8, d = 2560 2178 -> 2080; 16 nodes, k = 16, d = 4096
// 3479 -> 3427; 64 nodes, k = 64 2771 -> 2714; 3 x 11 nodes 591 -> 564; 8 x 32
// nodes and candidate sets (where the W_i GEMM beside it is longer) -0.5 %.
constexpr int kMergeCluster = 16;     // blocks per cluster, at most
constexpr int kMergeThreads = 1024;
constexpr int kGroupMaxK = 16;        // threshold from group maxima up to this k
constexpr int kMergeSearchP = 16;     // frontier by binary searches up to this many parents

__device__ __forceinline__ void st_cluster_u64(uint32_t local, uint32_t rank, uint64_t v) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(remote), "l"(v) : "memory");
}

// More than kRankMax keys reach the threshold (many equal scores): the kk
// largest of the n keys by radix select, into surv (unsorted).
__device__ __noinline__ void radix_survivors(const uint64_t* keys, int n, int kk, uint64_t* surv, uint32_t* hist,
                                             int* scal) {
    const uint64_t kth = block_kth_largest(keys, n, kk, hist, scal);
    if (threadIdx.x == 0) scal[2] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const uint64_t x = keys[i];
        if (x != 0ull && x >= kth) surv[atomicAdd(&scal[2], 1)] = x;
    }
    __syncthreads();
}

// Keys above x among l[0..m) (16-byte aligned; l[m] = 0 when m is odd).
__device__ __forceinline__ int count_above(const uint64_t* l, int m, uint64_t x) {
    const ulonglong2* l2 = reinterpret_cast<const ulonglong2*>(l);
    int r = 0;
#pragma unroll 4
    for (int j = 0; j < (m + 1) / 2; j++) {
        const ulonglong2 y = l2[j];
        r += (y.x > x) + (y.y > x);
    }
    return r;
}

// The first min(n, 4) keys of a list, zeros past them: one 32-byte load where
// every list starts on such a boundary (wide), since four 8-byte loads of
// lists that lie apart each take the load unit 32 cycles per warp.
__device__ __forceinline__ void load4(const uint64_t* l, int n, bool wide, uint64_t (&v)[4]) {
    if (wide) {
        asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(l));
        return;
    }
#pragma unroll
    for (int j = 0; j < 4; j++) v[j] = j < n ? __ldcg(reinterpret_cast<const unsigned long long*>(l) + j) : 0ull;
}

// Appends the keys of keys[0..n) that reach T (none is 0) to surv.
__device__ __forceinline__ void append_reaching(const uint64_t* keys, int n, uint64_t T, uint64_t* surv, int* cnt, int t0,
                                                int nt) {
#pragma unroll 1
    for (int i = t0; i < n; i += nt) {
        const uint64_t x = keys[i];
        if (x != 0ull && x >= T) {
            const int pos = atomicAdd(cnt, 1);
            if (pos < kRankMax) surv[pos] = x;
        }
    }
}

// npb nodes per block: block r of a cluster merges the nodes r * npb ...
// kFew: fewer lists than k (small vocabularies, large k), where no list head
// bounds the k-th key and a thread that walked its list would wait for a round
// trip per four keys.  The threshold then is the r-th largest of the lists'
// j-th keys, j the least with j * nV >= k and r = ceil(k / j): at least r * j
// keys reach it; and the node's keys, at most 63 * 64, are read eight per
// thread at once.  Measured on GB300 (µs, events around the launch; walking the
// lists, now): 10 nodes, k = 61, 49 lists 37.8, 15.3; 6 x 3 nodes, k = 57, 20
// lists 56.0, 11.0; 2 x 6 nodes, k = 41, 23 lists 41.5, 13.1.
// (One block per SM at least: left to itself the compiler may keep two blocks of
// threads by 32 registers a thread and spill, 3 x 11 nodes 493 -> 522 µs per round.)
template <int kPer, bool kFew>
__global__ void __launch_bounds__(kMergeThreads, 1) merge_select_kernel(const SelectArgs a, int cs, int npb) {
    pdl_trigger();
    cluster_started_arrive();
    constexpr int kNodes = kMergeThreads / kPer, kWarps = kPer / 32;
    extern __shared__ __align__(16) uint64_t survs[];  // [nh][kRankMax] keys that reach the threshold
    __shared__ __align__(16) uint64_t heads2[kNodes][kPer];  // list heads, or per-warp group maxima [kWarps][32]
    __shared__ float redm2[kNodes][kWarps], redf2[kNodes][kWarps];
    __shared__ uint32_t hist[256];
    __shared__ int scal[4];
    __shared__ int cnt2[kNodes];
    __shared__ uint64_t thr2[kNodes];
    const int nh = blockDim.x / kPer;  // nodes at once
    const int fk = (a.P * a.k + 1) & ~1, stride = part_stride(a.nV, a.klist);
    const int half = threadIdx.x / kPer, tid = threadIdx.x % kPer, lane = tid & 31, warp = tid >> 5;
    uint64_t* surv = survs + half * kRankMax;
    uint64_t* fkey = survs + nh * kRankMax;  // [P * k] block 0: the frontier's candidates, sorted per parent
    const bool search = a.P <= kMergeSearchP;
    int* ftok = reinterpret_cast<int*>(fkey + fk);  // [P * k] with `search`; else read from node_tok
    uint64_t* heads = heads2[half];
    const int rank = blockIdx.x % cs, s = blockIdx.x / cs;
    const float2 none = make_float2(-INFINITY, 0.0f);
    const bool wide = (a.klist & 3) == 0 && (reinterpret_cast<uintptr_t>(a.part_key) & 31u) == 0;
    pdl_wait();
    cluster_started_wait();  // block 0 runs before candidates are sent to it
    const int prev_count = a.dep == 1 ? 1 : __ldcg(a.tree_count + s * a.L + a.dep - 2);
    const uint32_t fk0 = smem_u32(fkey), ft0 = smem_u32(ftok);
#pragma unroll 1
    for (int it = 0; it * nh < npb; it++) {
        const int p = rank * npb + it * nh + half, n = s * a.P + p;
        const bool mine = it * nh + half < npb && p < a.P;
        // the loads of one round trip: partials, the first keys of this
        // thread's list, the bound, the parent's score
        const float2* ms = a.part_ms + static_cast<size_t>(n) * a.nV;
        const uint64_t* lists = a.part_key + static_cast<size_t>(n) * stride;
        const float2 m0 = mine && tid < a.nV ? __ldcg(ms + tid) : none;
        const float2 m1 = mine && tid + kPer < a.nV ? __ldcg(ms + tid + kPer) : none;
        constexpr int kKeys = kFew ? 8 : 4;  // keys of this thread
        uint64_t v[kKeys] = {};
        uint64_t g = 0ull;  // the key whose rank gives the threshold
        const int jth = kFew ? (a.k + a.nV - 1) / a.nV : 1;
        // (kFew: the node's keys i0 + 2 * (tid + u * kPer) and the next, u < 4)
        auto load_keys = [&](int i0) {
#pragma unroll
            for (int u = 0; u < kKeys / 2; u++) {
                const int i = i0 + 2 * (tid + u * kPer);
                ulonglong2 x = make_ulonglong2(0ull, 0ull);
                if (mine && i < a.nV * a.klist) x = __ldcg(reinterpret_cast<const ulonglong2*>(lists + i));
                v[2 * u] = x.x;
                v[2 * u + 1] = i + 1 < a.nV * a.klist ? x.y : 0ull;  // (an odd number of keys: past the end)
            }
        };
        if constexpr (kFew) {
            if (mine && tid < a.nV)
                g = __ldcg(reinterpret_cast<const unsigned long long*>(lists) + tid * a.klist + jth - 1);
            load_keys(0);
        } else {
            if (mine && tid < a.nV) load4(lists + tid * a.klist, a.klist, wide, v);
            g = v[0];
        }
        const uint64_t bound =
            a.gthr && mine ? __ldcg(reinterpret_cast<const unsigned long long*>(a.gthr) + n) : 0ull;
        const float ps = a.dep == 1 || !mine
                             ? 0.0f
                             : __ldcg(a.tree_score + (static_cast<size_t>(s) * a.L + a.dep - 2) * a.W + p);
        const float2 acc = lse_merge(m0, m1);
        const float wm = warp_max(acc.x);
        if (lane == 0) redm2[half][warp] = wm;
        if (tid == 0) {
            cnt2[half] = 0;
            thr2[half] = 0ull;
        }
        // threshold: a key that at least k keys reach.  Up to kGroupMaxK: the
        // heads are dealt into 2^q >= k groups, each of whose maxima reaches
        // the least of them; above: the k-th largest head.  (Lists past kPer,
        // which only candidate sets of more than 512 tokens have, are left out.)
        const bool groups = !kFew && a.k <= kGroupMaxK;
        const int q2 = a.k <= 1 ? 1 : 1 << (32 - __clz(a.k - 1));
        if (groups) {
#pragma unroll 1
            for (int o = 16; o >= q2; o >>= 1) {
                const uint64_t y = shfl_xor_u64(g, o);
                g = y > g ? y : g;
            }
        }
        heads[tid] = g;  // groups: of warp `warp`, group lane mod q2
        __syncthreads();
        const float gm = warp_max(redm2[half][lane % kWarps]);
        float part = acc.x == -INFINITY ? 0.0f : acc.y * __expf(acc.x - gm);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(kFull, part, o);
        if (lane == 0) redf2[half][warp] = part;
        uint64_t T = 0ull;
        if (groups) {
#pragma unroll 1
            for (int w = 0; w < kWarps; w++) {
                const uint64_t y = heads[w * 32 + (lane & (q2 - 1))];
                T = y > T ? y : T;
            }
#pragma unroll 1
            for (int o = q2 >> 1; o > 0; o >>= 1) {
                const uint64_t y = shfl_xor_u64(T, o);
                T = y < T ? y : T;
            }
        } else {
            const int nl = min(a.nV, kPer);
            if (g != 0ull && count_above(heads, nl, g) == (a.k + jth - 1) / jth - 1) thr2[half] = g;
            __syncthreads();
            T = thr2[half];
        }
        T = T > bound ? T : bound;
        {
            auto take = [&](uint64_t x) -> bool {
                if (x == 0ull || x < T) return false;
                const int pos = atomicAdd(&cnt2[half], 1);
                if (pos < kRankMax) surv[pos] = x;
                return true;
            };
            if constexpr (kFew) {
#pragma unroll 1
                for (int i0 = 0; i0 < a.nV * a.klist; i0 += kKeys * kPer) {
                    if (i0 > 0) load_keys(i0);
#pragma unroll
                    for (int u = 0; u < kKeys; u++) take(v[u]);
                }
            } else {
                bool more = take(v[0]) && take(v[1]) && take(v[2]) && take(v[3]);
#pragma unroll 1
                for (int r = tid, j = 4; mine && r < a.nV; r += kPer, j = 0, more = true) {
#pragma unroll 1
                    for (; more && j < a.klist; j += 4) {
                        load4(lists + r * a.klist + j, a.klist - j, wide, v);
                        more = take(v[0]) && take(v[1]) && take(v[2]) && take(v[3]);
                    }
                }
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int h = 0; h < nh; h++) {
            if (cnt2[h] > kRankMax) {
                radix_survivors(a.part_key + static_cast<size_t>(n + h - half) * stride, a.nV * a.klist, a.k,
                                survs + h * kRankMax, hist, scal);
                if (threadIdx.x == 0) cnt2[h] = a.k;
                __syncthreads();
            }
        }
        const int m = cnt2[half];
        if ((m & 1) && tid == 0) surv[m] = 0ull;  // (an odd m leaves room)
        float ssum = 0.0f;
#pragma unroll
        for (int i = 0; i < kWarps; i++) ssum += redf2[half][i];  // (in warp order)
        const float lse = gm == -INFINITY ? -INFINITY : gm + logf(ssum);
        const bool live = mine && p < prev_count;
        if (mine && tid == 0) {
            a.node_lse[n] = live ? lse : -INFINITY;
            if (a.lse_hist && live) a.lse_hist[static_cast<size_t>(n) * a.lse_hist_stride] = lse;
        }
        __syncthreads();
        if (live) {
#pragma unroll 1
            for (int i = tid; i < m; i += kPer) {
                const uint64_t x = surv[i];
                const int j = count_above(surv, m, x);
                if (j >= a.k) continue;
                const float z = key_val(x);
                const int tok = static_cast<int>(key_idx(x));
                const float lq = (lse != -INFINITY && z != -INFINITY) ? fminf(z - lse, 0.0f) : -INFINITY;
                a.node_logq[static_cast<size_t>(n) * a.k + j] = lq;
                a.node_tok[static_cast<size_t>(n) * a.k + j] = tok;
                const float sc = (ps + lq) + a.beta;  // Eq. 5, one more depth
                const int c = p * a.k + j;
                st_cluster_u64(fk0 + c * 8, 0, sc > -INFINITY ? make_key(sc, static_cast<uint32_t>(c)) : 0ull);
                if (search) st_cluster_s32(ft0 + c * 4, 0, tok);
            }
        } else if (mine && tid < a.k) {
            a.node_logq[static_cast<size_t>(n) * a.k + tid] = -INFINITY;
            a.node_tok[static_cast<size_t>(n) * a.k + tid] = -1;
        }
        __syncthreads();  // this node's buffers are free for the next
    }
    cluster_sync_all();
    if (rank != 0) return;
    // block 0: the top W of the candidates (p, j), sorted for every parent p
    const int t = threadIdx.x, nt = blockDim.x;
    const int ncand = prev_count * a.k;
    const size_t tb = (static_cast<size_t>(s) * a.L + a.dep - 1) * a.W;
    auto keep = [&](uint64_t x, int r) {
        const int c = static_cast<int>(key_idx(x));
        if (r >= a.W || !bounds_check(a.status, c < ncand)) return;
        const int pp = c / a.k, tok = search ? ftok[c] : __ldcg(a.node_tok + static_cast<size_t>(s) * a.P * a.k + c);
        a.tree_tok[tb + r] = tok;
        a.tree_parent[tb + r] = a.dep == 1 ? -1 : pp;
        a.tree_score[tb + r] = key_val(x);
        if (r < a.Pn) {
            a.child_prow[s * a.Pn + r] = s * a.P + pp;
            a.child_tok[s * a.Pn + r] = tok;
        }
    };
    int nvalid = 0;
    if (search) {
#pragma unroll 1
        for (int c0 = 0; c0 < ncand; c0 += nt) {
            const uint64_t x = c0 + t < ncand ? fkey[c0 + t] : 0ull;
            nvalid += __syncthreads_count(x != 0ull);
            if (x == 0ull) continue;
            int r = 0;
#pragma unroll 1
            for (int o = 0; o < prev_count; o++) r += count_greater(fkey + o * a.k, a.k, x);
            keep(x, r);
        }
    } else {
        // (nt >= P) at least W candidates reach the W-th largest list head
        if (t == 0) {
            cnt2[0] = 0;
            thr2[0] = 0ull;
        }
        uint64_t* fh = heads2[0];
        if (t < prev_count + 1) fh[t] = t < prev_count ? fkey[t * a.k] : 0ull;
        __syncthreads();
        if (t < prev_count && fh[t] != 0ull && count_above(fh, prev_count, fh[t]) == a.W - 1) thr2[0] = fh[t];
        for (int c0 = 0; c0 < ncand; c0 += nt) nvalid += __syncthreads_count(c0 + t < ncand && fkey[c0 + t] != 0ull);
        append_reaching(fkey, ncand, thr2[0], survs, &cnt2[0], t, nt);
        __syncthreads();
        int m = cnt2[0];
        if (m > kRankMax) {
            m = min(a.W, nvalid);
            radix_survivors(fkey, ncand, m, survs, hist, scal);
        }
        if ((m & 1) && t == 0) survs[m] = 0ull;
        __syncthreads();
        if (t < m) keep(survs[t], count_above(survs, m, survs[t]));
        if (t + nt < m) keep(survs[t + nt], count_above(survs, m, survs[t + nt]));
    }
    const int cnt = min(a.W, nvalid);
#pragma unroll 1
    for (int r = cnt + t; r < a.W; r += nt) {
        a.tree_tok[tb + r] = -1;
        a.tree_parent[tb + r] = -1;
        a.tree_score[tb + r] = -INFINITY;
        if (r < a.Pn) {
            a.child_prow[s * a.Pn + r] = -1;
            a.child_tok[s * a.Pn + r] = 0;
        }
    }
    if (t == 0) a.tree_count[s * a.L + a.dep - 1] = cnt;
}

// Only the log-sum-exp of each node (the same arithmetic), of the nodes with
// row_ent[n] >= 0, to lse[row_ent[n]] (sequential search).
__global__ void __launch_bounds__(kSelThreads) merge_lse_kernel(const float2* part_ms, int nV, const int* row_ent,
                                                                float* lse) {
    pdl_trigger();
    pdl_wait();
    __shared__ float redf[32];
    __shared__ float redm[32];
    const int n = blockIdx.x, tid = threadIdx.x;
    const int ent = __ldcg(row_ent + n);
    if (ent < 0) return;
    const float2* ms = part_ms + static_cast<size_t>(n) * nV;
    float2 acc = make_float2(-INFINITY, 0.0f);
    for (int r = tid + 2 * kSelThreads; r < nV; r += kSelThreads) acc = lse_merge(acc, __ldcg(ms + r));
    for (int r = tid; r < min(nV, 2 * kSelThreads); r += kSelThreads) acc = lse_merge(acc, __ldcg(ms + r));
    const float m = warp_max(acc.x);
    if ((tid & 31) == 0) redm[tid >> 5] = m;
    __syncthreads();
    float gm = -INFINITY;
    for (int i = 0; i < kSelThreads / 32; i++) gm = fmaxf(gm, redm[i]);
    const float ssum = block_sum_float(acc.x == -INFINITY ? 0.0f : acc.y * __expf(acc.x - gm), redf);
    if (tid == 0) lse[ent] = gm == -INFINITY ? -INFINITY : gm + logf(ssum);
}

__global__ void __launch_bounds__(kEmitThreads) prune_emit_kernel(const EmitArgs a) {
    pdl_trigger();
    pdl_wait();
    prune_emit_seq<kEmitThreads>(a, blockIdx.x);
}

// 4 consecutive floats -> 4 hi and 4 lo bf16 (8-byte stores)
__device__ __forceinline__ void split4(const float4 v, __nv_bfloat16* hi, __nv_bfloat16* lo) {
    __align__(8) __nv_bfloat16 h[4], l[4];
    split_bf16(v.x, h[0], l[0]);
    split_bf16(v.y, h[1], l[1]);
    split_bf16(v.z, h[2], l[2]);
    split_bf16(v.w, h[3], l[3]);
    *reinterpret_cast<uint2*>(hi) = *reinterpret_cast<const uint2*>(h);
    *reinterpret_cast<uint2*>(lo) = *reinterpret_cast<const uint2*>(l);
}

__global__ void prep_anchor_kernel(const float* anchor, int nseq, int d, float* h, __nv_bfloat16* HL, int bhalf,
                                   uint64_t* gthr_all, int n_gthr) {
    pdl_trigger();
    pdl_wait();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_gthr; i += gridDim.x * blockDim.x) gthr_all[i] = 0ull;
    const int q4 = d / 4;
    const int total = nseq * q4;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < total; u += gridDim.x * blockDim.x) {
        const int s = u / q4, j = (u % q4) * 4;
        const float4 x = *reinterpret_cast<const float4*>(anchor + static_cast<size_t>(s) * d + j);
        *reinterpret_cast<float4*>(h + static_cast<size_t>(s) * d + j) = x;
        if (HL) split4(x, HL + static_cast<size_t>(s) * d + j, HL + static_cast<size_t>(bhalf + s) * d + j);
    }
}

// X[c] = [h[prow[c]] ; E[tok[c]]]: one thread per 4 columns.
__global__ void gather_x_kernel(int Nc, int d, const int* prow, const int* tok, const float* h, const void* E,
                                int wbf16, __nv_bfloat16* XL, int bhalf, float* X32) {
    pdl_trigger();
    pdl_wait();
    const int q4 = (2 * d) / 4;
    const int total = Nc * q4;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < total; u += gridDim.x * blockDim.x) {
        const int c = u / q4, j = (u % q4) * 4;
        const int pr = prow[c];
        const size_t xo = static_cast<size_t>(c) * 2 * d + j;
        const size_t xl = static_cast<size_t>(bhalf + c) * 2 * d + j;
        if (j < d) {
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (pr >= 0) x = *reinterpret_cast<const float4*>(h + static_cast<size_t>(pr) * d + j);
            if (wbf16)
                split4(x, XL + xo, XL + xl);
            else
                *reinterpret_cast<float4*>(X32 + xo) = x;
        } else {
            const size_t eo = static_cast<size_t>(tok[c]) * d + (j - d);
            if (wbf16) {
                uint2 e = make_uint2(0u, 0u);
                if (pr >= 0) e = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(E) + eo);
                *reinterpret_cast<uint2*>(XL + xo) = e;
                *reinterpret_cast<uint2*>(XL + xl) = make_uint2(0u, 0u);
            } else {
                float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
                if (pr >= 0) e = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(E) + eo);
                *reinterpret_cast<float4*>(X32 + xo) = e;
            }
        }
    }
}

// v += p[0] + p[stride] + ... (n terms, in this order), with up to 8 of the
// 16-byte loads in flight at once (a plain loop issues them one at a time).
__device__ __forceinline__ void add_splits(float4& v, const float* p, size_t stride, int n) {
    constexpr int kBatch = 8;
    for (int s0 = 0; s0 < n; s0 += kBatch) {
        float4 w[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; u++)
            if (s0 + u < n) w[u] = *reinterpret_cast<const float4*>(p + static_cast<size_t>(s0 + u) * stride);
#pragma unroll
        for (int u = 0; u < kBatch; u++) {
            if (s0 + u < n) {
                v.x += w[u].x;
                v.y += w[u].y;
                v.z += w[u].z;
                v.w += w[u].w;
            }
        }
    }
}

__global__ void silu_split_kernel(int Nc, int d, int S, const float* part, __nv_bfloat16* AL, int bhalf, float* A32) {
    pdl_trigger();
    pdl_wait();
    const size_t total = static_cast<size_t>(Nc) * d;
    const size_t t4 = total / 4;
    for (size_t u = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; u < t4;
         u += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const size_t q = u * 4;
        float4 v = *reinterpret_cast<const float4*>(part + q);
        add_splits(v, part + total + q, total, S - 1);
        v.x = v.x / (1.0f + expf(-v.x));
        v.y = v.y / (1.0f + expf(-v.y));
        v.z = v.z / (1.0f + expf(-v.z));
        v.w = v.w / (1.0f + expf(-v.w));
        if (AL)
            split4(v, AL + q, AL + static_cast<size_t>(bhalf) * d + q);
        else
            *reinterpret_cast<float4*>(A32 + q) = v;
    }
}

// First head layer with the E half taken from the per-token table
// Q[t] = W_i[:, d:2d] . E[t] (computed once per handle):
//   a_c = SiLU(Q[tok[c]] + sum_s part[s][prow[c]]),
// where part holds the S k-split partials of W_i[:, 0:d] . h over the Np
// parents, then the hi/lo bf16 split of a_c (input of the W_o GEMM).  Empty
// child slots (prow < 0) and tokens outside [0, V) give a_c = 0.
__global__ void gather_silu_kernel(int Nc, int d, int S, int Np, const float* part, const int* prow, const int* tok,
                                   int V, const float* Q, __nv_bfloat16* AL, int bhalf, int* status) {
    pdl_trigger();
    pdl_wait();
    const size_t stride = static_cast<size_t>(Np) * d;
    const int q4 = d / 4;
    const int total = Nc * q4;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < total; u += gridDim.x * blockDim.x) {
        const int c = u / q4, j = (u % q4) * 4;
        int pr = prow[c];
        const int t = tok[c];
        if (pr >= 0 && !bounds_check(status, pr < Np && static_cast<unsigned>(t) < static_cast<unsigned>(V))) pr = -1;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (pr >= 0 && static_cast<unsigned>(t) < static_cast<unsigned>(V)) {
            v = *reinterpret_cast<const float4*>(Q + static_cast<size_t>(t) * d + j);
            add_splits(v, part + static_cast<size_t>(pr) * d + j, stride, S);
            v.x = v.x / (1.0f + expf(-v.x));
            v.y = v.y / (1.0f + expf(-v.y));
            v.z = v.z / (1.0f + expf(-v.z));
            v.w = v.w / (1.0f + expf(-v.w));
        }
        split4(v, AL + static_cast<size_t>(c) * d + j, AL + static_cast<size_t>(bhalf + c) * d + j);
    }
}

// One block per child: r = h[prow] + sum_s part[s], h_next = r / rms(r).
// NT = 1024 threads when S partial tiles are summed (many loads in flight),
// 256 for one summed tile (few registers, so blocks can become resident
// beside the GEMM before it ends).  kIt: float4 columns per thread, no more
// than d needs, since the code is cold at every depth (one kernel for every d
// was 20 to 55 KB).  Measured on GB300 against that one (µs per round, same
// box): 3 x 11 nodes, d = 1088 565 -> 533, 64 nodes, d = 2560 2703 -> 2689,
// 16 nodes, K = 64 466 -> 462; a cluster of four blocks per child was slower
// where the LM-head follows (8 nodes 2071 -> 2096).
template <int NT, int kIt>
__global__ void __launch_bounds__(NT) residual_norm_kernel(int d, int S, int Nc, const float* part, const int* prow,
                                                           const float* h, float eps, float* h_next,
                                                           __nv_bfloat16* HL, int bhalf) {
    pdl_trigger();
    pdl_wait();
    __shared__ float red[32];
    const int c = blockIdx.x, lane = threadIdx.x & 31;
    const int pr = prow[c];
    const size_t total = static_cast<size_t>(Nc) * d;
    float4 r[kIt], q[kIt];
#pragma unroll
    for (int it = 0; it < kIt; it++) {
        const int j = (it * NT + threadIdx.x) * 4;
        r[it] = q[it] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j < d && pr >= 0) {
            r[it] = *reinterpret_cast<const float4*>(h + static_cast<size_t>(pr) * d + j);
            q[it] = *reinterpret_cast<const float4*>(part + static_cast<size_t>(c) * d + j);
        }
    }
    float ss = 0.0f;
#pragma unroll
    for (int it = 0; it < kIt; it++) {
        const int j = (it * NT + threadIdx.x) * 4;
        float4 v = r[it];
        v.x += q[it].x;
        v.y += q[it].y;
        v.z += q[it].z;
        v.w += q[it].w;
        if (NT == 1024 && j < d && pr >= 0) add_splits(v, part + static_cast<size_t>(c) * d + j + total, total, S - 1);
        r[it] = v;
        ss = __fadd_rn(ss, fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.y, v.y, __fmul_rn(v.x, v.x)))));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(kFull, ss, o);
    if (lane == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.0f;
#pragma unroll 8
    for (int i = 0; i < NT / 32; i++) tot += red[i];
    const float inv = 1.0f / sqrtf(tot / static_cast<float>(d) + eps);
#pragma unroll
    for (int it = 0; it < kIt; it++) {
        const int j = (it * NT + threadIdx.x) * 4;
        if (j < d) {
            const float4 v = make_float4(r[it].x * inv, r[it].y * inv, r[it].z * inv, r[it].w * inv);
            *reinterpret_cast<float4*>(h_next + static_cast<size_t>(c) * d + j) = v;
            if (HL) split4(v, HL + static_cast<size_t>(c) * d + j, HL + static_cast<size_t>(bhalf + c) * d + j);
        }
    }
}

}  // namespace

bool pdl_enabled() { return true; }

// Launch shape: 256 threads per node up to 256 vocabulary ranges, else 512.
// Two nodes per block, so that a cluster is small (it starts when all of its
// blocks fit on one GPC at once), four where more than 16 blocks were needed.
// Measured on GB300 (µs per round): 16 nodes, k = 16: 3422 with one or two
// nodes per block, 3441 with four.
struct MergePlan {
    int per, nh, cs, npb, smem;
};
static MergePlan merge_plan(int P, int nV, int k) {
    MergePlan m;
    m.per = nV <= 256 ? 256 : 512;
    m.nh = std::min({P, P <= 2 * kMergeCluster ? 2 : 4, kMergeThreads / m.per});
    const int cs = std::min((P + m.nh - 1) / m.nh, kMergeCluster);
    m.npb = (P + cs - 1) / cs;
    m.cs = (P + m.npb - 1) / m.npb;
    m.smem = (m.nh * kRankMax + ((P * k + 1) & ~1)) * 8 + (P <= kMergeSearchP ? P * k * 4 : 0);
    return m;
}

int merge_select_smem(int P, int nV, int k) { return merge_plan(P, nV, k).smem; }

cudaError_t select_set_smem_limits() {
    cudaError_t e = cudaSuccess;
    for (const void* fn : {reinterpret_cast<const void*>(merge_select_kernel<256, false>),
                           reinterpret_cast<const void*>(merge_select_kernel<512, false>),
                           reinterpret_cast<const void*>(merge_select_kernel<256, true>)}) {
        if (e == cudaSuccess) e = set_max_dynamic_smem(fn);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    }
    return e;
}

cudaError_t launch_merge_select(const SelectArgs& a, cudaStream_t st) {
    const MergePlan m = merge_plan(a.P, a.nV, a.k);
    return launch_pdl_cluster(a.nV < a.k     ? merge_select_kernel<256, true>  // (k <= 64: m.per is 256)
                              : m.per == 256 ? merge_select_kernel<256, false>
                                             : merge_select_kernel<512, false>,
                              dim3(a.nseq * m.cs), dim3(m.nh * m.per), m.smem, st, m.cs, a, m.cs, m.npb);
}

cudaError_t launch_merge_lse(const float2* part_ms, int N, int nV, const int* row_ent, float* lse, cudaStream_t st) {
    return launch_pdl(merge_lse_kernel, dim3(N), dim3(kSelThreads), 0, st, part_ms, nV, row_ent, lse);
}

cudaError_t launch_prune_emit(const EmitArgs& a, cudaStream_t st) {
    return launch_pdl(prune_emit_kernel, dim3(a.nseq), dim3(kEmitThreads), 0, st, a);
}

static int grid_for(size_t units) {
    size_t b = (units + 255) / 256;
    return static_cast<int>(b < 1 ? 1 : (b > 2048 ? 2048 : b));
}

cudaError_t launch_prep_anchor(const float* anchor, int nseq, int d, float* h, __nv_bfloat16* HL, int bhalf,
                               uint64_t* gthr_all, int n_gthr, cudaStream_t st) {
    return launch_pdl(prep_anchor_kernel, dim3(grid_for(static_cast<size_t>(nseq) * d / 4)), dim3(256), 0, st, anchor,
                      nseq, d, h, HL, bhalf, gthr_all, n_gthr);
}

cudaError_t launch_gather_x(int Nc, int d, const int* prow, const int* tok, const float* h, const void* E,
                            int wbf16, __nv_bfloat16* XL, int bhalf, float* X32, cudaStream_t st) {
    return launch_pdl(gather_x_kernel, dim3(grid_for(static_cast<size_t>(Nc) * 2 * d / 4)), dim3(256), 0, st, Nc, d,
                      prow, tok, h, E, wbf16, XL, bhalf, X32);
}

cudaError_t launch_silu_split(int Nc, int d, int S, const float* part, __nv_bfloat16* AL, int bhalf, float* A32,
                              cudaStream_t st) {
    return launch_pdl(silu_split_kernel, dim3(grid_for(static_cast<size_t>(Nc) * d / 4)), dim3(256), 0, st, Nc, d, S,
                      part, AL, bhalf, A32);
}

cudaError_t launch_gather_silu(int Nc, int d, int S, int Np, const float* part, const int* prow, const int* tok,
                               int V, const float* Q, __nv_bfloat16* AL, int bhalf, int* status, cudaStream_t st) {
    return launch_pdl(gather_silu_kernel, dim3(grid_for(static_cast<size_t>(Nc) * d / 4)), dim3(256), 0, st, Nc, d, S,
                      Np, part, prow, tok, V, Q, AL, bhalf, status);
}

namespace {
// One thread evaluates one index check that fails (idx = n): the bounds bit
// is set in debug builds; nothing happens in release builds.  No memory but
// the status word is touched.
__global__ void bounds_probe_kernel(int* status, int idx, int n) { (void)bounds_check(status, idx < n); }
}  // namespace

cudaError_t launch_bounds_probe(int* status, cudaStream_t st) {
    bounds_probe_kernel<<<1, 1, 0, st>>>(status, 1, 1);
    return cudaGetLastError();
}

bool debug_build() {
#ifdef DART_DEBUG
    return true;
#else
    return false;
#endif
}

cudaError_t launch_residual_norm(int Nc, int d, int S, const float* part, const int* prow, const float* h,
                                 float eps, float* h_next, __nv_bfloat16* HL, int bhalf, cudaStream_t st) {
    const int NT = S > 1 ? 1024 : 256;
    const int its = (d / 4 + NT - 1) / NT;  // (d <= 16384)
    const auto fn = S > 1 ? (its <= 1   ? residual_norm_kernel<1024, 1>
                             : its <= 2 ? residual_norm_kernel<1024, 2>
                                        : residual_norm_kernel<1024, 4>)
                          : (its <= 2   ? residual_norm_kernel<256, 2>
                             : its <= 4 ? residual_norm_kernel<256, 4>
                                        : residual_norm_kernel<256, 16>);
    return launch_pdl(fn, dim3(Nc), dim3(NT), 0, st, d, S, Nc, part, prow, h, eps, h_next, HL, bhalf);
}

}  // namespace dart
