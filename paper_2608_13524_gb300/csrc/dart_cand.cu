// Candidate-restricted scoring (Algorithm 1 with a candidate-vocabulary size
// K > 0; the paper's default is K = 64):
//
//   cand_topk   C_d = TopK(L_d^base, K): for every (sequence, position) row
//               of the drafter logits, the K tokens with the largest base
//               logit (ties: token asc), written in ascending token order.
//               Once per round, for all L positions.
//   cand_score  for every node n of S_{d-1} and every candidate c of its
//               sequence's C_d: z = (Dlog[d-1][c] + E[c] . h_n) / T', in fp32
//               on CUDA cores (the dot products are K*N*d, far too small for
//               the tensor cores to matter).  Written in the LM-head's
//               partial format with one single-key list per candidate:
//               part_ms[n][i] = (z, 1), part_key[n][i] = key(z, c), so the
//               merge kernel computes log-sum-exp over C_d (q~ renormalised
//               over the candidates) and the node's top-k unchanged.
#include <algorithm>
#include <type_traits>

#include "dart_device.cuh"
#include "dart_kernels.h"

namespace dart {

namespace {

constexpr int kTopkThreads = 1024;
constexpr int kDigitBits = 12;
constexpr int kBins = 1 << kDigitBits;  // histogram bins per radix pass
constexpr int kCollCap = 8192;          // keys of the threshold bin finished in shared memory (radix path)

// Returns, in lanes of warp 0, the largest digit b with
// sum_{b' >= b} hist[b'] >= need (need >= 1), and the count above b.
__device__ __forceinline__ void find_digit(const uint32_t* hist, int need, int* out) {
    const int lane = threadIdx.x & 31;
    constexpr int kPer = kBins / 32;
    // lane l owns bins [kBins - (l+1)*kPer, kBins - l*kPer), highest first
    uint32_t sum = 0;
    for (int j = 0; j < kPer; j++) sum += hist[kBins - 1 - lane * kPer - j];
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
    }
    const unsigned hit = __ballot_sync(0xFFFFFFFFu, incl >= static_cast<uint32_t>(need));
    const int first = __ffs(hit) - 1;  // some lane always hits: the row holds >= need keys
    if (lane == first) {
        uint32_t cum = incl - sum;
        int b = kBins - 1 - lane * kPer;
        for (int j = 0; j < kPer; j++, b--) {
            const uint32_t c = hist[b];
            if (cum + c >= static_cast<uint32_t>(need)) break;
            cum += c;
        }
        out[0] = b;
        out[1] = static_cast<int>(cum);
    }
}

// Loads in flight per thread in the row passes (the row streams from HBM on
// the first pass; one load at a time would make it latency-bound).
constexpr int kRowBatch = 8;

// Calls f(value, token) for every element of this thread's strided share of
// the row, with kRowBatch 16-byte loads in flight when the row is 16-byte
// aligned (else 4-byte loads).
template <typename F>
__device__ __forceinline__ void for_row(const float* x, int V, F&& f) {
    const int tid = threadIdx.x;
    if ((V & 3) == 0 && (reinterpret_cast<uintptr_t>(x) & 15u) == 0) {
        const int V4 = V >> 2;
        const float4* x4 = reinterpret_cast<const float4*>(x);
        for (int q0 = tid; q0 < V4; q0 += kRowBatch * kTopkThreads) {
            float4 xs[kRowBatch];
#pragma unroll
            for (int u = 0; u < kRowBatch; u++) {
                const int q = q0 + u * kTopkThreads;
                xs[u] = q < V4 ? __ldg(x4 + q) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < kRowBatch; u++) {
                const int q = q0 + u * kTopkThreads;
                if (q < V4) {
                    f(xs[u].x, 4 * q);
                    f(xs[u].y, 4 * q + 1);
                    f(xs[u].z, 4 * q + 2);
                    f(xs[u].w, 4 * q + 3);
                }
            }
        }
    } else {
        for (int v0 = tid; v0 < V; v0 += 4 * kRowBatch * kTopkThreads) {
            float xs[4 * kRowBatch];
#pragma unroll
            for (int u = 0; u < 4 * kRowBatch; u++) {
                const int v = v0 + u * kTopkThreads;
                xs[u] = v < V ? __ldg(x + v) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4 * kRowBatch; u++) {
                const int v = v0 + u * kTopkThreads;
                if (v < V) f(xs[u], v);
            }
        }
    }
}

// S blocks per (sequence, position) row, block j taking the slice
// [V j / S, V (j + 1) / S) of the row; keys key(x, v) order by (value desc,
// token asc).  Every block finds the exact top min(K, slice) keys of its
// slice; the global top K is among them.  Pass 1: every thread finds the
// largest value of its share of the slice and makes a key of it.  Bound T: in every warp the m-th largest of these maxima
// (m = ceil(K/32), warp bitonic sort), minimised over the warps -- at least
// 32*m >= K threads hold a key >= T, so the K-th largest key is >= T, and
// only a small multiple of K keys reach it.  Pass 2 gathers the keys >= T
// (the slice is now in L2) and the top K of them are ranked in shared
// memory.  Both passes compare floats (with one block per row the instructions
// per element bound them: 128 rows of 151936, K = 64, on GB300: 40.9 µs with a
// key made and compared for every element, 34.1 now).  If more than kCollCap keys reach T (pathological rows, e.g. many
// equal values), an exact radix select over the slice decides instead: 12
// bits per pass from the top, the keys above the threshold digit taken, and
// once the threshold digit holds at most kCollCap keys they are gathered for
// an in-memory select.  With S > 1 each block publishes its keys (zeros past
// its count) and the last block of the row to finish (atomic ticket; nobody
// waits) selects the K largest of the S K published keys.
__global__ void __launch_bounds__(kTopkThreads)
    cand_topk_kernel(const float* dlog, int V, int K, int S, int* cand_tok, uint64_t* part, int* ticket,
                     int by_value, long long out_stride, float* out_val, const int* out_row) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ uint64_t csm[];
    uint64_t* coll = csm;                                       // [kCollCap]
    uint64_t* out = coll + kCollCap;                            // [K]
    uint64_t* surv = out + K;                                   // [kRankMax]
    uint32_t* hist = reinterpret_cast<uint32_t*>(surv + kRankMax);  // [kBins]
    __shared__ uint32_t hist8[256];
    __shared__ int scal[4];
    __shared__ uint64_t wmin[kTopkThreads / 32];
    __shared__ int dig[2];
    __shared__ int cnt[2];  // [0] keys taken into out, [1] keys gathered into coll
    __shared__ int last;
    const int row = blockIdx.x / S, sl = blockIdx.x % S;
    const int orow = out_row ? __ldcg(out_row + row) : row;
    if (orow < 0) return;  // nothing to select for this row
    const int v0 = static_cast<int>(static_cast<long long>(V) * sl / S);
    const int Vs = static_cast<int>(static_cast<long long>(V) * (sl + 1) / S) - v0;
    const int Kl = min(K, Vs);  // keys this block selects from its slice
    const float* x = dlog + static_cast<size_t>(row) * V + v0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) cnt[0] = cnt[1] = 0;
    // pass 1: the key of this thread's largest value (any of its keys would do for the bound)
    float best = 0.0f;
    int at = -1;
    for_row(x, Vs, [&](float xv, int v) {
        if (at < 0 || xv > best) {
            best = xv;
            at = v;
        }
    });
    const uint64_t mx = at < 0 ? 0ull : make_key(best, static_cast<uint32_t>(v0 + at));
    {
        const int m = (Kl + 31) / 32;
        uint64_t hv = mx;
#pragma unroll
        for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                const uint64_t y = shfl_xor_u64(hv, stride);
                const bool desc_block = (lane & size) == 0;
                const bool lower = (lane & stride) == 0;
                hv = (lower == desc_block) ? (hv > y ? hv : y) : (hv < y ? hv : y);
            }
        }
        const uint64_t mth = shfl_u64(hv, m - 1);
        if (lane == 0) wmin[warp] = mth;
    }
    __syncthreads();
    uint64_t T = wmin[0];
    for (int w = 1; w < kTopkThreads / 32; w++) T = wmin[w] < T ? wmin[w] : T;
    // pass 2: gather every key >= T
    const float tv = key_val(T);
    for_row(x, Vs, [&](float xv, int v) {
        if (xv < tv) return;  // (a NaN on either side is left to the keys)
        const uint64_t k = make_key(xv, static_cast<uint32_t>(v0 + v));
        if (k >= T) {
            const int pos = atomicAdd(&cnt[1], 1);
            if (pos < kCollCap) coll[pos] = k;
        }
    });
    __syncthreads();
    const int ng = cnt[1];
    const bool inexact = ng > kCollCap;
    __syncthreads();  // every thread has read the count before it is reused
    if (!inexact) {
        // the Kl largest of the ng gathered keys (ng >= Kl, keys distinct)
        if (ng <= kRankMax) {
            for (int i = tid; i < ng; i += kTopkThreads) {
                const uint64_t k = coll[i];
                int r = 0;
                for (int j = 0; j < ng; j++) r += coll[j] > k;
                if (r < Kl) out[r] = k;
            }
        } else {
            const uint64_t kth = block_kth_largest(coll, ng, Kl, hist8, scal);
            for (int i = tid; i < ng; i += kTopkThreads)
                if (coll[i] >= kth) out[atomicAdd(&cnt[0], 1)] = coll[i];
        }
        __syncthreads();
    }
    if (inexact) {
        if (tid == 0) cnt[0] = cnt[1] = 0;
        __syncthreads();
        uint64_t prefix = 0, mask = 0;
        int need = Kl;
        // at most 6 passes: after the 4-bit sixth digit the prefix is the whole
        // key, which is unique, so the threshold digit holds <= 1 key
        for (int level = 0, shift = 64 - kDigitBits; level < 6; level++, shift -= kDigitBits) {
            const int sh = shift > 0 ? shift : 0;
            const uint64_t dmask = (shift > 0 ? static_cast<uint64_t>(kBins - 1) : ((1ull << (kDigitBits + shift)) - 1));
            for (int i = tid; i < kBins; i += kTopkThreads) hist[i] = 0;
            __syncthreads();
            for (int v = tid; v < Vs; v += kTopkThreads) {
                const uint64_t k = make_key(__ldg(x + v), static_cast<uint32_t>(v0 + v));
                if ((k & mask) == prefix) atomicAdd(&hist[(k >> sh) & dmask], 1u);
            }
            __syncthreads();
            if (tid < 32) find_digit(hist, need, dig);
            __syncthreads();
            const uint64_t b = static_cast<uint64_t>(dig[0]);
            const int above = dig[1];
            const int m = static_cast<int>(hist[b]);
            const bool finish = m <= kCollCap;
            for (int v = tid; v < Vs; v += kTopkThreads) {
                const uint64_t k = make_key(__ldg(x + v), static_cast<uint32_t>(v0 + v));
                if ((k & mask) != prefix) continue;
                const uint64_t dg = (k >> sh) & dmask;
                if (dg > b)
                    out[atomicAdd(&cnt[0], 1)] = k;
                else if (dg == b && finish)
                    coll[atomicAdd(&cnt[1], 1)] = k;
            }
            __syncthreads();
            need -= above;
            if (finish) {
                // the `need` largest of the m gathered keys (keys are distinct)
                const uint64_t kth = need < m ? block_kth_largest(coll, m, need, hist8, scal) : 0ull;
                for (int i = tid; i < m; i += kTopkThreads)
                    if (coll[i] >= kth) out[atomicAdd(&cnt[0], 1)] = coll[i];
                __syncthreads();
                break;
            }
            prefix |= b << sh;
            mask |= dmask << sh;
            __syncthreads();
        }
    }
    if (S > 1) {
        // publish this slice's keys; the last block of the row merges
        uint64_t* pp = part + (static_cast<size_t>(row) * S + sl) * K;
        for (int i = tid; i < K; i += kTopkThreads) pp[i] = i < Kl ? out[i] : 0ull;
        __threadfence();
        __syncthreads();
        if (tid == 0) last = atomicAdd(&ticket[row], 1) == S - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (tid == 0) {
            ticket[row] = 0;
            cnt[0] = 0;
        }
        // S K <= kCollCap keys, non-zero ones distinct, at least K of them
        const int ng = S * K;
        const uint64_t* rp = part + static_cast<size_t>(row) * S * K;
        for (int i = tid; i < ng; i += kTopkThreads) coll[i] = __ldcg(rp + i);
        __syncthreads();
        const uint64_t kth = block_kth_largest(coll, ng, K, hist8, scal);
        for (int i = tid; i < ng; i += kTopkThreads)
            if (coll[i] >= kth && coll[i] != 0ull) out[atomicAdd(&cnt[0], 1)] = coll[i];
        __syncthreads();
    }
    // write the K tokens in ascending token order, or (by_value) best first
    // with their values (rank by counting; keys are distinct)
    for (int i = tid; i < K; i += kTopkThreads) {
        const uint32_t tk = key_idx(out[i]);
        int r = 0;
        if (by_value) {
            for (int j = 0; j < K; j++) r += out[j] > out[i];
        } else {
            for (int j = 0; j < K; j++) r += key_idx(out[j]) < tk;
        }
        cand_tok[static_cast<size_t>(orow) * out_stride + r] = static_cast<int>(tk);
        if (out_val) out_val[static_cast<size_t>(orow) * out_stride + r] = key_val(out[i]);
    }
}

constexpr int kScoreWarps = 8;  // candidates per group of cand_score_slices
constexpr int kScoreNodes = 8;  // nodes per warp tile
constexpr int kScoreThreads = 256;
constexpr int kScoreCluster = 16;

// A cluster of cs blocks per (sequence, G = 4 CT candidates); the d-slices
// ds = 0 .. DS - 1 are dealt to its blocks, DS / cs in a row each.  A block
// stages the slice of its sequence's node states in shared memory (PC nodes
// at a time), and each warp forms a tile of CT candidates x 8 nodes of
// partial dot products: a lane-strided partial sum in fixed order, then a
// butterfly.  After a cluster barrier the blocks sum the DS slices in order,
// through distributed shared memory, and write the merge kernel's lists:
// deterministic, and the same sums whatever CT, PC and cs.
// Bound by latency for few nodes (CT = 2: every warp of a small block has a
// tile) and by shared-memory reads and FMAs for many (CT = 4: 32 FMAs x 4 per
// 36 wavefronts); the E elements of a warp's next 4 x 128 columns are loaded
// before it waits or computes.  Measured on GB300, K = 64, d = 4096 (events
// around the launch, µs): 8 x 32 nodes 45.5 with one candidate x 8 nodes per
// warp and the slices summed by a last block through global memory, 16.6 now;
// 16 nodes 14.0, 10.6 now.
template <bool kBf16, int CT>
__global__ void __launch_bounds__(kScoreThreads) cand_score_kernel(const CandArgs a, int cs, int PC) {
    pdl_trigger();
    constexpr int G = 4 * CT, kST = kBf16 ? 4 : 2, kNw = kScoreThreads / 32;
    using Raw = typename std::conditional<kBf16, uint2, float4>::type;  // 4 elements of E
    extern __shared__ __align__(16) float hs[];  // [PC][dchunk], then the partial sums [spc][P][G + 1]
    __shared__ int tok[G];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ngroups = (a.K + G - 1) / G;
    const int r = blockIdx.x % cs, sg = blockIdx.x / cs;
    const int cg = sg % ngroups, s = sg / ngroups;
    const int d = a.d, P = a.P, dchunk = d / a.DS, q = dchunk / 4, spc = a.DS / cs;
    float* pt = hs + PC * dchunk;
    const size_t crow = (static_cast<size_t>(s) * a.L + a.dep - 1) * a.K;
    // Before the wait: E never changes, so the candidates' rows are requested
    // into L2 with whatever tokens the lists hold now (complete but at the
    // first depth; a stale one only warms the wrong row).
    constexpr int esz = kBf16 ? 2 : 4;
    const int lines = (spc * dchunk * esz + 127) / 128;
#pragma unroll 1
    for (int u = tid; u < G * lines; u += kScoreThreads) {
        const int ii = cg * G + u / lines;
        const int t = ii < a.K ? __ldcg(a.cand_tok + crow + ii) : -1;
        if (static_cast<unsigned>(t) < static_cast<unsigned>(a.V))
            asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char*>(a.E) +
                                                          (static_cast<size_t>(t) * d + r * spc * dchunk) * esz +
                                                          (u % lines) * 128));
    }
    pdl_wait();
    if (tid < G) {
        // a token outside the vocabulary would mean corrupted candidate lists:
        // it is never dereferenced (its score is -inf)
        const int t = cg * G + tid < a.K ? __ldcg(a.cand_tok + crow + cg * G + tid) : -1;
        tok[tid] = static_cast<unsigned>(t) < static_cast<unsigned>(a.V) ? t : -1;
    }
    __syncthreads();
    const int nb = (dchunk + 128 * kST - 1) / (128 * kST);  // column steps of a tile
#pragma unroll 1
    for (int u = 0; u < spc * ((P + PC - 1) / PC); u++) {
        const int sl = u % spc, pc0 = u / spc * PC, np = min(PC, P - pc0);
        const int j0 = (r * spc + sl) * dchunk;
        const float* src = a.h + (static_cast<size_t>(s) * P + pc0) * d + j0;
        const int tiles = 4 * ((np + kScoreNodes - 1) / kScoreNodes);
        const int items = warp < tiles ? ((tiles - 1 - warp) / kNw + 1) * nb : 0;
        Raw raw[kST][CT];
        auto load_e = [&](int it) {
            const int c0 = ((warp + it / nb * kNw) & 3) * CT, jb = it % nb * 128 * kST + lane * 4;
#pragma unroll
            for (int c = 0; c < CT; c++) {
                const char* row = static_cast<const char*>(a.E) + (static_cast<size_t>(max(tok[c0 + c], 0)) * d + j0) * esz;
#pragma unroll
                for (int st = 0; st < kST; st++)
                    if (jb + st * 128 < dchunk)
                        raw[st][c] = __ldg(reinterpret_cast<const Raw*>(row + (jb + st * 128) * esz));
            }
        };
        if (items > 0) load_e(0);
        if (u > 0) __syncthreads();  // the previous slice's states are no longer read
#pragma unroll 4
        for (int x = tid; x < np * q; x += kScoreThreads) {
            const int p = x / q, jj = (x - p * q) * 4;
            *reinterpret_cast<float4*>(hs + p * dchunk + jj) =
                *reinterpret_cast<const float4*>(src + static_cast<size_t>(p) * d + jj);
        }
        __syncthreads();
        float acc[CT * kScoreNodes];
#pragma unroll 1
        for (int it = 0; it < items; it++) {
            const int t = warp + it / nb * kNw, c0 = (t & 3) * CT, p0 = (t >> 2) * kScoreNodes;
            const int ib = it % nb, jb = ib * 128 * kST + lane * 4;
            if (ib == 0) {
#pragma unroll
                for (int x = 0; x < CT * kScoreNodes; x++) acc[x] = 0.0f;
            }
#pragma unroll
            for (int st = 0; st < kST; st++) {
                const int j = jb + st * 128;
                if (j >= dchunk) continue;
                float4 ev[CT];
#pragma unroll
                for (int c = 0; c < CT; c++) {
                    if constexpr (kBf16) {
                        const __nv_bfloat162 e01 = *reinterpret_cast<const __nv_bfloat162*>(&raw[st][c].x);
                        const __nv_bfloat162 e23 = *reinterpret_cast<const __nv_bfloat162*>(&raw[st][c].y);
                        ev[c] = make_float4(__low2float(e01), __high2float(e01), __low2float(e23), __high2float(e23));
                    } else {
                        ev[c] = raw[st][c];
                    }
                }
#pragma unroll
                for (int pp = 0; pp < kScoreNodes; pp++) {
                    const float4 hv = *reinterpret_cast<const float4*>(hs + min(p0 + pp, np - 1) * dchunk + j);
#pragma unroll
                    for (int c = 0; c < CT; c++) {
                        float v = acc[c * kScoreNodes + pp];
                        v = fmaf(ev[c].x, hv.x, v);
                        v = fmaf(ev[c].y, hv.y, v);
                        v = fmaf(ev[c].z, hv.z, v);
                        acc[c * kScoreNodes + pp] = fmaf(ev[c].w, hv.w, v);
                    }
                }
            }
            if (it + 1 < items) load_e(it + 1);
            if (ib + 1 < nb) continue;
            auto put = [&](int x, float v) {
                const int c = c0 + x / kScoreNodes, p = p0 + x % kScoreNodes;
                if (p < np) pt[(sl * P + pc0 + p) * (G + 1) + c] = v;
            };
            if constexpr (CT == 2) {
                const float v = bfly16<false>(acc, lane);
                if (!(lane & 1)) put(lane >> 1, v);
            } else {
                warp_reduce_scatter32(acc, lane);
                put(lane, acc[0]);
            }
        }
    }
    cluster_sync_all();  // every slice's partial sums are in place
    const int stride = part_stride(a.K, 1);
    const uint32_t base = smem_u32(pt);
    const int per = (P * G + cs - 1) / cs;  // (node, candidate) pairs summed by each block
#pragma unroll 1
    for (int u = r * per + tid; u < min(P * G, (r + 1) * per); u += kScoreThreads) {
        const int p = u / G, c = u % G, ii = cg * G + c;
        if (ii >= a.K) continue;
        float dot = 0.0f;
#pragma unroll 8
        for (int ds = 0; ds < a.DS; ds++)
            dot += ld_cluster_f32(base + (((ds % spc) * P + p) * (G + 1) + c) * 4, static_cast<uint32_t>(ds / spc));
        const int n = s * P + p, tk = tok[c];
        const float dl = tk >= 0 ? a.dlog[static_cast<size_t>(s) * a.dlog_seq_stride + a.dlog_row_off + tk] : -INFINITY;
        float z = tk >= 0 ? (dl + dot) * a.invT : -INFINITY;
        if (z == 0.0f) z = 0.0f;  // -0 -> +0
        a.part_ms[static_cast<size_t>(n) * a.K + ii] =
            z == -INFINITY ? make_float2(-INFINITY, 0.0f) : make_float2(z, 1.0f);
        a.part_key[static_cast<size_t>(n) * stride + ii] =
            make_key(z, static_cast<uint32_t>(tk >= 0 ? tk : __ldcg(a.cand_tok + crow + ii)));
    }
    cluster_sync_all();  // no block leaves while a peer reads its partial sums
}

}  // namespace

int cand_topk_smem(int K) { return (kCollCap + K + kRankMax) * 8 + kBins * 4; }

// Blocks per row of the candidate top-K: slices of at least 4096 logits
// (several per thread of the block), at most 8, S K keys within the merge's
// shared-memory buffer, and rows x S within one block per SM (measured on
// GB300: 8 slices of 16 rows -2 % per round at K = 64; 8 slices of 128 rows,
// several waves, +2.4 %).
int cand_topk_slices(int V, int K, int rows, int num_sms) {
    const int s = std::min(std::min(8, V / 4096), std::min(kCollCap / K, num_sms / std::max(rows, 1)));
    return std::max(1, s);
}

int cand_score_slices(int P, int d, int nseq, int K, int max_smem) {
    // Slices of d: enough (slice, group of 8 candidates) units to spread the
    // loads (>= 128; with kScoreManyNodes nodes the groups are of 16), a slice
    // of all P states within 64 KB, and d / DS a multiple of 4 floats.  A
    // slice of all P states above max_smem (d = 64 * an odd number, large) is
    // not supported, although the kernel stages PC of them at a time.
    const int ngroups = (K + kScoreWarps - 1) / kScoreWarps;
    int DS = 1;
    while (d % (8 * DS) == 0 &&
           (static_cast<long long>(P) * (d / DS) * 4 > 64 * 1024 || nseq * ngroups * DS < 128))
        DS *= 2;
    if (static_cast<long long>(P) * (d / DS) * 4 > max_smem) return 0;
    return DS;
}

// Tiles of 4 candidates for many nodes, of 2 (more blocks and warps) for few.
constexpr int kScoreManyNodes = 64;
constexpr int kScoreStage = 64 * 1024;  // shared memory for the staged states, at most

using ScoreKernel = void (*)(const CandArgs, int, int);
static ScoreKernel score_kernel(bool bf16, bool many) {
    if (bf16) return many ? cand_score_kernel<true, 4> : cand_score_kernel<true, 2>;
    return many ? cand_score_kernel<false, 4> : cand_score_kernel<false, 2>;
}

cudaError_t cand_set_smem_limits() {
    cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void*>(cand_topk_kernel));
    for (int i = 0; i < 4; i++) {
        const void* fn = reinterpret_cast<const void*>(score_kernel(i & 1, i & 2));
        if (e == cudaSuccess) e = set_max_dynamic_smem(fn);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    }
    return e;
}

cudaError_t launch_cand_topk(const float* dlog, int rows, int V, int K, int S, int* cand_tok, uint64_t* part,
                             int* ticket, cudaStream_t st) {
    return launch_pdl(cand_topk_kernel, dim3(rows * S), dim3(kTopkThreads), cand_topk_smem(K), st, dlog, V, K, S,
                      cand_tok, part, ticket, 0, static_cast<long long>(K), static_cast<float*>(nullptr),
                      static_cast<const int*>(nullptr));
}

cudaError_t launch_row_topk_by_value(const float* x, int rows, int V, int K, int S, int* tok, float* val,
                                     long long out_stride, uint64_t* part, int* ticket, cudaStream_t st,
                                     const int* out_row) {
    return launch_pdl(cand_topk_kernel, dim3(rows * S), dim3(kTopkThreads), cand_topk_smem(K), st, x, V, K, S, tok,
                      part, ticket, 1, out_stride, val, out_row);
}

// Candidates per group, blocks per cluster, node states staged at a time, and
// the shared memory of both these and the partial sums (at most 83 KB for any
// supported shape).
struct ScorePlan {
    bool many;
    int G, cs, PC, smem;
};
static ScorePlan score_plan(int nseq, int P, int d, int DS) {
    ScorePlan p;
    p.many = nseq * P >= kScoreManyNodes;
    p.G = p.many ? 16 : 8;
    p.cs = std::min(DS, kScoreCluster);  // (DS is a power of two)
    const int dchunk = d / DS;
    p.PC = std::max(1, std::min(P, kScoreStage / (dchunk * 4)));
    p.smem = (p.PC * dchunk + DS / p.cs * (p.G + 1) * P) * 4;
    return p;
}

int cand_score_smem(int nseq, int P, int d, int DS) { return score_plan(nseq, P, d, DS).smem; }

cudaError_t launch_cand_score(const CandArgs& a, cudaStream_t st) {
    const ScorePlan p = score_plan(a.nseq, a.P, a.d, a.DS);
    const int ngroups = (a.K + p.G - 1) / p.G;
    return launch_pdl_cluster(score_kernel(a.wbf16 != 0, p.many), dim3(a.nseq * ngroups * p.cs), dim3(kScoreThreads),
                              p.smem, st, p.cs, a, p.cs, p.PC);
}

}  // namespace dart
