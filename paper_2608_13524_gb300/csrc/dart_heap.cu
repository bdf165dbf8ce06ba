// Best-first (heap-order) tree constructions that Table 2 of the paper
// compares DARTree with, on the GPU:
//
//   Domino-chain + DDTree   causal correction along ONE draft chain (the
//       depth-wise path with W = k = 1, which also writes each depth's
//       scaled logits), then DDTree (Sec. 3.3) over the chain-conditioned
//       distributions: the prefixes are scored with those position-wise
//       marginals, sum_i log q~_i(u_i) + beta d, and the best B are taken
//       best first.  ddtree_kernel runs the best-first search.
//   Sequential correction with heap   exact node-wise best-first search under
//       the corrected scores (Sec. 4.1): every popped prefix is corrected
//       (head update + scoring of its children) before the next pop.
//       seqheap_step_kernel pops until a prefix must be corrected and
//       prepares the corrections of one pass (that prefix and the likely next
//       ones); the pass itself reuses the head-update, LM-head, merge and
//       top-K kernels.
//
// Both searches keep, for every popped node p (and the root), a cursor into
// its children sorted by log q~ (desc, token asc); p's "offer" is its best
// child not yet taken, scored s_p + log q~ + beta.  A pop takes the best offer
// by (score desc, node asc; the root first) -- DDTree's "next sibling / first
// child" pushes in another bookkeeping -- and the popped child becomes a node
// with its own offer.  Rows are emitted in pop order (parents first).
#include "dart_device.cuh"
#include "dart_kernels.h"

namespace dart {

namespace {

constexpr int kHeapThreads = 256;

// Key of an offer: score order, then the smaller slot (slot = node + 1, the
// root is slot 0).  An offer of score -inf is no offer (key 0).
__device__ __forceinline__ uint64_t offer_key(float v, int slot) {
    return v == -INFINITY ? 0ull : make_key(v, static_cast<uint32_t>(slot));
}

__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t y = shfl_xor_u64(v, o);
        v = y > v ? y : v;
    }
    return v;
}

// The best key among the offers of slots lane, lane + 32, ... < nslots.
__device__ __forceinline__ uint64_t lane_best(const float* offer, int nslots, int lane) {
    uint64_t b = 0ull;
    for (int o = lane; o < nslots; o += 32) {
        const uint64_t k = offer_key(offer[o], o);
        b = k > b ? k : b;
    }
    return b;
}

// Ancestor bit masks and padding of one sequence's emitted tree (rows in pop
// order, parents[] of its first n rows given).
__device__ void emit_masks(const int* par, int n, int B, size_t ob, int* tokens, int* parents, int* depths,
                           int* pos_ids, float* scores, uint64_t* mask) {
    const int nw = (B + 63) / 64;
    for (int i = n + static_cast<int>(threadIdx.x); i < B; i += blockDim.x) {
        tokens[ob + i] = -1;
        parents[ob + i] = -2;
        depths[ob + i] = 0;
        pos_ids[ob + i] = -1;
        scores[ob + i] = -INFINITY;
    }
    for (int q = threadIdx.x; q < B * nw; q += blockDim.x) {
        const int i = q / nw, wd = q % nw;
        uint64_t word = 0ull;
        if (i < n)
            for (int j = i; j >= 0; j = par[j])
                if ((j >> 6) == wd) word |= 1ull << (j & 63);
        mask[(ob + i) * nw + wd] = word;
    }
}

// 4 columns of row `row` of the head's input: fp32 and, for the tensor-core
// GEMMs, hi / lo bf16 rows.
__device__ __forceinline__ void sh_put_row(const SeqHeapArgs& a, int row, int j, const float4 v) {
    *reinterpret_cast<float4*>(a.hin + static_cast<size_t>(row) * a.d + j) = v;
    if (a.HL) {
        __align__(8) __nv_bfloat16 hi[4], lo[4];
        split_bf16(v.x, hi[0], lo[0]);
        split_bf16(v.y, hi[1], lo[1]);
        split_bf16(v.z, hi[2], lo[2]);
        split_bf16(v.w, hi[3], lo[3]);
        *reinterpret_cast<uint2*>(a.HL + static_cast<size_t>(row) * a.d + j) = *reinterpret_cast<const uint2*>(hi);
        *reinterpret_cast<uint2*>(a.HL + static_cast<size_t>(a.bhalf + row) * a.d + j) = *reinterpret_cast<const uint2*>(lo);
    }
}

// One block per sequence.  Shared memory: the chain's sorted children per
// depth as log q~ [L][Bp] and tokens [L][Bp]; per popped node its parent,
// depth and score; per slot its cursor and offer.
__global__ void __launch_bounds__(kHeapThreads) ddtree_kernel(const DdtArgs a) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ float hsm[];
    const int L = a.L, Bp = a.Bp, B = a.B;
    float* lq = hsm;                                          // [L][Bp]
    int* tk = reinterpret_cast<int*>(lq + L * Bp);            // [L][Bp]
    float* nsc = reinterpret_cast<float*>(tk + L * Bp);       // [B]
    int* npar = reinterpret_cast<int*>(nsc + B);              // [B]
    int* ndep = npar + B;                                     // [B]
    int* ntok = ndep + B;                                     // [B]
    int* next = ntok + B;                                     // [B + 1]
    float* offer = reinterpret_cast<float*>(next + B + 1);    // [B + 1]
    __shared__ int npop;
    const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    // log q~ = min(z - lse, 0) of the chain's best Bp children per depth
    for (int q = tid; q < L * Bp; q += blockDim.x) {
        const int dd = q / Bp;
        const size_t src = (static_cast<size_t>(s) * L + dd) * Bp + (q % Bp);
        const float z = a.zval[src], lse = a.lse[static_cast<size_t>(s) * L + dd];
        lq[q] = (z == -INFINITY || lse == -INFINITY) ? -INFINITY : fminf(z - lse, 0.0f);
        tk[q] = a.tok[src];
    }
    __syncthreads();
    if (tid < 32) {
        // best-first search, one warp; lane l owns the slots l, l + 32, ...
        if (lane == 0) {
            next[0] = 0;
            offer[0] = Bp > 0 ? lq[0] + a.beta : -INFINITY;
        }
        __syncwarp();
        uint64_t best = lane == 0 ? offer_key(offer[0], 0) : 0ull;
        int n = 0;
        while (n < B) {
            const uint64_t k = warp_max_u64(best);
            if (k == 0ull) break;
            const int o = static_cast<int>(key_idx(k));
            const float sc = key_val(k);
            const int dep = o == 0 ? 1 : ndep[o - 1] + 1;
            if (lane == 0) {
                int c = next[o];
                if (!bounds_check(a.status, c < Bp && dep <= L)) c = 0;
                ntok[n] = tk[(dep - 1) * Bp + c];
                npar[n] = o - 1;
                ndep[n] = dep;
                nsc[n] = sc;
                next[o] = c + 1;
                const float so = o == 0 ? 0.0f : nsc[o - 1];
                offer[o] = c + 1 < Bp ? so + lq[(dep - 1) * Bp + c + 1] + a.beta : -INFINITY;
                next[n + 1] = 0;
                offer[n + 1] = (dep < L && Bp > 0) ? sc + lq[dep * Bp] + a.beta : -INFINITY;
            }
            __syncwarp();
            n++;
            if (lane == (o & 31)) best = lane_best(offer, n + 1, lane);
            else if (lane == (n & 31)) {
                const uint64_t kn = offer_key(offer[n], n);
                best = kn > best ? kn : best;
            }
        }
        if (lane == 0) npop = n;
    }
    __syncthreads();
    const int n = npop;
    const size_t ob = static_cast<size_t>(s) * B;
    for (int i = tid; i < n; i += blockDim.x) {
        a.tokens[ob + i] = ntok[i];
        a.parents[ob + i] = npar[i];
        a.depths[ob + i] = ndep[i];
        a.pos_ids[ob + i] = a.pos_offset + ndep[i];
        a.scores[ob + i] = nsc[i];
    }
    emit_masks(npar, n, B, ob, a.tokens, a.parents, a.depths, a.pos_ids, a.scores, a.mask);
    if (tid == 0) a.n_nodes[s] = n;
}

// ---- sequential correction with heap
//
// The search pops prefixes best first; a popped prefix must be corrected (its
// state, and the distribution of its children over the vocabulary) before
// the next pop.  A correction streams the whole LM-head (HBM-bound) for one
// prefix as for sixteen, so each pass corrects, beside the prefix the search
// waits for, the prefixes it is most likely to need next: the step kernel
// runs the same best-first search ahead on what is known so far, and every
// uncorrected prefix it would pop becomes a target of the pass.  Nothing
// else changes: pops, their order, their scores and each prefix's own
// arithmetic (one column of the LM-head's node group) are those of the
// one-prefix-at-a-time search; a target that is never popped is wasted.
// Measured on GB300, V = 151936, d = 2560, L = 16, B = 64, one sequence:
// 10286 us per round with one prefix a pass (64 LM-head passes), 928 us with
// sixteen (the passes left take about 150 us each, 116 of them the LM-head).
//
// A corrected prefix is an entry (0 = the root) with its state, its best Bp
// children (sorted) and its log-sum-exp; the corrected children of an entry
// are always its best ones, ranks 0 .. ncorr - 1 (both searches take them
// in order), and lent[rank] names their entries.  A slot is a popped node
// (row + 1; slot 0 the root) with its entry, cursor, offer, depth and score.
// Both live in a state block per sequence that the kernel reads from one of
// two buffers and writes to the other, since M blocks per sequence run the
// same search (each then prepares one target's input).

constexpr int kShHead = 8;  // state words before the slot arrays: n, entries, pending, last pass's targets and first entry

__host__ __device__ __forceinline__ int sh_state_words(int B, int E) { return kShHead + 5 * (B + 1) + E; }

__global__ void __launch_bounds__(kHeapThreads) seqheap_init_kernel(const SeqHeapArgs a) {
    pdl_trigger();
    pdl_wait();
    const int s = blockIdx.x / a.M, m = blockIdx.x % a.M, row = blockIdx.x;
    for (int j = threadIdx.x * 4; j < a.d; j += blockDim.x * 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (m == 0) {
            v = *reinterpret_cast<const float4*>(a.anchor + static_cast<size_t>(s) * a.d + j);
            *reinterpret_cast<float4*>(a.tab + static_cast<size_t>(s) * a.E * a.d + j) = v;
        }
        sh_put_row(a, row, j, v);
    }
    if (threadIdx.x == 0) {
        a.dlog_row[row] = s * a.L;
        a.row_ent[row] = m == 0 ? s * a.E : -1;
        if (m == 0) {
            int* w = a.state[0] + static_cast<size_t>(s) * sh_state_words(a.B, a.E);
            const int S1 = a.B + 1;
            w[0] = 0;  // popped nodes
            w[1] = 1;  // entries: the root
            w[2] = 1;  // slot 0 waits for its children's scores
            w[3] = 0;
            w[4] = 0;
            int* sl = w + kShHead;
            sl[0] = 0;                                   // entry
            sl[S1] = 0;                                  // cursor
            sl[2 * S1] = 0;                              // depth
            sl[3 * S1] = __float_as_int(0.0f);           // score
            sl[4 * S1] = __float_as_int(-INFINITY);      // offer
            sl[5 * S1] = 0;                              // ncorr of the root
            if (s == 0) {
                a.sync[0] = a.sync[1] = 0;  // ticket, sequences with a target
                a.sync[2] = 0;              // state buffer to read
            }
        }
    }
}

// One step of the search between two passes, M blocks per sequence; see
// above.  Bound by the latency of the serial search (about 0.35 us a pop:
// a warp-wide maximum and a few shared-memory reads; the first children of
// every entry are staged in shared memory so that few pops wait for L2).
__global__ void __launch_bounds__(kHeapThreads) seqheap_step_kernel(const SeqHeapArgs a, cudaGraphConditionalHandle cond,
                                                                   int has_cond) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) int shs[];
    __shared__ int tpe[kSeqHeapMaxTargets], tc[kSeqHeapMaxTargets], tdep[kSeqHeapMaxTargets];
    __shared__ int res[4];  // real pops, targets, blocked
    const int s = blockIdx.x / a.M, m = blockIdx.x % a.M, row = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31;
    const int B = a.B, Bp = a.Bp, Bs = a.Bs, L = a.L, d = a.d, E = a.E, S1 = B + 1;
    const int buf = __ldcg(a.sync + 2);
    const int* win = a.state[buf] + static_cast<size_t>(s) * sh_state_words(B, E);
    int* wout = a.state[buf ^ 1] + static_cast<size_t>(s) * sh_state_words(B, E);
    const size_t eb = static_cast<size_t>(s) * E;
    float4* z4 = reinterpret_cast<float4*>(shs);       // [E] scaled logits of the first four children
    float* lse = reinterpret_cast<float*>(z4 + E);     // [E]
    int* ncorr = reinterpret_cast<int*>(lse + E);      // [E]
    int* ent = ncorr + E;                              // [B + 1]
    int* next = ent + S1;
    int* dep = next + S1;
    float* sc = reinterpret_cast<float*>(dep + S1);
    float* offer = sc + S1;
    int* rpe = reinterpret_cast<int*>(offer + S1);     // [B] rows popped now: parent's entry, child rank, parent's slot
    int* rc = rpe + B;
    int* ro = rc + B;
    const int n0 = win[0], ne = win[1], pending = win[2], pt = win[3], pbase = win[4];
    for (int i = tid; i <= n0; i += kHeapThreads) {
        const int* sl = win + kShHead + i;
        ent[i] = sl[0];
        next[i] = sl[S1];
        dep[i] = sl[2 * S1];
        sc[i] = __int_as_float(sl[3 * S1]);
        offer[i] = __int_as_float(sl[4 * S1]);
    }
    for (int e = tid; e < ne; e += kHeapThreads) {
        z4[e] = *reinterpret_cast<const float4*>(a.lz + (eb + e) * Bs);  // (Bs is a multiple of 4)
        lse[e] = a.llse[eb + e];
        ncorr[e] = win[kShHead + 5 * S1 + e];
    }
    __syncthreads();
    // log q~ of child c of entry e (-inf past its list)
    auto lq = [&](int e, int c) -> float {
        if (c >= Bp) return -INFINITY;
        const float z = c < 4 ? reinterpret_cast<const float*>(z4 + e)[c] : a.lz[(eb + e) * Bs + c];
        return (z == -INFINITY || lse[e] == -INFINITY) ? -INFINITY : fminf(z - lse[e], 0.0f);
    };
    // Pops until a prefix must be corrected (ahead = false: the rows of the
    // tree), or on past uncorrected prefixes, which become targets, up to
    // `most` of them (ahead = true: nothing but the targets is kept).
    int nt = 0;
    auto search = [&](int n, bool ahead, int most) -> int {
        uint64_t best = lane_best(offer, n + 1, lane);
        while (n < B && nt < most) {
            const uint64_t k = warp_max_u64(best);
            if (k == 0ull) break;
            const int o = static_cast<int>(key_idx(k));
            const float so = key_val(k);
            const int pe = ent[o], dp = dep[o] + 1;
            int c = next[o];
            if (!bounds_check(a.status, c < Bp && o <= n && dp <= L)) c = 0;
            const float po = sc[o] + lq(pe, c + 1) + a.beta;
            int e = -1;
            float no = -INFINITY;
            bool target = false;
            if (dp < L && n + 1 < B) {  // the last pop and nodes at depth L are not corrected
                if (c < ncorr[pe]) {
                    e = a.lent[(eb + pe) * Bs + c];
                    no = so + lq(e, 0) + a.beta;
                } else {
                    target = true;
                    e = ne + nt;
                }
            }
            __syncwarp();
            if (lane == 0) {
                if (!ahead) {
                    rpe[n] = pe;
                    rc[n] = c;
                    ro[n] = o;
                }
                next[o] = c + 1;
                offer[o] = po;
                n++;
                ent[n] = e;
                next[n] = 0;
                dep[n] = dp;
                sc[n] = so;
                offer[n] = no;
                if (target) {
                    tpe[nt] = pe;
                    tc[nt] = c;
                    tdep[nt] = dp;
                    ncorr[pe] = c + 1;
                    ncorr[e] = 0;
                    if (m == 0) a.lent[(eb + pe) * Bs + c] = e;  // read from the next step on
                }
            } else {
                n++;
            }
            __syncwarp();
            if (lane == (o & 31)) best = lane_best(offer, n + 1, lane);
            else if (lane == (n & 31)) {
                const uint64_t kn = offer_key(no, n);
                best = kn > best ? kn : best;
            }
            if (target) {
                nt++;
                if (!ahead) break;
            }
        }
        return n;
    };
    if (tid < 32) {
        if (pending && lane == 0) offer[n0] = sc[n0] + lq(ent[n0], 0) + a.beta;
        __syncwarp();
        const int n = search(n0, false, 1);
        if (lane == 0) {
            res[0] = n;
            res[2] = nt;
        }
    }
    __syncthreads();
    const int n1 = res[0], blocked = res[2];
    if (m == 0) {
        for (int i = tid; i <= n1; i += kHeapThreads) {
            int* sl = wout + kShHead + i;
            sl[0] = ent[i];
            sl[S1] = next[i];
            sl[2 * S1] = dep[i];
            sl[3 * S1] = __float_as_int(sc[i]);
            sl[4 * S1] = __float_as_int(offer[i]);
        }
        for (int i = n0 + tid; i < n1; i += kHeapThreads) {
            const size_t ob = static_cast<size_t>(s) * B + i;
            a.tokens[ob] = a.ltok[(eb + rpe[i]) * Bs + rc[i]];
            a.parents[ob] = ro[i] - 1;
            a.depths[ob] = dep[i + 1];
            a.pos_ids[ob] = a.pos_offset + dep[i + 1];
            a.scores[ob] = sc[i + 1];
        }
        if (tid == 0) a.npop[s] = n1;
    }
    __syncthreads();
    if (tid < 32) {
        // room for the corrections that the remaining pops may need is kept
        if (blocked) search(n1, true, min(a.M, max(1, E - ne - (B - n1))));
        if (lane == 0) res[1] = nt;
    }
    __syncthreads();
    nt = res[1];
    if (m == 0) {
        for (int e = tid; e < ne + nt; e += kHeapThreads) wout[kShHead + 5 * S1 + e] = ncorr[e];
        if (tid == 0) {
            wout[0] = n1;
            wout[1] = ne + nt;
            wout[2] = blocked;
            wout[3] = nt;
            wout[4] = ne;
        }
    }
    // the previous pass's target m: its state into the table
    if (m < pt)
        for (int j = tid * 4; j < d; j += kHeapThreads * 4)
            *reinterpret_cast<float4*>(a.tab + (eb + pbase + m) * d + j) =
                *reinterpret_cast<const float4*>(a.hout + static_cast<size_t>(row) * d + j);
    // this pass's target m: its parent's state (perhaps a target of the
    // previous pass, whose table row another block is writing), token and
    // drafter row
    if (m < nt) {
        const int pe = tpe[m];
        const float* src = pe >= pbase && pe < pbase + pt ? a.hout + (static_cast<size_t>(s) * a.M + pe - pbase) * d
                                                          : a.tab + (eb + pe) * d;
        for (int j = tid * 4; j < d; j += kHeapThreads * 4) sh_put_row(a, row, j, *reinterpret_cast<const float4*>(src + j));
    }
    if (tid == 0) {
        a.child_prow[row] = m < nt ? row : -1;
        a.child_tok[row] = m < nt ? a.ltok[(eb + tpe[m]) * Bs + tc[m]] : 0;
        a.dlog_row[row] = s * L + (m < nt ? min(tdep[m], L - 1) : 0);
        a.row_ent[row] = m < nt ? static_cast<int>(eb) + ne + m : -1;
        // the last block to get here (every block has read its state) turns
        // the buffers round and says whether another pass is needed
        if (m == 0 && nt > 0) atomicAdd(a.sync + 1, 1);
        __threadfence();
        if (atomicAdd(a.sync, 1) == a.nseq * a.M - 1) {
            __threadfence();
            const int any = atomicAdd(a.sync + 1, 0) > 0;
            a.sync[0] = a.sync[1] = 0;
            a.sync[2] = buf ^ 1;
            if (has_cond) cudaGraphSetConditional(cond, any ? 1u : 0u);
        }
    }
}

// Masks and padding after the last pop.
__global__ void __launch_bounds__(kHeapThreads) seqheap_emit_kernel(const SeqHeapArgs a) {
    pdl_trigger();
    pdl_wait();
    const int s = blockIdx.x;
    const int n = __ldcg(a.npop + s);
    const size_t ob = static_cast<size_t>(s) * a.B;
    emit_masks(a.parents + ob, n, a.B, ob, a.tokens, a.parents, a.depths, a.pos_ids, a.scores, a.mask);
    if (threadIdx.x == 0) a.n_nodes[s] = n;
}

}  // namespace

int ddtree_smem(int L, int Bp, int B) { return (L * Bp * 2 + B * 4 + (B + 1) * 2) * 4; }

int seqheap_step_smem(int B, int E) { return E * 24 + (B + 1) * 20 + B * 12; }
int seqheap_state_words(int B, int E) { return sh_state_words(B, E); }

cudaError_t heap_set_smem_limits() {
    cudaError_t e = set_max_dynamic_smem(reinterpret_cast<const void*>(ddtree_kernel));
    if (e == cudaSuccess) e = set_max_dynamic_smem(reinterpret_cast<const void*>(seqheap_step_kernel));
    return e;
}

cudaError_t launch_ddtree(const DdtArgs& a, cudaStream_t st) {
    return launch_pdl(ddtree_kernel, dim3(a.nseq), dim3(kHeapThreads), ddtree_smem(a.L, a.Bp, a.B), st, a);
}

cudaError_t launch_seqheap_init(const SeqHeapArgs& a, cudaStream_t st) {
    return launch_pdl(seqheap_init_kernel, dim3(a.nseq * a.M), dim3(kHeapThreads), 0, st, a);
}

cudaError_t launch_seqheap_step(const SeqHeapArgs& a, cudaGraphConditionalHandle cond, bool has_cond, cudaStream_t st) {
    return launch_pdl(seqheap_step_kernel, dim3(a.nseq * a.M), dim3(kHeapThreads), seqheap_step_smem(a.B, a.E), st, a,
                      cond, has_cond ? 1 : 0);
}

// (plain launch: it may follow a conditional node of a graph)
cudaError_t launch_seqheap_emit(const SeqHeapArgs& a, cudaStream_t st) {
    seqheap_emit_kernel<<<a.nseq, kHeapThreads, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace dart
