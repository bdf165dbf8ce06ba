// tcgen05 / TMA kernels of the DARTree construction path (sm_103a).
//
// One warp-specialised mainloop serves two contractions with bf16 operands
// in shared memory and fp32 accumulators in tensor memory:
//   * LM-head scoring: A = E tile [128 vocabulary rows x 64], B = node states
//     [NG nodes x 64] as hi + lo bf16 halves stored as 2*NG consecutive rows,
//     so ONE MMA with N = 2*NG computes both products (TMEM columns [0, NG)
//     = A.hi, [NG, 2NG) = A.lo; the epilogue adds them: states keep ~16
//     mantissa bits at half the MMA instruction count).  A persistent CTA
//     walks a contiguous range of vocabulary tiles; two TMEM accumulators let
//     the epilogue of tile i overlap the MMAs of tile i+1.  The epilogue adds
//     the drafter row, scales by 1/T and reduces on chip to a running
//     log-sum-exp and a top-k per node, so no [N,V] logits tensor is written.
//   * Correction-head GEMMs (split-K): A = W_i[:, 0:d] (or all of W_i) or
//     W_o tile, B = the node inputs; each CTA writes an fp32 partial tile, or
//     the k splits of a tile form a cluster that sums them on chip.  The same
//     kernel, with A = W_i[:, d:2d] and B = E rows as nodes, computes the
//     per-token table Q[t] = W_i[:, d:2d] . E[t] once per handle.
// Warp roles (192 threads): warp 0 = TMA producer, warp 1 = TMEM allocator
// and single-thread MMA issuer, warps 2-5 = epilogue (TMEM lane quarters
// warp%4).  Every wait is bounded: on timeout the CTA records kDevTimeout in
// the status word, drains its own copies/MMAs (bounded), frees TMEM and exits.
#include <algorithm>
#include <cstdio>
#include <cstdlib>

#include "dart_device.cuh"
#include "dart_kernels.h"

namespace dart {

namespace {

// 2 warps (producer, MMA) + 4 epilogue warps (one per TMEM lane quarter) per
// 16-node chunk of the group, at most 16 epilogue warps: in 128-node groups
// every epilogue warp handles two chunks.
template <int NG>
constexpr int epi_threads() {
    return 128 * (NG / 16 < 4 ? NG / 16 : 4);
}
template <int NG>
constexpr int epi_chunks() {
    return NG > 64 ? NG / 64 : 1;
}
// Candidate slots per node: a whole tile (nothing can overflow) up to 32-node
// groups; 64- and 128-node groups keep fewer (more pipeline stages fit) and
// merge in rounds when a tile overflows them.  Those groups come with the
// starting bound of the filter (seed pass before the launch), after which
// a tile rarely offers more than a few logits per node.  Measured on GB300
// at 64 nodes, k = 64 (µs per round, same box): 128 slots 3042, 64 slots
// 2806, 32 slots 2706 with the bound; without it 32 slots cost +6 %.  128-node
// groups keep 16 (cand_slots), which makes room for a fifth stage (389 instead
// of 403 µs per launch at 256 nodes; 8 slots change nothing more), but 32 where
// tiles offer more: without the bound, and in ranges of one tile.
// Measured on GB300 (µs per round of 3 depths at d = 5120, where there is no
// bound, and 4 at d = 4096; 16 slots, 32): 8 x 32 nodes, k = 32, V = 151936,
// d = 5120 1628, 1579; 16 x 6, k = 34, V = 30000, d = 5120 561, 465; 8 x 32, k = 32,
// d = 4096 V = 600 472, 451, V = 12000 485, 485, V = 32000 628, 646.
template <int NG>
constexpr int lm_cand_cap() {
    return NG >= 64 ? kCandCapLarge : kCandCap;
}
int cand_slots(int NG, bool bounded, bool one_tile) {
    return NG > 64 && bounded && !one_tile ? kCandCapLarge / 2 : NG >= 64 ? kCandCapLarge : kCandCap;
}
template <int NG>
constexpr int threads() {
    return 64 + epi_threads<NG>();
}
constexpr int kATileBytes = kTileM * kBlockK * 2;  // 16 KB

struct Work {
    int ntiles;     // consecutive A tiles handled by this CTA
    int row0;       // row coordinate of the first tile
    int kb0, kb1;   // k-block range
    int brow;       // B row of this node group (hi half); lo half at + bhalf
    int lo_kb_end;  // k-blocks >= this carry no lo half
    int tiled_kb;   // 0: A is row-major [rows][K]; else A is tiled, tile (rt, kb) at rows (rt * tiled_kb + kb) * 128
};

// TMA coordinates of A tile i (of this CTA's range), k-block kb: in the
// row-major layout (x = kb * 64, y = row), or in the tiled layout, where the
// 128 x 64 tile (rt, kb) is 16 KB of contiguous memory, viewed as rows of 64
// elements: (x = 0, y = (rt * KB + kb) * 128).
__device__ __forceinline__ int a_x(const Work& w, int kb) { return w.tiled_kb ? 0 : kb * kBlockK; }
__device__ __forceinline__ int a_y(const Work& w, int i, int kb) {
    return w.tiled_kb ? ((w.row0 / kTileM + i) * w.tiled_kb + kb) * kTileM : w.row0 + i * kTileM;
}

template <int NG>
struct Layout {
    static constexpr int kStage = kATileBytes + 2 * NG * 128;
};

__device__ __forceinline__ void record_timeout(int* status, volatile int* abort) {
    *abort = 1;
    atomicOr(status, kDevTimeout);
}

// Bounded wait that ignores the abort flag (used while draining).
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
    const unsigned long long t0 = globaltimer_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (globaltimer_ns() - t0 > kWaitLimitNs) return;
    }
}

template <int NG>
__device__ __forceinline__ void producer(const CUtensorMap* tmA, const CUtensorMap* tmB, const Work& w, int bhalf,
                                         uint8_t* ring, int stages, uint64_t* full, uint64_t* empty,
                                         volatile int* abort, int* status, int l2pf = 0, bool keep_a = false) {
    // A: streamed once (E), or kept for the next depth (head weights when
    // nothing else streams through L2)
    const uint64_t pol_a = keep_a ? l2_policy_evict_last() : l2_policy_evict_first();
    const uint64_t pol_b = l2_policy_evict_last();   // re-read by every tile
    const int kbs = w.kb1 - w.kb0;
    const uint32_t total = static_cast<uint32_t>(w.ntiles * kbs);
    // The A operand (E or a head weight) never depends on an earlier kernel:
    // its first `pre` stages are requested before waiting on the previous
    // kernel; the B operand (node states) only after.
    const uint32_t pre = total < static_cast<uint32_t>(stages) ? total : static_cast<uint32_t>(stages);
#pragma unroll 1
    for (uint32_t f = 0; f < pre; f++) {
        const int i = static_cast<int>(f) / kbs, kb = w.kb0 + static_cast<int>(f) % kbs;
        const bool lo = kb < w.lo_kb_end;
        mbar_arrive_expect_tx(&full[f], kATileBytes + NG * 128 * (lo ? 2 : 1));
        tma_load_2d(ring + f * Layout<NG>::kStage, tmA, &full[f], a_x(w, kb), a_y(w, i, kb), pol_a);
    }
    // and the next `l2pf` into L2, while the previous kernel still runs
#pragma unroll 1
    for (uint32_t f = pre; f < pre + static_cast<uint32_t>(l2pf) && f < total; f++) {
        const int i = static_cast<int>(f) / kbs, kb = w.kb0 + static_cast<int>(f) % kbs;
        tma_prefetch_2d(tmA, a_x(w, kb), a_y(w, i, kb));
    }
    pdl_wait();
#pragma unroll 1
    for (uint32_t f = 0; f < pre; f++) {
        const int kb = w.kb0 + static_cast<int>(f) % kbs;
        uint8_t* sH = ring + f * Layout<NG>::kStage + kATileBytes;
        tma_load_2d(sH, tmB, &full[f], kb * kBlockK, w.brow, pol_b);
        if (kb < w.lo_kb_end) tma_load_2d(sH + NG * 128, tmB, &full[f], kb * kBlockK, bhalf + w.brow, pol_b);
    }
    uint32_t stage = pre % stages, phase = (pre / stages) & 1u, fills = pre;
    bool ok = true;
    int i = static_cast<int>(pre) / kbs, kb = w.kb0 + static_cast<int>(pre) % kbs;
#pragma unroll 1
    for (uint32_t f = pre; f < total; f++, kb++) {
        if (kb == w.kb1) {
            kb = w.kb0;
            i++;
        }
        if (!mbar_wait(&empty[stage], phase ^ 1u, abort)) {
            record_timeout(status, abort);
            ok = false;
            break;
        }
        const bool lo = kb < w.lo_kb_end;
        uint8_t* sA = ring + stage * Layout<NG>::kStage;
        uint8_t* sH = sA + kATileBytes;
        mbar_arrive_expect_tx(&full[stage], kATileBytes + NG * 128 * (lo ? 2 : 1));
        tma_load_2d(sA, tmA, &full[stage], a_x(w, kb), a_y(w, i, kb), pol_a);
        tma_load_2d(sH, tmB, &full[stage], kb * kBlockK, w.brow, pol_b);
        if (lo) tma_load_2d(sH + NG * 128, tmB, &full[stage], kb * kBlockK, bhalf + w.brow, pol_b);
        fills++;
        if (++stage == static_cast<uint32_t>(stages)) {
            stage = 0;
            phase ^= 1u;
        }
    }
    if (!ok) {
        // wait for this thread's copies still in flight before the CTA exits
        const uint32_t first = fills > static_cast<uint32_t>(stages) ? fills - stages : 0;
        for (uint32_t f = first; f < fills; f++) drain_wait(&full[f % stages], (f / stages) & 1u);
    }
}

template <int NG>
__device__ __forceinline__ void mma_issuer(const Work& w, uint8_t* ring, int stages, uint64_t* full,
                                           uint64_t* empty, uint64_t* tfull, uint64_t* tempty, uint64_t* tdown,
                                           uint32_t tmem_base, int acc_stride, volatile int* abort,
                                           int* status, int nacc = 2) {
    constexpr uint32_t idesc2 = idesc_bf16_f32(kTileM, 2 * NG);  // hi and lo rows together
    constexpr uint32_t idesc1 = idesc_bf16_f32(kTileM, NG);      // hi rows only (no lo half)
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int i = 0; i < w.ntiles && ok; i++) {
        const int acc = i % nacc;
        const uint32_t aph = (i / nacc) & 1;
        if (!mbar_wait(&tempty[acc], aph ^ 1u, abort)) {
            record_timeout(status, abort);
            ok = false;
            break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * acc_stride;
#pragma unroll 1
        for (int kb = w.kb0; kb < w.kb1; kb++) {
            if (!mbar_wait(&full[stage], phase, abort)) {
                record_timeout(status, abort);
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t idesc = kb < w.lo_kb_end ? idesc2 : idesc1;
            const uint32_t a = smem_u32(ring + stage * Layout<NG>::kStage);
            const uint32_t hb = a + kATileBytes;
#pragma unroll
            for (int kk = 0; kk < kBlockK / 16; kk++)
                tc_mma_bf16(d_tmem, sdesc_sw128(a + kk * 32), sdesc_sw128(hb + kk * 32), idesc,
                            (kb > w.kb0 || kk > 0) ? 1u : 0u);
            tc_commit(&empty[stage]);  // frees the smem stage once these MMAs are done
            if (++stage == static_cast<uint32_t>(stages)) {
                stage = 0;
                phase ^= 1u;
            }
        }
        if (ok) tc_commit(&tfull[acc]);
    }
    if (!ok) {
        // make sure no MMA still reads smem / writes TMEM before teardown
        tc_commit(tdown);
        drain_wait(tdown, 0);
    }
}

// ---- the same roles for a CTA pair (lmhead_tc_kernel with kPair)
//
// Each CTA loads its own A tile (128 rows) and one half of the group's B
// rows: the leader the hi rows, its peer the lo rows.  A stage is full when
// all four copies have completed on the leader's barrier; it is empty when
// the leader's commit has arrived in both CTAs.
//
// A commit arrives in the peer's shared memory some time after the MMAs it
// tracks, and no barrier of threads orders that.  So every arrival is waited
// for where it lands, before the CTA leaves: the last ones of `empty` by the
// CTA's producer, that of an accumulator its epilogue does not read by the
// epilogue's first thread.

template <int NG>
struct PairLayout {
    static constexpr int kStage = kATileBytes + NG * 128;
};

template <int NG>
__device__ __forceinline__ void producer_pair(const CUtensorMap* tmA, const CUtensorMap* tmB, const Work& w,
                                              uint32_t rank, int bhalf, uint8_t* ring, int stages, uint64_t* full,
                                              uint64_t* empty, volatile int* abort, int* status) {
    const uint64_t pol_a = l2_policy_evict_first();  // streamed once
    const uint64_t pol_b = l2_policy_evict_last();   // re-read by every tile
    const int kbs = w.kb1 - w.kb0;
    const uint32_t total = static_cast<uint32_t>(w.ntiles * kbs);
    const uint32_t pre = total < static_cast<uint32_t>(stages) ? total : static_cast<uint32_t>(stages);
    const int brow = w.brow + (rank ? bhalf : 0);
    auto load_a = [&](uint32_t f, uint32_t st) {
        const int i = static_cast<int>(f) / kbs, kb = w.kb0 + static_cast<int>(f) % kbs;
        tma_load_2d_pair(ring + st * PairLayout<NG>::kStage, tmA, mapa_u32(smem_u32(&full[st]), 0), a_x(w, kb),
                         a_y(w, i, kb), pol_a);
    };
    auto load_b = [&](uint32_t f, uint32_t st) {
        tma_load_2d_pair(ring + st * PairLayout<NG>::kStage + kATileBytes, tmB, mapa_u32(smem_u32(&full[st]), 0),
                         (w.kb0 + static_cast<int>(f) % kbs) * kBlockK, brow, pol_b);
    };
    // (as in `producer`: A does not depend on an earlier kernel, B does)
#pragma unroll 1
    for (uint32_t f = 0; f < pre; f++) {
        if (rank == 0) mbar_arrive_expect_tx(&full[f], 2 * PairLayout<NG>::kStage);
        load_a(f, f);
    }
    pdl_wait();
#pragma unroll 1
    for (uint32_t f = 0; f < pre; f++) load_b(f, f);
    uint32_t stage = pre % stages, phase = (pre / stages) & 1u, fills = pre;
    bool ok = true;
#pragma unroll 1
    for (uint32_t f = pre; f < total; f++) {
        if (!mbar_wait(&empty[stage], phase ^ 1u, abort)) {
            record_timeout(status, abort);
            ok = false;
            break;
        }
        if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * PairLayout<NG>::kStage);
        load_a(f, stage);
        load_b(f, stage);
        fills++;
        if (++stage == static_cast<uint32_t>(stages)) {
            stage = 0;
            phase ^= 1u;
        }
    }
    // the fills that no later fill waited for
    const uint32_t first = fills > static_cast<uint32_t>(stages) ? fills - stages : 0;
#pragma unroll 1
    for (uint32_t f = first; f < fills && ok; f++) {
        if (!mbar_wait(&empty[f % stages], (f / stages) & 1u, abort)) {
            record_timeout(status, abort);
            ok = false;
        }
    }
    // copies still in flight must land before the pair leaves: the leader's
    // barriers track both CTAs' (the peer, which cannot wait on them, stays
    // with it: teardown)
    if (!ok && rank == 0) {
        for (uint32_t f = first; f < fills; f++) drain_wait(&full[f % stages], (f / stages) & 1u);
    }
}

// One thread of the leader.
template <int NG>
__device__ __forceinline__ void mma_issuer_pair(const Work& w, uint8_t* ring, int stages, uint64_t* full,
                                                uint64_t* empty, uint64_t* tfull, uint64_t* tempty, uint64_t* tdown,
                                                uint32_t tmem_base, int acc_stride, volatile int* abort, int* status,
                                                int nacc) {
    constexpr uint32_t idesc = idesc_bf16_f32(2 * kTileM, 2 * NG);
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int i = 0; i < w.ntiles && ok; i++) {
        const int acc = i % nacc;
        if (!mbar_wait(&tempty[acc], ((i / nacc) & 1) ^ 1u, abort)) {
            record_timeout(status, abort);
            ok = false;
            break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * acc_stride;
#pragma unroll 1
        for (int kb = w.kb0; kb < w.kb1; kb++) {
            if (!mbar_wait(&full[stage], phase, abort)) {
                record_timeout(status, abort);
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t a = smem_u32(ring + stage * PairLayout<NG>::kStage);
            const uint32_t hb = a + kATileBytes;
#pragma unroll
            for (int kk = 0; kk < kBlockK / 16; kk++)
                tc_mma_bf16_pair(d_tmem, sdesc_sw128(a + kk * 32), sdesc_sw128(hb + kk * 32), idesc,
                                 (kb > w.kb0 || kk > 0) ? 1u : 0u);
            tc_commit_pair(&empty[stage]);
            if (++stage == static_cast<uint32_t>(stages)) {
                stage = 0;
                phase ^= 1u;
            }
        }
        if (ok) tc_commit_pair(&tfull[acc]);
    }
    if (!ok) {
        tc_commit_pair(tdown);
        drain_wait(tdown, 0);
    }
}

struct Smem {
    uint8_t* ring;
    uint64_t *full, *empty, *tfull, *tempty, *tdown;
    int* misc;  // [0] tmem base, [1] abort flag, [2] epilogue flag, [3] pairs: the other CTA's abort flag
    uint8_t* tail;
};

template <int NG, bool kPair = false>
__device__ __forceinline__ Smem carve(uint8_t* raw, int stages, int nacc = 2) {
    Smem s;
    const uint32_t off = (1024u - (smem_u32(raw) & 1023u)) & 1023u;
    s.ring = raw + off;
    s.full = reinterpret_cast<uint64_t*>(s.ring + stages * (kPair ? PairLayout<NG>::kStage : Layout<NG>::kStage));
    s.empty = s.full + stages;
    s.tfull = s.empty + stages;
    s.tempty = s.tfull + nacc;
    s.tdown = s.tempty + nacc;
    s.misc = reinterpret_cast<int*>(s.tdown + 1);
    s.tail = reinterpret_cast<uint8_t*>(s.misc + 4);
    return s;
}

template <int NG, bool kPair = false>
__device__ __forceinline__ uint32_t setup(const Smem& s, int stages, int ncols, int nacc = 2) {
    constexpr int kEpi = epi_threads<NG>();
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int i = 0; i < stages; i++) {
            mbar_init(&s.full[i], 1);
            mbar_init(&s.empty[i], 1);
        }
        for (int i = 0; i < nacc; i++) {
            mbar_init(&s.tfull[i], 1);
            mbar_init(&s.tempty[i], kPair ? 2 * kEpi / 32 : kEpi);  // pairs: a lane of every warp of both CTAs
        }
        mbar_init(s.tdown, 1);
        s.misc[1] = 0;
        s.misc[2] = 0;
        s.misc[3] = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        if constexpr (kPair) {
            tmem_alloc_pair(reinterpret_cast<uint32_t*>(&s.misc[0]), ncols);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(reinterpret_cast<uint32_t*>(&s.misc[0]), ncols);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (kPair) cluster_sync_all();  // the peer's barriers are initialised
    tc_fence_after();
    return static_cast<uint32_t>(s.misc[0]);
}

// Debug builds: every phase of this CTA's `empty` and `tfull` barriers that
// the pair's commits end has ended when its threads are done (unless a wait
// gave up).
__device__ __forceinline__ void check_pair_quiet(const Smem& s, const Work& w, int stages, int nacc, int* status) {
#ifdef DART_DEBUG
    __syncthreads();
    if (threadIdx.x != 0 || s.misc[1] != 0) return;
    const int fills = w.ntiles * (w.kb1 - w.kb0);
    bool quiet = true;
    for (int f = max(fills - stages, 0); f < fills; f++)
        quiet = mbar_test_wait(&s.empty[f % stages], static_cast<uint32_t>(f / stages) & 1u) && quiet;
    for (int i = max(w.ntiles - nacc, 0); i < w.ntiles; i++)
        quiet = mbar_test_wait(&s.tfull[i % nacc], static_cast<uint32_t>(i / nacc) & 1u) && quiet;
    bounds_check(status, quiet);
#endif
}

template <bool kPair = false>
__device__ __forceinline__ void teardown(uint32_t tmem_base, int ncols, int* misc = nullptr) {
    tc_fence_before();
    __syncthreads();
    if constexpr (kPair) {
        // neither CTA leaves while the other's threads may still signal it,
        // and neither frees the TMEM that its MMAs write
        if (threadIdx.x == 0) st_cluster_s32(smem_u32(&misc[3]), cluster_ctarank() ^ 1u, misc[1]);
        cluster_sync_all();
    }
    if ((threadIdx.x >> 5) == 1) {
        __syncwarp();
        tc_fence_after();
        if constexpr (kPair) {
            // A wait gave up in one of the two: copies and arrivals that were
            // not waited for land within a millisecond (the leader has issued
            // its last commit and seen it complete before the barrier).
            if (misc[1] != 0 || misc[3] != 0) {
                const unsigned long long t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 1000000ull) {
                }
            }
            __syncwarp();
        }
        if constexpr (kPair) tmem_dealloc_pair(tmem_base, ncols);
        else tmem_dealloc(tmem_base, ncols);
    }
}

// One accumulator = 2*NG fp32 columns (hi products, then lo products).
template <int NG>
constexpr int acc_stride() {
    return 2 * NG < 32 ? 32 : 2 * NG;
}
// TMEM columns of a GEMM CTA: one tile, hence one accumulator (a power of two
// of at least 32 columns).
template <int NG>
constexpr int tmem_cols() {
    return acc_stride<NG>();
}

// Accumulators of the LM-head (a ring in TMEM): with 64-node groups four,
// so that the MMAs run up to three tiles ahead of the epilogue, whose cost
// per tile is uneven (the first tiles of a vocabulary range pass most
// logits to the top-k merges, later ones few).  All of TMEM then belongs to
// one CTA, which the plan's shared memory makes the only LM-head CTA of its SM.
template <int NG>
constexpr int lm_nacc() {
    return NG == 64 ? 4 : 2;
}
template <int NG>
constexpr int lm_tmem_cols() {
    return lm_nacc<NG>() * acc_stride<NG>() <= 32
               ? 32
               : (lm_nacc<NG>() * acc_stride<NG>() <= 64
                      ? 64
                      : (lm_nacc<NG>() * acc_stride<NG>() <= 128 ? 128
                                                                 : (lm_nacc<NG>() * acc_stride<NG>() <= 256 ? 256 : 512)));
}

// ------------------------------------------------------------ LM-head kernel

// kPair: two neighbouring vocabulary ranges of a node group as a CTA pair.
// With 128-node groups the L2 -> SM bytes bound the launch (an SM takes in
// about 64 bytes per clock): alone a CTA loads 16 KB of E and 32 KB of hi and
// lo states per k-block, in a pair 16 KB of each.  Ranges, tiles and the order
// of every sum are those of the single CTAs.  Measured on GB300, 256 nodes,
// V = 151936, d = 4096 (µs per launch): single CTAs 450 (0.45 µs per k-block,
// 107 GB/s into each SM), pairs with 4 stages 403, with 5 389.
// (kCap: candidate slots per node, cand_slots)
template <int NG, bool kPair, int kCap = lm_cand_cap<NG>()>
__global__ void __launch_bounds__(threads<NG>(), 1)
    lmhead_tc_kernel(const __grid_constant__ CUtensorMap tmE, const __grid_constant__ CUtensorMap tmH,
                     const LmheadArgs a) {
    extern __shared__ uint8_t smem_raw[];
    pdl_trigger();
    const int stages = a.stages;
    constexpr int kNacc = lm_nacc<NG>();
    Smem s = carve<NG, kPair>(smem_raw, stages, kNacc);
    EpiSmem e;
    e.cap = kCap;
    e.list = reinterpret_cast<uint64_t*>(s.tail);
    e.cand = e.list + NG * a.k;
    e.gcache = e.cand + NG * kCap;
    e.stats = reinterpret_cast<float2*>(e.gcache + NG);
    e.mref = reinterpret_cast<float*>(e.stats + 4 * NG);
    e.cnt = reinterpret_cast<int*>(e.mref + 4 * NG);
    e.more = e.cnt + NG;

    // (pairs: blocks 2 q and 2 q + 1 are ranges 2 r and 2 r + 1 of one group)
    const int g = (kPair ? blockIdx.x / 2 : blockIdx.x) % a.G;
    const int vr = kPair ? (blockIdx.x / 2 / a.G) * 2 + (blockIdx.x & 1) : blockIdx.x / a.G;
    const int t0 = static_cast<int>((static_cast<long long>(vr) * a.tiles) / a.nV);
    const int t1 = static_cast<int>((static_cast<long long>(vr + 1) * a.tiles) / a.nV);
    Work w;
    w.ntiles = t1 - t0;
    w.row0 = t0 * kTileM;
    w.kb0 = 0;
    w.kb1 = a.d / kBlockK;
    w.brow = g * NG;
    w.lo_kb_end = w.kb1;
    w.tiled_kb = a.e_tiled ? w.kb1 : 0;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem_base = setup<NG, kPair>(s, stages, lm_tmem_cols<NG>(), kNacc);
    volatile int* abort = &s.misc[1];
    // a pair walks as many tiles as its longer range: the shorter range's
    // last accumulator (rows of the next range, or past V: zeros) is not read
    const int own = w.ntiles;
    if constexpr (kPair) {
        const int o0 = static_cast<int>((static_cast<long long>(vr ^ 1) * a.tiles) / a.nV);
        const int o1 = static_cast<int>((static_cast<long long>((vr ^ 1) + 1) * a.tiles) / a.nV);
        w.ntiles = max(own, o1 - o0);
    }

    if (warp == 0) {
        if (lane == 0) {
            if constexpr (kPair)
                producer_pair<NG>(&tmE, &tmH, w, blockIdx.x & 1, a.bhalf, s.ring, stages, s.full, s.empty, abort, a.status);
            else
                producer<NG>(&tmE, &tmH, w, a.bhalf, s.ring, stages, s.full, s.empty, abort, a.status, a.l2pf);
        }
    } else if (warp == 1) {
        if constexpr (kPair) {
            if (lane == 0 && (blockIdx.x & 1) == 0)
                mma_issuer_pair<NG>(w, s.ring, stages, s.full, s.empty, s.tfull, s.tempty, s.tdown, tmem_base,
                                    acc_stride<NG>(), abort, a.status, kNacc);
        } else {
            if (lane == 0)
                mma_issuer<NG>(w, s.ring, stages, s.full, s.empty, s.tfull, s.tempty, s.tdown, tmem_base,
                               acc_stride<NG>(), abort, a.status, kNacc);
        }
    } else {
        // epilogue warp wi = warp - 2 reads TMEM lane quarter warp % 4 and
        // owns the 16-node chunks wi / 4 + 4 * ci (ci < kChunks) of the group
        constexpr int kEpi = epi_threads<NG>();
        constexpr int kChunks = epi_chunks<NG>();
        const int etid = threadIdx.x - 64;
        const int wi = warp - 2;
        const int quarter = warp & 3;
        pdl_wait();
        epi_init(e, NG, a.k, etid, kEpi, a.gthr, g * NG, a.N, a.seed_y, a.seed_R, vr == 0);
        float ssum[kChunks];
        uint32_t nodemask[kChunks];
#pragma unroll
        for (int ci = 0; ci < kChunks; ci++) {
            const int c0 = ((wi >> 2) + 4 * ci) * 16;
            ssum[ci] = 0.0f;
            // bit j: node c0 + j exists; bit 16 + j: it starts a sequence (or the chunk)
            nodemask[ci] = 0;
            int left = 0;
#pragma unroll 1
            for (int j = 0; j < 16; j++) {
                if (j == 0) left = a.P - (g * NG + c0) % a.P;
                if (g * NG + c0 + j < a.N) nodemask[ci] |= (j == 0 || left == 0 ? 0x10001u : 1u) << j;
                if (left == 0) left = a.P;
                left--;
            }
        }
        // scaled logits of this thread's row v for chunk ci from accumulator acc:
        // hi + lo products, drafter row added, 1/T applied
        auto load_z = [&](int acc, int ci, int v, bool valid, float (&z)[16]) {
            const int c0 = ((wi >> 2) + 4 * ci) * 16;
            float zl[16];
            const uint32_t tcol =
                tmem_base + acc * acc_stride<NG>() + c0 + (static_cast<uint32_t>(quarter * 32) << 16);
            tmem_ld16_pair(tcol, tcol + NG, z, zl);
#pragma unroll
            for (int j = 0; j < 16; j++) z[j] += zl[j];
            int seq = (g * NG + c0) / a.P - 1;
            float dl = 0.0f;
#pragma unroll
            for (int j = 0; j < 16; j++) {
                if ((nodemask[ci] >> j) & 1u) {
                    if ((nodemask[ci] >> (16 + j)) & 1u) {  // the first node of a sequence, or of the chunk
                        seq++;
                        const long long off = a.dlog_row ? static_cast<long long>(__ldg(a.dlog_row + seq)) * a.V
                                                         : a.dlog_row_off;
                        dl = valid ? __ldg(a.dlog + seq * a.dlog_seq_stride + off + v) : 0.0f;
                    }
                    z[j] = (z[j] + dl) * a.invT;
                }
            }
        };
        // the accumulator has been read: the (leader's) next MMAs may overwrite it
        auto release = [&](int acc) {
            tc_fence_before();
            if constexpr (kPair) {
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(mapa_u32(smem_u32(&s.tempty[acc]), 0));
            } else {
                mbar_arrive(&s.tempty[acc]);
            }
        };
        for (int i = 0; i < own; i++) {
            const int acc = i % kNacc;
            const uint32_t aph = (i / kNacc) & 1;
            if (etid == 0) {
                const bool ok = mbar_wait(&s.tfull[acc], aph, abort);
                if (!ok) record_timeout(a.status, abort);
                s.misc[2] = ok ? 1 : 0;
            }
            named_bar_sync(kEpiBarrier, kEpi);
            if (s.misc[2] == 0) break;
            tc_fence_after();
            const int v = w.row0 + i * kTileM + quarter * 32 + lane;
            const bool valid = v < a.V;
            if constexpr (kCap >= kTileM) {
                // every candidate of the tile fits: one merge, and the
                // accumulator is released as soon as it has been read
                float z[16];
                load_z(acc, 0, v, valid, z);
                release(acc);
                if (a.zout && valid) {
                    const int nb = g * NG + (wi >> 2) * 16;
#pragma unroll
                    for (int j = 0; j < 16; j++)
                        if ((nodemask[0] >> j) & 1u) a.zout[static_cast<long long>(nb + j) * a.zout_stride + v] = z[j];
                }
                (void)epi_chunk(e, NG, a.k, quarter, lane, (wi >> 2) * 16, z, nodemask[0], valid,
                                static_cast<uint32_t>(v), ssum[0]);
                epi_merge(e, NG, a.k, wi, lane, kEpi, etid, a.gthr, g * NG, a.N);
            } else {
                uint32_t pend[kChunks];
#pragma unroll
                for (int ci = 0; ci < kChunks; ci++) {
                    float z[16];
                    load_z(acc, ci, v, valid, z);
                    pend[ci] = epi_chunk(e, NG, a.k, quarter, lane, ((wi >> 2) + 4 * ci) * 16, z, nodemask[ci],
                                         valid, static_cast<uint32_t>(v), ssum[ci]);
                }
                // Merge rounds while some candidate found no free slot: those
                // still beating the raised thresholds are read again from the
                // accumulator (kept until the last round) and offered again.
                // A round's flag is set before epi_merge's first barrier, read
                // after its second, and cleared in the next round after that
                // round's first barrier.
                for (int round = 0;; round++) {
                    bool any = false;
#pragma unroll
                    for (int ci = 0; ci < kChunks; ci++) any |= pend[ci] != 0u;
                    if (__any_sync(kFull, any) && lane == 0) atomicOr(&e.more[round & 1], 1);
                    epi_merge(e, NG, a.k, wi, lane, kEpi, etid, a.gthr, g * NG, a.N,
                              round > 0 ? &e.more[(round + 1) & 1] : nullptr);
                    if (e.more[round & 1] == 0) break;
#pragma unroll
                    for (int ci = 0; ci < kChunks; ci++) {
                        if (__any_sync(kFull, pend[ci] != 0u)) {
                            const int c0 = ((wi >> 2) + 4 * ci) * 16;
                            float z[16];
                            load_z(acc, ci, v, valid, z);
                            pend[ci] = epi_offer(e, c0, z, epi_still_pass(e, a.k, c0, z, pend[ci], static_cast<uint32_t>(v)),
                                                 static_cast<uint32_t>(v), lane);
                        }
                    }
                }
                release(acc);
            }
        }
#pragma unroll
        for (int ci = 0; ci < kChunks; ci++) epi_stash(e, NG, quarter, lane, ((wi >> 2) + 4 * ci) * 16, ssum[ci]);
        epi_finalize(e, NG, a.k, etid, kEpi, g * NG, a.N, vr, a.nV, a.part_ms, a.part_key);
        if constexpr (kPair) {
            // the accumulator of the longer range's last tile is not read here, but its commit arrives here too
            if (etid == 0 && own < w.ntiles && s.misc[2] != 0 &&
                !mbar_wait(&s.tfull[own % kNacc], (own / kNacc) & 1, abort))
                record_timeout(a.status, abort);
        }
    }
    if constexpr (kPair) check_pair_quiet(s, w, stages, kNacc, a.status);
    teardown<kPair>(tmem_base, lm_tmem_cols<NG>(), s.misc);
}

// --------------------------------------------------------------- GEMM kernel
//
// Correction-head layer out = A . B^T with A = W_i or W_o [M x K] and B the
// node inputs [N x K], split over K into a.S parts.
//   kGemmPartials:  every CTA writes its fp32 partial tile to out[split]; the
//                   elementwise kernels that follow sum the splits.
//   kGemmSiluSplit, kGemmSum: the S splits of one (M tile, node group) form
//                   a thread-block cluster: every CTA stages its fp32 tile in
//                   shared memory, and after a cluster barrier CTA r sums
//                   rows [r*R, (r+1)*R) of the tile over the S CTAs in rank
//                   order (deterministic) and writes outL = hi/lo bf16 split
//                   of SiLU(sum) (input of W_o), or out = sum in fp32.

// (two CTAs per SM: at most 56 registers per thread)
template <int NG>
__global__ void __launch_bounds__(threads<NG>(), 2)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const GemmArgs a) {
    extern __shared__ uint8_t smem_raw[];
    pdl_trigger();
    const int stages = a.stages;
    Smem s = carve<NG>(smem_raw, stages);

    // block = (g * MT + mt) * S + split: the S splits of a tile are consecutive,
    // i.e. one cluster
    const int tile = blockIdx.x / a.S;
    const int mt_c = tile % a.MT, g_c = tile / a.MT, split_c = blockIdx.x % a.S;
    Work w;
    w.ntiles = 1;
    w.row0 = mt_c * kTileM;
    w.kb0 = static_cast<int>((static_cast<long long>(split_c) * a.KB) / a.S);
    w.kb1 = static_cast<int>((static_cast<long long>(split_c + 1) * a.KB) / a.S);
    w.brow = g_c * NG;
    w.lo_kb_end = a.lo_kb_end;
    w.tiled_kb = a.a_tiled_kb;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem_base = setup<NG>(s, stages, tmem_cols<NG>());
    volatile int* abort = &s.misc[1];
    // staging tile [NG nodes][128 rows] fp32, in the pipeline ring (free once
    // the last MMA has completed)
    float* stage_tile = reinterpret_cast<float*>(s.ring);

    if (warp == 0) {
        if (lane == 0)
            producer<NG>(&tmA, &tmB, w, a.bhalf, s.ring, stages, s.full, s.empty, abort, a.status, 0, a.keep_a != 0);
    } else if (warp == 1) {
        if (lane == 0)
            mma_issuer<NG>(w, s.ring, stages, s.full, s.empty, s.tfull, s.tempty, s.tdown, tmem_base,
                           acc_stride<NG>(), abort, a.status);
    } else {
        const int etid = threadIdx.x - 64;
        const int quarter = warp & 3;
        pdl_wait();
        if (etid == 0) {
            const bool ok = mbar_wait(&s.tfull[0], 0, abort);
            if (!ok) record_timeout(a.status, abort);
            s.misc[2] = ok ? 1 : 0;
        }
        named_bar_sync(kEpiBarrier, epi_threads<NG>());
        if (s.misc[2] != 0) {
            tc_fence_after();
            const int c0 = ((warp - 2) >> 2) * 16;
            float vals[16], lov[16];
            const uint32_t tcol = tmem_base + c0 + (static_cast<uint32_t>(quarter * 32) << 16);
            tmem_ld16_pair(tcol, tcol + NG, vals, lov);
            // lo columns were written only if this split saw a k-block with a lo half
            if (w.kb0 < w.lo_kb_end) {
#pragma unroll
                for (int j = 0; j < 16; j++) vals[j] += lov[j];
            }
            if (a.mode == kGemmPartials) {
                const int m = w.row0 + quarter * 32 + lane;
                float* out = a.out + static_cast<size_t>(split_c) * a.N * a.M;
#pragma unroll
                for (int j = 0; j < 16; j++) {
                    const int n = g_c * NG + c0 + j;
                    if (m < a.M && n < a.N) out[static_cast<size_t>(n) * a.M + m] = vals[j];
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; j++) stage_tile[(c0 + j) * kTileM + quarter * 32 + lane] = vals[j];
            }
        }
    }
    teardown(tmem_base, tmem_cols<NG>());
    if (a.mode == kGemmPartials) return;  // launched without clusters
    cluster_sync_all();  // every split's tile is staged
    {
        // units of 4 rows (M is a multiple of 64: a unit is inside or outside whole)
        const int S = a.S;
        const uint32_t r = cluster_ctarank();
        const int u0 = static_cast<int>(r) * (kTileM / 4) / S, nu = (static_cast<int>(r) + 1) * (kTileM / 4) / S - u0;
        const uint32_t base = smem_u32(stage_tile);
#pragma unroll 1
        for (int idx = threadIdx.x; idx < nu * NG; idx += threads<NG>()) {
            const int nl = idx / nu, row = (u0 + idx % nu) * 4;
            const int m = w.row0 + row, n = g_c * NG + nl;
            if (m >= a.M || n >= a.N) continue;
            const uint32_t off = base + static_cast<uint32_t>((nl * kTileM + row) * 4);
            float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 1
            for (int q0 = 0; q0 < S; q0 += 4) {  // four loads in flight
                float4 v[4];
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (q0 + q < S) v[q] = ld_cluster_f32x4(off, static_cast<uint32_t>(q0 + q));
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    if (q0 + q < S) {
                        acc.x += v[q].x;
                        acc.y += v[q].y;
                        acc.z += v[q].z;
                        acc.w += v[q].w;
                    }
                }
            }
            const size_t o = static_cast<size_t>(n) * a.M + m;
            if (a.mode == kGemmSiluSplit) {
                const float act[4] = {acc.x / (1.0f + expf(-acc.x)), acc.y / (1.0f + expf(-acc.y)),
                                      acc.z / (1.0f + expf(-acc.z)), acc.w / (1.0f + expf(-acc.w))};
                __align__(8) __nv_bfloat16 hi[4], lo[4];
#pragma unroll
                for (int e = 0; e < 4; e++) split_bf16(act[e], hi[e], lo[e]);
                *reinterpret_cast<uint2*>(a.outL + o) = *reinterpret_cast<const uint2*>(hi);
                *reinterpret_cast<uint2*>(a.outL + static_cast<size_t>(a.bhalf) * a.M + o) =
                    *reinterpret_cast<const uint2*>(lo);
            } else {
                *reinterpret_cast<float4*>(a.out + o) = acc;
            }
        }
    }
    cluster_sync_all();  // no CTA leaves while a peer still reads its staging tile
}

template <int NG>
int lmhead_fixed(int k, int stages, int cap) {
    return (2 * stages + 2 * lm_nacc<NG>() + 1) * 8 + 16 + NG * k * 8 + NG * cap * 8 + NG * 8 + 4 * NG * 8 + 4 * NG * 4 +
           NG * 4 + 8;
}

// The failure path of the bounded waits, exercised without a fault: two
// mbarriers that nothing ever completes (count 1, no arrival, no copy or MMA
// tracked by them).  Thread 0 waits with limit_ns, gives up and records the
// timeout exactly as the pipeline roles do (abort flag + status bit); thread
// 32 waits with the kernels' own limit and returns once it sees the abort
// flag.  Each records how long its wait took.
__global__ void __launch_bounds__(64) wait_probe_kernel(int* status, unsigned long long limit_ns,
                                                        long long* elapsed_ns) {
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    volatile int* abort = &abort_flag;
    const unsigned long long t0 = globaltimer_ns();
    long long took = -1;
    if (threadIdx.x == 0) {
        if (!mbar_wait(&bar[0], 0, abort, limit_ns)) record_timeout(status, abort);
        took = static_cast<long long>(globaltimer_ns() - t0);
    } else if (threadIdx.x == 32) {
        if (!mbar_wait(&bar[1], 0, abort)) took = static_cast<long long>(globaltimer_ns() - t0);
    }
    if (elapsed_ns && took >= 0) elapsed_ns[threadIdx.x == 0 ? 0 : 1] = took;
}

template <int NG>
cudaError_t launch_lmhead_ng(const CUtensorMap* tmE, const CUtensorMap* tmH, const LmheadArgs& a, int smem,
                             cudaStream_t st) {
    if constexpr (NG == 128) {
        constexpr int kFew = kCandCapLarge / 2;
        if (a.pair)
            return launch_pdl_cluster(a.cap == kFew ? lmhead_tc_kernel<NG, true, kFew> : lmhead_tc_kernel<NG, true>,
                                      dim3(a.nV * a.G), dim3(threads<NG>()), smem, st, 2, *tmE, *tmH, a);
        if (a.cap == kFew)
            return launch_pdl(lmhead_tc_kernel<NG, false, kFew>, dim3(a.nV * a.G), dim3(threads<NG>()), smem, st, *tmE,
                              *tmH, a);
    }
    return launch_pdl(lmhead_tc_kernel<NG, false>, dim3(a.nV * a.G), dim3(threads<NG>()), smem, st, *tmE, *tmH, a);
}
template <int NG>
cudaError_t launch_gemm_ng(const CUtensorMap* tmA, const CUtensorMap* tmB, const GemmArgs& a, int smem,
                           cudaStream_t st) {
    if (a.mode == kGemmPartials)
        return launch_pdl(gemm_tc_kernel<NG>, dim3(a.MT * a.G * a.S), dim3(threads<NG>()), smem, st, *tmA, *tmB, a);
    return launch_pdl_cluster(gemm_tc_kernel<NG>, dim3(a.MT * a.G * a.S), dim3(threads<NG>()), smem, st, a.S, *tmA,
                              *tmB, a);
}

template <int NG>
int max_clusters_ng(int smem, int cluster) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster * 1024);
    cfg.blockDim = dim3(threads<NG>());
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_tc_kernel<NG>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

}  // namespace

int tc_stage_bytes(int NG) { return kATileBytes + 2 * NG * 128; }

int lmhead_tc_tmem_cols(int NG) {
    switch (NG) {
        case 16: return lm_tmem_cols<16>();
        case 32: return lm_tmem_cols<32>();
        case 64: return lm_tmem_cols<64>();
        default: return lm_tmem_cols<128>();
    }
}

int lmhead_tc_fixed_smem(int NG, int k, int stages, int cap) {
    switch (NG) {
        case 16: return lmhead_fixed<16>(k, stages, cap) + 1024;
        case 32: return lmhead_fixed<32>(k, stages, cap) + 1024;
        case 64: return lmhead_fixed<64>(k, stages, cap) + 1024;
        default: return lmhead_fixed<128>(k, stages, cap) + 1024;
    }
}

int gemm_tc_fixed_smem(int stages) { return (2 * stages + 5) * 8 + 16 + 1024; }

// Resident CTAs per SM for a kernel with `smem` bytes of dynamic shared
// memory, from the device limits (shared memory with the per-block
// reservation, register file at 8-register granularity, threads).
static int ctas_per_sm(const void* fn, int nthreads, int smem) {
    int dev = 0, sm_smem = 0, reserved = 0, sm_regs = 0, sm_threads = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaFuncGetAttributes(&fa, fn) != cudaSuccess ||
        cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sm_regs, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sm_threads, cudaDevAttrMaxThreadsPerMultiProcessor, dev) != cudaSuccess)
        return 1;
    const int per_smem = smem + static_cast<int>(fa.sharedSizeBytes) + reserved;
    const int per_regs = ((fa.numRegs + 7) / 8) * 8 * nthreads;
    int n = per_smem > 0 ? sm_smem / per_smem : 1;
    if (per_regs > 0) n = std::min(n, sm_regs / per_regs);
    n = std::min(n, sm_threads / nthreads);
    return std::max(n, 1);
}

int gemm_tc_ctas_per_sm(int NG, int smem) {
    switch (NG) {
        case 16: return ctas_per_sm(reinterpret_cast<const void*>(gemm_tc_kernel<16>), threads<16>(), smem);
        case 32: return ctas_per_sm(reinterpret_cast<const void*>(gemm_tc_kernel<32>), threads<32>(), smem);
        default: return ctas_per_sm(reinterpret_cast<const void*>(gemm_tc_kernel<64>), threads<64>(), smem);
    }
}

int gemm_tc_max_clusters(int NG, int smem, int cluster) {
    switch (NG) {
        case 16: return max_clusters_ng<16>(smem, cluster);
        case 32: return max_clusters_ng<32>(smem, cluster);
        default: return max_clusters_ng<64>(smem, cluster);
    }
}

int lmhead_tc_ctas_per_sm(int NG, int smem) {
    switch (NG) {
        case 16: return ctas_per_sm(reinterpret_cast<const void*>(lmhead_tc_kernel<16, false>), threads<16>(), smem);
        case 32: return ctas_per_sm(reinterpret_cast<const void*>(lmhead_tc_kernel<32, false>), threads<32>(), smem);
        case 64: return ctas_per_sm(reinterpret_cast<const void*>(lmhead_tc_kernel<64, false>), threads<64>(), smem);
        default: return ctas_per_sm(reinterpret_cast<const void*>(lmhead_tc_kernel<128, false>), threads<128>(), smem);
    }
}

// Node groups from which two vocabulary ranges work as a CTA pair.  64-node
// groups (16 + 16 KB per k-block alone) gain nothing from it: 136 µs per launch
// either way at V = 151936, d = 2560, where HBM bounds them, and 3 x 11 nodes
// at V = 50021, d = 1088 lost 4 %.
constexpr int kLmheadPairNG = 128;

bool plan_lmhead_tc(int N, int V, int d, int k, int num_sms, int smem_optin, int ctas_per_sm_pref, bool e_tiled,
                    bool bounded, LmheadPlan* out) {
    LmheadPlan p;
    p.NG = N <= 16 ? 16 : (N <= 32 ? 32 : (N <= 64 ? 64 : 128));
    p.G = (N + p.NG - 1) / p.NG;
    const int tiles = (V + kTileM - 1) / kTileM;
    p.nV = std::max(1, std::min(num_sms / p.G, tiles));
    // CTA pairs: an even number of vocabulary ranges of at least one tile
    const int nv1 = std::max(1, std::min(num_sms / p.G, tiles));
    p.pair = p.NG >= kLmheadPairNG && nv1 % 2 == 0;
    const int sb = p.pair ? kATileBytes + p.NG * 128 : tc_stage_bytes(p.NG);
    p.cap = cand_slots(p.NG, bounded, nv1 >= tiles);
    const int fixed = lmhead_tc_fixed_smem(p.NG, k, 16, p.cap);
    auto stages_in = [&](int budget) { return std::min(16, (budget - fixed) / sb); };
    // Two CTAs per SM when both fit with >= 4 pipeline stages each: two
    // independent TMA streams per SM, and one CTA's epilogue / start-up /
    // tail overlaps the other's stream.  Measured on GB300 (A/B per round):
    // with E row-major it pays for short rows (d = 2560: -4 %) but not for
    // d = 4096 (+6 %), where the deeper single-CTA pipeline wins; with E in
    // contiguous 16 KB tiles two CTAs win at d = 4096 too (-3.6 % against
    // one CTA on the same tiles, -1.0 % against row-major with one).
    const int st2 = stages_in(smem_optin / 2 - 2048);
    const int smem2 = lmhead_tc_fixed_smem(p.NG, k, st2, p.cap) + st2 * sb;
    const bool want2 = ctas_per_sm_pref ? ctas_per_sm_pref == 2 : (e_tiled || d <= 3072);
    if (!p.pair && want2 && st2 >= 4 && 2 * lmhead_tc_tmem_cols(p.NG) <= 512 && lmhead_tc_ctas_per_sm(p.NG, smem2) >= 2) {
        p.stages = st2;
        p.nV = std::max(1, std::min(2 * num_sms / p.G, tiles));
    } else {
        p.stages = stages_in(smem_optin);
    }
    if (p.stages < 2) return false;
    p.smem = lmhead_tc_fixed_smem(p.NG, k, p.stages, p.cap) + p.stages * sb;
    *out = p;
    return true;
}

cudaError_t tc_set_smem_limits(int max_dyn) {
    cudaError_t e = cudaSuccess;
#define DART_SET(fn)                                                                                   \
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn); \
    if (e == cudaSuccess)                                                                              \
        e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    DART_SET((lmhead_tc_kernel<16, false>))
    DART_SET((lmhead_tc_kernel<32, false>))
    DART_SET((lmhead_tc_kernel<64, false>))
    DART_SET((lmhead_tc_kernel<128, false>))
    DART_SET((lmhead_tc_kernel<128, true>))
    DART_SET((lmhead_tc_kernel<128, false, kCandCapLarge / 2>))
    DART_SET((lmhead_tc_kernel<128, true, kCandCapLarge / 2>))
    DART_SET(gemm_tc_kernel<16>)
    DART_SET(gemm_tc_kernel<32>)
    DART_SET(gemm_tc_kernel<64>)
#undef DART_SET
    return e;
}

cudaError_t launch_lmhead_tc(const CUtensorMap* tmE, const CUtensorMap* tmH, const LmheadArgs& a, int smem,
                             cudaStream_t st) {
    switch (a.NG) {
        case 16: return launch_lmhead_ng<16>(tmE, tmH, a, smem, st);
        case 32: return launch_lmhead_ng<32>(tmE, tmH, a, smem, st);
        case 64: return launch_lmhead_ng<64>(tmE, tmH, a, smem, st);
        case 128: return launch_lmhead_ng<128>(tmE, tmH, a, smem, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_gemm_tc(const CUtensorMap* tmA, const CUtensorMap* tmB, const GemmArgs& a, int smem,
                           cudaStream_t st) {
    switch (a.NG) {
        case 16: return launch_gemm_ng<16>(tmA, tmB, a, smem, st);
        case 32: return launch_gemm_ng<32>(tmA, tmB, a, smem, st);
        case 64: return launch_gemm_ng<64>(tmA, tmB, a, smem, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_wait_probe(int* status, unsigned long long limit_ns, long long* elapsed_ns, cudaStream_t st) {
    wait_probe_kernel<<<1, 64, 0, st>>>(status, limit_ns, elapsed_ns);
    return cudaGetLastError();
}

namespace {

// dst = src [rows][cols] bf16 (row pitch `pitch`) re-laid as 128 x 64 tiles, tile (rt, kb)
// (rows 128 rt .., columns 64 kb ..) as 16 KB of contiguous memory at tile
// index rt * (cols / 64) + kb, rows 128-byte, rows past `rows` zero.  One
// thread per 16-byte chunk of dst.
__global__ void retile_kernel(const __nv_bfloat16* src, int rows, int cols, long long pitch, __nv_bfloat16* dst,
                              long long chunks) {
    const int KB = cols / kBlockK;
    for (long long q = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; q < chunks;
         q += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int c8 = static_cast<int>(q & 7);
        const int r = static_cast<int>((q >> 3) & (kTileM - 1));
        const long long tile = q >> 10;
        const long long rt = tile / KB;
        const int kb = static_cast<int>(tile % KB);
        const long long row = rt * kTileM + r;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (row < rows) v = *reinterpret_cast<const uint4*>(src + row * pitch + kb * kBlockK + c8 * 8);
        reinterpret_cast<uint4*>(dst)[q] = v;
    }
}

}  // namespace

cudaError_t launch_retile(const __nv_bfloat16* src, int rows, int cols, long long pitch, __nv_bfloat16* dst,
                          cudaStream_t st) {
    const long long rt = (rows + kTileM - 1) / kTileM;
    const long long chunks = rt * (cols / kBlockK) * kTileM * 8;
    retile_kernel<<<4096, 256, 0, st>>>(src, rows, cols, pitch, dst, chunks);
    return cudaGetLastError();
}

namespace {

// The first `count` E tiles of every CTA of an LM-head launch (nV vocabulary
// ranges of whole tiles, the same split as lmhead_tc_kernel) prefetched into
// L2, one block per range so that every SM's TMA unit issues its own share
// (one unit issuing them all takes hundreds of microseconds).  Launched beside
// the selection of the previous depth, while HBM would otherwise wait.
__global__ void lmhead_l2_prefetch_kernel(const __grid_constant__ CUtensorMap tmE, int tiles, int nV, int KB, int count,
                                          int tiled) {
    const int vr = blockIdx.x;
    if (threadIdx.x != 0 || vr >= nV) return;
    const int t0 = static_cast<int>((static_cast<long long>(vr) * tiles) / nV);
    const int t1 = static_cast<int>((static_cast<long long>(vr + 1) * tiles) / nV);
    Work w;
    w.ntiles = t1 - t0;
    w.row0 = t0 * kTileM;
    w.kb0 = 0;
    w.kb1 = KB;
    w.brow = 0;
    w.lo_kb_end = KB;
    w.tiled_kb = tiled ? KB : 0;
    const int total = w.ntiles * KB;
    for (int f = 0; f < count && f < total; f++) tma_prefetch_2d(&tmE, a_x(w, f % KB), a_y(w, f / KB, f % KB));
}

}  // namespace

cudaError_t launch_lmhead_l2_prefetch(const CUtensorMap* tmE, int tiles, int nV, int d, int count, int tiled,
                                      cudaStream_t st) {
    const int KB = d / kBlockK;
    lmhead_l2_prefetch_kernel<<<nV, 32, 0, st>>>(*tmE, tiles, nV, KB, count, tiled);
    return cudaGetLastError();
}

}  // namespace dart
