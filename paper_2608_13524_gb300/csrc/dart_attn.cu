// Tree-attention verification consumer of the emitted draft tree (Sec. 3.3,
// "Tree Verification and DDTree": every flattened tree node attends to the
// verified context and to the tokens on its root-to-node path; Sec. 4.3
// hands the pruned tree to that single forward pass).  Contract:
// include/dart_verify.h.
//
// Launches of a call:
//   attn_prep_kernel   the RoPE (cos, sin) table of every tree position and
//                      the rotated tree keys (rotate-half RoPE in fp32,
//                      rounded to bf16) in the workspace;
//   tree_attn_kernel   flash attention on the tensor cores (tcgen05, TMEM
//                      operands and accumulators, TMA-staged K/V).  A CTA
//                      owns 128 query rows = 128/G tree rows x the G query
//                      heads sharing one kv head, so each K/V tile feeds all
//                      G heads.  Its key tiles are the context tiles (all
//                      visible, ragged tail masked) followed by the tree
//                      tiles up to its last row (ancestors precede their
//                      descendants, so later tiles are invisible), masked by
//                      the ancestor bitmask.  When there are fewer (sequence,
//                      kv head, query tile) blocks than SMs, the key list is
//                      split over a thread-block cluster of up to 4 CTAs
//                      that merge their partial (max, sum, O) over
//                      distributed shared memory, in rank order;
//   tree_attn2_kernel  the same for two query tiles per CTA, when there are
//                      more query tiles than SMs and pairs_pay says so (and
//                      tree_attn_kernel for what its last wave would leave);
// and dart_ancestor_mask's own kernel, one block per sequence.
// tree_attn_kernel, 320 threads: warp 0 TMA producer (K ring 3 stages, V ring
// 3 stages), warp 1 TMEM allocator + single-thread MMA issuer, warps 2-9 two
// softmax warpgroups; thread = query row = TMEM lane, warpgroup wg owns key
// columns and O columns [64 wg, 64 wg + 64) of the rows, the pair of warps of
// a lane quarter exchanging row max and row sum through shared memory.
// TMEM (512 columns): S [0,128), O [128,256), P double buffer [256,384), the
// rotated query tile [384,448).  S = Q K^T and O += P V both take A from
// TMEM (K K-major, V MN-major from shared memory); the softmax reads S into
// registers at once, which frees it for the next tile's S while it works.
// O stays in TMEM for the whole key range; a row's running max is raised
// (and O, l rescaled through tcgen05.ld/st) only when a tile exceeds it by
// more than 2^8, so P = exp2(s - m) <= 256 and the rescale is rare.  Every
// wait is bounded (status bit on timeout, then drain and exit).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "../../include/dart.h"
#include "../../include/dart_verify.h"
#include "dart_device.cuh"
#include "dart_kernels.h"

namespace dart {
namespace {

constexpr int kDh = 128;                  // head dimension (two 64-element swizzle columns)
constexpr int kRows = 128;                // query rows per CTA (MMA M)
constexpr int kKeys = 128;                // keys per tile (MMA N of S = QK^T, K of O += PV)
constexpr int kSoftThreads = 256;             // two softmax warpgroups: key / O columns [0,64) and [64,128)
constexpr int kAttnThreads = 64 + kSoftThreads;
constexpr int kPairBarrier0 = 2;             // named barriers 2..5: the two warps of one TMEM lane quarter
constexpr int kKStages = 3;                  // K ring: the S MMA needs K two tiles ahead of its load
constexpr int kVStages = 3;
constexpr int kHalf = kRows * 64 * 2;     // 16 KB: 128 rows x 64 bf16, one 128-byte swizzle column
constexpr int kTileBytes = 2 * kHalf;     // 32 KB: 128 rows x dh bf16
constexpr int kMaxSplits = 4;                // cluster size: clusters of 4 fit a GPC in one wave beside each other
constexpr int kTmemCols = 512;            // S [0,128), O [128,256), P0 [256,320), P1 [320,384), Q [384,448)
constexpr int kSCol = 0;
constexpr int kOCol = 128;
constexpr int kPCol = 256;                // P tiles: 128 keys as 64 columns of bf16 pairs
constexpr int kQCol = 384;                // rotated query tile: dh = 128 as 64 columns of bf16 pairs
constexpr float kRescaleSlack = 8.0f;     // log2 units: P <= 2^8 between rescales
constexpr int kNumBars = 1 + 2 * kKStages + 2 * kVStages + 2 + 5;
constexpr int kSmemUsed = kTileBytes * (1 + kKStages + kVStages) + kNumBars * 8 + 4 * 4 + 2 * 128 * 4 + 8 * 4;  // Q, K/V rings, barriers, exchange
constexpr int kAttnSmem = kSmemUsed + 1024;  // + alignment slack of the 1024-byte swizzle atoms

struct AttnArgs {
    int B, C, Hq, Hkv, G, qpt, nqt, splits, mw, nct;
    int nunits;               // pairs of query tiles in all
    int u0;                   // tree_attn_kernel: >= 0: blocks 2 i, 2 i + 1 are the query tiles of pair unit u0 + i
    float sl2;                // scale * log2(e)
    const float2* cs;         // [nseq][B][dh/2] RoPE (cos, sin) of the tree positions
    const int32_t* n_nodes;   // [nseq]
    const uint64_t* mask;     // [nseq][B][mw]
    float* out;               // [nseq][B][Hq][dh]
    int* status;
};

// Pair unit u (two neighbouring query tiles of a kv head): the pairs of the
// last rows, which see the most tree keys, come first.
__device__ __forceinline__ void pair_unit(const AttnArgs& a, int u, int* qp, int* kvh, int* s) {
    const int nqp = (a.nqt + 1) / 2;
    const int nsk = a.nunits / nqp;
    *qp = nqp - 1 - u / nsk;
    *kvh = (u % nsk) % a.Hkv;
    *s = (u % nsk) / a.Hkv;
}

struct PrepArgs {
    int nseq, B, Hkv;
    const __nv_bfloat16* kt;  // [nseq][B][Hkv][dh]
    const int32_t* pos_ids;   // [nseq][B]
    __nv_bfloat16* kr;        // [nseq][B][Hkv][dh] rotated tree keys
    float2* cs;               // [nseq][B][dh/2] (cos, sin) of every tree position and frequency
    float inv_freq[kDh / 2];
};

// ------------------------------------------------------------ PTX helpers

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z,
                                            int w, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4, %5, %6}], [%2], %7;" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(w), "l"(policy)
        : "memory");
}

// Descriptor of an MN-major operand written by TMA with 128-byte swizzling:
// 64 MN elements (128 bytes) per row, 8 K rows per 1024-byte atom (stride
// byte offset), the next 64 MN elements `lbo` bytes further (leading byte
// offset).  Used for V (N = head dim contiguous, K = keys).
__device__ __forceinline__ uint64_t sdesc_sw128_mn(uint32_t saddr, uint32_t lbo) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr >> 4) & 0x3FFFu);
    d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
    d |= static_cast<uint64_t>((1024u >> 4) & 0x3FFFu) << 32;
    d |= static_cast<uint64_t>(1u) << 46;
    d |= static_cast<uint64_t>(2u) << 61;
    return d;
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
        "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
        "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
        "r"(__float_as_uint(v[15]))
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// D[tmem] (+)= A[tmem] * B[smem], bf16 inputs, fp32 accumulation (A: lane =
// row, K along columns as bf16 pairs).
__device__ __forceinline__ void tc_mma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// 16 consecutive 32-bit TMEM columns of this thread's lane from registers.
__device__ __forceinline__ void tmem_st16u(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}

// 32 consecutive 32-bit TMEM columns of this thread's lane from registers.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
        "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
        "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

__device__ __forceinline__ void attn_timeout(int* status, volatile int* abort) {
    *abort = 1;
    if (status) atomicOr(status, kDevTimeout);
}
__device__ __forceinline__ void attn_drain(uint64_t* bar, uint32_t parity) {
    const unsigned long long t0 = globaltimer_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (globaltimer_ns() - t0 > kWaitLimitNs) return;
    }
}

// Polls between two looks at the timer in tree_attn_kernel, whose eight softmax
// warps wait together for every key tile and are better kept apart: with 32,
// 0.5 to 1.2 % slower over long contexts (152 heads of 3 tiles, 8192 keys 217.0
// and 219.4 µs), at no length faster.
constexpr uint32_t kTilePolls = 1;

// A wait whose outcome is the same for every lane of the warp (the
// tcgen05.ld / st that follow are warp-collective).
template <uint32_t kPolls = kWaitPolls>
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
    const bool got = mbar_wait_inline<kPolls>(bar, parity, abort);
    return __all_sync(0xFFFFFFFFu, got);
}

// Stores into the shared memory of cluster CTA `rank` at the offset of the
// local shared address `local` (distributed shared memory).
__device__ __forceinline__ void st_cluster_f32x4(uint32_t local, int rank, float x, float y, float z, float w) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(remote), "f"(x), "f"(y), "f"(z), "f"(w)
                 : "memory");
}
__device__ __forceinline__ void st_cluster_f32x2(uint32_t local, int rank, float x, float y) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(remote), "f"(x), "f"(y) : "memory");
}

// Column slice [slice_lo(j), slice_lo(j + 1)) merged by cluster CTA j of
// `splits` (multiples of 4 columns), and the padded row stride (floats) of a
// received slice: an odd number of 16-byte units.
__device__ __forceinline__ int slice_lo(int j, int splits) { return 4 * ((j * (kDh / 4)) / splits); }
__device__ __forceinline__ int slice_stride(int ncol) { return ((ncol / 4) & 1) ? ncol : ncol + 4; }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// ------------------------------------------------------------ RoPE pre-pass

// sin and cos of x (|x| up to ~1e5): Cody-Waite reduction by 2*pi split
// into two floats (the high part exactly representable, so k * hi is exact
// inside the fma), then the hardware approximations on [-pi, pi] (absolute
// error ~2^-21, far below the bf16 rounding of the rotated values).
__device__ __forceinline__ void sincos_reduced(float x, float* sn, float* cs) {
    constexpr float kInv2Pi = 0.159154943091895336f;
    constexpr float k2PiHi = 6.28318548202514648f;  // float(2 pi)
    constexpr float k2PiLo = -1.74845560e-7f;       // 2 pi - k2PiHi
    const float k = rintf(x * kInv2Pi);
    float r = fmaf(-k, k2PiHi, x);
    r = fmaf(-k, k2PiLo, r);
    __sincosf(r, sn, cs);
}

// One warp per tree key row (s, b, kv head) -- every row's loads in flight at
// once: the row is rotated into kr (two of the 64 frequencies per lane), and
// the kv-head-0 warp of (s, b) writes the (cos, sin) of its position to the
// table the attention kernel rotates its queries with.
__global__ void __launch_bounds__(256) attn_prep_kernel(const PrepArgs a) {
    pdl_trigger();
    pdl_wait();
    const int lane = threadIdx.x & 31, t = lane * 2;
    const int rows = a.nseq * a.B * a.Hkv;
    const int wstride = gridDim.x * (blockDim.x >> 5);
    for (int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); row < rows; row += wstride) {
        const int sb = row / a.Hkv;
        const size_t off = static_cast<size_t>(row) * kDh;
        const __nv_bfloat162 x1 = *reinterpret_cast<const __nv_bfloat162*>(a.kt + off + t);
        const __nv_bfloat162 x2 = *reinterpret_cast<const __nv_bfloat162*>(a.kt + off + t + kDh / 2);
        const float pos = static_cast<float>(__ldg(a.pos_ids + sb));
        float s0, c0, s1, c1;
        sincos_reduced(pos * a.inv_freq[t], &s0, &c0);
        sincos_reduced(pos * a.inv_freq[t + 1], &s1, &c1);
        if (row % a.Hkv == 0)
            *reinterpret_cast<float4*>(a.cs + static_cast<size_t>(sb) * (kDh / 2) + t) = make_float4(c0, s0, c1, s1);
        const float a0 = __low2float(x1), a1 = __high2float(x1);
        const float b0 = __low2float(x2), b1 = __high2float(x2);
        *reinterpret_cast<__nv_bfloat162*>(a.kr + off + t) = __floats2bfloat162_rn(a0 * c0 - b0 * s0, a1 * c1 - b1 * s1);
        *reinterpret_cast<__nv_bfloat162*>(a.kr + off + t + kDh / 2) =
            __floats2bfloat162_rn(b0 * c0 + a0 * s0, b1 * c1 + a1 * s1);
    }
}

// ------------------------------------------------------------ attention

// 64 consecutive 32-bit TMEM columns of this thread's lane into registers
// (two x32 loads, one wait; the registers are tied to the wait so no use can
// move above it).
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float (&v)[64]) {
    uint32_t r[64];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr + 0));
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
                 : "r"(taddr + 32));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]), "+r"(r[32]), "+r"(r[33]), "+r"(r[34]), "+r"(r[35]), "+r"(r[36]), "+r"(r[37]), "+r"(r[38]), "+r"(r[39]), "+r"(r[40]), "+r"(r[41]), "+r"(r[42]), "+r"(r[43]), "+r"(r[44]), "+r"(r[45]), "+r"(r[46]), "+r"(r[47]), "+r"(r[48]), "+r"(r[49]), "+r"(r[50]), "+r"(r[51]), "+r"(r[52]), "+r"(r[53]), "+r"(r[54]), "+r"(r[55]), "+r"(r[56]), "+r"(r[57]), "+r"(r[58]), "+r"(r[59]), "+r"(r[60]), "+r"(r[61]), "+r"(r[62]), "+r"(r[63])
                 :
                 : "memory");
#pragma unroll
    for (int k = 0; k < 64; k++) v[k] = __uint_as_float(r[k]);
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__global__ void __launch_bounds__(kAttnThreads, 1)
    tree_attn_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmKc,
                     const __grid_constant__ CUtensorMap tmVc, const __grid_constant__ CUtensorMap tmKt,
                     const __grid_constant__ CUtensorMap tmVt, const AttnArgs a) {
    extern __shared__ uint8_t attn_smem_raw[];
    pdl_trigger();
    const uint32_t off = (1024u - (smem_u32(attn_smem_raw) & 1023u)) & 1023u;
    uint8_t* sQ = attn_smem_raw + off;
    uint8_t* sK = sQ + kTileBytes;                    // [kKStages] K stages
    uint8_t* sV = sK + kKStages * kTileBytes;         // [kVStages] V stages
    uint64_t* bars = reinterpret_cast<uint64_t*>(sV + kVStages * kTileBytes);
    uint64_t* q_full = bars;
    uint64_t* k_full = bars + 1;                      // [kKStages]
    uint64_t* k_empty = k_full + kKStages;            // [kKStages] S of the stage's tile done
    uint64_t* v_full = k_empty + kKStages;            // [kVStages]
    uint64_t* v_empty = v_full + kVStages;            // [kVStages] PV of the stage's tile done
    uint64_t* s_full = v_empty + kVStages;
    uint64_t* s_empty = s_full + 1;                   // softmax has S in registers
    uint64_t* p_full = s_empty + 1;
    uint64_t* pv_done = p_full + 1;                   // [2] PV of a tile using P buffer b done
    uint64_t* tdown = pv_done + 2;
    uint64_t* q_ready = tdown + 1;                    // queries rotated in place
    int* misc = reinterpret_cast<int*>(bars + kNumBars);  // [0] TMEM base, [1] abort
    volatile int* abort = &misc[1];

    // cluster of `splits` CTAs = one (sequence, kv head, query tile); the
    // cluster rank is the key-range split
    const int split = a.splits > 1 ? static_cast<int>(cluster_ctarank()) : 0;
    const int blk = blockIdx.x / a.splits;
    int qt = blk % a.nqt;
    int kvh = (blk / a.nqt) % a.Hkv;
    int s = blk / (a.nqt * a.Hkv);
    if (a.u0 >= 0) {
        pair_unit(a, a.u0 + blk / 2, &qt, &kvh, &s);
        qt = 2 * qt + (blk & 1);
        if (qt >= a.nqt) return;  // an odd number of query tiles: the last pair has one
    }
    const int q0 = qt * a.qpt;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        mbar_init(q_full, 1);
        for (int i = 0; i < kKStages; i++) {
            mbar_init(&k_full[i], 1);
            mbar_init(&k_empty[i], 1);
        }
        for (int i = 0; i < kVStages; i++) {
            mbar_init(&v_full[i], 1);
            mbar_init(&v_empty[i], 1);
        }
        mbar_init(s_full, 1);
        mbar_init(s_empty, kSoftThreads);
        mbar_init(p_full, kSoftThreads);
        mbar_init(&pv_done[0], 1);
        mbar_init(&pv_done[1], 1);
        mbar_init(tdown, 1);
        mbar_init(q_ready, kSoftThreads);
        misc[1] = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(reinterpret_cast<uint32_t*>(&misc[0]), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = static_cast<uint32_t>(misc[0]);
    pdl_wait();  // the key table, rotated keys and the tree arrays come from earlier kernels

    const int nn = min(max(__ldg(a.n_nodes + s), 0), a.B);
    const int qlast = min(q0 + a.qpt, nn) - 1;  // last tree row of this CTA with a query (-1: none)
    const int T = qlast >= 0 ? a.nct + qlast / kKeys + 1 : 0;
    const int j0 = (split * T) / a.splits;
    const int nt = ((split + 1) * T) / a.splits - j0;

    // softmax state (warps 2-9), kept for the epilogue.  Warps w and w + 4
    // share TMEM lane quarter w % 4 (the same 32 query rows); warpgroup wg
    // handles key columns and O columns [64 wg, 64 wg + 64).
    const int qd = warp & 3;
    const int wg = warp >= 2 ? (warp - 2) >> 2 : 0;
    const int cb = wg * 64;
    const int r = qd * 32 + lane;  // query row = TMEM lane
    const int b = q0 + r / a.G, g = r % a.G;
    const bool row_ok = b < nn;
    const uint32_t tl = tmem + (static_cast<uint32_t>(qd * 32) << 16);
    float* xch = reinterpret_cast<float*>(misc + 4);  // [2][128] row max / sum exchange of the two warpgroups
    int* xok = misc + 4 + 2 * kRows;                   // [2][4] per-warp "no wait failed" exchange
    float m_run = -INFINITY, l = 0.0f;
    bool ok = true;

    if (warp == 0) {
        // ---------------------------------------------------------- producer
        if (lane == 0 && nt > 0) {
            const uint64_t pol_q = l2_policy_evict_first();
            const uint64_t pol_kv = l2_policy_evict_last();  // re-read by the other query tiles
            // rows (tree row q0 + r / G, head kvh * G + r % G)
            mbar_arrive_expect_tx(q_full, kTileBytes);
            tma_load_4d(sQ, &tmQ, q_full, 0, kvh * a.G, q0, s, pol_q);
            tma_load_4d(sQ + kHalf, &tmQ, q_full, 64, kvh * a.G, q0, s, pol_q);
            // K runs up to kKStages tiles ahead, V up to kVStages: issue
            // whichever is due, K first
            int kdone = 0, vdone = 0;
            while ((kdone < nt || vdone < nt) && !*abort) {
                const bool do_k = kdone < nt && kdone < vdone + kKStages;
                const int i = do_k ? kdone : vdone;
                const int j = j0 + i;
                const bool ctx = j < a.nct;
                const int key0 = (ctx ? j : j - a.nct) * kKeys;
                if (do_k) {
                    const int st = i % kKStages;
                    if (!mbar_wait_inline<kTilePolls>(&k_empty[st], (static_cast<uint32_t>(i / kKStages) & 1u) ^ 1u, abort)) {
                        attn_timeout(a.status, abort);
                        break;
                    }
                    uint8_t* dk = sK + st * kTileBytes;
                    mbar_arrive_expect_tx(&k_full[st], kTileBytes);
                    tma_load_4d(dk, ctx ? &tmKc : &tmKt, &k_full[st], 0, kvh, key0, s, pol_kv);
                    tma_load_4d(dk + kHalf, ctx ? &tmKc : &tmKt, &k_full[st], 64, kvh, key0, s, pol_kv);
                    kdone++;
                } else {
                    const int st = i % kVStages;
                    if (!mbar_wait_inline<kTilePolls>(&v_empty[st], (static_cast<uint32_t>(i / kVStages) & 1u) ^ 1u, abort)) {
                        attn_timeout(a.status, abort);
                        break;
                    }
                    uint8_t* dv = sV + st * kTileBytes;
                    mbar_arrive_expect_tx(&v_full[st], kTileBytes);
                    tma_load_4d(dv, ctx ? &tmVc : &tmVt, &v_full[st], 0, kvh, key0, s, pol_kv);
                    tma_load_4d(dv + kHalf, ctx ? &tmVc : &tmVt, &v_full[st], 64, kvh, key0, s, pol_kv);
                    vdone++;
                }
            }
            if (*abort) {
                // copies still in flight must land before the CTA exits
                attn_drain(q_full, 0);
                for (int i = kdone > kKStages ? kdone - kKStages : 0; i < kdone; i++)
                    attn_drain(&k_full[i % kKStages], static_cast<uint32_t>(i / kKStages) & 1u);
                for (int i = vdone > kVStages ? vdone - kVStages : 0; i < vdone; i++)
                    attn_drain(&v_full[i % kVStages], static_cast<uint32_t>(i / kVStages) & 1u);
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issuer
        // Q (rotated) and P are tensor-memory operands, K and V come from the
        // shared-memory rings.  Order: S(0); then per tile i: S(i+1) once
        // softmax(i) holds S(i) in registers (it runs during softmax(i)),
        // PV(i) once P(i) is written (P is double-buffered).
        if (lane == 0 && nt > 0) {
            constexpr uint32_t idesc_s = idesc_bf16_f32(kRows, kKeys);
            constexpr uint32_t idesc_pv = idesc_bf16_f32(kRows, kDh) | (1u << 16);  // B (= V) MN-major
            bool mok = mbar_wait_inline<kTilePolls>(q_ready, 0, abort);
            auto issue_s = [&](int i) -> bool {
                const int st = i % kKStages;
                // the S columns were last read by softmax(i - 1)
                if (!mbar_wait_inline<kTilePolls>(&k_full[st], static_cast<uint32_t>(i / kKStages) & 1u, abort) ||
                    (i > 0 && !mbar_wait_inline<kTilePolls>(s_empty, static_cast<uint32_t>(i - 1) & 1u, abort)))
                    return false;
                tc_fence_after();
                const uint32_t k_addr = smem_u32(sK + st * kTileBytes);
#pragma unroll
                for (int kk = 0; kk < kDh / 16; kk++) {
                    const uint32_t o = (kk >> 2) * kHalf + (kk & 3) * 32;
                    tc_mma_bf16_ts(tmem + kSCol, tmem + kQCol + kk * 8, sdesc_sw128(k_addr + o), idesc_s,
                                   kk > 0 ? 1u : 0u);
                }
                tc_commit(s_full);
                tc_commit(&k_empty[st]);
                return true;
            };
            if (mok) tc_fence_after();
            if (mok) mok = issue_s(0);
            for (int i = 0; i < nt && mok; i++) {
                if (i + 1 < nt && !issue_s(i + 1)) {
                    mok = false;
                    break;
                }
                const int st = i % kVStages;
                if (!mbar_wait_inline<kTilePolls>(p_full, static_cast<uint32_t>(i) & 1u, abort) ||
                    !mbar_wait_inline<kTilePolls>(&v_full[st], static_cast<uint32_t>(i / kVStages) & 1u, abort)) {
                    mok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t v_addr = smem_u32(sV + st * kTileBytes);
                const uint32_t p_tmem = tmem + kPCol + (i & 1) * (kKeys / 2);
#pragma unroll
                for (int kk = 0; kk < kKeys / 16; kk++)  // 16 keys = 8 columns of bf16 pairs
                    tc_mma_bf16_ts(tmem + kOCol, p_tmem + kk * 8, sdesc_sw128_mn(v_addr + kk * 2048, kHalf), idesc_pv,
                                   (i > 0 || kk > 0) ? 1u : 0u);
                tc_commit(&v_empty[st]);
                tc_commit(&pv_done[i & 1]);
            }
            if (!mok) {
                attn_timeout(a.status, abort);
                tc_commit(tdown);
                attn_drain(tdown, 0);
            }
        }
    } else {
        // ---------------------------------------------------------- softmax
        const uint32_t swz = static_cast<uint32_t>(r & 7);
        const int pair_bar = kPairBarrier0 + qd;
        if (nt > 0) {
            // RoPE of this thread's query row, in place: element t of the
            // first 64 and element t of the second 64 sit at the same
            // swizzled position of the two 16 KB halves; warpgroup wg
            // rotates chunks 4 wg .. 4 wg + 3
            float4 f[16];  // (cos, sin) of this thread's 32 pairs, in flight while the queries load
            const float4* cs = reinterpret_cast<const float4*>(a.cs + (static_cast<size_t>(s) * a.B + min(b, a.B - 1)) * (kDh / 2));
#pragma unroll
            for (int e = 0; e < 16; e++) f[e] = __ldg(cs + wg * 16 + e);
            if (!warp_wait<kTilePolls>(q_full, 0, abort)) {
                attn_timeout(a.status, abort);
                ok = false;
            }
            // rotated elements t (first half) and t + 64 (second half) of this
            // warpgroup's t in [32 wg, 32 wg + 32), as bf16 pairs for the TMEM
            // columns kQCol + t / 2 and kQCol + 32 + t / 2 (zeros past row B)
            uint32_t q1[16], q2[16];
            if (ok && b < a.B) {
#pragma unroll
                for (int cc = 0; cc < 4; cc++) {
                    const int c = wg * 4 + cc;
                    const uint8_t* p1 = sQ + r * 128 + ((static_cast<uint32_t>(c) ^ swz) << 4);
                    const uint4 x1 = *reinterpret_cast<const uint4*>(p1);
                    const uint4 x2 = *reinterpret_cast<const uint4*>(p1 + kHalf);
                    const uint32_t* u1 = reinterpret_cast<const uint32_t*>(&x1);
                    const uint32_t* u2 = reinterpret_cast<const uint32_t*>(&x2);
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        const float4 cw = f[cc * 4 + e];  // pairs 8c+2e, 8c+2e+1
                        const __nv_bfloat162 h1 = *reinterpret_cast<const __nv_bfloat162*>(&u1[e]);
                        const __nv_bfloat162 h2 = *reinterpret_cast<const __nv_bfloat162*>(&u2[e]);
                        const float a0 = __low2float(h1), a1 = __high2float(h1);
                        const float b0 = __low2float(h2), b1 = __high2float(h2);
                        q1[cc * 4 + e] = pack_bf16(a0 * cw.x - b0 * cw.y, a1 * cw.z - b1 * cw.w);
                        q2[cc * 4 + e] = pack_bf16(b0 * cw.x + a0 * cw.y, b1 * cw.z + a1 * cw.w);
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < 16; k++) q1[k] = q2[k] = 0u;
            }
            tmem_st16u(tl + kQCol + wg * 16, q1);
            tmem_st16u(tl + kQCol + 32 + wg * 16, q2);
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(q_ready);
        }
        for (int i = 0; i < nt; i++) {
            const int j = j0 + i;
            // visible keys of this row among this warpgroup's 64 keys of the tile
            uint64_t w = 0ull;
            if (row_ok) {
                int kvalid;
                if (j < a.nct) {
                    kvalid = min(kKeys, a.C - j * kKeys);
                    w = ~0ull;
                } else {
                    const int t = j - a.nct;
                    kvalid = min(kKeys, nn - t * kKeys);
                    w = 2 * t + wg < a.mw ? __ldg(a.mask + (static_cast<size_t>(s) * a.B + b) * a.mw + 2 * t + wg) : 0ull;
                }
                kvalid -= cb;
                if (kvalid <= 0)
                    w = 0ull;
                else if (kvalid < 64)
                    w &= (1ull << kvalid) - 1ull;
            }
            const bool full = __all_sync(0xFFFFFFFFu, w == ~0ull);  // whole warp sees all 64 keys
            // Both warps of the lane quarter reach both pair barriers of every
            // iteration and leave the loop at the same point: a failed wait is
            // exchanged with the row max and acted on after the barriers.
            if (ok && !warp_wait<kTilePolls>(s_full, static_cast<uint32_t>(i) & 1u, abort)) {
                attn_timeout(a.status, abort);
                ok = false;
            }
            float sv[64];
            float mx = -INFINITY;
            if (ok) {
                tc_fence_after();
                tmem_ld64(tl + kSCol + cb, sv);
                // S is in registers: the buffer is free for S(i + 2)
                tc_fence_before();
                mbar_arrive(s_empty);
                if (full) {
#pragma unroll
                    for (int c = 0; c < 64; c += 2) mx = fmaxf(mx, fmaxf(sv[c], sv[c + 1]));
                } else {
#pragma unroll
                    for (int c = 0; c < 64; c++) {
                        if (!((w >> c) & 1ull)) sv[c] = -INFINITY;
                        mx = fmaxf(mx, sv[c]);
                    }
                }
            }
            xch[wg * kRows + r] = mx;
            if (lane == 0) xok[wg * 4 + qd] = ok ? 1 : 0;
            named_bar_sync(pair_bar, 64);
            mx = fmaxf(mx, xch[(1 - wg) * kRows + r]);
            ok = ok && xok[(1 - wg) * 4 + qd] != 0;
            named_bar_sync(pair_bar, 64);  // both read before the next tile's write
            if (!ok) break;
            const float mx2 = mx * a.sl2;
            const bool resc = mx2 > m_run + kRescaleSlack;
            const float m_new = resc ? mx2 : m_run;
            const float alpha = resc ? ex2(m_run - m_new) : 1.0f;
            // P buffer i & 1 was last read by PV(i - 2); O must be stable (PV(i - 1)
            // done) only when it is rescaled.  On a timeout this tile is
            // skipped; the pair leaves the loop together at the next exchange.
            if (i > 1 && !warp_wait<kTilePolls>(&pv_done[i & 1], (static_cast<uint32_t>(i >> 1) & 1u) ^ 1u, abort)) {
                attn_timeout(a.status, abort);
                ok = false;
                continue;
            }
            tc_fence_after();
            const bool any_resc = __any_sync(0xFFFFFFFFu, resc);
            if (i > 0 && any_resc) {
                if (!warp_wait<kTilePolls>(&pv_done[(i - 1) & 1], static_cast<uint32_t>((i - 1) >> 1) & 1u, abort)) {
                    attn_timeout(a.status, abort);
                    ok = false;
                    continue;
                }
                tc_fence_after();
                {
#pragma unroll
                    for (int c0 = 0; c0 < 64; c0 += 16) {
                        float o[16];
                        tmem_ld16(tl + kOCol + cb + c0, o);
#pragma unroll
                        for (int e = 0; e < 16; e++) o[e] *= alpha;
                        tmem_st16(tl + kOCol + cb + c0, o);
                    }
                    tmem_wait_st();
                }
            }
            l *= alpha;
            m_run = m_new;
            // P = 2^(s * scale * log2 e - m) as bf16 pairs into TMEM P buffer
            // i & 1 (lane = row, keys 64 wg .. 64 wg + 63 in 32 columns); masked
            // keys hold -inf and give 0 (so does every key of a row that has
            // seen no visible key: m = -inf)
            const float nm = m_run == -INFINITY ? 0.0f : -m_run;
            float lsum = 0.0f;
            uint32_t pk[32];
#pragma unroll
            for (int c = 0; c < 64; c += 2) {
                const float p0 = ex2(fmaf(sv[c], a.sl2, nm));
                const float p1 = ex2(fmaf(sv[c + 1], a.sl2, nm));
                lsum += p0 + p1;
                pk[c >> 1] = pack_bf16(p0, p1);
            }
            tmem_st32(tl + kPCol + (i & 1) * (kKeys / 2) + wg * 32, pk);
            tmem_wait_st();
            l += lsum;
            tc_fence_before();
            mbar_arrive(p_full);
        }
        if (ok && nt > 0) {
            if (!warp_wait<kTilePolls>(&pv_done[(nt - 1) & 1], static_cast<uint32_t>((nt - 1) >> 1) & 1u, abort)) {
                attn_timeout(a.status, abort);
                ok = false;
            }
            tc_fence_after();
        }
        // the row sum is split over the two warpgroups
        xch[wg * kRows + r] = l;
        named_bar_sync(pair_bar, 64);
        l += xch[(1 - wg) * kRows + r];
        ok = __all_sync(0xFFFFFFFFu, ok);
    }

    const int h = kvh * a.G + g;
    if (a.splits == 1) {
        if (warp >= 2 && ok) {
            float* orow = a.out + ((static_cast<size_t>(s) * a.B + b) * a.Hq + h) * kDh + cb;
            const float inv = (row_ok && l > 0.0f) ? 1.0f / l : 0.0f;
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 16) {
                float o[16];
                if (nt > 0) {
                    tmem_ld16(tl + kOCol + cb + c0, o);
                } else {
#pragma unroll
                    for (int e = 0; e < 16; e++) o[e] = 0.0f;
                }
                if (b < a.B) {
#pragma unroll
                    for (int e = 0; e < 16; e += 4)
                        *reinterpret_cast<float4*>(orow + c0 + e) =
                            make_float4(o[e] * inv, o[e + 1] * inv, o[e + 2] * inv, o[e + 3] * inv);
                }
            }
        }
    } else {
        // Split key range.  Columns are owned in groups of 4: CTA j merges
        // [c_lo(j), c_hi(j)).  After a cluster barrier (every CTA is past its
        // main loop, so the K and V rings are free), every CTA p pushes,
        // with 16-byte stores into the peers' shared memory, its (m, l) row
        // to every peer and its unnormalised O row slices to their owners
        // (row-major, row stride padded to an odd number of 16-byte units:
        // conflict-free); after a second barrier CTA j merges locally, in
        // rank order: O = sum_p 2^(m_p - M) O_p / sum_p 2^(m_p - M) l_p.
        float* rbuf = reinterpret_cast<float*>(sK);     // [p][128 rows][stride]
        float2* rml = reinterpret_cast<float2*>(sV);    // [p][128 rows]
        __syncwarp();
        cluster_sync_all();
        if (warp >= 2) {
            const bool have = ok && nt > 0;
            if (wg == 0)
                for (int jj = 0; jj < a.splits; jj++)
                    st_cluster_f32x2(smem_u32(rml + split * kRows + r), jj, m_run, have ? l : 0.0f);
            if (have) {
                float o[64];
                tmem_ld64(tl + kOCol + cb, o);
                for (int jj = 0; jj < a.splits; jj++) {
                    const int lo = slice_lo(jj, a.splits), ncol = slice_lo(jj + 1, a.splits) - lo;
                    const int stride = slice_stride(ncol);
                    const uint32_t dst = smem_u32(rbuf + (split * kRows + r) * stride);
#pragma unroll
                    for (int c = 0; c < 64; c += 4)
                        if (cb + c >= lo && cb + c < lo + ncol)
                            st_cluster_f32x4(dst + (cb + c - lo) * 4, jj, o[c], o[c + 1], o[c + 2], o[c + 3]);
                }
            }
        }
        __syncwarp();
        cluster_sync_all();  // every push has landed
        if (warp >= 2) {
            const int c_lo = slice_lo(split, a.splits), ncol = slice_lo(split + 1, a.splits) - c_lo;
            const int stride = slice_stride(ncol);
            float M = -INFINITY;
            for (int p = 0; p < a.splits; p++) {
                const float2 ml = rml[p * kRows + r];
                if (ml.y > 0.0f) M = fmaxf(M, ml.x);
            }
            float wp[kMaxSplits];
            float L = 0.0f;
#pragma unroll
            for (int p = 0; p < kMaxSplits; p++) {
                wp[p] = 0.0f;
                if (p < a.splits) {
                    const float2 ml = rml[p * kRows + r];
                    if (ml.y > 0.0f) {
                        wp[p] = ex2(ml.x - M);
                        L += wp[p] * ml.y;
                    }
                }
            }
            const float inv = (row_ok && L > 0.0f) ? 1.0f / L : 0.0f;
            if (b < a.B) {
                float* orow = a.out + ((static_cast<size_t>(s) * a.B + b) * a.Hq + h) * kDh + c_lo;
                // the two warpgroups take alternate 4-column groups of the slice
                for (int c = 4 * wg; c < ncol; c += 8) {
                    float4 o = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                    for (int p = 0; p < kMaxSplits; p++) {
                        if (wp[p] != 0.0f) {
                            const float4 v = *reinterpret_cast<const float4*>(rbuf + (p * kRows + r) * stride + c);
                            o.x += wp[p] * v.x;
                            o.y += wp[p] * v.y;
                            o.z += wp[p] * v.z;
                            o.w += wp[p] * v.w;
                        }
                    }
                    *reinterpret_cast<float4*>(orow + c) = make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ------------------------------------------------------------ attention, two query tiles
//
// The kernel for more (sequence, kv head, query tile) blocks than SMs: a CTA
// owns two neighbouring query tiles of a kv head, two softmax warpgroups each
// (thread = query row = TMEM lane, 64 keys of a tile), so that one tile's
// MMAs run during the other's softmax and every K/V tile is read once for
// both.  Order of the issuing thread: S0(0), S1(0); then per key tile i
// PV0(i), S0(i+1), PV1(i), S1(i+1).  The tensor pipe queues hardly anything,
// so all that this thread does besides (a wait takes it 100 cycles even when
// it is satisfied) leaves the pipe idle: two helper warps wait for the K and V
// tiles and free their slots, and it waits and commits once per tile.  P_t overwrites the first 64 columns of
// S_t (the MMAs are in order: PV_t(i) has read it before S_t(i+1) is
// written), and a tile's S being complete implies that its previous PV is, so
// O_t may be rescaled without another wait.  TMEM: S0 [0,128), S1 [128,256),
// O0 [256,384), O1 [384,512); the rotated queries stay in shared memory.
// Every row's maxima, probabilities and sums are those of tree_attn_kernel,
// tile by tile, so both give the same output.
// Measured on GB300, 8 x 512 rows, 32 / 8 heads, 2048 context keys: 190 µs per
// call with one query tile per CTA, 163 with pairs.  A key tile takes a pair
// 4000 cycles (2 x 1900 alone) of which the issuing thread spends 3250 on 32
// MMAs: beside the softmax's TMEM and shared-memory traffic one costs 100
// cycles instead of 65.  Tried: an issuing thread per query tile (223 µs),
// the waits and the freeing of slots in the issuing thread (198), one
// warpgroup per query tile (196).
constexpr int kK2Stages = 3, kV2Stages = 2;
constexpr int kNum2Bars = 1 + 2 * kK2Stages + 2 * kV2Stages + 2 * 4 + 1;
constexpr int kSmem2Used =
    kTileBytes * (2 + kK2Stages + kV2Stages) + kNum2Bars * 8 + 4 * 4 + 2 * 2 * 128 * 4 + 2 * 8 * 4;  // ... exchange
constexpr int kFirstSoft2 = 4;                       // first softmax warp
constexpr int kAttn2Threads = kFirstSoft2 * 32 + 512;
constexpr int kAttn2Smem = kSmem2Used;  // (the base is declared with the swizzle atoms' 1024-byte alignment)

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, const void* src, int x, int y, int z, int w) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z), "r"(w)
                 : "memory");
}

__global__ void __launch_bounds__(kAttn2Threads, 1)
    tree_attn2_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmKc,
                      const __grid_constant__ CUtensorMap tmVc, const __grid_constant__ CUtensorMap tmKt,
                      const __grid_constant__ CUtensorMap tmVt,
                      const __grid_constant__ CUtensorMap tmO, const AttnArgs a) {
    extern __shared__ __align__(1024) uint8_t attn2_smem[];
    pdl_trigger();
    uint8_t* sQ = attn2_smem;                         // [2] query tiles
    uint8_t* sK = sQ + 2 * kTileBytes;
    uint8_t* sV = sK + kK2Stages * kTileBytes;
    uint64_t* q_full = reinterpret_cast<uint64_t*>(sV + kV2Stages * kTileBytes);
    uint64_t* k_full = q_full + 1;
    uint64_t* k_empty = k_full + kK2Stages;
    uint64_t* v_full = k_empty + kK2Stages;
    uint64_t* v_empty = v_full + kV2Stages;
    uint64_t* q_ready = v_empty + kV2Stages;          // [2] the tile's queries are rotated
    uint64_t* s_full = q_ready + 2;                   // [2]
    uint64_t* p_full = s_full + 2;                    // [2]
    uint64_t* o_full = p_full + 2;                    // [2] the last PV of the tile is done
    uint64_t* tdown = o_full + 2;
    int* misc = reinterpret_cast<int*>(q_full + kNum2Bars);  // [0] TMEM base, [1] abort
    volatile int* abort = &misc[1];
    float* xch = reinterpret_cast<float*>(misc + 4);  // [2 tiles][2 warpgroups][128] row max / sum
    int* xok = reinterpret_cast<int*>(xch + 2 * 2 * kRows);  // [2][2][4] per-warp "no wait failed"

    int qp, kvh, s;
    pair_unit(a, blockIdx.x, &qp, &kvh, &s);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        mbar_init(q_full, 1);
        for (int i = 0; i < kK2Stages; i++) {
            mbar_init(&k_full[i], 1);
            mbar_init(&k_empty[i], 1);
        }
        for (int i = 0; i < kV2Stages; i++) {
            mbar_init(&v_full[i], 1);
            mbar_init(&v_empty[i], 1);
        }
        for (int t = 0; t < 2; t++) {
            mbar_init(&q_ready[t], 8);
            mbar_init(&s_full[t], 1);
            mbar_init(&p_full[t], 9);
            mbar_init(&o_full[t], 1);
        }
        mbar_init(tdown, 1);
        misc[1] = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(reinterpret_cast<uint32_t*>(&misc[0]), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = static_cast<uint32_t>(misc[0]);
    pdl_wait();

    const int nn = min(max(__ldg(a.n_nodes + s), 0), a.B);
    // key tiles of each query tile: 0 if none of its rows is a node
    int nt[2];
#pragma unroll
    for (int t = 0; t < 2; t++) {
        const int q0 = (2 * qp + t) * a.qpt, qlast = min(q0 + a.qpt, nn) - 1;
        nt[t] = qlast >= q0 ? a.nct + qlast / kKeys + 1 : 0;
    }
    const int ntm = max(nt[0], nt[1]);

    if (warp == 0) {
        if (lane == 0 && ntm > 0) {
            const uint64_t pol_q = l2_policy_evict_first();
            const uint64_t pol_kv = l2_policy_evict_last();  // re-read by the other query tiles
            mbar_arrive_expect_tx(q_full, 2 * kTileBytes);
            for (int t = 0; t < 2; t++)
                for (int hf = 0; hf < 2; hf++)  // (rows past B are filled with zeros)
                    tma_load_4d(sQ + t * kTileBytes + hf * kHalf, &tmQ, q_full, hf * 64, kvh * a.G, (2 * qp + t) * a.qpt, s,
                                pol_q);
            int kdone = 0, vdone = 0;
            while ((kdone < ntm || vdone < ntm) && !*abort) {
                const bool do_k = kdone < ntm && kdone < vdone + 2;  // K one tile ahead of V
                const int i = do_k ? kdone : vdone;
                const bool ctx = i < a.nct;
                const int key0 = (ctx ? i : i - a.nct) * kKeys;
                const int ns = do_k ? kK2Stages : kV2Stages;
                uint64_t* full = (do_k ? k_full : v_full) + i % ns;
                uint64_t* empty = (do_k ? k_empty : v_empty) + i % ns;
                if (!mbar_wait_inline(empty, (static_cast<uint32_t>(i / ns) & 1u) ^ 1u, abort)) {
                    attn_timeout(a.status, abort);
                    break;
                }
                uint8_t* dst = (do_k ? sK : sV) + (i % ns) * kTileBytes;
                const CUtensorMap* tm = do_k ? (ctx ? &tmKc : &tmKt) : (ctx ? &tmVc : &tmVt);
                mbar_arrive_expect_tx(full, kTileBytes);
                tma_load_4d(dst, tm, full, 0, kvh, key0, s, pol_kv);
                tma_load_4d(dst + kHalf, tm, full, 64, kvh, key0, s, pol_kv);
                (do_k ? kdone : vdone)++;
            }
            if (*abort) {
                // copies still in flight must land before the CTA exits
                attn_drain(q_full, 0);
                for (int i = max(kdone - kK2Stages, 0); i < kdone; i++)
                    attn_drain(&k_full[i % kK2Stages], static_cast<uint32_t>(i / kK2Stages) & 1u);
                for (int i = max(vdone - kV2Stages, 0); i < vdone; i++)
                    attn_drain(&v_full[i % kV2Stages], static_cast<uint32_t>(i / kV2Stages) & 1u);
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && ntm > 0) {
            constexpr uint32_t idesc_s = idesc_bf16_f32(kRows, kKeys);
            constexpr uint32_t idesc_pv = idesc_bf16_f32(kRows, kDh) | (1u << 16);  // B (= V) MN-major
            constexpr int kTile16 = kTileBytes >> 4, kHalf16 = kHalf >> 4;  // (descriptors address units of 16 bytes)
            const uint64_t q_desc = sdesc_sw128(smem_u32(sQ)), k_desc = sdesc_sw128(smem_u32(sK));
            const uint64_t v_desc = sdesc_sw128_mn(smem_u32(sV), kHalf);
            const int nt0 = nt[0], nt1 = nt[1];
            auto issue_s = [&](int t, int ks) {
                const uint64_t qd = q_desc + t * kTile16, kd = k_desc + ks * kTile16;
#pragma unroll
                for (int kk = 0; kk < kDh / 16; kk++) {
                    const int o = (kk >> 2) * kHalf16 + (kk & 3) * 2;
                    tc_mma_bf16(tmem + t * 128, qd + o, kd + o, idesc_s, kk > 0 ? 1u : 0u);
                }
                tc_commit(&s_full[t]);
            };
            auto step = [&](int t, int i, int my_nt, int ks, int vs) -> bool {
                // (P(i) written, V(i) and K(i + 1) loaded)
                if (!mbar_wait_inline(&p_full[t], static_cast<uint32_t>(i) & 1u, abort)) return false;
                tc_fence_after();
                const uint64_t vd = v_desc + vs * kTile16;
#pragma unroll
                for (int kk = 0; kk < kKeys / 16; kk++)  // 16 keys = 8 columns of bf16 pairs
                    tc_mma_bf16_ts(tmem + 256 + t * 128, tmem + t * 128 + kk * 8, vd + kk * (2048 >> 4), idesc_pv,
                                   (i > 0 || kk > 0) ? 1u : 0u);
                if (i + 1 < my_nt) issue_s(t, ks);
                else tc_commit(&o_full[t]);
                return true;
            };
            bool ok = mbar_wait_inline(&k_full[0], 0, abort);
            if (ok && nt0 > 0) {
                ok = mbar_wait_inline(&q_ready[0], 0, abort);
                tc_fence_after();
                if (ok) issue_s(0, 0);
            }
            if (ok && nt1 > 0) {
                ok = mbar_wait_inline(&q_ready[1], 0, abort);
                tc_fence_after();
                if (ok) issue_s(1, 0);
            }
            int ks = 0, vs = 0;
#pragma unroll 1
            for (int i = 0; i < ntm && ok; i++) {
                ks = ks + 1 == kK2Stages ? 0 : ks + 1;  // slot of K tile i + 1
                if (i < nt0) ok = step(0, i, nt0, ks, vs);
                if (ok && i < nt1) ok = step(1, i, nt1, ks, vs);
                vs = vs + 1 == kV2Stages ? 0 : vs + 1;
            }
            if (!ok) {
                attn_timeout(a.status, abort);
                tc_commit(tdown);
                attn_drain(tdown, 0);
            }
        }
    } else if (warp < kFirstSoft2) {
        // warp 2 + t waits, for the issuing thread, for the V and K tiles of
        // the next step of query tile t (a ninth arrival at p_full), and for
        // the last tile in issue order it frees the slots: S(i) complete
        // means that K(i) and V(i - 1) have been read
        const int t = warp - 2;
        const bool frees = t == (nt[1] > 0 ? 1 : 0);  // (nt[0] <= nt[1] unless nt[1] = 0)
        if (lane == 0) {
            bool ok = true;
#pragma unroll 1
            for (int i = 0; i < nt[t] && ok; i++) {
                if (frees) {
                    ok = mbar_wait_inline(&s_full[t], static_cast<uint32_t>(i) & 1u, abort);
                    if (!ok) break;
                    mbar_arrive(&k_empty[i % kK2Stages]);
                    if (i > 0) mbar_arrive(&v_empty[(i - 1) % kV2Stages]);
                }
                ok = mbar_wait_inline(&v_full[i % kV2Stages], static_cast<uint32_t>(i / kV2Stages) & 1u, abort) &&
                     (i + 1 >= ntm || mbar_wait_inline(&k_full[(i + 1) % kK2Stages],
                                                       static_cast<uint32_t>((i + 1) / kK2Stages) & 1u, abort));
                if (!ok) break;
                mbar_arrive(&p_full[t]);
                ok = mbar_wait_inline(&p_full[t], static_cast<uint32_t>(i) & 1u, abort);
            }
            if (!ok) attn_timeout(a.status, abort);
        }
    } else {
        // two warpgroups per query tile: warpgroup (t, wg) takes key and O
        // columns [64 wg, 64 wg + 64) of the rows of tile 2 qp + t; the two
        // warps of a lane quarter exchange their row maxima
        const int sw = warp - kFirstSoft2;
        const int t = sw >> 3, wg = (sw >> 2) & 1, qd = warp & 3, r = qd * 32 + lane;
        const int cb = wg * 64, pair_bar = kPairBarrier0 + t * 4 + qd;
        const int my_nt = t ? nt[1] : nt[0];
        const int b = (2 * qp + t) * a.qpt + r / a.G, g = r % a.G;
        const bool row_ok = b < nn;
        const uint32_t tS = tmem + t * 128 + (static_cast<uint32_t>(qd * 32) << 16), tO = tS + 256 + cb;
        float* xt = xch + t * 2 * kRows;       // [2 warpgroups][128]
        int* xk = xok + t * 8 + qd;            // [2 warpgroups][4]
        float m_run = -INFINITY, l = 0.0f;
        bool ok = true;
        if (my_nt > 0) {
            // rotate this row's chunks 4 wg .. 4 wg + 3 in place (element e of
            // the first 64 and of the second 64 sit at the same swizzled
            // position of the two 16 KB halves)
            float4 f[16];  // (cos, sin) of this thread's 32 pairs, in flight while the queries load
            const float4* cs = reinterpret_cast<const float4*>(a.cs + (static_cast<size_t>(s) * a.B + min(b, a.B - 1)) * (kDh / 2));
#pragma unroll
            for (int e = 0; e < 16; e++) f[e] = __ldg(cs + wg * 16 + e);
            ok = warp_wait(q_full, 0, abort);
            if (ok && b < a.B) {
#pragma unroll
                for (int cc = 0; cc < 4; cc++) {
                    const int c = wg * 4 + cc;
                    uint8_t* p1 = sQ + t * kTileBytes + r * 128 + ((static_cast<uint32_t>(c) ^ (r & 7)) << 4);
                    uint4 x1 = *reinterpret_cast<const uint4*>(p1);
                    uint4 x2 = *reinterpret_cast<const uint4*>(p1 + kHalf);
                    uint32_t* u1 = reinterpret_cast<uint32_t*>(&x1);
                    uint32_t* u2 = reinterpret_cast<uint32_t*>(&x2);
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        const float4 w = f[cc * 4 + e];  // pairs 8c+2e, 8c+2e+1
                        const __nv_bfloat162 h1 = *reinterpret_cast<const __nv_bfloat162*>(&u1[e]);
                        const __nv_bfloat162 h2 = *reinterpret_cast<const __nv_bfloat162*>(&u2[e]);
                        const float a0 = __low2float(h1), a1 = __high2float(h1);
                        const float b0 = __low2float(h2), b1 = __high2float(h2);
                        u1[e] = pack_bf16(a0 * w.x - b0 * w.y, a1 * w.z - b1 * w.w);
                        u2[e] = pack_bf16(b0 * w.x + a0 * w.y, b1 * w.z + a1 * w.w);
                    }
                    *reinterpret_cast<uint4*>(p1) = x1;
                    *reinterpret_cast<uint4*>(p1 + kHalf) = x2;
                }
            }
            if (!ok) attn_timeout(a.status, abort);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the MMAs read it
            __syncwarp();
            if (lane == 0) mbar_arrive(&q_ready[t]);
        }
#pragma unroll 1
        for (int i = 0; i < my_nt; i++) {
            uint64_t w = 0ull;  // visible keys of this row among this warpgroup's 64
            if (row_ok) {
                int kvalid;
                if (i < a.nct) {
                    kvalid = min(kKeys, a.C - i * kKeys) - cb;
                    w = ~0ull;
                } else {
                    const int wd = 2 * (i - a.nct) + wg;
                    kvalid = nn - wd * 64;
                    if (wd < a.mw) w = __ldg(a.mask + (static_cast<size_t>(s) * a.B + b) * a.mw + wd);
                }
                if (kvalid <= 0)
                    w = 0ull;
                else if (kvalid < 64)
                    w &= (1ull << kvalid) - 1ull;
            }
            const bool full = __all_sync(0xFFFFFFFFu, w == ~0ull);  // the whole warp sees all 64 keys
            // Both warps of a lane quarter reach the pair barrier of every
            // iteration and leave the loop together: a failed wait is
            // exchanged with the row max.
            if (ok && !warp_wait(&s_full[t], static_cast<uint32_t>(i) & 1u, abort)) {
                attn_timeout(a.status, abort);
                ok = false;
            }
            float sv[64];
            float mx = -INFINITY;
            if (ok) {
                tc_fence_after();
                tmem_ld64(tS + cb, sv);
                if (full) {
#pragma unroll
                    for (int c = 0; c < 64; c += 2) mx = fmaxf(mx, fmaxf(sv[c], sv[c + 1]));
                } else {
#pragma unroll
                    for (int c = 0; c < 64; c++) {
                        if (!((w >> c) & 1ull)) sv[c] = -INFINITY;
                        mx = fmaxf(mx, sv[c]);
                    }
                }
            }
            // (S(i) complete: the other warp has arrived at p_full(i - 1),
            // after it read the previous exchange)
            xt[wg * kRows + r] = mx;
            if (lane == 0) xk[wg * 4] = ok ? 1 : 0;
            named_bar_sync(pair_bar, 64);  // also: both halves of S are in registers (P overwrites them)
            mx = fmaxf(mx, xt[(1 - wg) * kRows + r]);
            ok = ok && xk[(1 - wg) * 4] != 0;
            if (!ok) break;
            const float mx2 = mx * a.sl2;
            const bool resc = mx2 > m_run + kRescaleSlack;
            const float m_new = resc ? mx2 : m_run;
            const float alpha = resc ? ex2(m_run - m_new) : 1.0f;
            if (i > 0 && __any_sync(0xFFFFFFFFu, resc)) {
                // (S(i) complete: PV(i - 1) is too)
#pragma unroll 1
                for (int c0 = 0; c0 < 64; c0 += 16) {
                    float o[16];
                    tmem_ld16(tO + c0, o);
#pragma unroll
                    for (int e = 0; e < 16; e++) o[e] *= alpha;
                    tmem_st16(tO + c0, o);
                }
            }
            l *= alpha;
            m_run = m_new;
            const float nm = m_run == -INFINITY ? 0.0f : -m_run;
            float lsum = 0.0f;
#pragma unroll
            for (int hf = 0; hf < 2; hf++) {
                uint32_t pk[16];
#pragma unroll
                for (int c = 0; c < 32; c += 2) {
                    const float p0 = ex2(fmaf(sv[hf * 32 + c], a.sl2, nm));
                    const float p1 = ex2(fmaf(sv[hf * 32 + c + 1], a.sl2, nm));
                    lsum += p0 + p1;
                    pk[c >> 1] = pack_bf16(p0, p1);
                }
                tmem_st16u(tS + wg * 32 + hf * 16, pk);
            }
            tmem_wait_st();
            l += lsum;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&p_full[t]);
        }
        // both tiles' MMAs done: queries and K/V are no longer read
#pragma unroll 1
        for (int u = 0; u < 2; u++) {
            if (ok && nt[u] > 0 && !warp_wait(&o_full[u], 0, abort)) {
                attn_timeout(a.status, abort);
                ok = false;
            }
        }
        tc_fence_after();
        // the row sum is split over the two warpgroups
        xt[wg * kRows + r] = l;
        named_bar_sync(pair_bar, 64);
        l += xt[(1 - wg) * kRows + r];
        const float inv = (row_ok && l > 0.0f) ? 1.0f / l : 0.0f;
        // O / l into shared memory (tile 0 over the queries, tile 1 over K) in
        // the swizzled layout of the store, which clips rows past B: four
        // boxes of 32 columns per tile, two per warpgroup.  (Rows lie 512 bytes
        // apart: stored by their own threads they took 4 µs of a CTA's 50.)
        uint8_t* ob = t ? sK : sQ;
#pragma unroll 1
        for (int c0 = 0; c0 < 64; c0 += 16) {
            float o[16];
            if (my_nt > 0) {
                tmem_ld16(tO + c0, o);
            } else {
#pragma unroll
                for (int e = 0; e < 16; e++) o[e] = 0.0f;
            }
            uint8_t* row = ob + (cb + c0) / 32 * kHalf + r * 128;
            const int ch = (c0 & 16) / 4;  // first 16-byte chunk of the row
#pragma unroll
            for (int e = 0; e < 4; e++)
                *reinterpret_cast<float4*>(row + (((ch + e) ^ (r & 7)) << 4)) =
                    make_float4(o[4 * e] * inv, o[4 * e + 1] * inv, o[4 * e + 2] * inv, o[4 * e + 3] * inv);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        named_bar_sync(kPairBarrier0 + 8 + t * 2 + wg, 128);
        const int q0 = (2 * qp + t) * a.qpt;
        if ((sw & 3) == 0 && lane == 0 && q0 < a.B) {
            for (int q = 2 * wg; q < 2 * wg + 2; q++) tma_store_4d(&tmO, ob + q * kHalf, q * 32, kvh * a.G, q0, s);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ------------------------------------------------------------ ancestor mask

constexpr int kMaskThreads = 1024;

__global__ void __launch_bounds__(kMaskThreads) ancestor_mask_kernel(const int32_t* parents, const int32_t* n_nodes,
                                                                      int B, uint64_t* mask) {
    pdl_trigger();
    pdl_wait();
    const int s = blockIdx.x, mw = (B + 63) / 64;
    const int nn = min(max(n_nodes[s], 0), B);
    const int32_t* par = parents + static_cast<size_t>(s) * B;
    for (int q = threadIdx.x; q < B * mw; q += kMaskThreads) {
        const int i = q / mw, wd = q % mw;
        uint64_t word = 0ull;
        if (i < nn) {
            int j = i;
            for (int steps = 0; steps <= i && j >= 0; steps++) {
                if ((j >> 6) == wd) word |= 1ull << (j & 63);
                const int pj = par[j];
                if (pj < -1 || pj >= j) break;
                j = pj;
            }
        }
        mask[(static_cast<size_t>(s) * B + i) * mw + wd] = word;
    }
}

// ------------------------------------------------------------ host helpers

struct Plan {
    int G, qpt, nqt, blocks, splits, mw, nct;
};

// Workspace: rotated tree keys, then the (cos, sin) table (no device query).
struct WsLayout {
    size_t off_kr, off_cs, total;
};

size_t align256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

bool valid_cfg(const dart_attn_config* c) {
    if (!c) return false;
    if (c->nseq < 1 || c->B < 1 || c->B > 1024 || c->C < 0 || c->Hkv < 1 || c->Hq < c->Hkv) return false;
    if (c->Hq % c->Hkv != 0) return false;
    const int G = c->Hq / c->Hkv;
    if (G != 1 && G != 2 && G != 4 && G != 8 && G != 16) return false;
    if (c->dh != kDh) return false;
    if (!(c->rope_theta > 1.0f) || !std::isfinite(c->rope_theta)) return false;
    if (!(c->scale > 0.0f) || !std::isfinite(c->scale)) return false;
    // TMA coordinates and element counts stay in int range
    if (static_cast<long long>(c->nseq) * c->B * (c->Hq + c->Hkv) > (1ll << 30)) return false;
    if (static_cast<long long>(c->C) * c->Hkv * kDh > (1ll << 40)) return false;
    return true;
}

// Splits of the key list (= cluster size): as many as keep every CTA in one
// wave (1 CTA per SM) with at least two key tiles per split.
int pick_splits(int blocks, int max_tiles, int nsm) {
    int sp = 1;
    while (sp < kMaxSplits && static_cast<long long>(blocks) * (sp + 1) <= nsm && max_tiles / (sp + 1) >= 2) sp++;
    return sp;
}

int key_tiles(const dart_attn_config& c) { return (c.C + kKeys - 1) / kKeys + (c.B + kKeys - 1) / kKeys; }

Plan make_plan(const dart_attn_config* c, int nsm) {
    Plan p;
    p.G = c->Hq / c->Hkv;
    p.qpt = kRows / p.G;
    p.nqt = (c->B + p.qpt - 1) / p.qpt;
    p.blocks = c->nseq * c->Hkv * p.nqt;
    p.mw = (c->B + 63) / 64;
    p.nct = (c->C + kKeys - 1) / kKeys;
    p.splits = pick_splits(p.blocks, key_tiles(*c), nsm);
    return p;
}

// Units of the pair route that go to tree_attn_kernel, one query tile per CTA:
// a last wave that would leave half of the SMs idle.  Measured on GB300, 512
// pairs on 152 SMs (8 x 512 rows, 2048 context keys): four waves of pairs
// 175 µs, three and 112 single tiles 163.
int pair_tail(int nunits, int nsm) {
    const int rem = nunits % nsm;
    return nunits > nsm && 2 * rem <= nsm ? rem : 0;
}

// Whether two query tiles per CTA (tree_attn2_kernel) take less time than one:
// with more tiles than SMs both run in waves, and a kv head with an odd number
// of tiles leaves a pair with one (all such units come first).  In units of one
// key tile a CTA with one query tile takes 4 + n for n key tiles, one with two
// 3 + 1.85 n, one with two of which one is empty 5 + 1.7 n (while those run,
// every SM streams another head's keys and values); the list schedule of the
// pairs against the waves of the single tiles.  The five constants are fitted
// to 530 calls timed both ways on GB300 (40 to 360 kv heads, 2 to 11 tiles
// each, 0 to 8192 context keys): the choice costs at most 3.4 % against the
// better side, 0.05 % on average, where pairs for all of them cost up to 37 %
// (µs, pairs and single tiles: 40 heads of 7 tiles, 2048 keys 74.4, 57.9; 88
// of 3 72.3, 57.3; 360 of 1 109, 99; 56 of 3 47, 54; 64 of 16 163, 190).
bool pairs_pay(const Plan& p, int nheads, int nkt, int nsm) {
    if (p.splits != 1 || p.blocks <= nsm || p.nqt < 2) return false;
    const double one = 4.0 + nkt, full = (3.0 + 1.85 * nkt) / one, half = (5.0 + 1.7 * nkt) / one;
    const int nunits = nheads * ((p.nqt + 1) / 2), tail = pair_tail(nunits, nsm);
    const int nhalf = p.nqt % 2 ? std::min(nheads, nunits - tail) : 0, nfull = nunits - tail - nhalf;
    // the half-empty units: nb SMs are done with them at t1, the others at t0
    const int nb = nhalf % nsm;
    const double t0 = nhalf / nsm * half, t1 = t0 + half;
    double end = 1e30;
    for (int i = std::max(0, nfull / nsm - 2); i <= nfull / nsm + 3; i++) {
        for (const double t : {t0 + i * full, t1 + i * full}) {
            if (t < (nb > 0 ? t1 : t0) - 1e-9) continue;
            const double done = (nsm - nb) * std::floor((t - t0) / full + 1e-9) +
                                nb * std::max(0.0, std::floor((t - t1) / full + 1e-9));
            if (done >= nfull) end = std::min(end, t);
        }
    }
    return end + (tail > 0 ? 1.0 : 0.0) < static_cast<double>((p.blocks + nsm - 1) / nsm);
}

WsLayout ws_layout(const dart_attn_config* c) {
    WsLayout w;
    const size_t kr = static_cast<size_t>(c->nseq) * c->B * c->Hkv * kDh * 2;
    const size_t cs = static_cast<size_t>(c->nseq) * c->B * (kDh / 2) * 8;
    w.off_kr = 0;
    w.off_cs = align256(w.off_kr + kr);
    w.total = align256(w.off_cs + cs);
    return w;
}

// Compute capability, shared-memory opt-in and SM count of a device, queried
// once per device.
struct DevInfo {
    int major, minor, optin, nsm;
};
bool dev_info(int dev, DevInfo* out) {
    constexpr int kMaxDev = 64;
    static DevInfo info[kMaxDev];
    static std::atomic<int> ready[kMaxDev];
    if (dev < 0 || dev >= kMaxDev) return false;
    if (ready[dev].load(std::memory_order_acquire) == 0) {
        DevInfo d{};
        if (cudaDeviceGetAttribute(&d.major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&d.minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&d.optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&d.nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return false;
        info[dev] = d;  // every thread that gets here writes the same values
        ready[dev].store(1, std::memory_order_release);
    }
    *out = info[dev];
    return true;
}

// Queries [nseq][B][Hq][dh] bf16 with a (64, G heads, qpt rows, 1) box: the
// 128 box rows are (tree row, head) pairs, heads fastest.
bool encode_q(CUtensorMap* m, const void* base, int nseq, int B, int Hq, int G, int qpt) {
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn) return false;
    cuuint64_t dims[4] = {static_cast<cuuint64_t>(kDh), static_cast<cuuint64_t>(Hq), static_cast<cuuint64_t>(B),
                          static_cast<cuuint64_t>(nseq)};
    cuuint64_t strides[3] = {static_cast<cuuint64_t>(kDh) * 2, static_cast<cuuint64_t>(Hq) * kDh * 2,
                             static_cast<cuuint64_t>(B) * Hq * kDh * 2};
    cuuint32_t box[4] = {64, static_cast<cuuint32_t>(G), static_cast<cuuint32_t>(qpt), 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The output [nseq][B][Hq][dh] fp32 with a (32, G heads, qpt rows, 1) box.
bool encode_out(CUtensorMap* m, void* base, int nseq, int B, int Hq, int G, int qpt) {
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn) return false;
    cuuint64_t dims[4] = {static_cast<cuuint64_t>(kDh), static_cast<cuuint64_t>(Hq), static_cast<cuuint64_t>(B),
                          static_cast<cuuint64_t>(nseq)};
    cuuint64_t strides[3] = {static_cast<cuuint64_t>(kDh) * 4, static_cast<cuuint64_t>(Hq) * kDh * 4,
                             static_cast<cuuint64_t>(B) * Hq * kDh * 4};
    cuuint32_t box[4] = {32, static_cast<cuuint32_t>(G), static_cast<cuuint32_t>(qpt), 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

// [nseq][len][Hkv][dh] bf16 with a (64, 1, 128 keys, 1) box.
bool encode_kv(CUtensorMap* m, const void* base, int nseq, int len, int Hkv) {
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn) return false;
    cuuint64_t dims[4] = {static_cast<cuuint64_t>(kDh), static_cast<cuuint64_t>(Hkv), static_cast<cuuint64_t>(len),
                          static_cast<cuuint64_t>(nseq)};
    cuuint64_t strides[3] = {static_cast<cuuint64_t>(kDh) * 2, static_cast<cuuint64_t>(Hkv) * kDh * 2,
                             static_cast<cuuint64_t>(len) * Hkv * kDh * 2};
    cuuint32_t box[4] = {64, 1, kKeys, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The kernel's shared-memory opt-in, set once per device (a host call that
// costs microseconds when repeated on every launch).
bool attn_attr_set(int dev) {
    static std::atomic<uint64_t> done{0};
    const uint64_t bit = dev < 64 ? (1ull << dev) : 0ull;
    if (bit && (done.load() & bit)) return true;
    if (cudaFuncSetAttribute(tree_attn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttnSmem) !=
            cudaSuccess ||
        cudaFuncSetAttribute(tree_attn2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttn2Smem) != cudaSuccess)
        return false;
    done.fetch_or(bit);
    return true;
}



// Validates, then enqueues the pre-pass and the attention kernel; ev[0..2]
// (optional) are recorded before the pre-pass, between the two and after.
int enqueue_tree_attention(const dart_attn_config* cfg, const void* q, const void* k_tree, const void* v_tree,
                           const void* k_ctx, const void* v_ctx, const int32_t* pos_ids, const uint64_t* mask,
                           const int32_t* n_nodes, float* out, void* workspace, size_t workspace_bytes,
                           int* status, void* stream, cudaEvent_t* ev) {
    if (!valid_cfg(cfg)) return DART_ERR_INVALID;
    const dart_attn_config& c = *cfg;
    if (!q || !k_tree || !v_tree || !pos_ids || !mask || !n_nodes || !out || !workspace) return DART_ERR_INVALID;
    if (c.C > 0 && (!k_ctx || !v_ctx)) return DART_ERR_INVALID;
    if (!al16(q) || !al16(k_tree) || !al16(v_tree) || !al16(out) || !al16(mask) || !al16(pos_ids) ||
        !al16(n_nodes) || (reinterpret_cast<uintptr_t>(workspace) & 255u))
        return DART_ERR_INVALID;
    if (c.C > 0 && (!al16(k_ctx) || !al16(v_ctx))) return DART_ERR_INVALID;
    if (status && !al16(status)) return DART_ERR_INVALID;
    const WsLayout wl = ws_layout(cfg);
    if (workspace_bytes < wl.total) return DART_ERR_INVALID;
    int dev = 0;
    DevInfo di;
    if (cudaGetDevice(&dev) != cudaSuccess || !dev_info(dev, &di)) return DART_ERR_CUDA;
    if (di.major != 10 || di.minor != 3 || di.optin < std::max(kAttnSmem, kAttn2Smem)) return DART_ERR_UNSUPPORTED;
    const int nsm = di.nsm > 0 ? di.nsm : 148;
    const Plan p = make_plan(cfg, nsm);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    __nv_bfloat16* kr = reinterpret_cast<__nv_bfloat16*>(ws + wl.off_kr);
    float2* cs = reinterpret_cast<float2*>(ws + wl.off_cs);

    const bool two = pairs_pay(p, c.nseq * c.Hkv, key_tiles(c), nsm);  // two query tiles per CTA (tree_attn2_kernel)
    CUtensorMap tmQ, tmKc, tmVc, tmKt, tmVt, tmO;
    if (two && !encode_out(&tmO, out, c.nseq, c.B, c.Hq, p.G, p.qpt)) return DART_ERR_CUDA;
    if (!encode_q(&tmQ, q, c.nseq, c.B, c.Hq, p.G, p.qpt)) return DART_ERR_CUDA;
    if (!encode_kv(&tmKt, kr, c.nseq, c.B, c.Hkv) || !encode_kv(&tmVt, v_tree, c.nseq, c.B, c.Hkv))
        return DART_ERR_CUDA;
    if (c.C > 0) {
        if (!encode_kv(&tmKc, k_ctx, c.nseq, c.C, c.Hkv) || !encode_kv(&tmVc, v_ctx, c.nseq, c.C, c.Hkv))
            return DART_ERR_CUDA;
    } else {
        tmKc = tmKt;  // never read: no context tiles
        tmVc = tmVt;
    }

    PrepArgs ra;
    std::memset(&ra, 0, sizeof ra);
    ra.nseq = c.nseq;
    ra.B = c.B;
    ra.Hkv = c.Hkv;
    ra.kt = static_cast<const __nv_bfloat16*>(k_tree);
    ra.pos_ids = pos_ids;
    ra.kr = kr;
    ra.cs = cs;
    for (int t = 0; t < kDh / 2; t++)
        ra.inv_freq[t] = static_cast<float>(std::pow(static_cast<double>(c.rope_theta), -2.0 * t / kDh));

    AttnArgs aa;
    std::memset(&aa, 0, sizeof aa);
    aa.B = c.B;
    aa.C = c.C;
    aa.Hq = c.Hq;
    aa.Hkv = c.Hkv;
    aa.G = p.G;
    aa.qpt = p.qpt;
    aa.nqt = p.nqt;
    aa.splits = p.splits;
    aa.mw = p.mw;
    aa.nct = p.nct;
    aa.nunits = c.nseq * c.Hkv * ((p.nqt + 1) / 2);
    aa.u0 = -1;
    aa.sl2 = static_cast<float>(static_cast<double>(c.scale) * 1.4426950408889634);
    aa.cs = cs;
    aa.n_nodes = n_nodes;
    aa.mask = mask;
    aa.out = out;
    aa.status = status;

    if (!attn_attr_set(dev)) return DART_ERR_CUDA;
    const int prep_blocks = static_cast<int>(std::min<long long>(
        (static_cast<long long>(c.nseq) * c.B * c.Hkv + 7) / 8, 16LL * nsm));  // 8 rows per block
    if (ev && cudaEventRecord(ev[0], st) != cudaSuccess) return DART_ERR_CUDA;
    if (launch_pdl(attn_prep_kernel, dim3(prep_blocks), dim3(256), 0, st, ra) != cudaSuccess) return DART_ERR_CUDA;
    if (ev && cudaEventRecord(ev[1], st) != cudaSuccess) return DART_ERR_CUDA;
    cudaError_t le;
    if (two) {
        const int single = pair_tail(aa.nunits, nsm);
        le = launch_pdl(tree_attn2_kernel, dim3(aa.nunits - single), dim3(kAttn2Threads), kAttn2Smem, st, tmQ, tmKc, tmVc,
                        tmKt, tmVt, tmO, aa);
        if (le == cudaSuccess && single > 0) {
            aa.u0 = aa.nunits - single;
            le = launch_pdl(tree_attn_kernel, dim3(2 * single), dim3(kAttnThreads), kAttnSmem, st, tmQ, tmKc, tmVc, tmKt,
                            tmVt, aa);
        }
    } else if (p.splits > 1) {
        le = launch_pdl_cluster(tree_attn_kernel, dim3(p.blocks * p.splits), dim3(kAttnThreads), kAttnSmem, st, p.splits,
                                tmQ, tmKc, tmVc, tmKt, tmVt, aa);
    } else {
        le = launch_pdl(tree_attn_kernel, dim3(p.blocks), dim3(kAttnThreads), kAttnSmem, st, tmQ, tmKc, tmVc, tmKt, tmVt,
                        aa);
    }
    if (le != cudaSuccess) return DART_ERR_CUDA;
    if (ev && cudaEventRecord(ev[2], st) != cudaSuccess) return DART_ERR_CUDA;
    return DART_OK;
}

}  // namespace
}  // namespace dart

using namespace dart;

extern "C" {

size_t dart_tree_attention_workspace(const dart_attn_config* cfg) {
    if (!valid_cfg(cfg)) return 0;
    return ws_layout(cfg).total;
}


int dart_tree_attention_tiles(const dart_attn_config* cfg, int num_sms) {
    if (!valid_cfg(cfg) || num_sms < 1) return 0;
    return pairs_pay(make_plan(cfg, num_sms), cfg->nseq * cfg->Hkv, key_tiles(*cfg), num_sms) ? 2 : 1;
}

int dart_tree_attention(const dart_attn_config* cfg, const void* q, const void* k_tree, const void* v_tree,
                        const void* k_ctx, const void* v_ctx, const int32_t* pos_ids, const uint64_t* mask,
                        const int32_t* n_nodes, float* out, void* workspace, size_t workspace_bytes, int* status,
                        void* stream) {
    return enqueue_tree_attention(cfg, q, k_tree, v_tree, k_ctx, v_ctx, pos_ids, mask, n_nodes, out, workspace,
                                  workspace_bytes, status, stream, nullptr);
}

int dart_tree_attention_timed(const dart_attn_config* cfg, const void* q, const void* k_tree, const void* v_tree,
                              const void* k_ctx, const void* v_ctx, const int32_t* pos_ids, const uint64_t* mask,
                              const int32_t* n_nodes, float* out, void* workspace, size_t workspace_bytes,
                              int* status, float* ms_rope, float* ms_attn, void* stream) {
    if (!ms_rope || !ms_attn) return DART_ERR_INVALID;
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    int rc = DART_OK;
    for (int i = 0; i < 3 && rc == DART_OK; i++)
        if (cudaEventCreate(&ev[i]) != cudaSuccess) rc = DART_ERR_CUDA;
    if (rc == DART_OK)
        rc = enqueue_tree_attention(cfg, q, k_tree, v_tree, k_ctx, v_ctx, pos_ids, mask, n_nodes, out, workspace,
                                    workspace_bytes, status, stream, ev);
    if (rc == DART_OK && cudaEventSynchronize(ev[2]) != cudaSuccess) rc = DART_ERR_CUDA;
    if (rc == DART_OK && (cudaEventElapsedTime(ms_rope, ev[0], ev[1]) != cudaSuccess ||
                          cudaEventElapsedTime(ms_attn, ev[1], ev[2]) != cudaSuccess))
        rc = DART_ERR_CUDA;
    for (int i = 0; i < 3; i++)
        if (ev[i]) cudaEventDestroy(ev[i]);
    return rc;
}

int dart_ancestor_mask(const int32_t* parents, const int32_t* n_nodes, int nseq, int B, uint64_t* mask,
                       void* stream) {
    if (!parents || !n_nodes || !mask || nseq < 1 || B < 1 || B > 1024) return DART_ERR_INVALID;
    if (reinterpret_cast<uintptr_t>(mask) & 7u) return DART_ERR_INVALID;
    if (launch_pdl(ancestor_mask_kernel, dim3(nseq), dim3(kMaskThreads), 0, static_cast<cudaStream_t>(stream),
                   parents, n_nodes, B, mask) != cudaSuccess)
        return DART_ERR_CUDA;
    return DART_OK;
}

}  // extern "C"
