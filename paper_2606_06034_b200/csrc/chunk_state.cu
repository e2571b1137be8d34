// State passing and output of chunk-wise Gated DeltaNet, given W (gated) and U of every chunk (tcgen05 + TMEM + TMA).
//
// What it computes, per (batch, value head), chunk after chunk (C = 64 tokens, S0 = state [d_v x d_k] carried in,
// g = chunk-local cumulative log-gate, W = T diag(beta exp(g)) K, U = T diag(beta) V from the chunk-prepare path):
//     U_new = U - W S0^T
//     o_i   = scale (exp(g_i) S0 q_i + sum_{j <= i} exp(g_i - g_j) <k_j, q_i> U_new_j)
//     S_end = exp(g_C) S0 + sum_j exp(g_C - g_j) U_new_j k_j^T
// This is the WY form of the gated delta rule that the chunk-prepare quantities exist for (Sec. 2.1); the chunks of
// one head are a serial chain, heads are independent.
//
// Everything is evaluated with the value dimension on the 128 TMEM lanes ("transposed"): one CTA per (batch, head)
// keeps the state S [d_v x d_k] as an fp32 accumulator in TMEM for the whole sequence, lane t = value feature t.
//     D1  = S0 W^T - U^T      A = S0 as hi + lo bf16 halves in TMEM (the state is O(1) while U_new can be small:
//                             a single bf16 copy costs 1e-2 on strongly correlated keys), B = W tile; the
//                             transpose of U comes from the tensor core as
//                             (-I) U^T with a constant A operand, so no thread ever transposes anything
//     PT  = K Q^T             an M = 64 product: token j = 16 (lane / 32) + lane mod 16 on the lower 16 lanes of every lane
//                             quadrant, columns = token i; lanes 16..31 of a warp read the upper 32 columns of the lower ones
//     O1  = S0 Q^T
//     O2  = U_new^T P^T       A = bf16(U_new^T) (written over D1's columns), B = P_ij = exp(g_i-g_j) PT_ji [j <= i]
//     S  += (U_new^T exp(g_C - g_j)) K     accumulated onto exp(g_C) S0 (the decay is a pass over the TMEM columns)
//     O^T = scale (exp(g_i) O1 + O2)  -> transposed through shared memory -> bulk tensor store
// Two MMA groups per chunk; Q, K, W, U tiles of the next chunk are in flight (two stages) while a chunk is worked on.
// All operand layouts are the ones the chunk-prepare kernel uses.
// Warps: 16 compute warps (four threads per TMEM lane), one that issues every MMA, one that issues the TMA loads and
// the output stores, two that form the gate tables and the norms a chunk ahead. The chain of a sequence is thread work (every phase runs on all 16 warps at once, so its
// instruction count is what it costs); hand-offs to the issuing warp are hardware barriers, completions come back
// through mbarriers (a poll costs ~200 cycles, so as few as possible are waited for).
// Instantiations: packed variable-length sequences (one CTA per (sequence, value head), starting at the sequence's
// first token; the tokens a short last chunk lacks decay nothing and write nothing); state only (no queries, no
// output: the first pass of the segmented call for few long sequences, see launch_chunk_state_segmented); keys and
// queries L2-normalised here (GDN_FLAG_K_L2NORM).
#include <cuda.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace gdn {
namespace {

using namespace sm100;

constexpr int kC = 64;         // chunk size
constexpr int kD = 128;        // d_k = d_v
constexpr int kThreads = 512;  // compute threads, four per TMEM lane; two more warps issue the MMAs and the TMA loads
constexpr int kTabThreads = 64;  // gate tables and norms, one thread per token of a chunk (four warps would cap the registers at 80)
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kMaxOrder = 512;  // sequences that a packed launch takes longest first (see launch_chunk_state)

// TMEM column map (512 columns: one CTA per SM)
constexpr uint32_t kSD = 0;    // 128: state S, fp32 accumulator
constexpr uint32_t kSA = 128;  // 64: bf16(S0) as A operand (K = d_k)
constexpr uint32_t kIA = 192;  // 64: -I as A operand (K = d_v), constant
constexpr uint32_t kD1 = 256;  // 64: S0 W^T - U^T, then the two bf16 forms of U_new^T as A operands
constexpr uint32_t kPT = 320;  // 64: K Q^T (half of the lanes); once read, the lo bf16 halves of the two forms of U_new^T
constexpr uint32_t kO1 = 384;  // 64: S0 Q^T
constexpr uint32_t kO2 = 448;  // 64: U_new^T P^T; between chunks it holds the lo bf16 half of S0 (A operand)
constexpr uint32_t kTmemCols = 512;

// shared memory map (bytes; 1 KB aligned). A [64 x 128] bf16 tile is two [64 x 64] sub-tiles of 8 KB (128B swizzle).
constexpr int kTileBytes = 16384;
constexpr int kStageBytes = 4 * kTileBytes;  // Q, K, W, U
constexpr int kOffQ = 0, kOffK = kTileBytes, kOffW = 2 * kTileBytes, kOffU = 3 * kTileBytes;
constexpr int kOffP = 2 * kStageBytes;       // 2 x 8 KB: P as B operand [64 x 64] (MN-major, no swizzle), hi and lo halves
constexpr int kOffO = kOffP + 16384;          // 2 x 16 KB: O tile staged for the bulk store (128B swizzle), two buffers
constexpr int kTab = 5 * 64;  // floats per table buffer: scale exp(g_i) / ||q_i||, -exp(g_C - g_j) / ||k_j||, g, -1 / ||k_j||, scale / ||q_i||
constexpr int kOffG = kOffO + 2 * kTileBytes;  // three table buffers
constexpr int kSmemTotal = kOffG + 3 * kTab * 4;


struct ParamsS {
    const float* g;
    const float* S_in;  // may be null
    float* S_out;       // may be null
    int* status;
    int H_k, H_v, T, group;
    float scale;
    unsigned flags;  // GDN_FLAG_G_RAW: g holds raw log-gates, prefix-summed inside every chunk here
    // packed variable-length sequences (B = 1): sequence s holds the tokens [seq_start[s], seq_end[s]) of tensors
    // with T tokens per head and is chunked from its own first token; null for dense tensors
    const int* seq_start;  // first token of sequence s
    const int* seq_end;    // one past its last token (the public call passes cu_seqlens and cu_seqlens + 1)
    const int* seq_no_u;   // optional: sequence s runs with U = 0 (the state map of a segment, see the segmented call)
    int n_order;             // sequences (the instantiations that take them longest first)
    int out_from;            // S_out holds the final states of the sequences from this one on
    __nv_bfloat16* O;  // output tensor (rows of a short last chunk are stored one by one)
};

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// bounded mbarrier wait (about a second), as in the chunk-prepare kernels
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    uint32_t i = 0;
    while (!mbar_try_wait_hint(bar, parity, 2000u)) {
        if ((++i & 63u) == 0 && clock64() - t0 > 2000000000LL) return false;
    }
    return true;
}

// The same for a whole warp, with one answer for all its lanes (the hardware barriers behind it count warps). It also gives
// up when another warp has: the lanes still polling then vote on one last poll. Lanes that have left the loop have seen the
// phase complete, so that poll sees it too. (A vote on every poll, or a look at `fail` before the first one, costs the chain of
// the sequence 20 to 40 cycles a chunk: 32 heads x 32768 tokens 1217 and 1207 us instead of 1199.) What follows the first poll is
// one function for the seven places that wait: in line it is code that a short call fetches for nothing (the same shape 1204
// instead of 1192 us, one chunk 34.8 instead of 34.5).
__device__ __noinline__ bool wait_bar_slow(uint64_t* bar, uint32_t parity, const volatile int* fail) {
    const long long t0 = clock64();
    uint32_t i = 0;
    while (!mbar_try_wait_hint(bar, parity, 2000u)) {
        if ((++i & 15u) == 0) {
            const uint32_t lanes = __activemask();
            if (__any_sync(lanes, *fail != 0 || clock64() - t0 > 2000000000LL)) return __all_sync(lanes, mbar_try_wait(bar, parity));
        }
    }
    return true;
}
__device__ __forceinline__ bool wait_bar_warp(uint64_t* bar, uint32_t parity, const volatile int* fail) {
    return mbar_try_wait(bar, parity) || wait_bar_slow(bar, parity, fail);
}

// Hand-offs over hardware barriers: the 16 compute warps arrive and go on, whoever needs their work waits. (An mbarrier poll
// costs the waiting warp ~200-300 cycles per hand-off on the chain of the sequence; this is a few tens.) Per chunk:
//   4  the state copies are in place: 16 compute warps arrive, the issuing warp and the two table warps wait (these stay one
//      chunk ahead)
//   5  U_new, P and the decayed state are in place: 16 compute warps arrive, the issuing warp waits
//   6  the output tile is staged: 16 compute warps arrive, the storing warp waits (not state only)
// These waits have no bound of their own. They end because every warp takes part in every one of them exactly once per chunk,
// also after a bounded wait has run out (s_fail): the issuing, storing and table warps go through all chunks without doing
// their work, and a compute warp that gives up does the rest of its hand-offs as waits (see the end of its loop). No warp
// arrives twice in one generation of a barrier: a warp that goes on has seen a product that was issued behind the generation
// before (D1 of a chunk behind its hand-off 4, O2 and the state behind its hand-off 5) or, for 6, the staging buffer of the chunk
// before released; one that has given up waits for 5, which the issuing warp takes behind 4, and looks whether the storing warp
// has taken 6 (s_taken). (The storing warp in hand-off 4 as well would say so without a look, but it reaches it late where many
// CTAs store at once: 256 heads x 4096 tokens 435 instead of 431 us.)
template <int ID>
__device__ __forceinline__ void handoff_arrive() {
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(kThreads + 32 + (ID == 4 ? kTabThreads : 0)) : "memory");
}
template <int ID>
__device__ __forceinline__ void handoff_wait() {
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(kThreads + 32 + (ID == 4 ? kTabThreads : 0)) : "memory");
}
// 8 columns of 16 lanes: threads 0..15 the columns from taddr on, threads 16..31 of the same lanes those 32 further
__device__ __forceinline__ void tmem_ld8_split32(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.16x32bx2.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], 32;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
typedef unsigned long long f2;  // two packed fp32
__device__ __forceinline__ f2 pair2(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint32_t pack_pair(f2 v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return pack_bf16x2(a, b);
}
// two values as bf16 pairs hi + lo
__device__ __forceinline__ void split_pair(f2 v, uint32_t& hi, uint32_t& lo) {
    hi = pack_pair(v);
    f2 rest;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rest) : "l"(v), "l"(pair2(bf16_lo(hi), bf16_hi(hi))));
    lo = pack_pair(rest);
}
// 16 lanes x 16 columns of an accumulator as the fragments of four 8 x 8 matrices: r[0..1] lanes 0..7, r[2..3] lanes 8..15
// of columns 0..7, r[4..7] the same of columns 8..15; thread l holds lane l / 4, columns 2 (l mod 4) and the next
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

// Sequence of rank `rank` among the p.n_order <= 32 G of a packed call, longest class first, in their order inside a class; one
// warp. Classes by the number of chunks: 0 .. 8, then four to a doubling. Bisection over the 32 classes, then the place inside
// the class. Every CTA does it for itself, in the shadow of the TMEM allocation and of the loads of the sequence's bounds, which
// it leaves in the L1 cache: 0.4 us a CTA up to 64 sequences, 0.7 at 256, 1.3 at 512. (A rank by comparison with every other
// sequence, two barriers more: 2.4 us at 256.)
template <int G>
__device__ __forceinline__ int ranked_sequence(const ParamsS& p, int rank, int lane) {
    int cls[G];
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const int s = i * 32 + lane;
        cls[i] = s < p.n_order ? __ldg(p.seq_end + s) - __ldg(p.seq_start + s) : -kC;
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const int n = (cls[i] + kC - 1) / kC, e = 31 - __clz(n | 8);
        cls[i] = i * 32 + lane >= p.n_order ? -1 : n < 8 ? max(n, 0) : min(8 + (e - 3) * 4 + ((n >> (e - 2)) & 3), 31);
    }
    int lo = 0, longer = 0;  // more than `rank` sequences are of class lo or above, `longer` of the one behind the last bisection
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
        int n = 0;
#pragma unroll
        for (int i = 0; i < G; ++i) n += cls[i] >= lo + step;
        n = __reduce_add_sync(0xFFFFFFFFu, n);
        if (n > rank) lo += step;
        else longer = n;
    }
    int at = rank - longer, found = 0;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const uint32_t members = __ballot_sync(0xFFFFFFFFu, cls[i] == lo);
        const bool me = cls[i] == lo && __popc(members & ((1u << lane) - 1u)) == at;
        const uint32_t hit = __ballot_sync(0xFFFFFFFFu, me);
        if (hit != 0) found = i * 32 + __ffs(hit) - 1;
        at -= __popc(members);
    }
    return found;
}

// VAR: packed variable-length sequences (own instantiation: its masks sit on the chain the dense case is bound by)
// SO: state only: no queries, no output (the first pass of the segmented call); U may be absent per sequence.
// NRM: GDN_FLAG_K_L2NORM (keys and queries normalised here): own instantiations, the plain chain pays nothing for it.
// ORD: packed sequences, longest first (own instantiations: the code in front of the roles costs every CTA of a launch that does
// not use it 0.1 to 0.4 us).
template <bool VAR, bool SO, bool NRM, bool ORD>
__global__ void __launch_bounds__(kThreads + 64 + kTabThreads, 1)
chunk_state_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmU,
                   const __grid_constant__ CUtensorMap tmO, const ParamsS p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    float* gtab = reinterpret_cast<float*>(smem + kOffG);  // (see kTab)

    // One mbarrier per MMA group that is waited for (never two pending phases on one barrier), two per-stage TMA
    // barriers, two on which the storing warp releases the output staging buffers, and one for products still in flight when
    // the CTA gives up. The hand-offs between the warps go over hardware barriers 4, 5 and 6 (handoff_arrive / _wait).
    __shared__ uint64_t bar_full[2], bar_pre, bar_d1, bar_o2, bar_g2, bar_stg[2], bar_end;
    __shared__ uint32_t tmem_base_s;
    __shared__ int s_fail;
    __shared__ int s_taken;  // output tiles that the storing warp has taken over (hand-off 6)
    __shared__ int s_seq;

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int t = tid & 127;  // TMEM lane: value feature (state rows, output columns); token j for PT
    const int h = (tid >> 7) & 3;  // column quarter: 16 of the 64 columns of a product, 32 of the 128 state columns
    const int wq = warp & 3;
    const int lane = tid & 31;
    const bool issuer = warp == kThreads / 32;        // every tcgen05.mma
    const bool producer = warp == kThreads / 32 + 1;  // every TMA load
    const bool tabler = warp >= kThreads / 32 + 2;    // gate tables, norms

    if (tid == 0) {
        mbar_init(&bar_full[0], 1);
        mbar_init(&bar_full[1], 1);
        mbar_init(&bar_pre, 1);
        mbar_init(&bar_d1, 1);
        mbar_init(&bar_o2, 1);
        mbar_init(&bar_g2, 1);
        mbar_init(&bar_stg[0], 1);
        mbar_init(&bar_stg[1], 1);
        mbar_init(&bar_end, 1);
        s_fail = 0;
        s_taken = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmQ);
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmW);
        tma_prefetch_desc(&tmU);
        tma_prefetch_desc(&tmO);
    }
    if (warp == 0) {
        tmem_alloc(&tmem_base_s, kTmemCols);
        tmem_relinquish();
    }
    if (ORD && producer) {
        // longest sequences first: the CTAs with block index k H_v .. take the sequence of rank k
        const int rank = static_cast<int>(blockIdx.x / p.H_v);
        const int s = p.n_order <= 64 ? ranked_sequence<2>(p, rank, lane) : p.n_order <= 128 ? ranked_sequence<4>(p, rank, lane)
                    : p.n_order <= 256 ? ranked_sequence<8>(p, rank, lane) : ranked_sequence<kMaxOrder / 32>(p, rank, lane);
        if (lane == 0) s_seq = s;
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_base_s;
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(wq * 32) << 16);

    // dense: one CTA per (batch, value head), bhv = row of the [B * H_v, T] tensors. Packed sequences: one CTA per
    // (sequence, value head); the tensors have one batch row per head and the sequence starts at token tok0
    int b = blockIdx.x / p.H_v;
    const int hv = blockIdx.x - b * p.H_v;
    if (ORD) b = s_seq;
    const int tok0 = VAR ? __ldg(p.seq_start + b) : 0;
    const int len = VAR ? __ldg(p.seq_end + b) - tok0 : p.T;
    const bool no_u = SO && p.seq_no_u != nullptr && __ldg(p.seq_no_u + b) != 0;
    const int bhv = VAR ? hv : blockIdx.x;
    const int bhk = VAR ? hv / p.group : b * p.H_k + hv / p.group;
    // Token-major tensors [B, T, H, d] (GDN_FLAG_LAYOUT_BTHD) are seen by TMA as (H * d, T, B): the head picks the first
    // column of a box, the batch its outermost index; consecutive tokens of g are H_v apart.
    const bool bthd = (p.flags & GDN_FLAG_LAYOUT_BTHD) != 0;
    const int bz = VAR ? 0 : b;
    const int kx = bthd ? (hv / p.group) * kD : 0, kz = bthd ? bz : bhk;  // Q, K boxes
    const int vx = bthd ? hv * kD : 0, vz = bthd ? bz : bhv;              // W, U, O boxes
    const long long grow0 = bthd ? ((long long)bz * p.T + tok0) * p.H_v + hv : (long long)bhv * p.T + tok0;  // first token's row
    const int gstep = bthd ? p.H_v : 1;
    const int n_c = (len + kC - 1) / kC;
    const float* gseq = p.g + grow0;
    const uint32_t smem_a = smem_u32(smem);
    volatile int* fail = reinterpret_cast<volatile int*>(&s_fail);

    if (tabler) {
        // ================= table threads, one per token. Before hand-off 4 of chunk c they have written the factors of
        // chunk c (read behind the completion of its first product, which that hand-off precedes) and the gates of chunk
        // c + 1 (read from its start on, behind the same completion one chunk earlier). Three buffers: the threads are done
        // with a chunk's tables when they arrive on the next hand-off 4, and the table threads wait for it.
        const int tt = tid - (kThreads + 64);
        const bool g_raw = (p.flags & GDN_FLAG_G_RAW) != 0;
        auto fetch = [&](int c) -> float { return (c < n_c && (!VAR || c * kC + tt < len)) ? __ldg(gseq + (c * kC + tt) * gstep) : 0.f; };
        auto put_gates = [&](int c, float gc) {
            float* tb = gtab + (c % 3) * kTab;
            const int left = len - c * kC;  // tokens of this chunk (>= 64 except for a short last chunk)
            if (g_raw) {
                // inclusive prefix sum over the chunk's 64 tokens: inside each of the two warps by shuffles ...
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const float v = __shfl_up_sync(0xFFFFFFFFu, gc, off);
                    if (lane >= off) gc += v;
                }
                if (tt == 31) tb[128 + 63] = gc;  // ... and the first warp's total through the table itself
                asm volatile("bar.sync 3, 64;" ::: "memory");
                if (tt >= 32) gc += tb[128 + 63];
                asm volatile("bar.sync 3, 64;" ::: "memory");
            }
            tb[128 + tt] = gc;
            asm volatile("bar.sync 3, 64;" ::: "memory");
            if (VAR && !g_raw && left < kC) {
                // cumulative gates: tokens past the end keep the gate of the last real token
                gc = tb[128 + (tt < left ? tt : left - 1)];
                asm volatile("bar.sync 3, 64;" ::: "memory");
                tb[128 + tt] = gc;
                asm volatile("bar.sync 3, 64;" ::: "memory");
            }
        };
        // 1 / ||row|| of row tt of a tile in shared memory (the sum does not care about the swizzle inside the row: each of
        // eight neighbouring threads starts at another 16-byte piece, free of bank conflicts)
        auto inv_norm = [&](const uint8_t* tile) -> float {
            f2 a[2] = {0ull, 0ull};
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const uint4 w4 = *reinterpret_cast<const uint4*>(tile + (i >> 3) * 8192 + tt * 128 + (((i + tt) & 7) << 4));
                const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const f2 x = pair2(bf16_lo(w[q]), bf16_hi(w[q]));
                    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(a[q & 1]) : "l"(x));
                }
            }
            float s0, s1, s2, s3;
            asm("mov.b64 {%0, %1}, %2;" : "=f"(s0), "=f"(s1) : "l"(a[0]));
            asm("mov.b64 {%0, %1}, %2;" : "=f"(s2), "=f"(s3) : "l"(a[1]));
            return rsqrtf(fmaxf((s0 + s1) + (s2 + s3), 1e-30f));
        };
        float g_next = fetch(0);
        if (n_c > 0) put_gates(0, g_next);
        g_next = fetch(1);
        asm volatile("bar.sync 1, %0;" ::"n"(kThreads + kTabThreads) : "memory");
        for (int c = 0; c < n_c; ++c) {
            if (c + 1 < n_c) put_gates(c + 1, g_next);
            g_next = fetch(c + 2);
            float* tb = gtab + (c % 3) * kTab;
            const float gc = tb[128 + tt], gC = tb[128 + 63];
            float rk = 1.f, so = p.scale;
            if (NRM) {
                if (!wait_bar_warp(&bar_full[c & 1], (c >> 1) & 1, fail)) *fail = 1;
                const uint8_t* st = smem + (c & 1) * kStageBytes;
                rk = (VAR && tt >= len - c * kC) ? 0.f : inv_norm(st + kOffK);
                if (!SO) so *= inv_norm(st + kOffQ);
            }
            tb[tt] = so * fast_exp2(gc * kLog2e);
            tb[256 + tt] = so;
            tb[192 + tt] = -rk;
            tb[64 + tt] = -rk * fast_exp2((gC - gc) * kLog2e);
            handoff_wait<4>();
        }
    } else if (producer) {
        // ================= loading / storing warp: the four tiles of chunk c into stage c & 1, as soon as the products
        // that read the stage's previous tiles are complete; and the bulk stores of the staged output tiles, so that
        // no compute thread waits for the others at the end of a chunk
        const bool lead = elect_one();
        auto load_stage = [&](int c) {
            uint8_t* st = smem + (c & 1) * kStageBytes;
            uint64_t* bar = &bar_full[c & 1];
            mbar_arrive_expect_tx(bar, SO ? 3 * kTileBytes : kStageBytes);
            const int t0 = tok0 + c * kC;
            if (!SO) {
                tma_load_3d(st + kOffQ, &tmQ, bar, kx, t0, kz);
                tma_load_3d(st + kOffQ + 8192, &tmQ, bar, kx + 64, t0, kz);
            }
            tma_load_3d(st + kOffK, &tmK, bar, kx, t0, kz);
            tma_load_3d(st + kOffK + 8192, &tmK, bar, kx + 64, t0, kz);
            tma_load_3d(st + kOffW, &tmW, bar, vx, t0, vz);
            tma_load_3d(st + kOffW + 8192, &tmW, bar, vx + 64, t0, vz);
            tma_load_3d(st + kOffU, &tmU, bar, vx, t0, vz);
            tma_load_3d(st + kOffU + 8192, &tmU, bar, vx + 64, t0, vz);
        };
        int loaded = n_c < 2 ? n_c : 2;  // chunks whose tiles have been asked for
        if (lead) {
            if (n_c > 0) load_stage(0);
            if (n_c > 1) load_stage(1);
        }
        uint32_t par = 0;
        for (int c = 0; c < n_c; ++c) {
            // the staged output tile of chunk c is complete (every compute thread has arrived)
            if (!SO) {
                handoff_wait<6>();
                *reinterpret_cast<volatile int*>(&s_taken) = c + 1;
            }
            if (lead && *fail == 0) {
                if (!SO && !(VAR && len - c * kC < kC)) {  // (a short last chunk is stored row by row by the compute threads)
                    tma_store_3d(&tmO, smem + kOffO + (c & 1) * kTileBytes, vx, tok0 + c * kC, vz);
                    tma_store_3d(&tmO, smem + kOffO + (c & 1) * kTileBytes + 8192, vx + 64, tok0 + c * kC, vz);
                    tma_store_commit();
                }
                if (c + 2 < n_c) {
                    if (!wait_bar(&bar_g2, par)) *fail = 1;
                    if (*fail == 0) {
                        load_stage(c + 2);
                        loaded = c + 3;
                    }
                }
                if (!SO) {
                    tma_store_wait_read<0>();
                    mbar_arrive(&bar_stg[c & 1]);  // the staging buffer may be written again (chunk c + 2)
                }
            }
            par ^= 1;
            __syncwarp();
        }
        if (lead) {
            tma_store_wait_all<0>();
            if (*fail != 0) {  // loads still in flight land before the CTA leaves
                for (int c = loaded < 2 ? 0 : loaded - 2; c < loaded; ++c) wait_bar(&bar_full[c & 1], (c >> 1) & 1);
            }
        }
        __syncwarp();
    } else if (issuer) {
        // ================= issuing warp: every tcgen05.mma, in the order the tensor pipe runs them
        const uint32_t idesc_kk64 = instr_desc(128, 64, 1, 1, 0, 0, 1);   // B K-major (a TMA tile as [N x K])
        const uint32_t idesc_mn64 = instr_desc(128, 64, 1, 1, 0, 1, 1);   // B MN-major
        const uint32_t idesc_mn128 = instr_desc(128, 128, 1, 1, 0, 1, 1);
        const uint32_t idesc_pt = instr_desc(64, 64, 1, 1, 0, 0, 1);
        // the products of chunk c that do not depend on the state: D1 <- (-I) U^T and PT = K Q^T
        auto issue_pre = [&](int c) {
            const uint32_t sa = smem_a + (c & 1) * kStageBytes;
            if (!wait_bar_warp(&bar_full[c & 1], (c >> 1) & 1, fail)) *fail = 1;
            tc_fence_after_sync();
            if (*fail == 0 && elect_one()) {
                if (!no_u) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint64_t bd = smem_desc(sa + kOffU + (ks >> 2) * 8192 + (ks & 3) * 32, 16, 1024, SWZ_128B);
                        mma_f16_ts(tmem + kD1, tmem + kIA + ks * 8, bd, idesc_kk64, ks > 0);
                    }
                }
                if (!SO) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint64_t ad = smem_desc(sa + kOffK + (ks >> 2) * 8192 + (ks & 3) * 32, 16, 1024, SWZ_128B);
                        const uint64_t bd = smem_desc(sa + kOffQ + (ks >> 2) * 8192 + (ks & 3) * 32, 16, 1024, SWZ_128B);
                        mma_f16_ss(tmem + kPT, ad, bd, idesc_pt, ks > 0);
                    }
                    mma_commit(&bar_pre);  // (state only: nothing of this group is waited for by itself)
                }
            }
            __syncwarp();
        };
        for (int c = 0; c < n_c; ++c) {
            const uint32_t st_a = smem_a + (c & 1) * kStageBytes;
            // the state copies (and, for the first chunk, the constant operand) are in place
            handoff_wait<4>();
            tc_fence_after_sync();
            if (c == 0) issue_pre(0);
            if (*fail == 0 && elect_one()) {
                // D1 += (S0_hi + S0_lo) W^T onto -U^T, with its own completion barrier
#pragma unroll
                for (int part = 0; part < 2; ++part) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint64_t bd = smem_desc(st_a + kOffW + (ks >> 2) * 8192 + (ks & 3) * 32, 16, 1024, SWZ_128B);
                        mma_f16_ts(tmem + kD1, tmem + (part == 0 ? kSA : kO2) + ks * 8, bd, idesc_kk64,
                                   !no_u || part > 0 || ks > 0);
                    }
                }
                mma_commit(&bar_d1);
                if (!SO) {
                    // O1 = (S0_hi + S0_lo) Q^T
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks) {
                            const uint64_t bd = smem_desc(st_a + kOffQ + (ks >> 2) * 8192 + (ks & 3) * 32, 16, 1024, SWZ_128B);
                            mma_f16_ts(tmem + kO1, tmem + (part == 0 ? kSA : kO2) + ks * 8, bd, idesc_kk64, part > 0 || ks > 0);
                        }
                    }
                }
                // (no completion barrier of its own: the commit behind the output product below covers it, and a wait
                // costs the threads ~200 cycles even on a completed phase)
            }
            __syncwarp();
            // U_new^T (hi, lo; plain, scaled), P (hi, lo) and the decayed accumulator are in place
            handoff_wait<5>();
            tc_fence_after_sync();
            if (*fail == 0 && elect_one()) {
                if (!SO) {
                    // O2 = U_new^T P^T = Uh Ph + Ul Ph + Uh Pl (K-dim = 64 tokens; the plain copy of tokens 16 ks.. sits
                    // at columns 16 ks .. 16 ks + 7 of its region, the gate-scaled one at 16 ks + 8 ..)
#pragma unroll
                    for (int part = 0; part < 3; ++part) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) {
                            const uint64_t bd = smem_desc(smem_a + kOffP + (part == 2 ? 8192 : 0) + ks * 256, 128, 1024, SWZ_NONE);
                            mma_f16_ts(tmem + kO2, tmem + (part == 1 ? kPT : kD1) + ks * 16, bd,
                                       idesc_mn64, part > 0 || ks > 0);
                        }
                    }
                    mma_commit(&bar_o2);  // the output is finished while the state update still runs
                }
                // S += (U_new^T exp(g_C - g_j)) K, hi + lo (the K tile as MN-major operand, N = 128)
#pragma unroll
                for (int part = 0; part < 2; ++part) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        const uint64_t bd = smem_desc(st_a + kOffK + ks * 2048, 8192, 1024, SWZ_128B);
                        mma_f16_ts(tmem + kSD, tmem + (part == 0 ? kD1 : kPT) + ks * 16 + 8, bd,
                                   idesc_mn128, true);
                    }
                }
                mma_commit(&bar_g2);
            }
            __syncwarp();
            // D1 and PT are only read by the products just issued, which the tensor pipe runs first: the
            // state-independent products of the next chunk follow them directly
            if (c + 1 < n_c) issue_pre(c + 1);
        }
        if (*fail != 0 && elect_one()) {  // products still in flight end before their operands go
            mma_commit(&bar_end);
            wait_bar(&bar_end, 0);
        }
        __syncwarp();
    } else {
        // ================= compute threads (512): four per TMEM lane
        uint32_t par_pre = 0, par_d1 = 0, par_o2 = 0, par_g2 = 0;
        // completion of an MMA group: every lane polls the mbarrier (no CTA-wide barrier on this path). A poll of a
        // completed phase costs ~200 cycles whoever issues it; polling from lane 0 alone added a divergent branch and a
        // shuffle, ~150 cycles more per wait.
        auto wait_group = [&](uint64_t* bar, uint32_t& par) -> bool {
            const bool good = wait_bar_warp(bar, par, fail);
            if (!good) *fail = 1;
            par ^= 1;
            tc_fence_after_sync();
            return good;
        };
        // ---- constant A operand -I, initial state, and its bf16 copies (hi in kSA, lo in kO2)
        {
            uint32_t r[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int col = h * 16 + i;  // packed column: features 2 col, 2 col + 1
                r[i] = (col == (t >> 1)) ? ((t & 1) ? 0xBF800000u : 0x0000BF80u) : 0u;
            }
            tmem_st16(lane_base + kIA + h * 16, r);
            // this thread's quarter of state row t: columns [32 h, 32 h + 32)
            const float* s0 = (p.S_in != nullptr) ? p.S_in + (((long long)b * p.H_v + hv) * kD + t) * kD + h * 32 : nullptr;
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                uint32_t v[16], pk[8];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = (s0 != nullptr) ? __float_as_uint(__ldg(s0 + part * 16 + i)) : 0u;
                tmem_st16(lane_base + kSD + h * 32 + part * 16, v);
#pragma unroll
                for (int i = 0; i < 8; ++i) pk[i] = pack_bf16x2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
                tmem_st8(lane_base + kSA + h * 16 + part * 8, pk);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    pk[i] = pack_bf16x2(__uint_as_float(v[2 * i]) - bf16_lo(pk[i]), __uint_as_float(v[2 * i + 1]) - bf16_hi(pk[i]));
                tmem_st8(lane_base + kO2 + h * 16 + part * 8, pk);
            }
            tmem_wait_st();
            tc_fence_before_sync();
            handoff_arrive<4>();
        }
        int gave_up = 0;  // 1, 2, 3: a wait of chunk c ran out before hand-off 5, before 6, behind 6
        asm volatile("bar.sync 1, %0;" ::"n"(kThreads + kTabThreads) : "memory");  // the gates of the first chunk
        int c = 0;
        for (; c < n_c; ++c) {
            const float* se = gtab + (c % 3) * kTab;  // scale exp(g_i) / ||q_i||
            const float* sf = se + 64;               // -exp(g_C - g_j) / ||k_j|| (D1 holds -U_new)
            const float* sg = se + 128;              // g_i (cumulative inside the chunk)
            const float gC = sg[63];
            const int left = len - c * kC;
            const bool short_chunk = VAR && left < kC;

            // ---- decay of the accumulator, S <- exp(g_C) S0 (the products of this chunk read the bf16 copies)
            {
                const float dec = fast_exp2(gC * kLog2e);
                uint32_t v[32];
                tmem_ld32(lane_base + kSD + h * 32, v);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * dec);
                uint32_t w16[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) w16[i] = v[i];
                tmem_st16(lane_base + kSD + h * 32, w16);
#pragma unroll
                for (int i = 0; i < 16; ++i) w16[i] = v[16 + i];
                tmem_st16(lane_base + kSD + h * 32 + 16, w16);
            }
            // ---- P_ij = exp(g_i - g_j) PT_ji for j <= i (hi + lo): this thread's token j and 8 columns i. (Keys and queries
            // normalised here: 1 / ||k_j|| rides on U_new_j, 1 / ||q_i|| on the output.)
            if (!SO && !wait_group(&bar_pre, par_pre)) { gave_up = 1; break; }
            if (!SO) {
                uint32_t d[8];
                tmem_ld8_split32(lane_base + kPT + h * 8, d);
                const int j = wq * 16 + (lane & 15), n8 = (lane >> 4) * 4 + h;  // columns i = 8 n8 ..
                const float gj = sg[j] * kLog2e;
                float gi[8];
#pragma unroll
                for (int i4 = 0; i4 < 2; ++i4) {
                    const float4 q4 = *reinterpret_cast<const float4*>(sg + n8 * 8 + i4 * 4);
                    gi[i4 * 4 + 0] = q4.x; gi[i4 * 4 + 1] = q4.y; gi[i4 * 4 + 2] = q4.z; gi[i4 * 4 + 3] = q4.w;
                }
                tmem_wait_ld();
                uint32_t w[4], wl[4];
#pragma unroll
                for (int i2 = 0; i2 < 4; ++i2) {
                    float v[2];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const float x = __uint_as_float(d[i2 * 2 + q]) * fast_exp2(fminf(fmaf(gi[i2 * 2 + q], kLog2e, -gj), 0.f));
                        v[q] = (j <= n8 * 8 + i2 * 2 + q) ? x : 0.f;
                    }
                    w[i2] = pack_bf16x2(v[0], v[1]);
                    wl[i2] = pack_bf16x2(v[0] - bf16_lo(w[i2]), v[1] - bf16_hi(w[i2]));
                }
                // B operand [K-dim = j][N = i], MN-major, no swizzle: the 16-byte piece of row j for column group n8
                *reinterpret_cast<uint4*>(smem + kOffP + n8 * 1024 + j * 16) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4*>(smem + kOffP + 8192 + n8 * 1024 + j * 16) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
            }
            // ---- U_new^T = -D1 as bf16 hi + lo, plain and gate-scaled (the sums over the tokens of a chunk telescope
            // on correlated keys, so single bf16 copies cost 1e-2 there). This thread's 16 tokens are one k-step of the
            // products that consume them: the hi halves are written over its own D1 columns (plain -> 16 h .. 16 h + 7,
            // scaled -> 16 h + 8 ..), the lo halves at the same offsets of the PT region.
            if (!wait_group(&bar_d1, par_d1)) { gave_up = 1; break; }
            // (the four warps of a lane quadrant have read their columns of PT)
            if (!SO) asm volatile("bar.sync %0, 128;" ::"r"(8 + wq) : "memory");
            {
                uint32_t d[16];
                tmem_ld16(lane_base + kD1 + h * 16, d);
                tmem_wait_ld();
                uint32_t hi[16], lo[16];
#pragma unroll
                for (int i = 0; i < 8; i += 2) {
                    const ulonglong2 f4 = *reinterpret_cast<const ulonglong2*>(sf + h * 16 + 2 * i);
                    ulonglong2 k4;
                    if (NRM && !SO) k4 = *reinterpret_cast<const ulonglong2*>(sg + 64 + h * 16 + 2 * i);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        float d0 = __uint_as_float(d[2 * (i + q)]), d1 = __uint_as_float(d[2 * (i + q) + 1]);
                        if (short_chunk) {  // rows past the sequence's end hold another sequence's W, U
                            if (h * 16 + 2 * (i + q) >= left) d0 = 0.f;
                            if (h * 16 + 2 * (i + q) + 1 >= left) d1 = 0.f;
                        }
                        const f2 u = pair2(d0, d1);
                        split_pair(mul2(u, q == 0 ? f4.x : f4.y), hi[8 + i + q], lo[8 + i + q]);
                        if (!SO) split_pair(NRM ? mul2(u, q == 0 ? k4.x : k4.y) : pair2(-d0, -d1), hi[i + q], lo[i + q]);
                        else hi[i + q] = lo[i + q] = 0u;  // (only the output product reads the plain form)
                    }
                }
                tmem_st16(lane_base + kD1 + h * 16, hi);
                tmem_st16(lane_base + kPT + h * 16, lo);
            }
            fence_proxy_async_smem();
            tmem_wait_st();
            tc_fence_before_sync();
            handoff_arrive<5>();
            if (!SO) {
                // The storing warp has released the PREVIOUS chunk's staging buffer (polled here, in the shadow of the
                // output product; the store was issued most of a chunk ago). That is one chunk later than this chunk's
                // own buffer needs (chunk c - 2 used it, and the stores are read in order), but it also says that the
                // storing warp has taken the previous chunk's hand-off: the threads must not arrive on that hardware
                // barrier a second time before it has, however long a store may be held up.
                if (c >= 1 && !wait_bar_warp(&bar_stg[(c - 1) & 1], ((c - 1) >> 1) & 1, fail)) { *fail = 1; gave_up = 2; break; }
                // ---- O^T = scale (exp(g_i) O1 + O2), in fragments of 8 x 8: this warp's 32 features x 16 tokens, transposed
                // on the way to the staged tile (O1 is complete with O2: products finish in the order they were issued)
                if (!wait_group(&bar_o2, par_o2)) { gave_up = 2; break; }
                {
                    const int t2 = h * 16 + 2 * (lane & 3);
                    const float2 e0 = *reinterpret_cast<const float2*>(se + t2), e1 = *reinterpret_cast<const float2*>(se + t2 + 8);
                    float2 q0 = make_float2(p.scale, p.scale), q1 = q0;
                    if (NRM) {
                        q0 = *reinterpret_cast<const float2*>(se + 256 + t2);
                        q1 = *reinterpret_cast<const float2*>(se + 256 + t2 + 8);
                    }
                    const int tok = h * 16 + ((lane >> 4) << 3) + (lane & 7);  // row of the staged tile this lane addresses
#pragma unroll
                    for (int lh = 0; lh < 2; ++lh) {
                        uint32_t a[8], d[8];
                        tmem_ld_frag(lane_base + (static_cast<uint32_t>(lh * 16) << 16) + kO1 + h * 16, a);
                        tmem_ld_frag(lane_base + (static_cast<uint32_t>(lh * 16) << 16) + kO2 + h * 16, d);
                        tmem_wait_ld();
                        uint32_t m[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const float2 e = k < 2 ? e0 : e1, q = k < 2 ? q0 : q1;
                            m[k] = pack_bf16x2(fmaf(__uint_as_float(a[2 * k]), e.x, __uint_as_float(d[2 * k]) * q.x),
                                               fmaf(__uint_as_float(a[2 * k + 1]), e.y, __uint_as_float(d[2 * k + 1]) * q.y));
                        }
                        const int fb = wq * 4 + lh * 2 + ((lane >> 3) & 1);  // block of 8 features
                        const uint32_t at = smem_a + kOffO + (c & 1) * kTileBytes + (fb >> 3) * 8192 + tok * 128 + (((fb & 7) ^ (tok & 7)) << 4);
                        asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(m[0]), "r"(m[1]),
                                     "r"(m[2]), "r"(m[3])
                                     : "memory");
                    }
                }
                // the tile goes to the storing warp: no compute thread waits for the others here
                fence_proxy_async_smem();
                handoff_arrive<6>();
            }
            // ---- bf16 copies (hi, lo) of the new state for the next chunk's products; the lo half goes where O2 was
            // (this thread has read its O2 columns above)
            if (!wait_group(&bar_g2, par_g2)) { gave_up = 3; break; }
            {
                uint32_t v[32], pk[16];
                tmem_ld32(lane_base + kSD + h * 32, v);
                tmem_wait_ld();
                uint32_t lo[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) split_pair(pair2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), pk[i], lo[i]);
                tmem_st16(lane_base + kSA + h * 16, pk);
                tmem_st16(lane_base + kO2 + h * 16, lo);
                tmem_wait_st();
                tc_fence_before_sync();
                handoff_arrive<4>();
            }
            if (!SO && short_chunk) {
                // only the rows of real tokens leave, 16 bytes per thread and step, from the staged (swizzled) tile
                asm volatile("bar.sync 1, 512;" ::: "memory");  // (last chunk of a packed sequence only)
                for (int q = tid; q < left * 16; q += kThreads) {
                    const int tok = q >> 4, ch = q & 15;  // 16-byte piece ch of the token's 256-byte row
                    const uint4 v = *reinterpret_cast<const uint4*>(smem + kOffO + (c & 1) * kTileBytes + (ch >> 3) * 8192 +
                                                                    tok * 128 + (((ch & 7) ^ (tok & 7)) << 4));
                    *reinterpret_cast<uint4*>(p.O + (grow0 + (long long)(c * kC + tok) * gstep) * kD + ch * 8) = v;
                }
            }
        }
        if (gave_up != 0) {
            // A bounded wait ran out (s_fail is set): this warp's remaining barriers of chunk c and of the chunks behind it, in
            // the order of the loop above and as waits, so that no generation counts it twice.
            for (; c < n_c; ++c, gave_up = 1) {
                if (gave_up < 2) {
                    if (!SO) asm volatile("bar.sync %0, 128;" ::"r"(8 + wq) : "memory");
                    handoff_wait<5>();
                }
                if (!SO && gave_up < 3) {
                    // (it will: this warp has arrived there, the others arrive or wait there too; bounded as every wait)
                    const long long t0 = clock64();
                    while (__any_sync(0xFFFFFFFFu, *reinterpret_cast<volatile int*>(&s_taken) < c && clock64() - t0 < 2000000000LL)) {
                    }
                    handoff_wait<6>();
                }
                if (c + 1 < n_c) handoff_wait<4>();
                if (VAR && !SO && len - c * kC < kC) asm volatile("bar.sync 1, 512;" ::: "memory");
            }
            gave_up = 1;
        }
        // ---- final state
        // (the run's place among the states is formed again here: it is not held over the chunks)
        const int seq = ORD ? *reinterpret_cast<volatile int*>(&s_seq) : static_cast<int>(blockIdx.x / p.H_v);
        if (gave_up == 0 && p.S_out != nullptr && seq >= p.out_from) {
            float* so = p.S_out + (((long long)(seq - p.out_from) * p.H_v + blockIdx.x % p.H_v) * kD + t) * kD + h * 32;
            uint32_t v[32];
            tmem_ld32(lane_base + kSD + h * 32, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float4*>(so + i * 4) =
                    make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]), __uint_as_float(v[4 * i + 2]),
                                __uint_as_float(v[4 * i + 3]));
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (tid == 0 && *fail != 0) atomicExch(p.status, GDN_ERR_TIMEOUT);
    if (warp == 0) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, kTmemCols);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (fn == nullptr) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

// [heads][T][cols] bf16 tensor (cols = 128, or H * 128 for token-major tensors with heads = B), boxes of 64 rows x 64
// columns, 128-byte swizzle
bool make_map(CUtensorMap* tm, const void* base, long long heads, int T, int cols) {
    EncodeTiledFn enc = get_encode_fn();
    if (enc == nullptr) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(T), static_cast<cuuint64_t>(heads)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(cols) * 2, static_cast<cuuint64_t>(T) * cols * 2};
    cuuint32_t box[3] = {64, static_cast<cuuint32_t>(kC), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---- the segmented call: a long sequence cut into P segments whose state maps are formed in parallel
// Set-up of the first pass: the token ranges of its 2P - 3 runs (runs 0 .. P-2: segment s from a zero state, segment 0
// from the caller's; runs P-1 .. 2P-4: segments 1 .. P-2 from the identity with U = 0, which gives the matrix M of
// S_end = S_start M + N), their initial states, the token ranges of the second pass and its first initial state.
// Grid (value heads, n1 + 1 states): one state of 128 x 128 per CTA. (The heads along x: y ends at 65535.)
__global__ void __launch_bounds__(256) segmented_setup_kernel(int P, int H_v, int n_chunks, const float* S_user, float* S_in1,
                                                              float* S_start, int* start1, int* end1, int* no_u1, int* start3,
                                                              int* end3) {
    const int n1 = 2 * P - 3;
    const int run = blockIdx.y, hv = blockIdx.x;
    if (run == 0 && hv == 0) {
        for (int s_ = threadIdx.x; s_ < n1; s_ += 256) {
            const int seg = (s_ <= P - 2) ? s_ : s_ - (P - 2);
            start1[s_] = (int)((long long)n_chunks * seg / P) * kC;
            end1[s_] = (int)((long long)n_chunks * (seg + 1) / P) * kC;
            no_u1[s_] = (s_ <= P - 2) ? 0 : 1;
        }
        for (int s_ = threadIdx.x; s_ < P; s_ += 256) {
            start3[s_] = (int)((long long)n_chunks * s_ / P) * kC;
            end3[s_] = (int)((long long)n_chunks * (s_ + 1) / P) * kC;
        }
    }
    const bool user = (run == 0 || run == n1) && S_user != nullptr;
    const bool eye = run > P - 2 && run < n1;
    const float4* src = reinterpret_cast<const float4*>(S_user + (user ? (long long)hv * kD * kD : 0));
    float4* dst = reinterpret_cast<float4*>((run < n1 ? S_in1 + (long long)run * H_v * kD * kD : S_start) + (long long)hv * kD * kD);
#pragma unroll 4
    for (int i = threadIdx.x; i < kD * kD / 4; i += 256) {
        float4 v = user ? src[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        if (eye) {
            const int row = i / (kD / 4), c = row - (i % (kD / 4)) * 4;  // the diagonal's place among these four
            v = make_float4(c == 0, c == 1, c == 2, c == 3);
        }
        dst[i] = v;
    }
}

// S_start[k] = S_start[k-1] M_{k-1} + N_{k-1} for k = 2 .. P-1, S_start[1] = N_0 (the first segment ran from the caller's
// state). One CTA per (value head, block of 32 state rows): the rows of the state are independent. fp32 FMAs, every sum
// in the order of the state's columns. M (64 KB) comes into shared memory while the step before is worked on; a thread
// holds 4 rows x 4 columns. What a step costs is the chain load -> product: 3 us (one thread column per output, M read from
// L2 in the loop: 13 us).
constexpr int kCombRows = 32;
constexpr int kCombSmem = 2 * kD * kD * 4;
__global__ void __launch_bounds__(256) segmented_combine_kernel(int P, int H_v, const float* S_out1, float* S_start) {
    extern __shared__ __align__(16) float comb_m[];  // two buffers of M
    __shared__ __align__(16) float cur[kCombRows][kD + 4];
    const int hv = blockIdx.x, r0 = blockIdx.y * kCombRows;
    const long long per = (long long)H_v * kD * kD;
    const float* base = S_out1 + (long long)hv * kD * kD;  // N of segment s at s * per, M of segment s (1 <= s <= P - 2) at (P - 2 + s) * per
    float* out = S_start + (long long)hv * kD * kD;
    const int col = (threadIdx.x & 31) * 4, rw = (threadIdx.x >> 5) * 4;  // this thread: rows r0 + rw .., columns col ..
    auto fetch = [&](int s) {
        const float* M = base + (long long)(P - 2 + s) * per;
        float* dst = comb_m + (s & 1) * (kD * kD);
        for (int i = threadIdx.x * 4; i < kD * kD; i += 1024) {
            const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(dst + i));
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(M + i) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (P > 2) fetch(1);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(base + (r0 + rw + r) * kD + col);
        *reinterpret_cast<float4*>(&cur[rw + r][col]) = v;
        *reinterpret_cast<float4*>(out + per + (r0 + rw + r) * kD + col) = v;
    }
    for (int k = 2; k < P; ++k) {
        float4 acc[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = *reinterpret_cast<const float4*>(base + (long long)(k - 1) * per + (r0 + rw + r) * kD + col);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();  // M of this step and the state rows are in place, the other buffer is free
        if (k + 1 < P) fetch(k);
        const float* M = comb_m + ((k - 1) & 1) * (kD * kD);
#pragma unroll 2
        for (int d = 0; d < kD; d += 4) {
            float4 c[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) c[r] = *reinterpret_cast<const float4*>(&cur[rw + r][d]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 m = *reinterpret_cast<const float4*>(M + (d + q) * kD + col);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float x = q == 0 ? c[r].x : q == 1 ? c[r].y : q == 2 ? c[r].z : c[r].w;
                    acc[r].x = fmaf(x, m.x, acc[r].x);
                    acc[r].y = fmaf(x, m.y, acc[r].y);
                    acc[r].z = fmaf(x, m.z, acc[r].z);
                    acc[r].w = fmaf(x, m.w, acc[r].w);
                }
            }
        }
        __syncwarp();  // (a warp reads and writes its own four rows of the state only)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            *reinterpret_cast<float4*>(&cur[rw + r][col]) = acc[r];
            *reinterpret_cast<float4*>(out + (long long)k * per + (r0 + rw + r) * kD + col) = acc[r];
        }
    }
}

}  // namespace

size_t chunk_state_segmented_workspace(int H_v, int P) {
    if (P < 2) return 0;
    const size_t per = (size_t)H_v * kD * kD * sizeof(float);
    const size_t n1 = (size_t)(2 * P - 3);
    // (P states more than the passes use: what callers allocate, and what the built-in array takes, stays as it was published)
    return (2 * n1 + 2 * (size_t)P) * per + (3 * n1 + 2 * (size_t)P) * sizeof(int) + 256;
}

int chunk_state_auto_segments(long long H_v) {
    int n_sm = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    int P = 1;
    while (P < 8 && H_v * (2 * (P + 1) - 3) <= n_sm) ++P;
    return P;
}

// One sequence per value head (B = 1), cut into P segments: first pass = every segment's state map in parallel (state
// only), then the segments' initial states by a short recurrence, then every segment in parallel with its output.
int launch_chunk_state_segmented(const ProblemS& q, int P, void* workspace, cudaStream_t stream) {
    if (q.B != 1 || q.seq_start != nullptr) return GDN_ERR_UNSUPPORTED;
    const int n_chunks = q.T / kC;
    if (P > n_chunks) P = n_chunks;
    if (P < 2) return launch_chunk_state(q, stream);
    const size_t per = (size_t)q.H_v * kD * kD;
    const size_t n1 = (size_t)(2 * P - 3);
    float* S_in1 = static_cast<float*>(workspace);
    float* S_out1 = S_in1 + n1 * per;
    float* S_start = S_out1 + n1 * per;
    int* start1 = reinterpret_cast<int*>(S_start + (size_t)P * per);
    int* end1 = start1 + n1;
    int* no_u1 = end1 + n1;
    int* start3 = no_u1 + n1;
    int* end3 = start3 + P;
    segmented_setup_kernel<<<dim3(q.H_v, static_cast<unsigned>(n1) + 1), 256, 0, stream>>>(P, q.H_v, n_chunks, q.S_in, S_in1, S_start, start1, end1, no_u1, start3, end3);
    if (cudaGetLastError() != cudaSuccess) return GDN_ERR_LAUNCH;  // (the passes read the token ranges it writes)
    count_launch();
    ProblemS a = q;
    a.B = static_cast<int>(n1);
    a.S_in = S_in1;
    a.S_out = S_out1;
    a.O = q.O;  // not written
    a.seq_start = start1;
    a.seq_end = end1;
    a.seq_no_u = no_u1;
    a.state_only = true;
    int rc = launch_chunk_state(a, stream);
    if (rc != GDN_OK) return rc;
    if (cudaFuncSetAttribute(segmented_combine_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCombSmem) != cudaSuccess)
        return GDN_ERR_LAUNCH;
    segmented_combine_kernel<<<dim3(q.H_v, kD / kCombRows), 256, kCombSmem, stream>>>(P, q.H_v, S_out1, S_start);
    if (cudaGetLastError() != cudaSuccess) return GDN_ERR_LAUNCH;
    count_launch();
    ProblemS b = q;
    b.B = P;
    b.S_in = S_start;
    b.out_from = P - 1;  // (only the last segment's state leaves)
    b.seq_start = start3;
    b.seq_end = end3;
    rc = launch_chunk_state(b, stream);
    if (rc != GDN_OK) return rc;
    return cudaGetLastError() == cudaSuccess ? GDN_OK : GDN_ERR_LAUNCH;
}

// ---- the segmented call on built-in scratch memory (for callers that cannot allocate device memory)
// The scratch lives in this file-scope device array: every GPU that loads the library holds it until the process
// exits. In host code the array's name is only a handle; the device address comes from cudaGetSymbolAddress, once per
// device, with that device current.
namespace {
constexpr size_t kBuiltinStateBlocks = 128;  // state-sized blocks of 128 x 128 fp32 (64 KB each): 8 MB
constexpr size_t kBuiltinScratchBytes = kBuiltinStateBlocks * kD * kD * sizeof(float) + 4096;
static __device__ __align__(256) unsigned char g_builtin_scratch[kBuiltinScratchBytes];
constexpr int kMaxDev = 64;
void* g_builtin_scratch_addr[kMaxDev] = {nullptr};
}  // namespace

int launch_chunk_state_segmented_builtin(const ProblemS& q, int P, cudaStream_t stream) {
    const int n_chunks = q.T / kC;
    const int p_eff = P > n_chunks ? n_chunks : P;
    if (p_eff >= 2 && chunk_state_segmented_workspace(q.H_v, p_eff) > kBuiltinScratchBytes) return GDN_ERR_SCRATCH;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return GDN_ERR_LAUNCH;
    if (g_builtin_scratch_addr[dev] == nullptr) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_builtin_scratch) != cudaSuccess || ptr == nullptr) {
            cudaGetLastError();
            return GDN_ERR_LAUNCH;
        }
        g_builtin_scratch_addr[dev] = ptr;
    }
    return launch_chunk_state_segmented(q, P, g_builtin_scratch_addr[dev], stream);
}


int launch_chunk_state(const ProblemS& q, cudaStream_t stream) {
    if (q.d_k != kD || q.d_v != kD || q.C != kC) return GDN_ERR_UNSUPPORTED;
    // packed sequences: B counts the sequences, the tensors have one row of T tokens per head
    const bool var = q.seq_start != nullptr;
    if (q.state_only && !var) return GDN_ERR_UNSUPPORTED;
    const long long hk = var ? q.H_k : (long long)q.B * q.H_k, hv = var ? q.H_v : (long long)q.B * q.H_v;
    const long long n_cta = (long long)q.B * q.H_v;
    if (n_cta == 0) return GDN_OK;
    if (q.T == 0) {
        // no tokens: every sequence hands its initial state on (zeros without one)
        if (q.S_out != nullptr && !q.state_only) {
            const size_t bytes = static_cast<size_t>(n_cta) * kD * kD * sizeof(float);
            const cudaError_t e = (q.S_in != nullptr) ? cudaMemcpyAsync(q.S_out, q.S_in, bytes, cudaMemcpyDeviceToDevice, stream)
                                                      : cudaMemsetAsync(q.S_out, 0, bytes, stream);
            if (e != cudaSuccess) return GDN_ERR_LAUNCH;
        }
        return GDN_OK;
    }
    if (n_cta >= (1LL << 31)) return GDN_ERR_UNSUPPORTED;
    if (hv >= (1LL << 31)) return GDN_ERR_UNSUPPORTED;
    int* status = device_status_word();
    if (status == nullptr) return GDN_ERR_LAUNCH;
    CUtensorMap mQ, mK, mW, mU, mO;
    const bool bthd = (q.flags & GDN_FLAG_LAYOUT_BTHD) != 0;
    const long long nb = var ? 1 : q.B;
    const long long zk = bthd ? nb : hk, zv = bthd ? nb : hv;
    const int ck = bthd ? q.H_k * kD : kD, cv = bthd ? q.H_v * kD : kD;
    if (!make_map(&mQ, q.Q, zk, q.T, ck) || !make_map(&mK, q.K, zk, q.T, ck) || !make_map(&mW, q.W, zv, q.T, cv) ||
        !make_map(&mU, q.U, zv, q.T, cv) || !make_map(&mO, q.O, zv, q.T, cv))
        return GDN_ERR_LAUNCH;
    ParamsS prm;
    prm.g = q.g;
    prm.S_in = q.S_in;
    prm.S_out = q.S_out;
    prm.status = status;
    prm.H_k = q.H_k;
    prm.H_v = q.H_v;
    prm.T = q.T;
    prm.group = q.H_v / q.H_k;
    prm.scale = q.scale;
    prm.flags = q.flags;
    prm.seq_start = q.seq_start;
    prm.seq_end = q.seq_end;
    prm.seq_no_u = q.seq_no_u;
    prm.out_from = q.out_from;
    prm.O = static_cast<__nv_bfloat16*>(q.O);
    // More runs than SMs (one CTA each): the long ones may start first, so that none of them is left for the end. That saves a
    // share of the longest run once, in proportion to the mean run, and costs every CTA (0.25 + 0.002 n) us for finding its
    // sequence. It is done where the waves of CTAs times that are at most 1.5 us per chunk of the mean run. State passing,
    // log-normal lengths (gain) and equal ones (cost), with the order / without: 61 sequences of 500 tokens, 8 heads, 131 / 181 us
    // and 131 / 129; 256 of 128, 2 heads, 70 / 99 and 57 / 54. Beyond the line: 256 of 64, 128 heads, 2780 / 2560 us.
    const double chunks = q.T / 64.0 + 0.5 * q.B;  // of all sequences
    const bool ordered = var && !q.state_only && n_cta > kSMs && q.B > 1 && q.B <= kMaxOrder &&
                         static_cast<double>(n_cta) * q.B * (125 + q.B) <= 750.0 * kSMs * chunks;
    prm.n_order = q.B;
    const int smem = kSmemTotal + 1024;
    const bool nrm = (q.flags & GDN_FLAG_K_L2NORM) != 0;
    auto kern = q.state_only ? (nrm ? chunk_state_kernel<true, true, true, false> : chunk_state_kernel<true, true, false, false>)
                : ordered    ? (nrm ? chunk_state_kernel<true, false, true, true> : chunk_state_kernel<true, false, false, true>)
                : var        ? (nrm ? chunk_state_kernel<true, false, true, false> : chunk_state_kernel<true, false, false, false>)
                             : (nrm ? chunk_state_kernel<false, false, true, false> : chunk_state_kernel<false, false, false, false>);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return GDN_ERR_LAUNCH;
    kern<<<static_cast<int>(n_cta), kThreads + 64 + kTabThreads, smem, stream>>>(mQ, mK, mW, mU, mO, prm);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? GDN_OK : GDN_ERR_LAUNCH;
}

}  // namespace gdn
