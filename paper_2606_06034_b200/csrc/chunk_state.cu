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
//     D1  = S0 W^T            A = S0 as hi + lo bf16 halves in TMEM (the state is O(1) while U_new can be small:
//                             a single bf16 copy costs 1e-2 on strongly correlated keys), B = W tile
//     U_new^T = U^T - D1      by threads: ldmatrix transposes 8 x 8 blocks of the U tile into the fragments in which D1 is read
//     PT  = K Q^T             an M = 64 product: token j = 16 (lane / 32) + lane mod 16 on the lower 16 lanes of every lane
//                             quadrant, columns = token i; lanes 16..31 of a warp read other columns of the lower ones
//     O1  = S0 Q^T
//     O2  = U_new^T P^T       A = bf16(U_new^T) (written over D1's columns), B = P_ij = exp(g_i-g_j) PT_ji [j <= i]
//     S  += (U_new^T exp(g_C - g_j)) K     accumulated onto exp(g_C) S0 (the decay is a pass over the TMEM columns)
//     O^T = scale (exp(g_i) O1 + O2)  -> transposed through shared memory -> bulk tensor store
// All operand layouts are the ones the chunk-prepare kernel uses.
// Warps: 8 chain warps (the state's copies, U_new, the decay), 8 output warps (P, O and the norms: nothing of theirs is on the chain),
// one that issues every MMA, one that issues the TMA loads and stores, two that form the gate tables.
// What bounds it: the chain of a sequence is D1 (16 products, 700 cycles with its completion) -> U_new (800) -> state update (first
// half 500) -> copies (650), 2900 cycles a chunk; and beside it the SM's shared memory, of which a chunk's products, TMA
// copies and fragments move 335 KB, 2600 cycles at its full rate. So the state's columns go through the update, the copies
// and D1 in two halves (the tensor pipe works on one while threads work on the other), what a phase reads from shared memory is
// fetched before its products start, and a hi + lo split takes four instructions (see split_neg). us per chunk of 32
// sequences of 256 chunks, before (16 warps that did everything in turn) and now: 2.33 and 1.61, with norms 2.60 and 1.97 (the norms read 32 KB
// of shared memory a chunk: 0.2 of that).
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
constexpr int kChain = 256;    // threads that carry the state's chain, two per TMEM lane
constexpr int kAux = 256;      // threads that form P, the output and the norms, two per TMEM lane
constexpr int kThreads = 512;  // both; two more warps issue the MMAs and the TMA copies
static_assert(kThreads == kChain + kAux, "");
constexpr int kTabThreads = 64;  // gate tables, one thread per token of a chunk
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kMaxOrder = 512;  // sequences that a packed launch takes longest first (see launch_chunk_state)

// TMEM column map (512 columns: one CTA per SM)
constexpr uint32_t kSD = 0;    // 128: state S, fp32 accumulator
constexpr uint32_t kSA = 128;  // 64: bf16(S0) as A operand (K = d_k)
constexpr uint32_t kSL = 192;  // 64: the rest bf16(S0) leaves, negated (A operand)
constexpr uint32_t kD1 = 256;  // 64: S0 W^T, then the hi halves of the two forms of U_new^T as A operands
constexpr uint32_t kUL = 320;  // 64: the lo halves of the two forms of U_new^T, negated
constexpr uint32_t kO1 = 384;  // 64: S0 Q^T
constexpr uint32_t kO2 = 448;  // 64: U_new^T P^T
constexpr uint32_t kPT = kO2;  // K Q^T (half of the lanes): read before O2 of the same chunk is issued
constexpr uint32_t kTmemCols = 512;
// A lo half is kept negated, as the difference comes out of a mixed-precision subtraction: its products subtract
constexpr uint32_t kNegA = 1u << 13, kNegB = 1u << 14;  // instruction descriptor: A or B negated

// shared memory map (bytes; 1 KB aligned). A [64 x 128] bf16 tile is two [64 x 64] sub-tiles of 8 KB (128B swizzle).
constexpr int kTileBytes = 16384;
constexpr int kRing = 3;  // K and Q tiles: in use from the norms on until the state update, so they are asked for three chunks ahead
constexpr int kOffK = 0, kOffQ = kRing * kTileBytes;
constexpr int kOffW = 2 * kRing * kTileBytes, kOffU = kOffW + 2 * kTileBytes;  // two each
constexpr int kOffP = kOffU + 2 * kTileBytes;  // 2 x 8 KB: P as B operand [64 x 64] (MN-major, no swizzle), hi and lo halves
constexpr int kOffO = kOffP + 16384;          // 2 x 16 KB: O tile staged for the bulk store (128B swizzle), two buffers
constexpr int kTab = 5 * 64;  // floats per table buffer: scale exp(g_i) / ||q_i||, exp(g_C - g_j) / ||k_j||, g, 1 / ||k_j||, scale / ||q_i||
constexpr int kOffG = kOffO + 2 * kTileBytes;  // four table buffers
constexpr int kSmemTotal = kOffG + 4 * kTab * 4;
static_assert(kSmemTotal + 1024 <= 227 * 1024, "");


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
// phase complete, so that poll sees it too. (A vote on every poll gives the same times.) What follows the first poll is
// one function for the places that wait. In line it is twice the code: layer calls of 8 x 4096 tokens 730 instead of 715 us, 32768
// tokens 1026 instead of 1038, one chunk 22.6 instead of 22.9.
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

// Hand-offs to the issuing warp over hardware barriers: the warps whose work it needs arrive and go on, it waits. (A poll of an
// mbarrier, though its phase be complete, costs the issuing warp 100 to 200 cycles behind the products it has just issued, this 20 to 40.)
//   4, 6  the copies of either half of the state's columns are in place (8 chain warps); 4 also: the tiles and the tables of the
//         chunk are (2 table warps, which wait too and so stay one chunk ahead)
//   5     U_new and the decayed state are in place (8 chain warps)
//   7, 8  P is in place; O1 and O2 have been read (8 output warps)
// These waits have no bound of their own. They end because every warp takes part in every one of its hand-offs exactly
// once per chunk, also after a bounded wait has run out (s_fail): the issuing and table warps go through all chunks without doing their
// work, and a chain or output warp that gives up does the rest of its hand-offs as waits (see the end of its loop). No warp
// arrives twice in one generation of a barrier: a warp that goes on has seen a product that was issued behind the generation
// before (D1 of a chunk behind its hand-offs 4 and 6, the state update behind 5, O2 behind 7, the next P^T behind 8).
static_assert(kChain == kAux, "");
template <int ID>
__device__ __forceinline__ void handoff_arrive() {
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(kChain + 32 + (ID == 4 ? kTabThreads : 0)) : "memory");
}
template <int ID>
__device__ __forceinline__ void handoff_wait() {
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(kChain + 32 + (ID == 4 ? kTabThreads : 0)) : "memory");
}
// 16 columns of 16 lanes: threads 0..15 the columns from taddr on, threads 16..31 of the same lanes those 32 further
__device__ __forceinline__ void tmem_ld16_split32(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.16x32bx2.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16], 32;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                   "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr)
                 : "memory");
}
// 8 columns of 16 lanes: threads 0..15 the columns from taddr on, threads 16..31 of the same lanes the next 8
__device__ __forceinline__ void tmem_ld8_split8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.16x32bx2.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], 8;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ uint32_t pack_pair(f2 v) {
    float a, b;
    unpair2(v, a, b);
    return pack_bf16x2(a, b);
}
// half HI of a bf16 pair minus x, in fp32 (one instruction, no unpacking)
template <int HI>
__device__ __forceinline__ float bf16_minus(uint32_t w, float x) {
    float r;
    if (HI) asm("{\n\t.reg .b16 a, b;\n\tmov.b32 {a, b}, %1;\n\tsub.f32.bf16 %0, b, %2;\n\t}" : "=f"(r) : "r"(w), "f"(x));
    else asm("{\n\t.reg .b16 a, b;\n\tmov.b32 {a, b}, %1;\n\tsub.f32.bf16 %0, a, %2;\n\t}" : "=f"(r) : "r"(w), "f"(x));
    return r;
}
// s0 += lo^2, s1 += hi^2 of a bf16 pair
__device__ __forceinline__ void bf16_square_add(uint32_t w, float& s0, float& s1) {
    asm("{\n\t.reg .b16 a, b;\n\tmov.b32 {a, b}, %2;\n\tfma.rn.f32.bf16 %0, a, a, %0;\n\tfma.rn.f32.bf16 %1, b, b, %1;\n\t}"
        : "+f"(s0), "+f"(s1)
        : "r"(w));
}
// two values as bf16 pairs, v = hi - neg_lo. 5.9 issue cycles per warp and pair; with the unpacked hi half subtracted from v (hi + lo)
// 10.2, which is what the phases of the chain were bound by.
__device__ __forceinline__ void split_neg(float v0, float v1, uint32_t& hi, uint32_t& neg_lo) {
    hi = pack_bf16x2(v0, v1);
    neg_lo = pack_bf16x2(bf16_minus<0>(hi, v0), bf16_minus<1>(hi, v1));
}
__device__ __forceinline__ void split_neg(f2 v, uint32_t& hi, uint32_t& neg_lo) {
    split_neg(__uint_as_float(static_cast<uint32_t>(v)), __uint_as_float(static_cast<uint32_t>(v >> 32)), hi, neg_lo);
}
// 16 lanes x 16 columns of an accumulator as the fragments of four 8 x 8 matrices: r[0..1] lanes 0..7, r[2..3] lanes 8..15
// of columns 0..7, r[4..7] the same of columns 8..15; thread l holds lane l / 4, columns 2 (l mod 4) and the next
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
// the reverse for packed operands: 16 lanes x 16 columns, r[2 k], r[2 k + 1] lanes 0..7 and 8..15 of columns 4 k .. 4 k + 3; thread l
// holds lane l / 4, column l mod 4
__device__ __forceinline__ void tmem_st_frag16(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.16x128b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]),
                 "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}

// the same with 8 columns
__device__ __forceinline__ void tmem_st_frag8(uint32_t taddr, const uint32_t (&r)[4]) {
    asm volatile("tcgen05.st.sync.aligned.16x128b.x2.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
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
    // (an offset, so that the compiler goes on to know it as shared memory: 32768 tokens, 32 heads 1052 -> 1038 us for the layer call, 8 x 4096
    // tokens 740 -> 715, 61 packed prompts 482 -> 470)
    uint8_t* smem = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);
    float* gtab = reinterpret_cast<float*>(smem + kOffG);  // (see kTab)

    // Never two pending phases on one barrier for anyone who waits on it: what a barrier's next phase needs, and who has to be past
    // the present one for that, stands at each.
    __shared__ uint64_t bar_kq[kRing], bar_w[2], bar_u[2];  // tiles: loaded again behind a product that every reader precedes (see the loading warp)
    __shared__ uint64_t bar_nrm[4], bar_tab[4];  // norms (eight warps), tables (two warps) of chunk c: again behind hand-off 8 of chunk c + 1
    __shared__ uint64_t bar_pt, bar_o2;  // products: the next one waits for a hand-off that every reader makes behind this one
    __shared__ uint64_t bar_d1[2];  // S0 W^T: the one of chunk c + 2 needs a W tile that is asked for behind this one
    // State update, either half of the state's columns. The chain warps, which alone wait for the first, precede the next one of either. The
    // loading warp waits for the second too, and asks for nothing behind it that chunk c + 2 needs: it may be two chunks late there (three
    // it may not: the W tile of chunk c + 3 is asked for behind it).
    __shared__ uint64_t bar_su0[2], bar_su1[4];
    __shared__ uint64_t bar_ost[2], bar_stg[2];  // output tile staged (eight warps); staging buffer free again
    __shared__ uint64_t bar_end;      // products still in flight when the CTA gives up
    __shared__ uint32_t tmem_base_s;
    __shared__ int s_fail;
    __shared__ int s_seq;

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int t = tid & 127;  // TMEM lane: value feature (state rows, output columns)
    const int h = (tid >> 7) & 1;  // half: 32 of the 64 tokens of a product, 32 of every 64 state columns
    const int wq = warp & 3;
    const int lane = tid & 31;
    const bool aux = warp >= kChain / 32 && warp < kThreads / 32;  // P, the output, the norms
    const bool issuer = warp == kThreads / 32;        // every tcgen05.mma
    const bool producer = warp == kThreads / 32 + 1;  // every TMA load and store
    const bool tabler = warp >= kThreads / 32 + 2;    // gate tables

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bar_w[i], 1);
            mbar_init(&bar_u[i], 1);
            mbar_init(&bar_d1[i], 1);
            mbar_init(&bar_su0[i], 1);
            mbar_init(&bar_ost[i], kAux / 32);
            mbar_init(&bar_stg[i], 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(&bar_su1[i], 1);
            mbar_init(&bar_nrm[i], kAux / 32);
            mbar_init(&bar_tab[i], kTabThreads / 32);
        }
        for (int i = 0; i < kRing; ++i) mbar_init(&bar_kq[i], 1);
        mbar_init(&bar_pt, 1);
        mbar_init(&bar_o2, 1);
        mbar_init(&bar_end, 1);
        s_fail = 0;
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
    grid_dependency_wait();  // (the set-up above runs beside the end of the kernel before; W and U are its output)
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
    const uint32_t smem_a = smem_u32(smem);
    volatile int* fail = reinterpret_cast<volatile int*>(&s_fail);

    // a wait of a whole warp that marks the CTA as failed when it runs out
    auto wait_for = [&](uint64_t* bar, uint32_t parity) -> bool {
        const bool good = wait_bar_warp(bar, parity, fail);
        if (!good) *fail = 1;
        return good;
    };
    // one arrival per warp, behind what all of its lanes have done
    auto warp_arrive = [&](uint64_t* bar) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };

    if (tabler) {
        // ================= table threads, one per token: the gates and factors of chunk c. They wait in hand-off 4 of the chunk, for
        // its tiles too, so they are one chunk ahead at most: behind hand-off 4 of chunk c - 1 the state update of chunk c - 2 is complete,
        // that was issued when the output warps were done with chunk c - 3 (hand-off 8), and nobody reads buffer c mod 4 any more.
        const int tt = tid - (kThreads + 64);
        const bool g_raw = (p.flags & GDN_FLAG_G_RAW) != 0;
        const float* gseq = p.g + grow0;
        auto fetch = [&](int c) -> float { return (c < n_c && (!VAR || c * kC + tt < len)) ? __ldg(gseq + (c * kC + tt) * gstep) : 0.f; };
        auto put_gates = [&](int c, float gc) {
            float* tb = gtab + (c & 3) * kTab;
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
        float g_next = fetch(0);
        for (int c = 0; c < n_c; ++c) {
            const float g_c = g_next;
            g_next = fetch(c + 1);
            put_gates(c, g_c);
            float* tb = gtab + (c & 3) * kTab;
            const float gc = tb[128 + tt], gC = tb[128 + 63];
            float rk = 1.f, so = p.scale;
            if (NRM) {  // (a wait that runs out sets the flag, and the others' waits end by it)
                wait_for(&bar_nrm[c & 3], (c >> 2) & 1);
                rk = (VAR && tt >= len - c * kC) ? 0.f : tb[192 + tt];
                if (!SO) so *= tb[256 + tt];
            }
            tb[tt] = so * fast_exp2(gc * kLog2e);
            tb[256 + tt] = so;
            tb[192 + tt] = rk;
            tb[64 + tt] = rk * fast_exp2((gC - gc) * kLog2e);
            warp_arrive(&bar_tab[c & 3]);
            wait_for(&bar_kq[c % kRing], (c / kRing) & 1);
            wait_for(&bar_w[c & 1], (c >> 1) & 1);
            handoff_wait<4>();
        }
    } else if (producer) {
        // ================= loading / storing warp. W and U of a chunk are asked for when D1 of the chunk two before is complete (its U is
        // in registers by then: the chain warps fetch it before they make the copies that this D1 waits for; that of the first chunk
        // behind its D1), K and Q when the state update of the chunk three before is. And the bulk stores of the staged output tiles.
        const bool lead = elect_one();
        auto load_tile = [&](int off, const CUtensorMap* tm, uint64_t* bar, int x, int c, int z) {
            tma_load_3d(smem + off, tm, bar, x, tok0 + c * kC, z);
            tma_load_3d(smem + off + 8192, tm, bar, x + 64, tok0 + c * kC, z);
        };
        auto load_kq = [&](int c) {
            if (c >= n_c) return;
            uint64_t* bar = &bar_kq[c % kRing];
            mbar_arrive_expect_tx(bar, (SO ? 1 : 2) * kTileBytes);
            load_tile(kOffK + (c % kRing) * kTileBytes, &tmK, bar, kx, c, kz);
            if (!SO) load_tile(kOffQ + (c % kRing) * kTileBytes, &tmQ, bar, kx, c, kz);
        };
        auto load_v = [&](int off, const CUtensorMap* tm, uint64_t* bars, int c) {  // a tile of W or U
            if (c >= n_c) return;
            mbar_arrive_expect_tx(&bars[c & 1], kTileBytes);
            load_tile(off + (c & 1) * kTileBytes, tm, &bars[c & 1], vx, c, vz);
        };
        if (lead) {
            int n_kq = kRing, n_w = 2, n_u = 2;  // chunks whose tiles have been asked for
            for (int c = 0; c < kRing; ++c) {
                load_kq(c);
                if (c < 2) load_v(kOffW, &tmW, bar_w, c);
                if (c < 2) load_v(kOffU, &tmU, bar_u, c);
            }
            for (int c = 0; c < n_c && *fail == 0; ++c) {
                if (c + 2 < n_c) {
                    if (!wait_bar(&bar_d1[c & 1], (c >> 1) & 1)) *fail = 1;
                    if (*fail != 0) break;
                    load_v(kOffW, &tmW, bar_w, n_w++);
                    if (c > 0) load_v(kOffU, &tmU, bar_u, n_u++);
                    if (!wait_bar(&bar_su1[c & 3], (c >> 2) & 1)) *fail = 1;
                    if (*fail != 0) break;
                    if (c == 0) load_v(kOffU, &tmU, bar_u, n_u++);
                    load_kq(n_kq++);
                }
                if (!SO) {
                    if (!wait_bar(&bar_ost[c & 1], (c >> 1) & 1)) *fail = 1;
                    if (*fail != 0) break;
                    if (!(VAR && len - c * kC < kC)) {  // (a short last chunk is stored row by row by the output warps)
                        tma_store_3d(&tmO, smem + kOffO + (c & 1) * kTileBytes, vx, tok0 + c * kC, vz);
                        tma_store_3d(&tmO, smem + kOffO + (c & 1) * kTileBytes + 8192, vx + 64, tok0 + c * kC, vz);
                        tma_store_commit();
                        tma_store_wait_read<0>();
                    }
                    mbar_arrive(&bar_stg[c & 1]);  // the staging buffer may be written again (chunk c + 2)
                }
            }
            tma_store_wait_all<0>();
            if (*fail != 0) {  // loads still in flight land before the CTA leaves
                for (int i = 1; i <= kRing; ++i) {
                    if (n_kq - i >= 0 && n_kq - i < n_c) wait_bar(&bar_kq[(n_kq - i) % kRing], ((n_kq - i) / kRing) & 1);
                    if (i <= 2 && n_w - i < n_c) wait_bar(&bar_w[(n_w - i) & 1], ((n_w - i) >> 1) & 1);
                    if (i <= 2 && n_u - i < n_c) wait_bar(&bar_u[(n_u - i) & 1], ((n_u - i) >> 1) & 1);
                }
            }
        }
        __syncwarp();
    } else if (issuer) {
        // ================= issuing warp: every tcgen05.mma, in the order the tensor pipe runs them. On the chain of the sequence are
        // D1 and the state update; P^T and O1 run while U_new is formed, O2 while the state is copied.
        const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem, 0);  // (a uniform register: every operand address of a product derives from it)
        const uint32_t idesc_kk64 = instr_desc(128, 64, 1, 1, 0, 0, 1);   // B K-major (a TMA tile as [N x K])
        const uint32_t idesc_mn64 = instr_desc(128, 64, 1, 1, 0, 1, 1);   // B MN-major
        const uint32_t idesc_pt = instr_desc(64, 64, 1, 1, 0, 0, 1);
        const uint64_t desc_p = smem_desc(smem_a + kOffP, 128, 1024, SWZ_NONE);
        for (int c = 0; c < n_c; ++c) {
            // descriptors of the tiles; a step inside a tile adds its bytes / 16
            const uint64_t desc_w = smem_desc(smem_a + kOffW + (c & 1) * kTileBytes, 16, 1024, SWZ_128B);
            const uint64_t desc_k = smem_desc(smem_a + kOffK + (c % kRing) * kTileBytes, 16, 1024, SWZ_128B), desc_q = desc_k + (kOffQ - kOffK) / 16;
            const uint64_t desc_kt = smem_desc(smem_a + kOffK + (c % kRing) * kTileBytes, 8192, 1024, SWZ_128B);
            // D1 = (S0_hi + S0_lo) W^T, the first half of the state's columns as soon as its copies are in place
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                if (half == 0) handoff_wait<4>();
                else handoff_wait<6>();
                tc_fence_after_sync();
                if (*fail == 0 && elect_one()) {
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4)
                            mma_f16_ts(tm + kD1, tm + (part == 0 ? kSA : kSL) + half * 32 + k4 * 8, desc_w + (half * 8192 + k4 * 32) / 16,
                                       part == 0 ? idesc_kk64 : idesc_kk64 | kNegA, half > 0 || part > 0 || k4 > 0);
                    }
                    if (half == 1) mma_commit(&bar_d1[c & 1]);
                }
                __syncwarp();
            }
            if (!SO) {
                if (c > 0) handoff_wait<8>();  // the output warps have read O1, O2 of the chunk before
                tc_fence_after_sync();
                if (*fail == 0 && elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        mma_f16_ss(tm + kPT, desc_k + ((ks >> 2) * 8192 + (ks & 3) * 32) / 16, desc_q + ((ks >> 2) * 8192 + (ks & 3) * 32) / 16,
                                   idesc_pt, ks > 0);
                    mma_commit(&bar_pt);
                    // O1 = (S0_hi + S0_lo) Q^T (no completion barrier of its own: the commit behind the output product covers it)
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            mma_f16_ts(tm + kO1, tm + (part == 0 ? kSA : kSL) + ks * 8, desc_q + ((ks >> 2) * 8192 + (ks & 3) * 32) / 16,
                                       part == 0 ? idesc_kk64 : idesc_kk64 | kNegA, part > 0 || ks > 0);
                    }
                }
                __syncwarp();
            }
            // the forms of U_new^T and the decayed accumulator are in place: S += (U_new^T exp(g_C - g_j)) K, hi + lo (the K tile as
            // MN-major operand), one half of the state's columns after the other
            handoff_wait<5>();
            tc_fence_after_sync();
            if (*fail == 0 && elect_one()) {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_f16_ts(tm + kSD + half * 64, tm + (part == 0 ? kD1 : kUL) + ks * 16 + 8, desc_kt + (half * 8192 + ks * 2048) / 16,
                                       part == 0 ? idesc_mn64 : idesc_mn64 | kNegA, true);
                    }
                    mma_commit(half == 0 ? &bar_su0[c & 1] : &bar_su1[c & 3]);
                }
            }
            __syncwarp();
            if (!SO) {
                // O2 = U_new^T P^T = Uh Ph + Ul Ph + Uh Pl (K-dim = 64 tokens; the plain copy of tokens 16 ks.. sits
                // at columns 16 ks .. 16 ks + 7 of its region, the gate-scaled one at 16 ks + 8 ..)
                handoff_wait<7>();
                tc_fence_after_sync();
                if (*fail == 0 && elect_one()) {
#pragma unroll
                    for (int part = 0; part < 3; ++part) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_f16_ts(tm + kO2, tm + (part == 1 ? kUL : kD1) + ks * 16, desc_p + ((part == 2 ? 8192 : 0) + ks * 256) / 16,
                                       part == 0 ? idesc_mn64 : part == 1 ? idesc_mn64 | kNegA : idesc_mn64 | kNegB, part > 0 || ks > 0);
                    }
                    mma_commit(&bar_o2);
                }
                __syncwarp();
            }
        }
        if (*fail != 0 && elect_one()) {  // products still in flight end before their operands go
            mma_commit(&bar_end);
            wait_bar(&bar_end, 0);
        }
        __syncwarp();
    } else if (aux) {
        // ================= output warps (eight, two per lane quadrant): P, the output tile and the norms, beside the chain of the state
        // 1 / ||k||, 1 / ||q|| of chunk c into its table buffer: four warps the rows of K, four those of Q, two threads a row. (The sum does
        // not care about the swizzle inside the row: eight neighbouring threads read eight different 16-byte pieces, free of bank
        // conflicts.) Two chunks ahead: the table threads and the chain want them before this chunk is done, and here is where warps wait.
        auto put_norms = [&](int c) -> bool {
            if (!NRM || c >= n_c) return true;
            if (SO && warp >= (kChain + kAux / 2) / 32) {  // (no queries)
                warp_arrive(&bar_nrm[c & 3]);
                return true;
            }
            if (!wait_for(&bar_kq[c % kRing], (c / kRing) & 1)) return false;
            const int at = tid - kChain, r = (at >> 1) & 63, half = at & 1;
            const uint8_t* rp = smem + (at < kAux / 2 ? kOffK : kOffQ) + (c % kRing) * kTileBytes + half * 8192 + r * 128;
            float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint4 w4 = *reinterpret_cast<const uint4*>(rp + (((i + lane) & 7) << 4));
                bf16_square_add(w4.x, a[0], a[1]);
                bf16_square_add(w4.y, a[2], a[3]);
                bf16_square_add(w4.z, a[0], a[1]);
                bf16_square_add(w4.w, a[2], a[3]);
            }
            float sum = (a[0] + a[1]) + (a[2] + a[3]);
            sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 1);
            if (half == 0) gtab[(c & 3) * kTab + (at < kAux / 2 ? 192 : 256) + r] = rsqrtf(fmaxf(sum, 1e-30f));
            warp_arrive(&bar_nrm[c & 3]);
            return true;
        };
        int taken = 0;  // hand-offs this warp has made (7, 8 of a chunk, in this order; no 8 for the last)
        bool good = put_norms(0);
        if (SO) {  // the norms only: of chunk c when the table of chunk c - 2 has been formed, which is behind the last reader of buffer c mod 4
            for (int c = 1; good && NRM && c < n_c; ++c) {
                good = (c < 2 || wait_for(&bar_tab[(c - 2) & 3], ((c - 2) >> 2) & 1)) && put_norms(c);
            }
        } else {  // P is zero above its diagonal: the blocks that no thread writes below
            uint4* pz = reinterpret_cast<uint4*>(smem + kOffP);
#pragma unroll
            for (int i = 0; i < 4; ++i) pz[i * kAux + tid - kChain] = make_uint4(0u, 0u, 0u, 0u);
            asm volatile("bar.sync 1, %0;" ::"n"(kAux) : "memory");
        }
        for (int c = 0; good && c < (SO ? 0 : n_c); ++c) {
            const float* se = gtab + (c & 3) * kTab;  // scale exp(g_i) / ||q_i||
            const float* sg = se + 128;              // g_i (cumulative inside the chunk)
            const int left = len - c * kC;
            // ---- P_ij = exp(g_i - g_j) PT_ji for j <= i (hi + lo): this thread's token j and 16 or 8 columns i. (Keys and
            // queries normalised here: 1 / ||k_j|| rides on P and on the scaled form of U_new_j, 1 / ||q_i|| on the output.)
            if (!(good = wait_for(&bar_pt, c & 1))) break;  // (issued behind hand-off 4: the tables are there too)
            tc_fence_after_sync();
            const int j = wq * 16 + (lane & 15);
            const float gj = sg[j] * kLog2e, rk = NRM ? sg[64 + j] : 1.f;
            auto put_p = [&](const uint32_t* d, int i0) {  // columns i0 .. i0 + 7 of this thread's row j
                float gi[8];
#pragma unroll
                for (int i4 = 0; i4 < 2; ++i4) {
                    const float4 q4 = *reinterpret_cast<const float4*>(sg + i0 + i4 * 4);
                    gi[i4 * 4 + 0] = q4.x; gi[i4 * 4 + 1] = q4.y; gi[i4 * 4 + 2] = q4.z; gi[i4 * 4 + 3] = q4.w;
                }
                uint32_t w[4], wl[4];
#pragma unroll
                for (int i2 = 0; i2 < 4; ++i2) {
                    float v[2];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        float x = __uint_as_float(d[i2 * 2 + q]) * fast_exp2(fminf(fmaf(gi[i2 * 2 + q], kLog2e, -gj), 0.f));
                        if (NRM) x *= rk;
                        v[q] = (j <= i0 + i2 * 2 + q) ? x : 0.f;
                    }
                    split_neg(v[0], v[1], w[i2], wl[i2]);
                }
                // B operand [K-dim = j][N = i], MN-major, no swizzle: the 16-byte piece of row j for a group of 8 columns
                uint8_t* at = smem + kOffP + (i0 >> 3) * 1024 + j * 16;
                *reinterpret_cast<uint4*>(at) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4*>(at + 8192) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
            };
            if (wq < 2) {
                uint32_t d[16];
                tmem_ld16_split32(lane_base + kPT + h * 16, d);
                tmem_wait_ld();
                put_p(d, (lane >> 4) * 32 + h * 16);
                put_p(d + 8, (lane >> 4) * 32 + h * 16 + 8);
            } else if (wq == 2 || h == 1) {  // rows j from 32 on: columns from 32 on, rows from 48 on: columns from 48 on; zeros elsewhere stay as written once
                uint32_t d[8];
                tmem_ld8_split8(lane_base + kPT + 32 + h * 16, d);
                tmem_wait_ld();
                put_p(d, 32 + h * 16 + (lane >> 4) * 8);
            }
            fence_proxy_async_smem();
            tc_fence_before_sync();
            handoff_arrive<7>();
            ++taken;
            if (c == 0 && !(good = put_norms(1))) break;
            if (!(good = put_norms(c + 2))) break;
            // ---- O^T = scale (exp(g_i) O1 + O2), in fragments of 8 x 8: this warp's 32 features x 32 tokens, transposed
            // on the way to the staged tile (O1 is complete with O2: products finish in the order they were issued)
            if (!(good = wait_for(&bar_o2, c & 1))) break;
            tc_fence_after_sync();
            uint32_t m[2][2][4];
#pragma unroll
            for (int tg = 0; tg < 2; ++tg) {
                uint32_t a[2][8], d[2][8];
#pragma unroll
                for (int lh = 0; lh < 2; ++lh) {
                    tmem_ld_frag(lane_base + (static_cast<uint32_t>(lh * 16) << 16) + kO1 + h * 32 + tg * 16, a[lh]);
                    tmem_ld_frag(lane_base + (static_cast<uint32_t>(lh * 16) << 16) + kO2 + h * 32 + tg * 16, d[lh]);
                }
                const int t2 = h * 32 + tg * 16 + 2 * (lane & 3);
                const f2 e[2] = {*reinterpret_cast<const f2*>(se + t2), *reinterpret_cast<const f2*>(se + t2 + 8)};
                const f2 q[2] = {*reinterpret_cast<const f2*>(se + 256 + t2), *reinterpret_cast<const f2*>(se + 256 + t2 + 8)};  // scale / ||q_i||
                tmem_wait_ld();
#pragma unroll
                for (int lh = 0; lh < 2; ++lh) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const f2 o1 = pair2(__uint_as_float(a[lh][2 * k]), __uint_as_float(a[lh][2 * k + 1]));
                        const f2 o2 = pair2(__uint_as_float(d[lh][2 * k]), __uint_as_float(d[lh][2 * k + 1]));
                        m[tg][lh][k] = pack_pair(fma2(o1, e[k >> 1], mul2(o2, q[k >> 1])));
                    }
                }
            }
            tc_fence_before_sync();
            if (c + 1 < n_c) {  // the columns and the tables of this chunk are read
                handoff_arrive<8>();
                ++taken;
            }
            if (c >= 2 && !(good = wait_for(&bar_stg[c & 1], ((c - 2) >> 1) & 1))) break;
#pragma unroll
            for (int tg = 0; tg < 2; ++tg) {
                const int tok = h * 32 + tg * 16 + ((lane >> 4) << 3) + (lane & 7);  // row of the staged tile this lane addresses
#pragma unroll
                for (int lh = 0; lh < 2; ++lh) {
                    const int fb = wq * 4 + lh * 2 + ((lane >> 3) & 1);  // block of 8 features
                    const uint32_t at = smem_a + kOffO + (c & 1) * kTileBytes + (fb >> 3) * 8192 + tok * 128 + (((fb & 7) ^ (tok & 7)) << 4);
                    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(m[tg][lh][0]),
                                 "r"(m[tg][lh][1]), "r"(m[tg][lh][2]), "r"(m[tg][lh][3])
                                 : "memory");
                }
            }
            if (VAR && left < kC) {
                // only the rows of real tokens leave, from the staged (swizzled) tile: every warp its own 32 tokens x 64 bytes
                __syncwarp();
#pragma unroll
                for (int q = lane; q < 128; q += 32) {
                    const int tok = h * 32 + (q >> 2), ch = wq * 4 + (q & 3);  // 16-byte piece ch of the token's 256-byte row
                    if (tok < left) {
                        const uint4 v = *reinterpret_cast<const uint4*>(smem + kOffO + (c & 1) * kTileBytes + (ch >> 3) * 8192 +
                                                                        tok * 128 + (((ch & 7) ^ (tok & 7)) << 4));
                        *reinterpret_cast<uint4*>(p.O + (grow0 + (long long)(c * kC + tok) * gstep) * kD + ch * 8) = v;
                    }
                }
            }
            // the tile goes to the storing warp
            fence_proxy_async_smem();
            warp_arrive(&bar_ost[c & 1]);
        }
        if (!SO && !good) {  // a bounded wait ran out (s_fail is set): the remaining hand-offs, as waits
            for (; taken < 2 * n_c - 1; ++taken) {
                if ((taken & 1) == 0) handoff_wait<7>();
                else handoff_wait<8>();
            }
        }
    } else {
        // ================= chain warps (eight, two per lane quadrant): the state's copies, its decay, U_new
        const uint32_t row = lane_base;
        const int tq = h * 32 + 2 * (lane & 3);  // this thread's tokens: tq + 8 k and the next one
        // What U_new of a chunk needs beside D1: U in the fragments in which D1 is read (tokens tq + 16 ks + 8 x and the next one of
        // feature lane / 4 of each block of 8), the tokens' factors exp(g_C - g_j) / ||k_j||, and the decay exp(g_C) of the state. Fetched
        // while the state update of the chunk before runs: behind D1 the products read shared memory at up to its full rate.
        uint32_t u[2][2][4];
        f2 f[2][2], dec2;
        auto prefetch = [&](int c) -> bool {
            if (!(wait_for(&bar_tab[c & 3], (c >> 2) & 1) && wait_for(&bar_u[c & 1], (c >> 1) & 1))) return false;
            const float* sf = gtab + (c & 3) * kTab + 64;
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
#pragma unroll
                for (int lh = 0; lh < 2; ++lh) {
                    const int tok = h * 32 + 16 * ks + ((lane >> 4) << 3) + (lane & 7), fb = wq * 4 + lh * 2 + ((lane >> 3) & 1);
                    const uint32_t at = smem_a + kOffU + (c & 1) * kTileBytes + (fb >> 3) * 8192 + tok * 128 + (((fb & 7) ^ (tok & 7)) << 4);
                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(u[ks][lh][0]), "=r"(u[ks][lh][1]), "=r"(u[ks][lh][2]), "=r"(u[ks][lh][3])
                                 : "r"(at)
                                 : "memory");
                }
#pragma unroll
                for (int x = 0; x < 2; ++x) f[ks][x] = *reinterpret_cast<const f2*>(sf + tq + 16 * ks + 8 * x);
            }
            const float dec = fast_exp2(sf[64 + 63] * kLog2e);
            dec2 = pair2(dec, dec);
            return true;
        };
        // bf16 copies (hi, -lo) of 32 state columns
        auto put_copies = [&](const uint32_t (&v)[32], int half) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t hi[8], lo[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) split_neg(__uint_as_float(v[16 * q + 2 * i]), __uint_as_float(v[16 * q + 2 * i + 1]), hi[i], lo[i]);
                tmem_st8(row + kSA + half * 32 + h * 16 + q * 8, hi);
                tmem_st8(row + kSL + half * 32 + h * 16 + q * 8, lo);
            }
            tmem_wait_st();
            tc_fence_before_sync();
        };
        // the accumulator for the coming chunk, S <- exp(g_C) S0 (its products read the bf16 copies)
        auto put_decayed = [&](uint32_t (&v)[32], int half) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const f2 x = mul2(pair2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), dec2);
                v[2 * i] = static_cast<uint32_t>(x);
                v[2 * i + 1] = static_cast<uint32_t>(x >> 32);
            }
            tmem_st32(row + kSD + half * 64 + h * 32, v);
        };
        int taken = 0;  // hand-offs this warp has made (4, 6, 5 of a chunk, in this order)
        bool good = true;
        {
            // this thread's part of state row t: columns [64 half + 32 h, + 32)
            const float* s0 = (p.S_in != nullptr) ? p.S_in + (((long long)b * p.H_v + hv) * kD + t) * kD + h * 32 : nullptr;
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                uint32_t v[32];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 x = (s0 != nullptr) ? __ldg(reinterpret_cast<const float4*>(s0 + half * 64) + i) : make_float4(0.f, 0.f, 0.f, 0.f);
                    v[4 * i] = __float_as_uint(x.x); v[4 * i + 1] = __float_as_uint(x.y);
                    v[4 * i + 2] = __float_as_uint(x.z); v[4 * i + 3] = __float_as_uint(x.w);
                }
                tmem_st32(row + kSD + half * 64 + h * 32, v);
                if (n_c == 0) continue;  // no tokens: the state is handed on
                put_copies(v, half);
                if (half == 0) handoff_arrive<4>();
                else handoff_arrive<6>();
                ++taken;
            }
            tmem_wait_st();
            if (n_c > 0 && (good = prefetch(0))) {
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    uint32_t v[32];
                    tmem_ld32(row + kSD + half * 64 + h * 32, v);
                    tmem_wait_ld();
                    put_decayed(v, half);
                }
            }
        }
        for (int c = 0; good && c < n_c; ++c) {
            const int left = len - c * kC;
            const bool short_chunk = VAR && left < kC;
            // ---- U_new^T = U^T - D1 as bf16 hi - lo, plain and gate-scaled (the sums over the tokens of a chunk telescope
            // on correlated keys, so single bf16 copies cost 1e-2 there). 16 tokens are one k-step of the
            // products that consume them: the hi halves are written over their own D1 columns (plain -> 16 ks .. 16 ks + 7,
            // scaled -> 16 ks + 8 ..), the lo halves at the same offsets of a region of their own.
            if (!(good = wait_for(&bar_d1[c & 1], (c >> 1) & 1))) break;
            tc_fence_after_sync();
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
                uint32_t d[2][8];
#pragma unroll
                for (int lh = 0; lh < 2; ++lh) tmem_ld_frag(row + (static_cast<uint32_t>(lh * 16) << 16) + kD1 + h * 32 + ks * 16, d[lh]);
                tmem_wait_ld();
#pragma unroll
                for (int lh = 0; lh < 2; ++lh) {
                    uint32_t hi[8], lo[8], shi[4], slo[4];  // (state only: the scaled form alone, the output product reads the plain one)
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
#pragma unroll
                        for (int fb = 0; fb < 2; ++fb) {
                            const uint32_t w = (SO && no_u) ? 0u : u[ks][lh][2 * x + fb];
                            float u0 = bf16_minus<0>(w, __uint_as_float(d[lh][4 * x + 2 * fb]));
                            float u1 = bf16_minus<1>(w, __uint_as_float(d[lh][4 * x + 2 * fb + 1]));
                            if (short_chunk) {  // rows past the sequence's end hold another sequence's W, U
                                if (tq + 16 * ks + 8 * x >= left) u0 = 0.f;
                                if (tq + 16 * ks + 8 * x + 1 >= left) u1 = 0.f;
                            }
                            if (SO) {
                                split_neg(mul2(pair2(u0, u1), f[ks][x]), shi[2 * x + fb], slo[2 * x + fb]);
                            } else {
                                split_neg(mul2(pair2(u0, u1), f[ks][x]), hi[4 + 2 * x + fb], lo[4 + 2 * x + fb]);
                                split_neg(u0, u1, hi[2 * x + fb], lo[2 * x + fb]);
                            }
                        }
                    }
                    const uint32_t at = row + (static_cast<uint32_t>(lh * 16) << 16) + h * 32 + ks * 16;
                    if (SO) {
                        tmem_st_frag8(at + kD1 + 8, shi);
                        tmem_st_frag8(at + kUL + 8, slo);
                    } else {
                        tmem_st_frag16(at + kD1, hi);
                        tmem_st_frag16(at + kUL, lo);
                    }
                }
            }
            tmem_wait_st();
            tc_fence_before_sync();
            handoff_arrive<5>();
            ++taken;
            if (c + 1 < n_c) {
                if (!(good = prefetch(c + 1))) break;
                // ---- bf16 copies (hi, -lo) of the new state for the next chunk's products, and its decay
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    if (!(good = half == 0 ? wait_for(&bar_su0[c & 1], (c >> 1) & 1) : wait_for(&bar_su1[c & 3], (c >> 2) & 1))) break;
                    tc_fence_after_sync();
                    uint32_t v[32];
                    tmem_ld32(row + kSD + half * 64 + h * 32, v);
                    tmem_wait_ld();
                    put_copies(v, half);
                    if (half == 0) handoff_arrive<4>();
                    else handoff_arrive<6>();
                    ++taken;
                    put_decayed(v, half);
                }
                if (!good) break;
            } else {
                good = wait_for(&bar_su1[c & 3], (c >> 2) & 1);
                tc_fence_after_sync();
            }
        }
        if (!good) {
            // A bounded wait ran out (s_fail is set): this warp's remaining hand-offs, as waits, so that no generation counts it twice.
            for (; taken < 3 * n_c; ++taken) {
                if (taken % 3 == 0) handoff_wait<4>();
                else if (taken % 3 == 1) handoff_wait<6>();
                else handoff_wait<5>();
            }
        }
        // ---- final state
        // (the run's place among the states is formed again here: it is not held over the chunks)
        const int seq = ORD ? *reinterpret_cast<volatile int*>(&s_seq) : static_cast<int>(blockIdx.x / p.H_v);
        if (good && p.S_out != nullptr && seq >= p.out_from) {
            float* so = p.S_out + (((long long)(seq - p.out_from) * p.H_v + blockIdx.x % p.H_v) * kD + t) * kD + h * 32;
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                uint32_t v[32];
                tmem_ld32(row + kSD + half * 64 + h * 32, v);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    *reinterpret_cast<float4*>(so + half * 64 + i * 4) =
                        make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]), __uint_as_float(v[4 * i + 2]),
                                    __uint_as_float(v[4 * i + 3]));
            }
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
    return P == 2 ? 1 : P;  // (two never pay: 64 heads x 256 chunks 512 us, 464 as one run each; a state-only chunk costs 0.85 of one with output)
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
    if (!launch_behind(kern, dim3(static_cast<unsigned>(n_cta)), kThreads + 64 + kTabThreads, smem, stream, mQ, mK, mW, mU, mO, prm)) return GDN_ERR_LAUNCH;
    count_launch();
    return GDN_OK;
}

}  // namespace gdn
