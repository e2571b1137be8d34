// Tensor-core kernel (tcgen05 + TMEM + TMA) for the bf16 chunk-prepare path.
//
// Work item = one tile of 128 consecutive tokens of one (batch, value head): 128 / C chunks, which sit as diagonal
// blocks of every 128 x 128 operand (chunks are independent, so the tile's matrices are block diagonal). Threads t and
// t + 128 share row t of the tile (TMEM lane t) and split its chunk columns; one elected lane of warp 0 issues the TMA
// loads and every tcgen05.mma. Two CTAs per SM, persistent over the tiles.
//
// Per tile (paper's notation, Abar = -A, Sec. 3 / Alg. 1):
//   G = K K^T                         tcgen05.mma, K tile staged by TMA (128B swizzle)      -> TMEM
//   Abar_ij = -beta_i e^{g_i-g_j} G_ij (i > j)                                  registers, fp32
//   L = T0 - I = band_{1<=i-j<=N}(sum_n Abar^n)  (Eq. 7, 10, 11), by the distance recursion
//       L_d[i] = Abar[i,i-d] + sum_{e<d} Abar[i,i-e] L_{d-e}[i-e], which equals the masked sum exactly
//   E = Abar + Abar L  on i-j > N, exactly 0 inside the band (Eq. 13)               registers, fp32
//   residual sum (Eq. 13): Z_0 = 0, Z_{k+1} = (T0 + Z_k) E, k < S, so that T = T0 + Z_S; chunks stacked along M,
//       A operand = bf16(T0 + Z_k) in TMEM, B operand = E in shared memory. For S = 8 and S = 15 at C = 64 the same
//       sum by four doubling levels (X_{2m+1} = X_m + X_m E^{m+1}), see the kernel body.
//   T = I + L + Z_S  -> Tinv
//   W = (T diag(beta)) K, U = (T diag(beta)) V: T diag(beta) as hi + lo bf16 A operands (lo on band and diagonal),
//       the K / V tile itself as MN-major B operand
//   C = 128: the two 64-blocks as above, then the block formula of App. E for the lower-left block (hi + lo operands).
// The identity and the O(1) band never pass through a single bf16 operand, which keeps the result within bf16 output
// rounding of the fp64 definition even for strongly correlated keys.
//
// The forward-substitution comparisons (Eq. 2-3; App. E for the blocked form) replace the L / E / residual steps by a
// column-parallel substitution in shared memory and reuse everything else.
#include <cuda.h>
#include <cstdlib>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace gdn {
namespace {

using namespace sm100;

constexpr int kTile = 128;            // rows per work item
constexpr int kThreads = 256;            // two threads per tile row
constexpr int kD = 128;               // d_k = d_v
constexpr float kLog2e = 1.4426950408889634f;

// TMEM column map (256 columns allocated):
//   R0..R1 (128 columns)  Gram matrix, then the accumulator of the residual rounds, of W and of U
//   R2     (64 columns)   low-half bf16 A operand of W/U (block diagonal)
//   AS     (64 columns)   bf16 A operand of the residual rounds (chunks stacked along M) and of W/U
//                         (high half, block diagonal)
constexpr uint32_t kR0 = 0, kR2 = 128, kAS = 192, kTmemCols = 256;


// (New fields go at the END: the struct's layout decides which parameters ptxas fetches with one wide load, and a
// field inserted in the middle moved the default instantiation from 36 to 96 bytes of spill, 10 % of its speed.)
struct Params {
    const float* beta;
    const float* g;
    __nv_bfloat16* W;
    __nv_bfloat16* U;
    __nv_bfloat16* Tinv;
    int* status;
    int H_k, H_v, T, group, n_tt;  // n_tt: tiles per head
    int N, S;
    unsigned flags;  // GDN_FLAG_*
    long long n_tiles;
    // packed variable-length sequences (EX instantiations only, B = 1): first token and length of every chunk; T is
    // then the padded token count n_tt * 128 and T_total the real one
    const int* chunk_start;
    const int* chunk_len;
    int n_chunks, T_total;
    int s_gi, s_tt, s_bhk;  // the grid size as a step in (value head of the group, token tile, key-head row) digits
    int n_mid;  // EX instantiations: range of the middle digit of the tile walk, n_tt (head-major tensors) or H_k (token-major)
};

template <int C, int NB>
struct Smem {
    static constexpr int kK = 0;                        // 32 KB, two [128][64] bf16 sub-tiles, 128B swizzle
    static constexpr int kV = 32768;                    // 32 KB
    // scratch: [EB | BR]. EB = E as the B operand of the residual rounds (128 x C bf16, core-matrix
    // layout); BR = one private packed-bf16 row per thread. Before EB/BR are in use the whole region
    // holds one private fp32 row per thread (Abar row, or the forward-substitution matrix).
    static constexpr int kEB = 65536;
    static constexpr int kEBBytes = kTile * C * 2;
    static constexpr int kBR = kEB + kEBBytes;
    static constexpr int NBP = (NB <= 3) ? 4 : 8;
    static constexpr int kScratchBytes = 32768;         // >= kEBBytes + kTile * C * 2 (BR); also the 4 x 8 KB store staging slices
    static constexpr int kSH = kEB + kScratchBytes;     // column form of the band: [128 + 8][NBP] floats
    static constexpr int kSHBytes = (kTile + 8) * NBP * 4;
    static constexpr int kRB = kSH + kSHBytes;          // row form of the band: [128][NBP] floats
    static constexpr int kRBBytes = kTile * NBP * 4;
    static constexpr int kBeta = kRB + kRBBytes;        // 128 floats
    static constexpr int kG = kBeta + 512;              // 128 floats
    static constexpr int kRn = kG + 512;                // 128 floats: 1 / ||K_row|| (GDN_FLAG_K_L2NORM)
    static constexpr int kBRn = kRn + 512;              // 128 floats: beta / ||K_row||
    static constexpr int kWt = kBRn + 512;              // 4 floats: warp totals of the gate prefix sum (GDN_FLAG_G_RAW)
    static constexpr int kDummy = kWt + 64;             // one word per thread: target of band entries a thread does not own
    static constexpr int kTotal = kDummy + kThreads * 4;
};

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void compute_barrier() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// bounded mbarrier wait: polls, and every 1024 polls compares the clock with a budget of about a second
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    uint32_t i = 0;
    while (!mbar_try_wait_hint(bar, parity, 2000u)) {
        if ((++i & 63u) == 0 && clock64() - t0 > 2000000000LL) return false;
    }
    return true;
}

// ---- private shared-memory rows (each thread touches only its own row; inline asm keeps the order)
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void sts16(uint32_t addr, uint16_t v) {
    asm volatile("st.shared.b16 [%0], %1;" ::"r"(addr), "h"(v) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float4 lds128f(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float lds32f(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
// 16-byte chunk index after the bank swizzle, for rows of CPR chunks
template <int CPR>
__device__ __forceinline__ int swz(int t, int c) {
    if constexpr (CPR >= 8) return c ^ (t & 7);
    else if constexpr (CPR == 4) return c ^ ((t >> 1) & 3);
    else if constexpr (CPR == 2) return c ^ ((t >> 2) & 1);
    else return c;
}

// Column split: for C >= 32 two threads share a tile row, thread half h owns the chunk-local columns
// [h * C/2, (h+1) * C/2); for C = 16 only the h = 0 thread works on the row (h = 1 joins for W/U).
template <int C>
struct Split {
    static constexpr bool kSplit = (C >= 32);
    static constexpr int HC = kSplit ? C / 2 : C;  // columns per thread
    static constexpr int PCH = HC / 2;             // packed bf16x2 words per thread
};

// Packed bf16 rows that are zero except for the band (vals[e] at column il - e) are assembled through a private
// shared-memory line per thread: registers cannot be indexed by a per-thread position, shared memory can.
// The line of tile row t is stored chunk-major (16-byte chunk c of row t at c * 2048 + t * 16), so a warp's
// accesses fall on consecutive addresses; the two halves of a row own disjoint chunks. Where column il - e lies
// does not change from tile to tile: band_slots() computes the byte address of each band entry once per thread
// (entries outside the thread's columns or beyond the band width point at a per-thread dummy word).
template <int C, int NB>
__device__ __forceinline__ void band_slots(uint32_t br_base, uint32_t dummy, int t, int il, int col0, int n_valid,
                                           uint32_t (&slot)[NB + 1]) {
#pragma unroll
    for (int e = 0; e <= NB; ++e) {
        const int j = il - e;
        const bool in = (j >= col0 && j < col0 + Split<C>::HC && e <= n_valid);
        slot[e] = in ? br_base + (j >> 3) * (kTile * 16) + t * 16 + (j & 7) * 2 : dummy;
    }
}
// line = address of the thread's first chunk (br_base + (col0 / 8) * 2048 + t * 16)
template <int C, int NB>
__device__ __forceinline__ void build_band_row(uint32_t line, const uint32_t (&slot)[NB + 1], const uint16_t (&vals)[NB + 1],
                                               uint32_t (&out)[Split<C>::PCH]) {
    constexpr int CPT = Split<C>::HC / 8;  // chunks owned by this thread
#pragma unroll
    for (int c = 0; c < CPT; ++c) sts128(line + c * (kTile * 16), 0u, 0u, 0u, 0u);
#pragma unroll
    for (int e = 0; e <= NB; ++e) sts16(slot[e], vals[e]);
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        const uint4 v = lds128(line + c * (kTile * 16));
        out[c * 4 + 0] = v.x;
        out[c * 4 + 1] = v.y;
        out[c * 4 + 2] = v.z;
        out[c * 4 + 3] = v.w;
    }
}

__device__ __forceinline__ uint16_t bf16_bits(float x) { return __bfloat16_as_ushort(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float bf16_bits_to_f32(uint16_t b) { return __uint_as_float(static_cast<uint32_t>(b) << 16); }

// Writes the thread's packed bf16 part of its row's diagonal block into a 64-column A-operand slot
// (block of row t: columns [cb/2, cb/2 + C/2)). tcgen05.st takes one address per warp; for C = 16 a warp
// holds two chunks, so the warp stores a 16-column window in which each half-warp fills its own half
// and zero-fills the other. FULL: the h = 0 thread also zero-fills the columns outside the block.
template <int C, bool FULL>
__device__ __forceinline__ void store_a_operand(uint32_t slot_addr, int t, int h, const uint32_t (&pk)[Split<C>::PCH]) {
    if constexpr (C == 64) {
        const int cb = t & 64;
        uint32_t r16[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) r16[i] = pk[i];
        tmem_st16(slot_addr + cb / 2 + h * 16, r16);
        if (FULL && h == 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i) r16[i] = 0u;
            tmem_st16(slot_addr + (32 - cb / 2), r16);
            tmem_st16(slot_addr + (32 - cb / 2) + 16, r16);
        }
    } else if constexpr (C == 32) {
        const int cb = t & 96;
        uint32_t r8[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) r8[i] = pk[i];
        tmem_st8(slot_addr + cb / 2 + h * 8, r8);
        if (FULL && h == 0) {
            uint32_t z[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) z[i] = 0u;
#pragma unroll
            for (int g = 1; g < 4; ++g) tmem_st16(slot_addr + ((cb / 2 + g * 16) & 63), z);
        }
    } else {
        if (h == 0) {
            const int wb = t & ~31;
            const bool upper = (t & 16) != 0;
            uint32_t r16[16];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                r16[i] = upper ? 0u : pk[i];
                r16[8 + i] = upper ? pk[i] : 0u;
            }
            tmem_st16(slot_addr + wb / 2, r16);
            if (FULL) {
#pragma unroll
                for (int i = 0; i < 16; ++i) r16[i] = 0u;
#pragma unroll
                for (int g = 1; g < 4; ++g) tmem_st16(slot_addr + ((wb / 2 + g * 16) & 63), r16);
            }
        }
    }
}

// Writes the thread's packed bf16 part of its row at its chunk-local position (columns [col0/2, col0/2 + PCH)
// of the slot): the A operand of the residual rounds, where the chunks of a tile are stacked along M.
template <int C>
__device__ __forceinline__ void store_stacked_operand(uint32_t slot_addr, int h, const uint32_t (&pk)[Split<C>::PCH]) {
    if constexpr (C == 64) {
        uint32_t r16[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) r16[i] = pk[i];
        tmem_st16(slot_addr + h * 16, r16);
    } else {
        uint32_t r8[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) r8[i] = pk[i];
        tmem_st8(slot_addr + ((C == 32) ? h * 8 : 0), r8);
    }
}

// Reads the thread's columns of its row's diagonal block of a 128-column accumulator (the Gram matrix).
template <int C>
__device__ __forceinline__ void load_diag_block(uint32_t lane_base, uint32_t col0, int t, int h, float (&a)[Split<C>::HC]) {
    if constexpr (C == 64) {
        uint32_t r[32];
        tmem_ld32(lane_base + col0 + (t & 64) + h * 32, r);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; ++i) a[i] = __uint_as_float(r[i]);
    } else if constexpr (C == 32) {
        uint32_t r[16];
        tmem_ld16(lane_base + col0 + (t & 96) + h * 16, r);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) a[i] = __uint_as_float(r[i]);
    } else {
        const int wb = t & ~31;
        const bool upper = (t & 16) != 0;
        uint32_t r[32];
        tmem_ld32(lane_base + col0 + wb, r);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) a[i] = __uint_as_float(upper ? r[16 + i] : r[i]);
    }
}

// Builds the two bf16 A operands of the W/U products for this thread's part of its row and stores them to TMEM:
// hi (slot AS) = bf16(T diag(scale)) over the whole row, lo (slot R2) = bf16 of what hi loses on the diagonal and
// the band, where entries are O(1). `sc` is the per-token scale in shared memory, `sc_i` the row's own scale;
// a[] = far part of the row, lb[] = band, y[] = T21 part (second block of a 128-chunk).
template <int C, int NB, bool MERGE, bool YPART = MERGE, bool KEEP = true, bool PERM = false>
__device__ __forceinline__ void build_wu_operands(uint32_t lane_base, uint32_t br_line, const uint32_t (&slot)[NB + 1], int t, int h,
                                                  int il, int cb, int col0, int wq, const float* sc, float sc_i,
                                                  const float (&a)[Split<C>::HC],
                                                  const uint32_t (&keep)[Split<C>::PCH], const float (&lb)[NB + 1],
                                                  const float (&y)[YPART ? Split<C>::HC : 1]) {
    constexpr int PCH = Split<C>::PCH;
    float tb[NB + 1];
    tb[0] = sc_i;
#pragma unroll
    for (int e = 1; e <= NB; ++e) tb[e] = (il - e >= 0) ? lb[e] * sc[(t - e) > 0 ? (t - e) : 0] : 0.f;
    uint16_t hi[NB + 1], lo[NB + 1];
#pragma unroll
    for (int e = 0; e <= NB; ++e) {
        hi[e] = bf16_bits(tb[e]);
        lo[e] = bf16_bits(tb[e] - bf16_bits_to_f32(hi[e]));
    }
    uint32_t bp[PCH], pk[PCH];
    build_band_row<C, NB>(br_line, slot, hi, bp);
    const uint32_t sb_a = smem_u32(sc + cb + col0);
#pragma unroll
    for (int i = 0; i < PCH / 2; ++i) {
        const float4 bb = lds128f(sb_a + i * 16);
        float p0, p1, p2, p3;
        unpair2(mul2(pair2(a[4 * i], a[4 * i + 1]), pair2(bb.x, bb.y)), p0, p1);
        unpair2(mul2(pair2(a[4 * i + 2], a[4 * i + 3]), pair2(bb.z, bb.w)), p2, p3);
        const uint32_t w0 = pack_bf16x2(p0, p1), w1 = pack_bf16x2(p2, p3);
        pk[2 * i] = (KEEP ? (w0 & keep[2 * i]) : w0) | bp[2 * i];
        pk[2 * i + 1] = (KEEP ? (w1 & keep[2 * i + 1]) : w1) | bp[2 * i + 1];
    }
    bool plain = true;
    if constexpr (MERGE) {
        if (wq >= 2) {
            // second block of a 128-chunk: columns of the first block carry T21 diag(scale) instead of zeros
            plain = false;
            store_a_operand<C, false>(lane_base + kAS, t, h, pk);
            if constexpr (YPART) {
                const float2* sb1 = reinterpret_cast<const float2*>(sc + col0);
                uint32_t po[PCH], pl[PCH];
#pragma unroll
                for (int i = 0; i < PCH; ++i) {
                    const float2 bb = sb1[i];
                    const float v0 = y[2 * i] * bb.x, v1 = y[2 * i + 1] * bb.y;
                    po[i] = pack_bf16x2(v0, v1);
                    pl[i] = pack_bf16x2(v0 - bf16_lo(po[i]), v1 - bf16_hi(po[i]));
                }
                store_stacked_operand<C>(lane_base + kAS, h, po);
                store_stacked_operand<C>(lane_base + kR2, h, pl);
            }
        }
    }
    if constexpr (PERM) {
        // (M = 64 products per chunk: no zero columns of the other chunk to fill, columns 0..31 for both chunks)
        store_a_operand<C, false>(lane_base + kAS, 0, h, pk);
        build_band_row<C, NB>(br_line, slot, lo, bp);
        store_a_operand<C, false>(lane_base + kR2, 0, h, bp);
        return;
    }
    if (plain) store_a_operand<C, true>(lane_base + kAS, t, h, pk);
    build_band_row<C, NB>(br_line, slot, lo, bp);
    // rows of the second block of a 128-chunk keep the lo half of T21 diag(scale) in the first block's columns
    if (plain) store_a_operand<C, true>(lane_base + kR2, t, h, bp);
    else store_a_operand<C, false>(lane_base + kR2, t, h, bp);
}

struct TileCoord {
    int bhk, bhv;
    int t0;
    // where the tile sits in memory: first TMA coordinates of the K tile (feature column, outermost index) and of the
    // V / W / U tiles, index of the tile's first token in beta / g, and the stride between tokens there
    int kx, kz, vx, vz;
    long long r0;
    int rs;
};
// A tile index in mixed-radix digits: tile = (bhk * n_tt + tt) * group + gi, so that tiles sharing a key tile are
// adjacent. A CTA walks its tiles by adding the grid size digit by digit (one carry per digit is enough because
// every digit of the step is below its radix), which avoids integer divisions inside the tile loop.
// All counts fit 32 bits (checked by the launcher).
struct TilePos {
    int gi, tt, bhk;
};
template <int EX>
__device__ __forceinline__ TilePos tile_pos(uint32_t tile, const Params& p) {
    TilePos c;
    const int n_mid = EX ? p.n_mid : p.n_tt;
    const uint32_t y = tile / static_cast<uint32_t>(p.group);
    c.gi = static_cast<int>(tile - y * p.group);
    c.bhk = static_cast<int>(y / static_cast<uint32_t>(n_mid));
    c.tt = static_cast<int>(y - static_cast<uint32_t>(c.bhk) * n_mid);
    return c;
}
template <int EX>
__device__ __forceinline__ void tile_advance(TilePos& c, const Params& p) {
    const int n_mid = EX ? p.n_mid : p.n_tt;
    c.gi += p.s_gi;
    const int c1 = (c.gi >= p.group) ? 1 : 0;
    c.gi -= c1 ? p.group : 0;
    c.tt += p.s_tt + c1;
    const int c2 = (c.tt >= n_mid) ? 1 : 0;
    c.tt -= c2 ? n_mid : 0;
    c.bhk += p.s_bhk + c2;
}
// (key head row, value head row, first token): value head row = bhk * group + gi because H_v = H_k * group.
// Head-major tensors [B, H, T, d] are seen by TMA as (d, T, B * H); token-major ones [B, T, H, d]
// (GDN_FLAG_LAYOUT_BTHD, only in the EX instantiations) as (H * d, T, B), the head selecting a column range.
// There the walk is (value head of the group, key head, batch * n_tt + token tile) instead, so that the CTAs running
// at one time read all heads of the same tokens: a token's heads are contiguous in memory.
template <int EX>
__device__ __forceinline__ TileCoord tile_coord(const TilePos& c, const Params& p) {
    TileCoord r;
    r.bhk = c.bhk;
    r.bhv = c.bhk * p.group + c.gi;
    r.t0 = c.tt * kTile;
    if (EX && (p.flags & GDN_FLAG_LAYOUT_BTHD)) {
        const int hk = c.tt;
        const int b = c.bhk / p.n_tt;
        const int hv = hk * p.group + c.gi;
        r.bhk = b * p.H_k + hk;
        r.bhv = b * p.H_v + hv;
        r.t0 = (c.bhk - b * p.n_tt) * kTile;
        r.kx = hk * kD;
        r.kz = b;
        r.vx = hv * kD;
        r.vz = b;
        r.r0 = ((long long)b * p.T + r.t0) * p.H_v + hv;
        r.rs = p.H_v;
    } else {
        r.kx = 0;
        r.kz = r.bhk;
        r.vx = 0;
        r.vz = r.bhv;
        r.r0 = (long long)r.bhv * p.T + r.t0;
        r.rs = 1;
    }
    return r;
}

// MERGE: the tile is ONE chunk of 128 tokens whose two 64 x 64 diagonal blocks are inverted by the scheme above
// (C = 64 is then the block size) and whose lower-left block follows from App. E, Eq. 28:
// T21 = -T22 A21 T11, evaluated as Y = A21 + A21 X11, T21 = -(Y + X22 Y) with X = T - I of the blocks, so that
// the identity parts stay in fp32 and only the small products pass through bf16 operands.
// EX: 1 = the optional prologue, layouts and packed sequences of gdn_chunk_prepare_ex / _varlen are compiled in (flags
// read at run time); 2 = also the fp32 outputs (parity debugging); 3 = 1 for packed variable-length sequences. The
// last two cost registers, so each has its own code.
// DBL: 8 or 15 = the residual sum for that S is evaluated by the four-level doubling scheme (C = 64 only); 0 = one
// product per term.
template <int C, int NB, int MODE, bool MERGE, int EX, int DBL, bool PERM = false>
__global__ void __launch_bounds__(kThreads, 2)
chunk_tc_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmU,
                const __grid_constant__ CUtensorMap tmT, const Params p) {
    static_assert(!MERGE || C == 64, "the block merge is built for 64-blocks");
    static_assert(DBL == 0 || ((DBL == 8 || DBL == 15) && C == 64 && MODE == INV_NEUMANN), "the doubling scheme is built for 64-blocks");
    using L = Smem<C, NB>;
    using SP = Split<C>;
    constexpr int NBP = L::NBP;
    constexpr int HC = SP::HC;     // columns of the chunk handled by this thread
    constexpr int PCH = SP::PCH;   // packed words handled by this thread
    constexpr int CPRF = C / 4;    // 16-byte chunks of an fp32 row
    constexpr int CPT = HC / 8;    // packed chunks owned by this thread
    constexpr int CPTF = HC / 4;   // fp32 chunks owned by this thread
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);  // (an offset: the compiler goes on to know it as shared memory)
    uint8_t* sK = smem + L::kK;
    uint8_t* sV = smem + L::kV;
    uint8_t* sEB = smem + L::kEB;
    float* sSH = reinterpret_cast<float*>(smem + L::kSH);
    float* sRB = reinterpret_cast<float*>(smem + L::kRB);
    float* sbeta = reinterpret_cast<float*>(smem + L::kBeta);
    float* sg = reinterpret_cast<float*>(smem + L::kG);
    float* srn = reinterpret_cast<float*>(smem + L::kRn);
    float* sbrn = reinterpret_cast<float*>(smem + L::kBRn);
    float* swt = reinterpret_cast<float*>(smem + L::kWt);
    const bool f_graw = EX && (p.flags & GDN_FLAG_G_RAW) != 0;
    const bool f_l2 = EX && (p.flags & GDN_FLAG_K_L2NORM) != 0;
    const bool f_wg = EX && (p.flags & GDN_FLAG_W_GATED) != 0;
    const bool two_scales = f_l2 || f_wg;  // the W operand is scaled by something other than beta
    const bool f_f32 = EX == 2 && (p.flags & GDN_FLAG_OUT_FP32) != 0;
    constexpr bool f_var = EX == 3;
    constexpr int CR = MERGE ? kTile : C;  // tokens of a chunk

    __shared__ uint64_t bar_k, bar_v, bar_mma;
    __shared__ uint32_t tmem_base_s;
    __shared__ int s_fail;  // set by warp 0 when one of its bounded waits ran out
    // the first tile's loads go out before the set-up in the 128-chunk instantiations (few tiles per CTA there); in the
    // others the change of code shape cost more (1.3 % on the prefill shapes) than the overlap gains
    constexpr bool kEarlyLoad = MERGE && EX == 0;

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;

    if constexpr (EX == 1 || EX == 3) {
        // The layer call's state passing follows and waits for this kernel's end itself. It takes all of an SM's TMEM at its start: none of its
        // CTAs (more than 200 KB of shared memory) may have room beside one of these that has not allocated its own columns yet.
        static_assert(L::kTotal >= 64 * 1024, "the next kernel's CTAs must not fit beside these");
        launch_dependents();
    }
    if (tid == 0) {
        mbar_init(&bar_k, 1);
        mbar_init(&bar_v, 1);
        mbar_init(&bar_mma, 1);
        s_fail = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmV);
        tma_prefetch_desc(&tmW);
        tma_prefetch_desc(&tmU);
        tma_prefetch_desc(&tmT);
        // the first tile's K and V are asked for right away, so that they travel while TMEM is allocated and the
        // tile-invariant values are set up (packed sequences need the chunk table: they load after the set-up)
        if (kEarlyLoad && blockIdx.x < static_cast<uint32_t>(p.n_tiles)) {
            const TileCoord c = tile_coord<EX>(tile_pos<EX>(blockIdx.x, p), p);
            mbar_arrive_expect_tx(&bar_k, 32768);
            tma_load_3d(sK, &tmK, &bar_k, c.kx, c.t0, c.kz);
            tma_load_3d(sK + 16384, &tmK, &bar_k, c.kx + 64, c.t0, c.kz);
            mbar_arrive_expect_tx(&bar_v, 32768);
            tma_load_3d(sV, &tmV, &bar_v, c.vx, c.t0, c.vz);
            tma_load_3d(sV + 16384, &tmV, &bar_v, c.vx + 64, c.t0, c.vz);
        }
    }
    if (warp == 0) {
        tmem_alloc(&tmem_base_s, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_base_s;

    // (S is known where the doubling form was chosen; as a constant it saves a register: chunks of 128, 4 x 16 heads x 4096 tokens, 115.5 ->
    // 108.1 us, layer call of 8 x 4096 tokens 724 -> 715, 61 packed prompts 482 -> 472)
    const int N = p.N, S = DBL != 0 && (MERGE || EX != 0) ? DBL : p.S;
    // width of the band kept in fp32 (lb[]): the order N, or all of NB for forward substitution
    const int n_band = (MODE == INV_NEUMANN) ? N : NB;
    const uint32_t n_tiles = static_cast<uint32_t>(p.n_tiles);

    // Threads t and t + 128 share tile row t (TMEM lane t): half h owns the chunk-local columns
    // [h * HC, (h + 1) * HC) when C >= 32; for C = 16 only h = 0 works on the row (h = 1 joins for W/U).
    // One elected lane of warp 0 also issues every TMA load and every tcgen05.mma, right after the CTA barrier
    // that says all rows of the operand are in place.
    // kPerm (PERM instantiations of the default 64-chunk path): every tensor-core product is an M = 64 instruction on ONE chunk, so
    // that none multiplies the structural zeros an M = 128 instruction spanning both chunks of the tile would (half of
    // the Gram product, half of the K steps of the block-diagonal W / U operands; that work is what drives the launch
    // into the power cap). An M = 64 accumulator (and A operand) occupies 16 lanes of every lane quadrant: rows
    // 16 q .. 16 q + 15 on lanes 32 q .. 32 q + 15, and with a lane offset of 16 the other half-lanes. So chunk 0 lives on
    // the lanes [0, 16) of every quadrant and chunk 1 on the lanes [16, 32): the thread on TMEM lane l works on tile row
    // t = 64 ((l / 16) % 2) + 16 (l / 32) + l % 16 instead of t = l. Everything indexed by a token (shared arrays, global
    // rows, B operands) keeps using t; TMEM columns no longer depend on the chunk (the two chunks sit on different
    // lanes of the same columns); a warp holds two groups of 16 consecutive rows, which leave as two bulk stores.
    // M = 64 instructions take as long as M = 128 ones (and the doubling levels need twice as many of them), so at full
    // clocks this form is 3 % slower; it draws less power, and on a GPU that runs at the power cap it is 3.5 % faster. The
    // host picks it for large launches (launch_tc_bf16).
    static_assert(!PERM || (C == 64 && !MERGE && MODE == INV_NEUMANN && EX == 0 && DBL != 0), "built for the default 64-chunk path");
    constexpr bool kPerm = PERM;
    const int lrow = tid & 127;  // TMEM lane of this thread's row
    const int t = kPerm ? ((((lrow >> 4) & 1) << 6) + ((lrow >> 5) << 4) + (lrow & 15)) : lrow;
    const int h = tid >> 7;
    const bool active = SP::kSplit || (h == 0);
    const int col0 = SP::kSplit ? h * HC : 0;  // first chunk-local column of this thread
    const int il = t % C;                      // row inside its chunk
    const int cb = t - il;                     // first tile row of the chunk
    const int wq = warp & 3;                   // TMEM lane quadrant of the warp
    const int wrow0 = wq * 32;                 // first tile row of the warp
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(wq * 32) << 16);
    const uint32_t scratch_a = smem_u32(smem + L::kEB);
    const uint32_t br_line = smem_u32(smem + L::kBR) + (col0 >> 3) * (kTile * 16) + t * 16;
    const uint32_t rowf = scratch_a + t * (4 * C);  // private fp32 row (shared by the two halves)
    const uint32_t sK_a = smem_u32(sK), sV_a = smem_u32(sV), sEB_a = smem_u32(sEB);
    const uint32_t sSH_a = smem_u32(smem + L::kSH), sg_a = smem_u32(smem + L::kG);
    const uint32_t idesc_g = instr_desc(128, 128, 1, 1, 0, 0, 1);
    const uint32_t idesc_c = instr_desc(128, 128, 1, 1, 0, 1, 1);
    const uint32_t idesc_w = instr_desc(128, 128, 1, 1, 0, 1, 1);
    uint32_t par_mma = 0, par_kv = 0;
    bool ok = true;
    // Completion of the MMAs committed to bar_mma: warp 0 polls the mbarrier, the other warps sleep on a hardware
    // barrier that warp 0 joins afterwards (no polling instructions from 7 of the 8 warps). A timeout is published
    // in s_fail, so that every thread leaves the tile loop at the same point.
    // kPerm: W (or U) of chunk m = (hi + lo operand of the chunk, 4 + 4 K steps of its own 64 tokens) x (the chunk's rows
    // of the K (V) tile), an M = 64, N = 128 product on the chunk's half-lanes
    auto issue_wu64 = [&](uint32_t tile_a) {
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const uint32_t lm = static_cast<uint32_t>(16 * m) << 16;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                const uint64_t bd = smem_desc(tile_a + (4 * m + (ks & 3)) * 2048, 16384, 1024, SWZ_128B);
                mma_f16_ts(tmem + kR0 + lm, tmem + ((ks < 4) ? kAS : kR2) + (ks & 3) * 8 + lm, bd, instr_desc(64, 128, 1, 1, 0, 1, 1), ks > 0);
            }
        }
    };
    auto wait_mma = [&]() -> bool {
        if (warp == 0 && !wait_bar(&bar_mma, par_mma)) *reinterpret_cast<volatile int*>(&s_fail) = 1;
        asm volatile("bar.sync 2, 256;" ::: "memory");
        par_mma ^= 1;
        return *reinterpret_cast<volatile int*>(&s_fail) == 0;
    };

    // tile-invariant per-thread band positions and keep-mask (0 on the band and the diagonal, ones elsewhere).
    // The mask cuts the band out of the packed far part of a row before the band words are OR-ed in. At C >= 32 (every
    // thread works on its row) it is not needed, and its 16 registers are: in the Neumann path a[] only ever holds E and
    // sums of products with E or its powers, which are exactly zero on the band, the diagonal and above (E is zero for
    // i - j <= N, every left factor is lower triangular, sums of exact zeros are zero); after a forward substitution
    // a[] is zeroed there when the rows are read back. At C = 16 it also blanks the rows of the idle half.
    constexpr bool kKeepMask = C < 32;
    uint32_t slot[NB + 1];
    uint32_t keep[PCH];
    band_slots<C, NB>(smem_u32(smem + L::kBR), smem_u32(smem + L::kDummy) + tid * 4, t, il, col0, n_band, slot);
    if (!kKeepMask) {
#pragma unroll
        for (int i = 0; i < PCH; ++i) keep[i] = 0xFFFFFFFFu;
    } else if (active) {
        uint16_t vals[NB + 1];
#pragma unroll
        for (int e = 0; e <= NB; ++e) vals[e] = 0xFFFFu;
        build_band_row<C, NB>(br_line, slot, vals, keep);
#pragma unroll
        for (int i = 0; i < PCH; ++i) keep[i] = ~keep[i];
    } else {
#pragma unroll
        for (int i = 0; i < PCH; ++i) keep[i] = 0u;
    }

    // K (or V) rows of a tile: one box of 128 tokens per 64-column half, or, with variable-length sequences, one box
    // per chunk from the chunk's own first token (rows past its length belong to the next sequence or are filled
    // with zeros past the end of the tensor: beta = 0 below keeps them out of every result)
    auto load_tile = [&](uint8_t* dst, const CUtensorMap* tm, uint64_t* bar, int x, int t0, int z) {
        mbar_arrive_expect_tx(bar, 32768);
        if (EX && f_var) {
            const int cid0 = (t0 / kTile) * (kTile / CR);
#pragma unroll 1
            for (int m = 0; m < kTile / CR; ++m) {
                const int st = (cid0 + m < p.n_chunks) ? __ldg(p.chunk_start + cid0 + m) : 0;
                tma_load_3d(dst + m * (CR * 128), tm, bar, x, st, z);
                tma_load_3d(dst + 16384 + m * (CR * 128), tm, bar, x + 64, st, z);
            }
        } else {
            tma_load_3d(dst, tm, bar, x, t0, z);
            tma_load_3d(dst + 16384, tm, bar, x + 64, t0, z);
        }
    };
    // beta and g of this thread's row of a tile, and (variable-length sequences) the row's token in the packed
    // tensors, -1 for a row past its chunk's length: such a row has beta = 0 and the gate of the chunk's last token
    auto fetch_row = [&](const TilePos& pos, float& b_out, float& g_out, int& tok_out) {
        const TileCoord c = tile_coord<EX>(pos, p);
        b_out = 0.f;
        g_out = 0.f;
        tok_out = -1;
        if (EX && f_var) {
            const int cid = (c.t0 / kTile) * (kTile / CR) + t / CR;
            const int r = t % CR;
            int st = 0, len = 0;
            if (cid < p.n_chunks) {
                st = __ldg(p.chunk_start + cid);
                len = __ldg(p.chunk_len + cid);
            }
            const bool bthd = (p.flags & GDN_FLAG_LAYOUT_BTHD) != 0;
            const long long base = bthd ? c.bhv : (long long)c.bhv * p.T_total;
            const long long stride = bthd ? p.H_v : 1;
            if (r < len) {
                tok_out = st + r;
                const long long row = base + (long long)tok_out * stride;
                b_out = __ldg(p.beta + row);
                g_out = __ldg(p.g + row);
            } else if (len > 0 && !f_graw) {
                g_out = __ldg(p.g + base + (long long)(st + len - 1) * stride);
            }
        } else if (c.t0 + t < p.T) {
            const long long r = c.r0 + (long long)t * c.rs;
            b_out = __ldg(p.beta + r);
            g_out = __ldg(p.g + r);
        }
    };
    // Token-major tensors: beta and g of consecutive tokens are H_v floats apart, one 32-byte sector per row and array.
    // Only the thread of a row's first column half fetches them; the other takes them from the shared arrays.
    constexpr bool kRowHalf = EX == 1 && C >= 32;
    TilePos pos_next = tile_pos<EX>(blockIdx.x, p);  // position of the tile after the one being worked on
    if (!kEarlyLoad && tid == 0 && blockIdx.x < n_tiles) {
        const TileCoord c = tile_coord<EX>(pos_next, p);
        load_tile(sK, &tmK, &bar_k, c.kx, c.t0, c.kz);
        load_tile(sV, &tmV, &bar_v, c.vx, c.t0, c.vz);
    }
    // beta and g of the row are fetched one tile ahead
    float bi_next = 0.f, gi_next = 0.f;
    int gtok_next = -1;
    if (blockIdx.x < n_tiles && !(kRowHalf && (p.flags & GDN_FLAG_LAYOUT_BTHD) && (threadIdx.x >> 7) == 1))
        fetch_row(pos_next, bi_next, gi_next, gtok_next);

    for (uint32_t rem = blockIdx.x < n_tiles ? (n_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0u; rem > 0 && ok; --rem) {  // tiles left for this CTA
        // The tile's coordinates are only needed by the stores at its end. With the optional layouts they are six values:
        // those instantiations keep the tile's position (three) and form the coordinates there.
        const TilePos pos_cur = pos_next;
        TileCoord tc;
        if constexpr (EX == 0) tc = tile_coord<EX>(pos_next, p);
        tile_advance<EX>(pos_next, p);
        const bool has_next = rem > 1;

        float bi = bi_next;  // loaded during the previous tile
        float gi_ = gi_next;
        const int gtok = gtok_next;
        constexpr int kWarpsPerChunk = MERGE ? 4 : (C >= 32 ? C / 32 : 1);
        if (f_graw) {
            // g holds the raw per-token log-gates: inclusive prefix sum inside the chunk, by shuffles inside the warp
            // (segments of C lanes when C = 16) and through shared memory across the chunk's warps
            constexpr int SEG = (C < 32) ? C : 32;
#pragma unroll
            for (int off = 1; off < SEG; off <<= 1) {
                const float v = __shfl_up_sync(0xFFFFFFFFu, gi_, off);
                if ((lane & (SEG - 1)) >= off) gi_ += v;
            }
        }
        // (the warp totals of the previous tile were read right after that tile's first barrier: free to overwrite)
        if (f_graw && kWarpsPerChunk > 1 && h == 0 && lane == 31) swt[wq] = gi_;
        // the previous tile's bulk stores have finished reading the staging slices
        if (lane == 0) tma_store_wait_read<0>();
        tc_fence_before_sync();
        compute_barrier();  // everyone is done with the previous tile's shared arrays and accumulators
        if (f_graw && kWarpsPerChunk > 1) {
            const int first = wq - (wq % kWarpsPerChunk);
            for (int w = first; w < wq; ++w) gi_ += swt[w];
        }
        if (C == 64 && EX == 0 && !PERM && !MERGE && warp == 0 && has_next && elect_one()) {
            // The next tile's K can only land in shared memory once this tile's W products are done with the buffer,
            // which leaves its load little time before the next Gram product wants it: ask for it in L2 now. Only in the default
            // form (4 x 16 heads x 4096 tokens 85.1 us with, 85.7 without): the others gain nothing by it (chunks of 128 109.0 and 108.1, layer
            // call of 8 x 4096 tokens 721 and 715, the M = 64 form 2423 and 2417 for 65536 tiles).
            const TileCoord nc = tile_coord<EX>(pos_next, p);
            tma_prefetch_l2_3d(&tmK, nc.kx, nc.t0, nc.kz);
            tma_prefetch_l2_3d(&tmK, nc.kx + 64, nc.t0, nc.kz);
        }
        if (warp == 0) {
            // G = K K^T into R0..R1 (128 columns)
            if (!wait_bar(&bar_k, par_kv)) ok = false;
            if (ok) {
                tc_fence_after_sync();
                if (elect_one()) {
#pragma unroll
                    if constexpr (kPerm) {
                        // one 64 x 64 Gram block per chunk, on the chunk's half-lanes, both in columns 0..63
#pragma unroll
                        for (int m = 0; m < 2; ++m) {
#pragma unroll
                            for (int ks = 0; ks < 8; ++ks) {
                                const uint64_t d = smem_desc(sK_a + (ks >> 2) * 16384 + m * 8192 + (ks & 3) * 32, 16, 1024, SWZ_128B);
                                mma_f16_ss(tmem + kR0 + (static_cast<uint32_t>(16 * m) << 16), d, d, instr_desc(64, 64, 1, 1, 0, 0, 1), ks > 0);
                            }
                        }
                    } else {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint64_t d = smem_desc(sK_a + (ks >> 2) * 16384 + (ks & 3) * 32, 16, 1024, SWZ_128B);
                        mma_f16_ss(tmem + kR0, d, d, idesc_g, ks > 0);
                    }
                    }
                    mma_commit(&bar_mma);
                }
            }
        }
        if (h == 0) {
            sbeta[t] = bi;
            sg[t] = gi_;
#pragma unroll
            for (int e = 0; e < NBP; ++e) sSH[t * NBP + e] = 0.f;
            if (t < 8) {
#pragma unroll
                for (int e = 0; e < NBP; ++e) sSH[(kTile + t) * NBP + e] = 0.f;
            }
        }
        compute_barrier();
        if (kRowHalf && (p.flags & GDN_FLAG_LAYOUT_BTHD) && h == 1) {
            bi = sbeta[t];
            gi_ = sg[t];
        }

        // ---- A-build: this thread's part of the row of Abar, from the Gram block in TMEM
        if (!wait_mma()) { ok = false; break; }
        tc_fence_after_sync();
        float a[HC];
        if constexpr (MERGE) {
            // rows of the second block keep their part of the lower-left Gram block (columns 0..63) in R2:
            // R0..R1 is overwritten by the residual rounds. Either half of a row keeps it in the very columns that its part of
            // X22 (hi, lo) goes to later: no thread writes over what the other half has yet to read.
            if (wq >= 2) {
                uint32_t r[32], r16[16];
                tmem_ld32(lane_base + kR0 + h * 32, r);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) r16[i] = r[i];
                tmem_st16(lane_base + kR2 + h * 16, r16);
#pragma unroll
                for (int i = 0; i < 16; ++i) r16[i] = r[16 + i];
                tmem_st16(lane_base + kR2 + 32 + h * 16, r16);
                tmem_wait_st();
            }
        }
        if (active) load_diag_block<C>(lane_base, kR0, kPerm ? (t & 63) : t, h, a);
        float rni = 1.f;
        if (f_l2) {
            // keys are normalised on the fly: 1 / ||K_i|| from the diagonal of the Gram matrix
            if (active && il >= col0 && il < col0 + HC) {
                float gd = 0.f;
#pragma unroll
                for (int jl = 0; jl < HC; ++jl)
                    if (col0 + jl == il) gd = a[jl];
                const float rn = (f_var && gtok < 0) ? 0.f : rsqrtf(fmaxf(gd, 1e-30f));
                srn[t] = rn;
                sbrn[t] = bi * rn * (f_wg ? fast_exp2(gi_ * kLog2e) : 1.f);
            }
            compute_barrier();
            rni = srn[t];
        } else if (f_wg) {
            // gated W: the column scale of the W operand is beta_j exp(g_j) (read after the barriers of the stages
            // below)
            if (h == 0) sbrn[t] = bi * fast_exp2(gi_ * kLog2e);
        }
        if (active) {
            const float gs = gi_ * kLog2e;
            const float nbi = -bi * rni;
            const float4* sr4 = reinterpret_cast<const float4*>(srn + cb + col0);
#pragma unroll
            for (int j4 = 0; j4 < HC / 4; ++j4) {
                const float4 gq = lds128f(sg_a + (cb + col0 + j4 * 4) * 4);
                const float gj[4] = {gq.x, gq.y, gq.z, gq.w};
                float rj[4] = {1.f, 1.f, 1.f, 1.f};
                if (f_l2) {
                    const float4 rq = sr4[j4];
                    rj[0] = rq.x; rj[1] = rq.y; rj[2] = rq.z; rj[3] = rq.w;
                }
                if constexpr (C == 64) {
                    // (see below: entries on and above the diagonal only have to be finite. Two elements an instruction here, in the sums of
                    // the levels and in the scaling of the W / U operands: 4 x 16 heads x 4096 tokens 86.0 -> 85.1 us, layer call of 8 x 4096
                    // tokens 721 -> 715.)
#pragma unroll
                    for (int q = 0; q < 4; q += 2) {
                        const int jl = j4 * 4 + q;
                        float x0, x1;
                        unpair2(fma2(pair2(gj[q], gj[q + 1]), pair2(-kLog2e, -kLog2e), pair2(gs, gs)), x0, x1);
                        f2 v = mul2(mul2(pair2(nbi, nbi), pair2(fast_exp2(fminf(x0, 64.f)), fast_exp2(fminf(x1, 64.f)))), pair2(a[jl], a[jl + 1]));
                        if (f_l2) v = mul2(v, pair2(rj[q], rj[q + 1]));
                        unpair2(v, a[jl], a[jl + 1]);
                    }
                    continue;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int jl = j4 * 4 + q;
                    // Entries on and above the diagonal are NOT zeroed here: every later use either reads strictly
                    // lower entries only or multiplies them by a band entry that is zero, so they only have to be
                    // finite, which the clamp of the exponent (<= 0 for every lower entry) guarantees.
                    float v = nbi * fast_exp2(fminf(fmaf(-gj[q], kLog2e, gs), 64.f)) * a[jl];
                    if (f_l2) v *= rj[q];
                    a[jl] = (C < 64 && !(col0 + jl < il)) ? 0.f : v;  // (for C < 64 the mask is kept: it costs less there than it saves)
                }
            }
            // the row of Abar goes to its private fp32 line: entries next to the diagonal (and, for the
            // left half, the first entries of the right half) are read back from there
#pragma unroll
            for (int c = 0; c < CPTF; ++c)
                sts128(rowf + (swz<CPRF>(t, (col0 >> 2) + c) << 4), __float_as_uint(a[c * 4 + 0]), __float_as_uint(a[c * 4 + 1]),
                       __float_as_uint(a[c * 4 + 2]), __float_as_uint(a[c * 4 + 3]));
        } else {
#pragma unroll
            for (int j = 0; j < HC; ++j) a[j] = 0.f;
        }
        bi_next = 0.f;
        gi_next = 0.f;
        if (has_next && !(kRowHalf && (p.flags & GDN_FLAG_LAYOUT_BTHD) && h == 1)) fetch_row(pos_next, bi_next, gi_next, gtok_next);
        compute_barrier();  // both halves of every fp32 row are written

        float lb[NB + 1];  // lb[d] = L[i][i-d], the band of T0 - I (or of T - I after forward substitution)
#pragma unroll
        for (int e = 0; e <= NB; ++e) lb[e] = 0.f;

        if constexpr (MODE == INV_NEUMANN) {
            float ab[NB + 1];     // ab[e] = Abar[i][i-e]
            float anext[NB + 1];  // anext[e] = Abar[i][col0 + HC + e]: the entries just right of this thread's part
            ab[0] = 0.f;
#pragma unroll
            for (int e = 1; e <= NB; ++e) {
                const int j = il - e;
                ab[e] = (j >= 0) ? lds32f(rowf + (swz<CPRF>(t, j >> 2) << 4) + (j & 3) * 4) : 0.f;
            }
#pragma unroll
            for (int e = 0; e < NB; ++e) {
                const int j = col0 + HC + e;
                anext[e] = (SP::kSplit && j < C) ? lds32f(rowf + (swz<CPRF>(t, j >> 2) << 4) + (j & 3) * 4) : 0.f;
            }
            anext[NB] = 0.f;
            // ---- band of the masked Neumann sum by distance recursion (both halves compute it, h = 0 publishes it)
            lb[1] = ab[1];
            if (h == 0) sRB[t * NBP + 0] = lb[1];
#pragma unroll
            for (int d = 2; d <= NB; ++d) {
                compute_barrier();
                float v = ab[d];
#pragma unroll
                for (int e = 1; e < d; ++e) {
                    const int r = (t - e) > 0 ? (t - e) : 0;
                    v = fmaf(ab[e], sRB[r * NBP + (d - e - 1)], v);
                }
                lb[d] = (d <= N) ? v : 0.f;
                if (d < NB && h == 0) sRB[t * NBP + (d - 1)] = lb[d];
            }
            // column form: SH[j][e-1] = L[j+e][j]
            if (h == 0) {
#pragma unroll
                for (int e = 1; e <= NB; ++e)
                    if (il - e >= 0) sSH[(t - e) * NBP + (e - 1)] = lb[e];
            }
            compute_barrier();

            if (active) {
                // ---- E = Abar + Abar L on i-j > N (in place over a[])
#pragma unroll
                for (int jl = 0; jl < HC; ++jl) {
                    float v = a[jl];
                    float cc[NBP];
                    if constexpr (NBP == 4) {
                        const float4 c4 = lds128f(sSH_a + (cb + col0 + jl) * 16);
                        cc[0] = c4.x; cc[1] = c4.y; cc[2] = c4.z; cc[3] = c4.w;
                    } else {
                        const float4 c4 = lds128f(sSH_a + (cb + col0 + jl) * 32);
                        const float4 d4 = lds128f(sSH_a + (cb + col0 + jl) * 32 + 16);
                        cc[0] = c4.x; cc[1] = c4.y; cc[2] = c4.z; cc[3] = c4.w;
                        cc[4] = d4.x; cc[5] = d4.y; cc[6] = d4.z; cc[7] = d4.w;
                    }
#pragma unroll
                    for (int e = 1; e <= NB; ++e) {
                        const int k = jl + e;
                        const float ak = (k < HC) ? a[(k < HC) ? k : 0] : anext[(k >= HC) ? k - HC : 0];
                        v = fmaf(ak, cc[e - 1], v);
                    }
                    a[jl] = (il - (col0 + jl) > N) ? v : 0.f;
                }
                // E as B operand [E_1 | E_2 | ...] (C x 128, MN-major, no swizzle): the 16-byte piece of chunk-row il
                // for global column group n8 sits at n8 * (16 C) + il * 16
                if (S >= 1) {
#pragma unroll
                    for (int c = 0; c < CPT; ++c) {
                        uint4 v;
                        v.x = pack_bf16x2(a[c * 8 + 0], a[c * 8 + 1]);
                        v.y = pack_bf16x2(a[c * 8 + 2], a[c * 8 + 3]);
                        v.z = pack_bf16x2(a[c * 8 + 4], a[c * 8 + 5]);
                        v.w = pack_bf16x2(a[c * 8 + 6], a[c * 8 + 7]);
                        *reinterpret_cast<uint4*>(sEB + (((cb + col0) >> 3) + c) * (16 * C) + il * 16) = v;
                    }
                }
            }
        } else {
            // ---- forward substitution (Eq. 2-3). The private fp32 rows hold Abar; thread (h = 0, t) solves
            // column il of its chunk, which has no dependence on other columns.
            if constexpr (MODE == INV_FWDSUBST_TC) {
                // Blocked form with the block merge on the tensor cores (App. E, Eq. 28 inside every 64-chunk): the two
                // 32 x 32 diagonal blocks by substitution (32 sequential rows instead of 64, 128 column threads), then
                // T21 = T22 Abar21 T11 (Abar = -A) as Y = Abar21 + Abar21 X11, T21 = Y + X22 Y with X = T - I: two products with hi + lo
                // bf16 operands (they cancel on correlated keys, as in the C = 128 merge), identity parts in fp32, all 256
                // threads taking part in the operand work. M = 128, N = 64, K = 32: rows 32..63 of both chunks are the
                // A operands, [X11 of chunk 0 | X11 of chunk 1] (then Y) the B operand.
                static_assert(C == 64 && !MERGE, "built for 64-chunks");
                const int b0 = il >> 5;        // diagonal block of this row / column (uniform per warp)
                const int ci2 = t >> 6;        // chunk of the tile
                if (h == 0) {
                    float xcol[32];  // xcol[r] = T[32 b0 + r][il]
#pragma unroll
                    for (int r = 0; r < 32; ++r) {
                        const int i = 32 * b0 + r;
                        float acc = 0.f;
                        const uint32_t ri = scratch_a + (cb + i) * (4 * C);
#pragma unroll
                        for (int q4 = 0; q4 < (r + 3) / 4; ++q4) {
                            const uint4 q = lds128(ri + (swz<CPRF>(i, 8 * b0 + q4) << 4));
                            if (q4 * 4 + 0 < r) acc = fmaf(__uint_as_float(q.x), xcol[q4 * 4 + 0], acc);
                            if (q4 * 4 + 1 < r) acc = fmaf(__uint_as_float(q.y), xcol[(q4 * 4 + 1 < 32) ? q4 * 4 + 1 : 0], acc);
                            if (q4 * 4 + 2 < r) acc = fmaf(__uint_as_float(q.z), xcol[(q4 * 4 + 2 < 32) ? q4 * 4 + 2 : 0], acc);
                            if (q4 * 4 + 3 < r) acc = fmaf(__uint_as_float(q.w), xcol[(q4 * 4 + 3 < 32) ? q4 * 4 + 3 : 0], acc);
                        }
                        xcol[r] = (i > il) ? acc : ((i == il) ? 1.f : 0.f);
                    }
                    compute_barrier();  // everyone has read Abar of the diagonal blocks
#pragma unroll
                    for (int r = 0; r < 32; ++r) {
                        const int i = 32 * b0 + r;
                        const uint32_t addr = scratch_a + (cb + i) * (4 * C) + (swz<CPRF>(i, il >> 2) << 4) + (il & 3) * 4;
                        asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(xcol[r]) : "memory");
                    }
                    if (b0 == 1) {
                        // rows above the second block: zeros (the entries above the diagonal were never masked)
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            const uint32_t addr = scratch_a + (cb + i) * (4 * C) + (swz<CPRF>(i, il >> 2) << 4) + (il & 3) * 4;
                            asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(0.f) : "memory");
                        }
                    }
                } else {
                    compute_barrier();
                }
                compute_barrier();
                // every thread takes its half row: T11 / zeros (first block), Abar21 / T22 (second block)
#pragma unroll
                for (int c = 0; c < CPTF; ++c) {
                    const uint4 q = lds128(rowf + (swz<CPRF>(t, (col0 >> 2) + c) << 4));
                    a[c * 4 + 0] = __uint_as_float(q.x);
                    a[c * 4 + 1] = __uint_as_float(q.y);
                    a[c * 4 + 2] = __uint_as_float(q.z);
                    a[c * 4 + 3] = __uint_as_float(q.w);
                }
                compute_barrier();  // the fp32 rows are dead: the B operands overlay them
                const uint32_t idesc_t = instr_desc(128, 64, 1, 1, 0, 1, 1);
                // one B piece = 8 columns of one row (16 bytes) at n8 * 512 + k * 16, hi plane at 0, lo plane at 4 KB
                auto store_b = [&](int krow) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint32_t wh[4], wl[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float v0 = a[8 * c + 2 * i], v1 = a[8 * c + 2 * i + 1];
                            wh[i] = pack_bf16x2(v0, v1);
                            wl[i] = pack_bf16x2(v0 - bf16_lo(wh[i]), v1 - bf16_hi(wh[i]));
                        }
                        const uint32_t off = (4 * ci2 + c) * 512 + krow * 16;
                        *reinterpret_cast<uint4*>(sEB + off) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
                        *reinterpret_cast<uint4*>(sEB + 4096 + off) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
                    }
                };
                auto store_a = [&](uint32_t slot_cols) {
                    uint32_t ph[16], pl[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        ph[i] = pack_bf16x2(a[2 * i], a[2 * i + 1]);
                        pl[i] = pack_bf16x2(a[2 * i] - bf16_lo(ph[i]), a[2 * i + 1] - bf16_hi(ph[i]));
                    }
                    tmem_st16(lane_base + slot_cols, ph);
                    tmem_st16(lane_base + slot_cols + 16, pl);
                };
                auto issue = [&](uint32_t slot_cols) {
                    if (warp == 0) {
                        tc_fence_after_sync();
                        if (elect_one()) {
#pragma unroll
                            for (int part = 0; part < 3; ++part) {
                                // hi*hi, lo*hi, hi*lo
#pragma unroll
                                for (int ks = 0; ks < 2; ++ks) {
                                    const uint64_t bd = smem_desc(sEB_a + (part == 2 ? 4096 : 0) + ks * 256, 128, 512, SWZ_NONE);
                                    mma_f16_ts(tmem + kR0, tmem + slot_cols + (part == 1 ? 16 : 0) + ks * 8, bd, idesc_t, part > 0 || ks > 0);
                                }
                            }
                            mma_commit(&bar_mma);
                        }
                    }
                };
                if (b0 == 0) {
                    if (h == 0) {
                        // X11 = T11 - I: the B operand of the first product
#pragma unroll
                        for (int jl = 0; jl < HC; ++jl) a[jl] -= (jl == il) ? 1.f : 0.f;
                        store_b(il);
#pragma unroll
                        for (int jl = 0; jl < HC; ++jl) a[jl] += (jl == il) ? 1.f : 0.f;
                    }
                } else if (h == 0) {
                    store_a(kAS);  // Abar21 (hi, lo): A operand of the first product
                } else {
                    // X22 = T22 - I (hi, lo): A operand of the second product
#pragma unroll
                    for (int jl = 0; jl < HC; ++jl) a[jl] -= (col0 + jl == il) ? 1.f : 0.f;
                    store_a(kR2);
#pragma unroll
                    for (int jl = 0; jl < HC; ++jl) a[jl] += (col0 + jl == il) ? 1.f : 0.f;
                }
                tmem_wait_st();
                fence_proxy_async_smem();
                tc_fence_before_sync();
                compute_barrier();
                issue(kAS);
                if (!wait_mma()) { ok = false; break; }
                tc_fence_after_sync();
                if (b0 == 1 && h == 0) {
                    // Y = Abar21 + Abar21 X11: the B operand of the second product
                    uint32_t d[32];
                    tmem_ld32(lane_base + kR0 + 32 * ci2, d);
                    tmem_wait_ld();
#pragma unroll
                    for (int jl = 0; jl < HC; ++jl) a[jl] += __uint_as_float(d[jl]);
                    store_b(il - 32);
                }
                fence_proxy_async_smem();
                tc_fence_before_sync();
                compute_barrier();
                issue(kR2);
                if (!wait_mma()) { ok = false; break; }
                tc_fence_after_sync();
                if (b0 == 1 && h == 0) {
                    // T21 = Y + X22 Y
                    uint32_t d[32];
                    tmem_ld32(lane_base + kR0 + 32 * ci2, d);
                    tmem_wait_ld();
#pragma unroll
                    for (int jl = 0; jl < HC; ++jl) a[jl] += __uint_as_float(d[jl]);
                }
                // the finished rows go back to the fp32 lines (the operand planes overlaid some of them)
#pragma unroll
                for (int c = 0; c < CPTF; ++c)
                    sts128(rowf + (swz<CPRF>(t, (col0 >> 2) + c) << 4), __float_as_uint(a[c * 4 + 0]), __float_as_uint(a[c * 4 + 1]),
                           __float_as_uint(a[c * 4 + 2]), __float_as_uint(a[c * 4 + 3]));
            } else {
            if (h == 0) {
                float xcol[C];  // xcol[k] = T[k][il]
                if constexpr (MODE == INV_FWDSUBST_BLOCKED) {
                    // Blocked form (App. E): the 16 x 16 diagonal blocks are inverted by substitution independently
                    // (Eq. 25), then block row bi follows from S_ij = S_ii sum_{k<i} Abar_ik S_kj (Eq. 27 with
                    // T_ik = -Abar_ik). The inverted diagonal blocks go through shared memory (strictly lower
                    // parts, 120 floats per block) because a column's thread needs the blocks of other columns.
                    float* sDi = sSH;  // [8 blocks of the tile][120]; the band arrays are unused in this mode
                    const int b0 = il >> 4, c16 = il & 15;
#pragma unroll
                    for (int i = 0; i < C; ++i) {
                        float acc = 0.f;
                        const uint32_t ri = scratch_a + (cb + i) * (4 * C);
#pragma unroll
                        for (int k4 = (i & ~15) / 4; k4 < (i + 3) / 4; ++k4) {
                            const uint4 q = lds128(ri + (swz<CPRF>(i, k4) << 4));
                            if (k4 * 4 + 0 < i) acc = fmaf(__uint_as_float(q.x), xcol[k4 * 4 + 0], acc);
                            if (k4 * 4 + 1 < i) acc = fmaf(__uint_as_float(q.y), xcol[(k4 * 4 + 1 < C) ? k4 * 4 + 1 : 0], acc);
                            if (k4 * 4 + 2 < i) acc = fmaf(__uint_as_float(q.z), xcol[(k4 * 4 + 2 < C) ? k4 * 4 + 2 : 0], acc);
                            if (k4 * 4 + 3 < i) acc = fmaf(__uint_as_float(q.w), xcol[(k4 * 4 + 3 < C) ? k4 * 4 + 3 : 0], acc);
                        }
                        xcol[i] = ((i >> 4) == b0 && i > il) ? acc : ((i == il) ? 1.f : 0.f);
                        if ((i >> 4) == b0 && (i & 15) > c16)
                            sDi[((cb >> 4) + (i >> 4)) * 120 + ((i & 15) * ((i & 15) - 1)) / 2 + c16] = xcol[i];
                    }
                    compute_barrier();  // the inverted diagonal blocks are published
#pragma unroll
                    for (int bi = 1; bi < C / 16; ++bi) {
                        float tmp[16];
#pragma unroll
                        for (int r = 0; r < 16; ++r) {
                            float acc = 0.f;
                            const int i = bi * 16 + r;
                            const uint32_t ri = scratch_a + (cb + i) * (4 * C);
#pragma unroll
                            for (int k4 = 0; k4 < bi * 4; ++k4) {
                                const uint4 q = lds128(ri + (swz<CPRF>(i, k4) << 4));
                                acc = fmaf(__uint_as_float(q.x), xcol[k4 * 4 + 0], acc);
                                acc = fmaf(__uint_as_float(q.y), xcol[k4 * 4 + 1], acc);
                                acc = fmaf(__uint_as_float(q.z), xcol[k4 * 4 + 2], acc);
                                acc = fmaf(__uint_as_float(q.w), xcol[k4 * 4 + 3], acc);
                            }
                            tmp[r] = acc;
                        }
                        const float* Sd = sDi + ((cb >> 4) + bi) * 120;
#pragma unroll
                        for (int r = 0; r < 16; ++r) {
                            float acc = tmp[r];
#pragma unroll
                            for (int q = 0; q < r; ++q) acc = fmaf(Sd[(r * (r - 1)) / 2 + q], tmp[q], acc);
                            if (bi > b0) xcol[bi * 16 + r] = acc;
                        }
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < C; ++i) {
                        float acc = 0.f;
                        const uint32_t ri = scratch_a + (cb + i) * (4 * C);
#pragma unroll
                        for (int k4 = 0; k4 < (i + 3) / 4; ++k4) {
                            const uint4 q = lds128(ri + (swz<CPRF>(i, k4) << 4));  // (cb + i) and i agree in the swizzle bits
                            if (k4 * 4 + 0 < i) acc = fmaf(__uint_as_float(q.x), xcol[k4 * 4 + 0], acc);
                            if (k4 * 4 + 1 < i) acc = fmaf(__uint_as_float(q.y), xcol[(k4 * 4 + 1 < C) ? k4 * 4 + 1 : 0], acc);
                            if (k4 * 4 + 2 < i) acc = fmaf(__uint_as_float(q.z), xcol[(k4 * 4 + 2 < C) ? k4 * 4 + 2 : 0], acc);
                            if (k4 * 4 + 3 < i) acc = fmaf(__uint_as_float(q.w), xcol[(k4 * 4 + 3 < C) ? k4 * 4 + 3 : 0], acc);
                        }
                        xcol[i] = (i > il) ? acc : ((i == il) ? 1.f : 0.f);
                    }
                }
                compute_barrier();  // everyone has read Abar
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    const uint32_t addr = scratch_a + (cb + i) * (4 * C) + (swz<CPRF>(i, il >> 2) << 4) + (il & 3) * 4;
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(xcol[i]) : "memory");
                }
            } else {
                if constexpr (MODE == INV_FWDSUBST_BLOCKED) compute_barrier();
                compute_barrier();
            }
            }
            compute_barrier();
            // back to rows: a[] = far part of this thread's columns, lb[] = band part
            if (active) {
#pragma unroll
                for (int c = 0; c < CPTF; ++c) {
                    const uint4 q = lds128(rowf + (swz<CPRF>(t, (col0 >> 2) + c) << 4));
                    a[c * 4 + 0] = __uint_as_float(q.x);
                    a[c * 4 + 1] = __uint_as_float(q.y);
                    a[c * 4 + 2] = __uint_as_float(q.z);
                    a[c * 4 + 3] = __uint_as_float(q.w);
                }
#pragma unroll
                for (int jl = 0; jl < HC; ++jl) a[jl] = (il - (col0 + jl) > NB) ? a[jl] : 0.f;
            }
#pragma unroll
            for (int e = 1; e <= NB; ++e) {
                const int j = il - e;
                lb[e] = (j >= 0) ? lds32f(rowf + (swz<CPRF>(t, j >> 2) << 4) + (j & 3) * 4) : 0.f;
            }
            compute_barrier();  // the fp32 rows are dead; the packed rows may overwrite them
        }

        // ---- packed bf16 form of the band: I + L (the keep-mask, 0 on the band and diagonal, was built before the loop)
        uint32_t bpT[PCH];
        if (active) {
            uint16_t vals[NB + 1];
            vals[0] = 0x3F80u;  // 1.0
#pragma unroll
            for (int e = 1; e <= NB; ++e) vals[e] = bf16_bits(lb[e]);
            build_band_row<C, NB>(br_line, slot, vals, bpT);
        } else {
#pragma unroll
            for (int i = 0; i < PCH; ++i) bpT[i] = 0u;
        }

        if constexpr (MODE == INV_NEUMANN) {
            // ---- residual correction T = T0 sum_{s<=S} E^s (Eq. 13). With X_m = T0 sum_{s<=m} E^s:
            //   X_{m+1} = T0 + X_m E   and   X_{2m+1} = X_m + X_m E^{m+1}.
            if constexpr (DBL != 0) {
                {
                    constexpr bool kFull = (DBL == 15);
                    // Four dependent products instead of eight: X_1 = T0 + T0 E and E^2; X_3 = X_1 + X_1 E^2 and E^4;
                    // X_4 = T0 + X_3 E; X_8 = X_3 + X_4 E^4. With S = 15 (kFull) the last two levels are
                    // X_7 = X_3 + X_3 E^4 and E^8; X_15 = X_7 + X_7 E^8, which is the exact inverse at N = 3
                    // because E^16 = 0 (the Newton-Schulz / factorised form of Eq. 12-13 with the same four levels).
                    // Each level is one MMA per chunk m (M = 128, N = 64,
                    // K = 64) whose A operand holds the X rows of chunk m on the chunk's own 64 lanes and the rows of
                    // the power of E_m on the other 64 lanes, so the product of both with the level's B operand
                    // (E_m, E_m^2 or E_m^4) comes out of the same instruction. A thread therefore owns, besides its
                    // part of row il of X of its chunk, the same part of row il of the powers of the OTHER chunk's E.
                    const int co = cb ^ 64;  // first tile row of the other chunk
                    const uint32_t a_own = lane_base + kAS + (kPerm ? 0 : (cb >> 1)) + h * 16;
                    const uint32_t a_oth = lane_base + kAS + (kPerm ? 32 : (co >> 1)) + h * 16;
                    const uint32_t d_own = lane_base + kR0 + (kPerm ? 0 : cb) + h * 32;
                    const uint32_t d_oth = lane_base + kR0 + (kPerm ? 64 : co) + h * 32;
                    uint8_t* sQB = sEB + 16384;  // powers of E as B operand, same layout as E
                    const uint32_t b_oth = ((co + col0) >> 3) * 1024 + il * 16;
                    const uint32_t idesc_h = instr_desc(128, 64, 1, 1, 0, 1, 1);
                    tmem_st16(a_own, bpT);
                    // the band words are parked in the idle R2 columns of the row's own lane during the levels (they come
                    // back 8 at a time with the accumulator reads, and as a whole afterwards): 16 registers less there
                    constexpr bool kParkBand = !MERGE && EX != 0;  // (in the default instantiation, which has no spills, the extra TMEM reads cost more than they save)
                    if constexpr (kParkBand) tmem_st16(lane_base + kR2 + h * 16, bpT);
                    compute_barrier();  // E of every row is in shared memory
                    {
                        uint32_t r16[16];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint4 v = *reinterpret_cast<const uint4*>(sEB + b_oth + j * 1024);
                            r16[4 * j + 0] = v.x; r16[4 * j + 1] = v.y; r16[4 * j + 2] = v.z; r16[4 * j + 3] = v.w;
                        }
                        tmem_st16(a_oth, r16);
                    }
                    fence_proxy_async_smem();
                    tmem_wait_st();
#pragma unroll
                    for (int lv = 0; lv < 4; ++lv) {
                        tc_fence_before_sync();
                        compute_barrier();
                        if (warp == 0) {
                            tc_fence_after_sync();
                            const uint32_t bb = (lv == 0 || (lv == 2 && !kFull)) ? sEB_a : sEB_a + 16384;
                            if (elect_one()) {
                            if constexpr (kPerm) {
                                // with B_m (E_m or one of its powers): the X rows of chunk m, on that chunk's half-lanes
                                // (operand columns 0..31 -> accumulator columns 0..63), and the rows of the power of E_m,
                                // which the threads of the OTHER chunk hold (columns 32..63 -> 64..127), while a power is
                                // still needed
                                constexpr uint32_t idesc_p = instr_desc(64, 64, 1, 1, 0, 1, 1);
                                const bool powers = lv < (kFull ? 3 : 2);
#pragma unroll
                                for (int m = 0; m < 2; ++m) {
                                    const uint32_t lm = static_cast<uint32_t>(16 * m) << 16, lo = static_cast<uint32_t>(16 * (1 - m)) << 16;
#pragma unroll
                                    for (int ks = 0; ks < 4; ++ks) {
                                        const uint64_t bd = smem_desc(bb + m * 8192 + ks * 256, 128, 1024, SWZ_NONE);
                                        mma_f16_ts(tmem + kR0 + lm, tmem + kAS + ks * 8 + lm, bd, idesc_p, ks > 0);
                                    }
                                    if (powers) {
#pragma unroll
                                        for (int ks = 0; ks < 4; ++ks) {
                                            const uint64_t bd = smem_desc(bb + m * 8192 + ks * 256, 128, 1024, SWZ_NONE);
                                            mma_f16_ts(tmem + kR0 + 64 + lo, tmem + kAS + 32 + ks * 8 + lo, bd, idesc_p, ks > 0);
                                        }
                                    }
                                }
                            } else {
#pragma unroll
                            for (int m = 0; m < 2; ++m) {
#pragma unroll
                                for (int ks = 0; ks < 4; ++ks) {
                                    const uint64_t bd = smem_desc(bb + m * 8192 + ks * 256, 128, 1024, SWZ_NONE);
                                    mma_f16_ts(tmem + kR0 + 64 * m, tmem + kAS + 32 * m + ks * 8, bd, idesc_h, ks > 0);
                                }
                            }
                            }
                            mma_commit(&bar_mma);
                            }
                        }
                        if (!wait_mma()) { ok = false; break; }
                        tc_fence_after_sync();
                        // in two halves of 16 columns, to keep the live registers down
#pragma unroll
                        for (int hh = 0; hh < 2; ++hh) {
                            uint32_t d[16], bph[8];
                            tmem_ld16(d_own + hh * 16, d);
                            if constexpr (kParkBand) {
                                if (lv < 3) tmem_ld8(lane_base + kR2 + h * 16 + hh * 8, bph);
                            } else {
#pragma unroll
                                for (int i = 0; i < 8; ++i) bph[i] = bpT[hh * 8 + i];
                            }
                            tmem_wait_ld();
                            if (lv == 0) {
#pragma unroll
                                for (int j = 0; j < 16; ++j) a[hh * 16 + j] = __uint_as_float(d[j]);
                            } else if (lv != 2 || kFull) {
#pragma unroll
                                for (int j = 0; j < 16; j += 2)
                                    unpair2(add2(pair2(a[hh * 16 + j], a[hh * 16 + j + 1]), pair2(__uint_as_float(d[j]), __uint_as_float(d[j + 1]))),
                                            a[hh * 16 + j], a[hh * 16 + j + 1]);
                            }
                            if (lv < 3) {
                                uint32_t pk[8];
#pragma unroll
                                for (int i = 0; i < 8; ++i) {
                                    const uint32_t w = (lv == 2 && !kFull) ? pack_bf16x2(__uint_as_float(d[2 * i]), __uint_as_float(d[2 * i + 1]))
                                                                 : pack_bf16x2(a[hh * 16 + 2 * i], a[hh * 16 + 2 * i + 1]);
                                    pk[i] = (kKeepMask ? (w & keep[hh * 8 + i]) : w) | bph[i];
                                }
                                tmem_st8(a_own + hh * 8, pk);
                            }
                        }
                        if (lv < (kFull ? 3 : 2)) {
#pragma unroll
                            for (int hh = 0; hh < 2; ++hh) {
                                uint32_t q[16], pq[8];
                                tmem_ld16(d_oth + hh * 16, q);
                                tmem_wait_ld();
#pragma unroll
                                for (int i = 0; i < 8; ++i) pq[i] = pack_bf16x2(__uint_as_float(q[2 * i]), __uint_as_float(q[2 * i + 1]));
                                if (lv < (kFull ? 2 : 1)) tmem_st8(a_oth + hh * 8, pq);
#pragma unroll
                                for (int j2 = 0; j2 < 2; ++j2)
                                    *reinterpret_cast<uint4*>(sQB + b_oth + (hh * 2 + j2) * 1024) =
                                        make_uint4(pq[4 * j2], pq[4 * j2 + 1], pq[4 * j2 + 2], pq[4 * j2 + 3]);
                            }
                            fence_proxy_async_smem();
                        }
                        if (lv < 3) tmem_wait_st();
                    }
                    if (!ok) break;
                    if constexpr (kParkBand) {
                        tmem_ld16(lane_base + kR2 + h * 16, bpT);
                        tmem_wait_ld();
                    }
                }
            } else {
            // one product per term: A_k = T0 + Z_k (bf16, TMEM), Z_{k+1} = A_k E, T = T0 + Z_S
            for (int k = 0; k < S; ++k) {
                if (active) {
                    uint32_t pk[PCH];
                    if (k == 0) {
#pragma unroll
                        for (int i = 0; i < PCH; ++i) pk[i] = bpT[i];
                    } else {
#pragma unroll
                        for (int i = 0; i < PCH; ++i) {
                            const uint32_t w = pack_bf16x2(a[2 * i], a[2 * i + 1]);
                            pk[i] = (kKeepMask ? (w & keep[i]) : w) | bpT[i];
                        }
                    }
                    store_stacked_operand<C>(lane_base + kAS, h, pk);
                    fence_proxy_async_smem();
                    tmem_wait_st();
                }
                tc_fence_before_sync();
                compute_barrier();
                if (warp == 0) {
                    // [Z_1; Z_2; ...] <- [A_1; A_2; ...] [E_1 | E_2 | ...]: M = 128, N = 128, K = C; row t keeps
                    // the C columns of its own chunk
                    tc_fence_after_sync();
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < C / 16; ++ks) {
                            const uint64_t bd = smem_desc(sEB_a + ks * 256, 128, 16 * C, SWZ_NONE);
                            mma_f16_ts(tmem + kR0, tmem + kAS + ks * 8, bd, idesc_c, ks > 0);
                        }
                        mma_commit(&bar_mma);
                    }
                }
                if (!wait_mma()) { ok = false; break; }
                tc_fence_after_sync();
                if (active) load_diag_block<C>(lane_base, kR0, t, h, a);
            }
            }
            if (!ok) break;
            if (S == 0) {
#pragma unroll
                for (int j = 0; j < HC; ++j) a[j] = 0.f;
            }
        }
        // a[] = this thread's part of the far row (T - I - L)

        // MERGE, rows of the second block: A21 part, then Y, then T21 (columns of the first block). Without the optional
        // prologue the T21 part is consumed (Tinv staging, W/U operand) at the end of the merge, which ends its live
        // range there; with it the operand is rebuilt for U, so the values stay in registers (y[]).
        constexpr bool Y_EARLY = MERGE && !EX;
        constexpr int YN = (MERGE && !Y_EARLY) ? HC : 1;
        float y[YN];
#pragma unroll
        for (int j = 0; j < YN; ++j) y[j] = 0.f;
        uint32_t yp[Y_EARLY ? PCH : 1];  // Y_EARLY: the T21 part as packed bf16, for the Tinv staging line
        yp[0] = 0u;
        if constexpr (MERGE) {
            float yl[Y_EARLY ? HC : 1];
            float* ym;
            if constexpr (Y_EARLY) {
                ym = yl;
#pragma unroll
                for (int j = 0; j < HC; ++j) yl[j] = 0.f;
            } else {
                ym = y;
            }
            const uint32_t idesc_m = instr_desc(128, 64, 1, 1, 0, 1, 1);
            // Both products of the merge cancel strongly when the keys of a chunk are correlated (A21 has entries
            // near 1, Y = A21 T11 is small), so every operand goes in as hi + lo (two bf16 halves) and each product
            // is hi*hi + lo*hi + hi*lo; the identity parts stay in fp32.
            if (wq >= 2) {
                // second block: A21_ij = beta_i e^{g_i - g_j} G_ij, j in the first block (fp32); its hi and lo halves
                // are the A operands (AS columns 0..31 and 32..63). In two halves of 16 columns to keep the live
                // registers down.
                const float gs = gi_ * kLog2e;
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    uint32_t gq[16];
                    tmem_ld16(lane_base + kR2 + hh * 32 + h * 16, gq);
                    tmem_wait_ld();
#pragma unroll
                    for (int j4 = 0; j4 < 4; ++j4) {
                        const int j0 = hh * 16 + j4 * 4;
                        const float4 gv = lds128f(sg_a + (col0 + j0) * 4);
                        const float gj[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            ym[j0 + q] = bi * rni * (f_l2 ? srn[col0 + j0 + q] : 1.f) * fast_exp2(fmaf(-gj[q], kLog2e, gs)) *
                                         __uint_as_float(gq[j4 * 4 + q]);
                    }
                    uint32_t ph[8], pl[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float v0 = ym[hh * 16 + 2 * i], v1 = ym[hh * 16 + 2 * i + 1];
                        ph[i] = pack_bf16x2(v0, v1);
                        pl[i] = pack_bf16x2(v0 - bf16_lo(ph[i]), v1 - bf16_hi(ph[i]));
                    }
                    tmem_st8(lane_base + kAS + h * 16 + hh * 8, ph);
                    tmem_st8(lane_base + kAS + 32 + h * 16 + hh * 8, pl);
                }
            }
            // X = T - I of the row's diagonal block (band without the unit diagonal + far part) as hi and lo halves:
            // X11 rows are the B operands of the first product ([64 x 64], MN-major, no swizzle; hi at 0, lo at 8 KB),
            // X22 rows the A operands of the second (R2 columns 0..31 and 32..63; this half's part of the Gram block there has been read).
            // One half (hi, then lo) and 16 columns at a time, stored at once, to keep the live registers down.
            {
                uint16_t vals[NB + 1];
                vals[0] = 0;
#pragma unroll
                for (int e = 1; e <= NB; ++e) vals[e] = bf16_bits(lb[e]);
#pragma unroll
                for (int part = 0; part < 2; ++part) {
                    uint32_t bp[PCH];
                    if (part == 1) {
#pragma unroll
                        for (int e = 1; e <= NB; ++e) vals[e] = bf16_bits(lb[e] - bf16_bits_to_f32(vals[e]));
                    }
                    build_band_row<C, NB>(br_line, slot, vals, bp);
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        uint32_t x[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int k = hh * 8 + i;
                            uint32_t w = pack_bf16x2(a[2 * k], a[2 * k + 1]);
                            if (part == 1) w = pack_bf16x2(a[2 * k] - bf16_lo(w), a[2 * k + 1] - bf16_hi(w));
                            x[i] = (kKeepMask ? (w & keep[k]) : w) | bp[k];
                        }
                        if (wq < 2) {
#pragma unroll
                            for (int c = 0; c < 2; ++c)
                                *reinterpret_cast<uint4*>(sEB + part * 8192 + ((col0 >> 3) + hh * 2 + c) * 1024 + t * 16) =
                                    make_uint4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
                        } else {
                            tmem_st8(lane_base + kR2 + part * 32 + h * 16 + hh * 8, x);
                        }
                    }
                }
            }
            // The far part a[] is not needed during the two products: it is parked in accumulator columns 64..127 of the
            // row's own lane (the products have N = 64) and comes back for the W / U operands, which frees 32 registers
            // where the T21 part, its packed halves and the accumulator reads are live.
            if constexpr (Y_EARLY) {
                uint32_t pa[HC];
#pragma unroll
                for (int j = 0; j < HC; ++j) pa[j] = __float_as_uint(a[j]);
                tmem_st32(lane_base + kR0 + 64 + h * 32, pa);
            }
            tmem_wait_st();
#pragma unroll 1
            for (int step = 0; step < 2; ++step) {
                fence_proxy_async_smem();
                tc_fence_before_sync();
                compute_barrier();
                if (warp == 0) {
                    tc_fence_after_sync();
                    if (elect_one()) {
                        const uint32_t a_hi = tmem + (step == 0 ? kAS : kR2), a_lo = a_hi + 32;
#pragma unroll
                        for (int part = 0; part < 3; ++part) {
                            // hi*hi, lo*hi, hi*lo
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks) {
                                const uint64_t bd = smem_desc(sEB_a + (part == 2 ? 8192 : 0) + ks * 256, 128, 1024, SWZ_NONE);
                                mma_f16_ts(tmem + kR0, (part == 1 ? a_lo : a_hi) + ks * 8, bd, idesc_m, part > 0 || ks > 0);
                            }
                        }
                        mma_commit(&bar_mma);
                    }
                }
                if (!wait_mma()) { ok = false; break; }
                tc_fence_after_sync();
                if (wq >= 2) {
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        uint32_t d[16];
                        tmem_ld16(lane_base + kR0 + h * 32 + hh * 16, d);
                        tmem_wait_ld();
                        if (step == 0) {
                            // Y = A21 + A21 X11; Y rows (hi, lo) become the B operands of X22 Y
#pragma unroll
                            for (int j = 0; j < 16; ++j) ym[hh * 16 + j] += __uint_as_float(d[j]);
#pragma unroll
                            for (int c = 0; c < 2; ++c) {
                                const int j0 = hh * 16 + c * 8;
                                uint32_t wh[4], wl[4];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const float v0 = ym[j0 + 2 * i], v1 = ym[j0 + 2 * i + 1];
                                    wh[i] = pack_bf16x2(v0, v1);
                                    wl[i] = pack_bf16x2(v0 - bf16_lo(wh[i]), v1 - bf16_hi(wh[i]));
                                }
                                const uint32_t off = ((col0 >> 3) + hh * 2 + c) * 1024 + il * 16;
                                *reinterpret_cast<uint4*>(sEB + off) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
                                *reinterpret_cast<uint4*>(sEB + 8192 + off) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
                            }
                        } else {
                            // T21 = -(Y + X22 Y)
#pragma unroll
                            for (int j = 0; j < 16; ++j) ym[hh * 16 + j] = -(ym[hh * 16 + j] + __uint_as_float(d[j]));
                        }
                    }
                }
            }
            if (!ok) break;
            if constexpr (Y_EARLY) {
                // the row's part of the other block column of Tinv (T21, or the zeros above it), packed for the
                // staging line (which overlaps the band-row lines that the W/U operands still need)
#pragma unroll
                for (int i = 0; i < PCH; ++i) yp[i] = pack_bf16x2(ym[2 * i], ym[2 * i + 1]);
                // T21 diag(beta): the first-block columns of the W/U operand of the second block's rows
                if (wq >= 2) {
                    const uint32_t sb_a = smem_u32(sbeta + col0);
                    uint32_t po[PCH], pl[PCH];
#pragma unroll
                    for (int i = 0; i < PCH / 2; ++i) {
                        const float4 bb = lds128f(sb_a + i * 16);
                        const float v0 = ym[4 * i] * bb.x, v1 = ym[4 * i + 1] * bb.y, v2 = ym[4 * i + 2] * bb.z, v3 = ym[4 * i + 3] * bb.w;
                        po[2 * i] = pack_bf16x2(v0, v1);
                        po[2 * i + 1] = pack_bf16x2(v2, v3);
                        pl[2 * i] = pack_bf16x2(v0 - bf16_lo(po[2 * i]), v1 - bf16_hi(po[2 * i]));
                        pl[2 * i + 1] = pack_bf16x2(v2 - bf16_lo(po[2 * i + 1]), v3 - bf16_hi(po[2 * i + 1]));
                    }
                    store_stacked_operand<C>(lane_base + kAS, h, po);
                    store_stacked_operand<C>(lane_base + kR2, h, pl);  // the lo operand keeps these columns (see build_wu_operands)
                }
            }
        }

        if constexpr (MERGE && !EX) {
            uint32_t pa[HC];
            tmem_ld32(lane_base + kR0 + 64 + h * 32, pa);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < HC; ++j) a[j] = __uint_as_float(pa[j]);
        }
        // ---- A operands for W/U: T diag(scale) = hi + lo, hi over the whole row, lo only on band + diagonal.
        // scale = beta for U; for W it is beta / ||K|| when the keys are normalised on the fly, else beta as well
        if (active) {
            build_wu_operands<C, NB, MERGE, MERGE && !Y_EARLY, kKeepMask, kPerm>(lane_base, br_line, slot, t, h, il, cb, col0, wq, two_scales ? sbrn : sbeta,
                                            two_scales ? sbrn[t] : bi, a, keep, lb, y);
            if constexpr (MERGE) {
                // I + L again for the Tinv rows: rebuilt here instead of being carried across the merge, where
                // registers are scarce (it must be built before the barrier below: the Tinv staging lines of other
                // rows overlap this row's private line)
                uint16_t vals[NB + 1];
                vals[0] = 0x3F80u;
#pragma unroll
                for (int e = 1; e <= NB; ++e) vals[e] = bf16_bits(lb[e]);
                build_band_row<C, NB>(br_line, slot, vals, bpT);
            }
            tmem_wait_st();
        }
        tc_fence_before_sync();
        compute_barrier();
        if (warp == 0) {
            // W = (hi + lo) K: A operands in TMEM (AS: high bf16 half, R2: low half of the band),
            // B = the K tile read as an MN-major operand (both 64-column sub-tiles, N = 128)
            tc_fence_after_sync();
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < (kPerm ? 0 : 16); ++ks) {
                    const uint64_t bd = smem_desc(sK_a + (ks & 7) * 2048, 16384, 1024, SWZ_128B);
                    mma_f16_ts(tmem + kR0, tmem + ((ks < 8) ? kAS : kR2) + (ks & 7) * 8, bd, idesc_w, ks > 0);
                }
                if constexpr (kPerm) issue_wu64(sK_a);
                mma_commit(&bar_mma);
            }
        }

        if constexpr (EX != 0) {
            TilePos pc = pos_cur;
            asm volatile("" : "+r"(pc.gi), "+r"(pc.tt), "+r"(pc.bhk));  // (formed here, not carried from the tile's top)
            tc = tile_coord<EX>(pc, p);
        }
        // With the optional prologue the U operand can differ from the W operand (two_scales) and is rebuilt from the row.
        // That happens right after the W product completes and BEFORE its accumulator is read, so that the row's
        // registers are dead while the epilogue holds its 64; the band-row lines must survive until then, so the Tinv
        // rows are staged in the E-operand region (dead since the last round) instead of over the band-row lines.
        constexpr bool kEarlyU = EX != 0 && !MERGE;
        constexpr int kTinvStage = kEarlyU ? L::kEB : L::kBR;
        // ---- T row -> Tinv: each half-row goes to a staging line in the TMA swizzle layout (the band-row
        // region is free now); one bulk tensor store of 32 rows x HC columns per warp, overlapping the W products
        if (f_f32 && p.Tinv != nullptr && active) {
            // fp32 outputs (parity debugging): the row part straight from registers, 16-byte stores
            const bool rv = (tc.t0 + t) < p.T;
            constexpr int COUT = MERGE ? 128 : C;
            float* trow = reinterpret_cast<float*>(p.Tinv) + ((long long)tc.bhv * p.T + tc.t0 + t) * COUT;
            if (rv) {
                const int dcol = (MERGE ? cb : 0) + col0;  // first output column of the diagonal-block part
#pragma unroll
                for (int c = 0; c < HC / 4; ++c) {
                    float v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int jl = c * 4 + q;
                        const int d = il - (col0 + jl);
                        float x = a[jl];
                        if (d == 0) x = 1.f;
#pragma unroll
                        for (int e = 1; e <= NB; ++e)
                            if (d == e && e <= n_band) x = lb[e];
                        v[q] = x;
                    }
                    *reinterpret_cast<float4*>(trow + dcol + c * 4) = make_float4(v[0], v[1], v[2], v[3]);
                }
                if constexpr (MERGE && !Y_EARLY) {
                    const int ocol = (wq >= 2 ? 0 : 64) + col0;  // T21 part, or the zero block above it
#pragma unroll
                    for (int c = 0; c < HC / 4; ++c)
                        *reinterpret_cast<float4*>(trow + ocol + c * 4) = make_float4(y[c * 4], y[c * 4 + 1], y[c * 4 + 2], y[c * 4 + 3]);
                }
            }
        } else if (MERGE && p.Tinv != nullptr) {
          if constexpr (MERGE) {
            // rows of the 128 x 128 inverse in four column groups of 32 (64-byte lines, 64-byte TMA swizzle):
            // the row's diagonal-block part, and its part of the other block column (T21, or zeros above it)
            const int gd = (cb >> 5) + h;                  // group of the diagonal-block part
            const int go = (wq >= 2) ? h : (2 + h);        // group of the off-diagonal part
            const uint32_t rowd = scratch_a + gd * 8192 + t * 64;
            const uint32_t rowo = scratch_a + go * 8192 + t * 64;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                sts128(rowd + (swz<4>(t, c) << 4),
                       (kKeepMask ? (pack_bf16x2(a[c * 8 + 0], a[c * 8 + 1]) & keep[c * 4 + 0]) : pack_bf16x2(a[c * 8 + 0], a[c * 8 + 1])) | bpT[c * 4 + 0],
                       (kKeepMask ? (pack_bf16x2(a[c * 8 + 2], a[c * 8 + 3]) & keep[c * 4 + 1]) : pack_bf16x2(a[c * 8 + 2], a[c * 8 + 3])) | bpT[c * 4 + 1],
                       (kKeepMask ? (pack_bf16x2(a[c * 8 + 4], a[c * 8 + 5]) & keep[c * 4 + 2]) : pack_bf16x2(a[c * 8 + 4], a[c * 8 + 5])) | bpT[c * 4 + 2],
                       (kKeepMask ? (pack_bf16x2(a[c * 8 + 6], a[c * 8 + 7]) & keep[c * 4 + 3]) : pack_bf16x2(a[c * 8 + 6], a[c * 8 + 7])) | bpT[c * 4 + 3]);
                if constexpr (Y_EARLY)
                    sts128(rowo + (swz<4>(t, c) << 4), yp[c * 4 + 0], yp[c * 4 + 1], yp[c * 4 + 2], yp[c * 4 + 3]);
                else
                    sts128(rowo + (swz<4>(t, c) << 4), pack_bf16x2(y[c * 8 + 0], y[c * 8 + 1]), pack_bf16x2(y[c * 8 + 2], y[c * 8 + 3]),
                           pack_bf16x2(y[c * 8 + 4], y[c * 8 + 5]), pack_bf16x2(y[c * 8 + 6], y[c * 8 + 7]));
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                tma_store_3d(&tmT, smem + L::kEB + gd * 8192 + wrow0 * 64, gd * 32, tc.t0 + wrow0, tc.bhv);
                tma_store_3d(&tmT, smem + L::kEB + go * 8192 + wrow0 * 64, go * 32, tc.t0 + wrow0, tc.bhv);
                tma_store_commit();
            }
          }
        } else if (p.Tinv != nullptr && active) {
            constexpr int RB = HC * 2;  // bytes per staged half-row
            const uint32_t stage = smem_u32(smem + kTinvStage) + h * (kTile * RB);
            const int srow = kPerm ? lrow : t;  // (kPerm: a warp's 32 lanes hold 16 rows of each chunk; staged in lane order)
            const uint32_t trow = stage + srow * RB;
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                sts128(trow + (swz<CPT>(srow, c) << 4),
                       (kKeepMask ? (pack_bf16x2(a[c * 8 + 0], a[c * 8 + 1]) & keep[c * 4 + 0]) : pack_bf16x2(a[c * 8 + 0], a[c * 8 + 1])) | bpT[c * 4 + 0],
                       (kKeepMask ? (pack_bf16x2(a[c * 8 + 2], a[c * 8 + 3]) & keep[c * 4 + 1]) : pack_bf16x2(a[c * 8 + 2], a[c * 8 + 3])) | bpT[c * 4 + 1],
                       (kKeepMask ? (pack_bf16x2(a[c * 8 + 4], a[c * 8 + 5]) & keep[c * 4 + 2]) : pack_bf16x2(a[c * 8 + 4], a[c * 8 + 5])) | bpT[c * 4 + 2],
                       (kKeepMask ? (pack_bf16x2(a[c * 8 + 6], a[c * 8 + 7]) & keep[c * 4 + 3]) : pack_bf16x2(a[c * 8 + 6], a[c * 8 + 7])) | bpT[c * 4 + 3]);
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                if constexpr (kPerm) {
#pragma unroll
                    for (int m = 0; m < 2; ++m)
                        tma_store_3d(&tmT, smem + kTinvStage + h * (kTile * RB) + (wrow0 + 16 * m) * RB, col0, tc.t0 + 64 * m + 16 * wq, tc.bhv);
                } else {
                    tma_store_3d(&tmT, smem + kTinvStage + h * (kTile * RB) + wrow0 * RB, col0, tc.t0 + wrow0, tc.bhv);
                }
                tma_store_commit();
            }
        }

        // ---- W, then U: each thread reads 64 accumulator columns of its row -> bf16 -> swizzled staging
        // sub-tile of its warp -> one bulk tensor store (32 rows x 64 columns) per warp
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            if (!wait_mma()) { ok = false; break; }
            tc_fence_after_sync();
            if (warp == 0 && has_next && elect_one()) {
                // the products that read this tile's K (half 0) or V (half 1) are complete: prefetch the next tile's
                const TileCoord nc = tile_coord<EX>(pos_next, p);
                if (half == 0)
                    load_tile(sK, &tmK, &bar_k, nc.kx, nc.t0, nc.kz);
                else
                    load_tile(sV, &tmV, &bar_v, nc.vx, nc.t0, nc.vz);
            }
            if constexpr (kEarlyU) {
                if (half == 0 && two_scales && active) {
                    // U uses beta where W used beta / ||K|| (or beta exp(g)): both A operands again (the W product has
                    // completed; the hand-over to the issuing thread is the barrier below)
                    build_wu_operands<C, NB, MERGE, MERGE && !Y_EARLY, kKeepMask, kPerm>(lane_base, br_line, slot, t, h, il, cb, col0, wq, sbeta, bi, a, keep, lb, y);
                    tmem_wait_st();
                }
            }
            uint32_t o[32];
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 32) {
                uint32_t r[32];
                tmem_ld32(lane_base + kR0 + h * 64 + c0, r);
                tmem_wait_ld();
                if (f_f32) {
                    if ((tc.t0 + t) < p.T) {
                        float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(half == 0 ? p.W : p.U) +
                                                               (tc.r0 + (long long)t * tc.rs) * kD + h * 64 + c0);
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            dst[i] = make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]), __uint_as_float(r[4 * i + 2]),
                                                 __uint_as_float(r[4 * i + 3]));
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[c0 / 2 + i] = pack_bf16x2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
                }
            }
            if (half == 0) {
                // this warp's Tinv store has been read (the staging slices below overlap other warps' lines)
                if (lane == 0) tma_store_wait_read<0>();
                tc_fence_before_sync();
                compute_barrier();  // every row of the W accumulator has been read
                if (!kEarlyU && two_scales) {
                    // U uses beta where W used beta / ||K|| (or beta exp(g)): rebuild both A operands
                    if (active) {
                        build_wu_operands<C, NB, MERGE, MERGE && !Y_EARLY, kKeepMask, kPerm>(lane_base, br_line, slot, t, h, il, cb, col0, wq, sbeta, bi, a, keep, lb, y);
                        tmem_wait_st();
                    }
                    tc_fence_before_sync();
                    compute_barrier();
                }
                if (warp == 0) {
                    if (!wait_bar(&bar_v, par_kv)) ok = false;
                    if (ok) {
                        tc_fence_after_sync();
                        if (elect_one()) {
#pragma unroll
                            for (int ks = 0; ks < (kPerm ? 0 : 16); ++ks) {
                                const uint64_t bd = smem_desc(sV_a + (ks & 7) * 2048, 16384, 1024, SWZ_128B);
                                mma_f16_ts(tmem + kR0, tmem + ((ks < 8) ? kAS : kR2) + (ks & 7) * 8, bd, idesc_w, ks > 0);
                            }
                            if constexpr (kPerm) issue_wu64(sV_a);
                            mma_commit(&bar_mma);
                        }
                    }
                }
            }
            // variable-length sequences: a warp whose 32 rows are 32 consecutive real tokens stores them like the dense
            // path (token coordinate of its first row); otherwise (a short chunk, or two chunks that are not adjacent in
            // memory) every row of a real token goes out by itself, so that nothing reaches a neighbouring sequence
            bool bulk = true;
            int tok0 = tc.t0 + wrow0;
            if (f_var) {
                tok0 = __shfl_sync(0xFFFFFFFFu, gtok, 0);
                bulk = __all_sync(0xFFFFFFFFu, gtok >= 0 && gtok == tok0 + lane);
            }
            if (!f_f32 && !bulk) {
                if (gtok >= 0) {
                    const bool bthd = (p.flags & GDN_FLAG_LAYOUT_BTHD) != 0;
                    const long long row = bthd ? (long long)gtok * p.H_v + tc.bhv : (long long)tc.bhv * p.T_total + gtok;
                    uint4* dst = reinterpret_cast<uint4*>((half == 0 ? p.W : p.U) + row * kD + h * 64);
#pragma unroll
                    for (int c = 0; c < 8; ++c) dst[c] = make_uint4(o[c * 4 + 0], o[c * 4 + 1], o[c * 4 + 2], o[c * 4 + 3]);
                }
            } else if (!f_f32) {
                // 32 rows x 64 columns of this warp in the 128-byte TMA swizzle: 4 KB at slice(wq) + h * 4 KB
                const uint32_t sub = scratch_a + wq * 8192 + h * 4096;
                if (lane == 0) tma_store_wait_read<0>();  // earlier stores from this sub-tile have been read
                __syncwarp();
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    sts128(sub + lane * 128 + ((c ^ (lane & 7)) << 4), o[c * 4 + 0], o[c * 4 + 1], o[c * 4 + 2], o[c * 4 + 3]);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if constexpr (kPerm) {
#pragma unroll
                        for (int m = 0; m < 2; ++m)
                            tma_store_3d((half == 0) ? &tmW : &tmU, smem + L::kEB + wq * 8192 + h * 4096 + m * 2048, tc.vx + h * 64,
                                         tc.t0 + 64 * m + 16 * wq, tc.vz);
                    } else {
                        tma_store_3d((half == 0) ? &tmW : &tmU, smem + L::kEB + wq * 8192 + h * 4096, tc.vx + h * 64, tok0, tc.vz);
                    }
                    tma_store_commit();
                }
            }
        }
        par_kv ^= 1;
    }
    if (lane == 0) tma_store_wait_all<0>();
    if (!ok) atomicExch(p.status, GDN_ERR_TIMEOUT);

    tc_fence_before_sync();
    __syncthreads();
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

// [heads][T][cols] bf16 tensor, boxes of `box_rows` rows x `box_cols` columns with the given swizzle
bool make_map(CUtensorMap* tm, const void* base, long long heads, int T, int cols, int box_cols, int box_rows,
              CUtensorMapSwizzle swizzle) {
    EncodeTiledFn enc = get_encode_fn();
    if (enc == nullptr) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(T), static_cast<cuuint64_t>(heads)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(cols) * 2, static_cast<cuuint64_t>(T) * cols * 2};
    cuuint32_t box[3] = {static_cast<cuuint32_t>(box_cols), static_cast<cuuint32_t>(box_rows), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct Maps {
    CUtensorMap K, V, W, U, T;
};

template <int C, int NB, int MODE, bool MERGE, int EX, int DBL, bool PERM = false>
int launch_ex(const Maps& m, const Params& prm, cudaStream_t stream) {
    using L = Smem<C, NB>;
    const int smem = L::kTotal + 1024;
    auto kern = chunk_tc_kernel<C, NB, MODE, MERGE, EX, DBL, PERM>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return GDN_ERR_LAUNCH;
    long long grid = prm.n_tiles < 2 * kSMs ? prm.n_tiles : 2 * kSMs;
    Params q = prm;
    const long long y = grid / prm.group;
    q.s_gi = static_cast<int>(grid - y * prm.group);
    q.s_bhk = static_cast<int>(y / prm.n_mid);
    q.s_tt = static_cast<int>(y - static_cast<long long>(q.s_bhk) * prm.n_mid);
    kern<<<static_cast<int>(grid), kThreads, smem, stream>>>(m.K, m.V, m.W, m.U, m.T, q);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? GDN_OK : GDN_ERR_LAUNCH;
}

template <int C, int NB, int MODE, bool MERGE>
int launch_one(const Maps& m, const Params& prm, cudaStream_t stream, bool perm) {
    constexpr bool kNeu = (MODE == INV_NEUMANN);
    constexpr bool kDbl = kNeu && C == 64;
    const int dbl = !kDbl ? 0 : (prm.S == 8 ? 8 : (prm.S == 15 ? 15 : 0));
    if (kNeu && (prm.flags & GDN_FLAG_OUT_FP32) != 0) {
        if (dbl == 8) return launch_ex<C, NB, MODE, MERGE, kNeu ? 2 : 0, kDbl ? 8 : 0>(m, prm, stream);
        if (dbl == 15) return launch_ex<C, NB, MODE, MERGE, kNeu ? 2 : 0, kDbl ? 15 : 0>(m, prm, stream);
        return launch_ex<C, NB, MODE, MERGE, kNeu ? 2 : 0, 0>(m, prm, stream);
    }
    if (kNeu && prm.chunk_start != nullptr) {
        if (dbl == 8) return launch_ex<C, NB, MODE, MERGE, kNeu ? 3 : 0, kDbl ? 8 : 0>(m, prm, stream);
        if (dbl == 15) return launch_ex<C, NB, MODE, MERGE, kNeu ? 3 : 0, kDbl ? 15 : 0>(m, prm, stream);
        return launch_ex<C, NB, MODE, MERGE, kNeu ? 3 : 0, 0>(m, prm, stream);
    }
    if (kNeu && prm.flags != 0) {
        if (dbl == 8) return launch_ex<C, NB, MODE, MERGE, kNeu ? 1 : 0, kDbl ? 8 : 0>(m, prm, stream);
        if (dbl == 15) return launch_ex<C, NB, MODE, MERGE, kNeu ? 1 : 0, kDbl ? 15 : 0>(m, prm, stream);
        return launch_ex<C, NB, MODE, MERGE, kNeu ? 1 : 0, 0>(m, prm, stream);
    }
    if constexpr (kDbl && !MERGE) {
        // (the tensor maps of W, U and Tinv were built with 16-row boxes when `perm` is set: see launch_tc_bf16)
        if (perm && dbl == 8) return launch_ex<C, NB, MODE, MERGE, 0, 8, true>(m, prm, stream);
        if (perm && dbl == 15) return launch_ex<C, NB, MODE, MERGE, 0, 15, true>(m, prm, stream);
    }
    if (perm) return GDN_ERR_LAUNCH;  // (not reached: `perm` is only set for the cases above)
    if (dbl == 8) return launch_ex<C, NB, MODE, MERGE, 0, kDbl ? 8 : 0>(m, prm, stream);
    if (dbl == 15) return launch_ex<C, NB, MODE, MERGE, 0, kDbl ? 15 : 0>(m, prm, stream);
    return launch_ex<C, NB, MODE, MERGE, 0, 0>(m, prm, stream);
}

template <int C, int MODE, bool MERGE = false>
int launch_c(const Maps& m, const Params& prm, cudaStream_t stream, bool perm = false) {
    if (MODE != INV_NEUMANN || prm.N <= 3) return launch_one<C, 3, MODE, MERGE>(m, prm, stream, perm);
    return launch_one<C, 7, MODE, MERGE>(m, prm, stream, perm);
}

}  // namespace


namespace {
constexpr long long kM64MinTiles = 32768;  // 65 536 chunks of 64 tokens: a launch of 1.1 to 1.25 ms
// waits on an mbarrier that never completes: wait_bar must give up after its budget and report it
__global__ void wait_selftest_kernel(int* status) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    if (!wait_bar(&bar, 0) && threadIdx.x == 0) atomicExch(status, GDN_ERR_TIMEOUT);
}
}  // namespace

int launch_wait_selftest(cudaStream_t stream) {
    int* status = device_status_word();
    if (status == nullptr) return GDN_ERR_LAUNCH;
    wait_selftest_kernel<<<1, 32, 0, stream>>>(status);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? GDN_OK : GDN_ERR_LAUNCH;
}

int launch_tc_bf16(const Problem& p, InverseMode mode, cudaStream_t stream) {
    if (p.d_k != kD || p.d_v != kD) return GDN_ERR_UNSUPPORTED;
    if (!(p.C == 16 || p.C == 32 || p.C == 64 || p.C == 128)) return GDN_ERR_UNSUPPORTED;
    if (mode == INV_NEUMANN && (p.order < 1 || p.order > 7)) return GDN_ERR_UNSUPPORTED;
    if ((long long)p.B * p.H_v * p.T == 0) return GDN_OK;
    const bool varlen = p.chunk_start != nullptr;
    if (varlen && (mode != INV_NEUMANN || p.B != 1 || p.T % kTile != 0)) return GDN_ERR_UNSUPPORTED;
    int* status = device_status_word();
    if (status == nullptr) return GDN_ERR_LAUNCH;
    Maps m;
    const long long hk = (long long)p.B * p.H_k, hv = (long long)p.B * p.H_v;
    // Tinv leaves in boxes of 32 rows x (C/2 columns for C >= 32, else C columns): 64-, 32- and 32-byte lines
    const int tbox = (p.C == 128) ? 32 : ((p.C >= 32) ? p.C / 2 : p.C);
    const CUtensorMapSwizzle tsw = (tbox * 2 == 64) ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
    // head-major [B, H, T, d]: (d, T, B * H); token-major [B, T, H, d]: (H * d, T, B), the head picks the columns
    const bool bthd = (p.flags & GDN_FLAG_LAYOUT_BTHD) != 0;
    if (bthd && mode != INV_NEUMANN) return GDN_ERR_UNSUPPORTED;
    const long long zk = bthd ? p.B : hk, zv = bthd ? p.B : hv;
    const int ck = bthd ? p.H_k * kD : kD, cv = bthd ? p.H_v * kD : kD;
    // variable-length sequences: the inputs hold T_total tokens and are loaded one chunk per box (W and U leave
    // by plain stores there, their maps are not used)
    const int t_in = varlen ? p.T_total : p.T;
    const int in_rows = varlen ? p.C : 128;
    if (!make_map(&m.K, p.K, zk, t_in, ck, 64, in_rows, CU_TENSOR_MAP_SWIZZLE_128B)) return GDN_ERR_LAUNCH;
    if (!make_map(&m.V, p.V, zv, t_in, cv, 64, in_rows, CU_TENSOR_MAP_SWIZZLE_128B)) return GDN_ERR_LAUNCH;
    // Large launches of the default 64-chunk path (no flags, S = 8 or 15) run the form whose tensor-core products are
    // M = 64 instructions per chunk (kPerm in the kernel): it draws less power. Which form is faster depends on the state of
    // the GPU more than on the size. Default and M = 64, us, one launch after idle (full clocks) | launches back to back at
    // the power cap (1627 to 1770 and 1770 to 1920 MHz): 2048 tiles 85, 87 | 85.5, 82.7; 8192 296, 307 | 320, 310; 32768 1092, 1126 | 1257,
    // 1215; 131072 4182, 4314 | 4981, 4809; 1024 tiles do not reach the cap (45.5, 46.1). A launch of a millisecond or more
    // is taken for work that keeps the GPU at the cap, a shorter one not. Its warps hold 16 rows
    // of each of a tile's two chunks, so its W, U and Tinv rows leave in boxes of 16 rows. (GDN_FORCE_M64 = 1 / 0 in the
    // environment forces the choice: the tests run both forms on small cases.)
    const long long n_tiles_all = (long long)p.B * p.H_v * ((p.T + kTile - 1) / kTile);
    bool perm = p.C == 64 && mode == INV_NEUMANN && p.flags == 0 && !varlen && (p.steps == 8 || p.steps == 15);
    if (perm) {
        const char* force = getenv("GDN_FORCE_M64");
        perm = (force != nullptr) ? (force[0] == '1') : (n_tiles_all >= kM64MinTiles);
    }
    const int obox = perm ? 16 : 32;
    if (!make_map(&m.W, p.W, zv, t_in, cv, 64, obox, CU_TENSOR_MAP_SWIZZLE_128B)) return GDN_ERR_LAUNCH;
    if (!make_map(&m.U, p.U, zv, t_in, cv, 64, obox, CU_TENSOR_MAP_SWIZZLE_128B)) return GDN_ERR_LAUNCH;
    // Tinv rows are C wide; without a Tinv output the map points at W (never used by the kernel then)
    if (!make_map(&m.T, p.Tinv != nullptr ? p.Tinv : p.W, hv, p.T, p.Tinv != nullptr ? p.C : kD, p.Tinv != nullptr ? tbox : 64, obox,
                  p.Tinv != nullptr ? tsw : CU_TENSOR_MAP_SWIZZLE_128B))
        return GDN_ERR_LAUNCH;
    Params prm;
    prm.beta = p.beta;
    prm.g = p.g;
    prm.W = static_cast<__nv_bfloat16*>(p.W);
    prm.U = static_cast<__nv_bfloat16*>(p.U);
    prm.Tinv = static_cast<__nv_bfloat16*>(p.Tinv);
    prm.status = status;
    prm.H_k = p.H_k;
    prm.H_v = p.H_v;
    prm.T = p.T;
    prm.group = p.H_v / p.H_k;
    prm.n_tt = (p.T + kTile - 1) / kTile;
    prm.n_mid = bthd ? p.H_k : prm.n_tt;
    prm.N = p.order;
    prm.S = p.steps;
    prm.flags = p.flags;
    prm.chunk_start = p.chunk_start;
    prm.chunk_len = p.chunk_len;
    prm.n_chunks = p.n_chunks;
    prm.T_total = p.T_total;
    prm.n_tiles = (long long)p.B * p.H_v * prm.n_tt;
    if (prm.n_tiles >= (1LL << 31) - 4096 || (long long)p.B * p.H_v >= (1LL << 31)) return GDN_ERR_UNSUPPORTED;
    if (mode == INV_NEUMANN) {
        switch (p.C) {
            case 16: return launch_c<16, INV_NEUMANN>(m, prm, stream);
            case 32: return launch_c<32, INV_NEUMANN>(m, prm, stream);
            case 128: return launch_c<64, INV_NEUMANN, true>(m, prm, stream);
            default: return launch_c<64, INV_NEUMANN>(m, prm, stream, perm);
        }
    }
    if (mode == INV_FWDSUBST_TC) {
        if (p.C != 64) return GDN_ERR_UNSUPPORTED;
        return launch_c<64, INV_FWDSUBST_TC>(m, prm, stream);
    }
    if (mode == INV_FWDSUBST_BLOCKED) {
        switch (p.C) {
            case 16: return launch_c<16, INV_FWDSUBST_BLOCKED>(m, prm, stream);
            case 32: return launch_c<32, INV_FWDSUBST_BLOCKED>(m, prm, stream);
            case 128: return launch_c<64, INV_FWDSUBST_BLOCKED, true>(m, prm, stream);
            default: return launch_c<64, INV_FWDSUBST_BLOCKED>(m, prm, stream);
        }
    }
    switch (p.C) {
        case 16: return launch_c<16, INV_FWDSUBST_ROWS>(m, prm, stream);
        case 32: return launch_c<32, INV_FWDSUBST_ROWS>(m, prm, stream);
        case 128: return launch_c<64, INV_FWDSUBST_ROWS, true>(m, prm, stream);  // 64-blocks by substitution, merged by App. E
        default: return launch_c<64, INV_FWDSUBST_ROWS>(m, prm, stream);
    }
}

}  // namespace gdn
