// Plain-FMA (no tensor core) kernel for the chunk-prepare path: one chunk per CTA (or one chunk per few CTAs when a
// launch has fewer chunks than the chip has SMs), every matrix of the chunk in shared memory, fp32 arithmetic throughout.
//
// It serves the fp32 configuration (tolerance 1e-5 against the fp64 definition), small and
// odd chunk sizes, and the forward-substitution comparisons (Eq. 2-3, App. E). The scheme of
// Sec. 3 is evaluated through its structure rather than as dense products:
//   * the band L = T0 - I (1 <= i-j <= N) by the distance recursion
//       L_d[i] = Abar[i][i-d] + sum_{e<d} Abar[i][i-e] L_{d-e}[i-e],
//     which equals the band of sum_{n<=N} Abar^n (a band entry at distance d only receives powers n <= d);
//   * E = Abar + Abar L on i-j > N (Eq. 13 with T0 = I + L; exactly zero inside the band), N multiply-adds per entry;
//   * X_0 = T0, X_{k+1} = T0 + X_k E for k < S (so X_S = T0 sum_{s<=S} E^s); round k changes entries with i - j >= (k+1)(N+1)
//     only, so block diagonals leave the rounds one by one (114 instead of 160 block products at C = 64, N = 3, S = 8; the
//     doubling form with powers of E needs 90 but squares E: where the series has not converged its fp32 error is up to
//     100 times larger, so it is not used);
//   * App. E's two-block formula for C = 128.
//
// What bounds it: the shared-memory reads that feed the FMA pipe (two thirds of their peak, the pipe at 41 %), and in short
// launches the chain of a chunk. Every product is a dot product of two ROWS held in shared memory (E is kept transposed), so
// one 16-byte read brings four terms of the sum: a thread holds the entries (ti + G r, tj + G s), r >= s, reads R + R rows per
// four terms and does 2 * 10 packed multiply-adds (fma.rn.f32x2) with them at R = 4. The stride of G between a thread's rows
// keeps the triangle's zero blocks the same for every thread (10 of 16 block pairs, 20 of 64 block triples) and the row pitch
// of 4 (mod 8) words keeps the reads free of bank conflicts. C = 64, d = 128: 1024 chunks 111 us (one entry per thread and
// step, two scalar reads per multiply-add: 1016 us), 8 chunks 21 us (216 us).
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace gdn {
namespace {

constexpr int kSliceW = 128;  // features of K (V) held in shared memory at a time
constexpr int kLdk = kSliceW + 4;

__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16* p, float4 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}
__device__ __forceinline__ void st(float* p, float v) { *p = v; }
__device__ __forceinline__ void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

using sm100::f2;
using sm100::pair2;
__device__ __forceinline__ void fma2(f2& acc, f2 a, f2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }
__device__ __forceinline__ float2 split2(f2 v) {
    float2 r;
    sm100::unpair2(v, r.x, r.y);
    return r;
}
__device__ __forceinline__ float sum2(f2 v) {
    const float2 r = split2(v);
    return r.x + r.y;
}

// Columns [0, w) of `rows` rows of a [rows, d] tile into shared memory as fp32 (row pitch kLdk), rows up to `pad` zero, columns
// up to the end of the last unit of UW too: the products run over whole units, and what an earlier kernel has left there must
// not reach the test for results that are not finite (d = 96 after a launch that left NaN: C = 64 173 instead of 81 us,
// C = 128 1112 instead of 241).
// fp32 arrives asynchronously: the caller waits (load_wait) and synchronises.
template <int NT, int UW>
__device__ __forceinline__ void load_tile(float* dst, const float* src, int rows, int pad, int d, int w) {
    const int c = (threadIdx.x & 31) << 2;
    if (c < (w + UW - 1) / UW * UW) {
        uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(dst + (threadIdx.x >> 5) * kLdk + c));
        src += (long long)(threadIdx.x >> 5) * d + c;
        for (int i = threadIdx.x >> 5; i < pad; i += NT / 32) {
            if (i < rows && c < w) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src) : "memory");
            else *reinterpret_cast<float4*>(dst + i * kLdk + c) = make_float4(0.f, 0.f, 0.f, 0.f);
            a += (NT / 32) * kLdk * 4;
            src += (NT / 32) * d;
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int NT, int UW>
__device__ __forceinline__ void load_tile(float* dst, const __nv_bfloat16* src, int rows, int pad, int d, int w) {
    const int c = (threadIdx.x & 15) << 3;
    if (c >= (w + UW - 1) / UW * UW) return;
    for (int i = threadIdx.x >> 4; i < pad; i += NT / 16) {
        uint4 v = make_uint4(0, 0, 0, 0);
        if (i < rows && c < w) v = *reinterpret_cast<const uint4*>(src + (long long)i * d + c);
        const uint32_t x[4] = {v.x, v.y, v.z, v.w};
        float f[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            f[2 * q] = __uint_as_float(x[q] << 16);
            f[2 * q + 1] = __uint_as_float(x[q] & 0xFFFF0000u);
        }
        *reinterpret_cast<float4*>(dst + i * kLdk + c) = make_float4(f[0], f[1], f[2], f[3]);
        *reinterpret_cast<float4*>(dst + i * kLdk + c + 4) = make_float4(f[4], f[5], f[6], f[7]);
    }
}
__device__ __forceinline__ void load_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Row j of the tile times scale[j].
template <int NT>
__device__ __forceinline__ void scale_rows(float* buf, const float* scale, int rows, int w) {
    const int per = w >> 2;
    for (int idx = threadIdx.x; idx < rows * per; idx += NT) {
        const int i = idx / per, c = (idx - i * per) << 2;
        float4* p = reinterpret_cast<float4*>(buf + i * kLdk + c);
        float4 v = *p;
        const float s = scale[i];
        v.x *= s; v.y *= s; v.z *= s; v.w *= s;
        *p = v;
    }
}

// v[r][s] = sum_k X[ti + G r][k] Et[tj + G s][k] for the pairs r - s >= DS, over the blocks q of k with s <= q <= r (X and E
// lower triangular).
template <int G, int R, int DS>
__device__ __forceinline__ void prod_tri(float (&v)[R][R], const float* X, const float* Et, int ti, int tj) {
    constexpr int ld = G * R + 4;
    f2 acc[R][R];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int s = 0; s < R; ++s) acc[r][s] = 0ull;
#pragma unroll
    for (int q = 0; q < R; ++q) {
#pragma unroll 4
        for (int k = q * G; k < q * G + G; k += 4) {
            ulonglong2 b[R];
#pragma unroll
            for (int s = 0; s <= q && s < R - DS; ++s) b[s] = *reinterpret_cast<const ulonglong2*>(Et + (tj + G * s) * ld + k);
#pragma unroll
            for (int r = (q > DS ? q : DS); r < R; ++r) {
                const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(X + (ti + G * r) * ld + k);
#pragma unroll
                for (int s = 0; s <= q && s <= r - DS; ++s) {
                    fma2(acc[r][s], a.x, b[s].x);
                    fma2(acc[r][s], a.y, b[s].y);
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int s = 0; s <= r - DS; ++s) v[r][s] = sum2(acc[r][s]);
}

// acc[r][c] += sum_j X[ti + G r][j] B[j][col_c .. col_c + 3] over the j of one block matrix: j blocks q <= r (X lower
// triangular) or all (FULL). Each thread: R rows, NC pieces of four columns, 4 G apart.
template <int G, int R, int NC, bool FULL>
__device__ __forceinline__ void prod_rows(f2 (&acc)[R][NC * 2], const float* X, const float* B, int ti, int col) {
    constexpr int ld = G * R + 4;
#pragma unroll
    for (int q = 0; q < R; ++q) {
#pragma unroll 2
        for (int j = q * G; j < q * G + G; j += 4) {
            float4 a[R];
#pragma unroll
            for (int r = FULL ? 0 : q; r < R; ++r) a[r] = *reinterpret_cast<const float4*>(X + (ti + G * r) * ld + j);
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                ulonglong2 b[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) b[c] = *reinterpret_cast<const ulonglong2*>(B + (j + jj) * kLdk + col + c * 4 * G);
#pragma unroll
                for (int r = FULL ? 0 : q; r < R; ++r) {
                    const float e = jj == 0 ? a[r].x : jj == 1 ? a[r].y : jj == 2 ? a[r].z : a[r].w;
                    const f2 x = pair2(e, e);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        fma2(acc[r][2 * c], x, b[c].x);
                        fma2(acc[r][2 * c + 1], x, b[c].y);
                    }
                }
            }
        }
    }
}

// Columns [c0, c0 + 4 G NC) of X B (X = T diag(beta), B: a tile of K or V in shared memory whose first column is column s0
// of the output) for block rows [nb0, nb1) of one chunk; columns from `d` on do not exist. `bad`: NaN once a result is not finite.
template <typename IO, int G, int R, int NB, int NC>
__device__ __forceinline__ void out_columns(IO* out, const float* X, const float* X22, const float* X21, const float* B, int C, int d, int s0,
                                            int c0, int ti, int tj, int nb0, int nb1, f2& bad) {
    constexpr int M = G * R;
    const int col = c0 + 4 * tj;
#pragma unroll 1
    for (int nb = nb0; nb < nb1; ++nb) {
        f2 acc[R][NC * 2];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < NC * 2; ++c) acc[r][c] = 0ull;
        if (nb == 0) {
            prod_rows<G, R, NC, false>(acc, X, B, ti, col - s0);
        } else {
            prod_rows<G, R, NC, true>(acc, X21, B, ti, col - s0);
            prod_rows<G, R, NC, false>(acc, X22, B + M * kLdk, ti, col - s0);
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < NC * 2; ++c) fma2(bad, acc[r][c], 0ull);  // NaN from here on if a result is not finite
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = nb * M + ti + G * r;
            if (i >= C) continue;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if (col + c * 4 * G >= d) continue;
                const float2 lo = split2(acc[r][2 * c]), hi = split2(acc[r][2 * c + 1]);
                st4(out + (long long)i * d + col + c * 4 * G, make_float4(lo.x, lo.y, hi.x, hi.y));
            }
        }
    }
}

// E = Abar + Abar L on i - j > N (w0: Abar on entry, E on return, Et its transpose) and X_1 = T0 + T0 E, N multiply-adds per
// entry each as T0 = I + L. NC: the order as a constant, 0 where it is not known.
template <int G, int R, int NC, class Sync>
__device__ __forceinline__ void first_term(float* X, float* w0, float* Et, int ti, int tj, int order, Sync sync) {
    constexpr int ld = G * R + 4;
    const int N = NC > 0 ? NC : order;
    float ev[R][R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = ti + G * r;
#pragma unroll
        for (int s = 0; s <= r; ++s) {
            const int j = tj + G * s;
            float v = 0.f;
            if (i - j > N) {
                // Abar[i][j] + sum_{e=1..N} Abar[i][j+e] L[j+e][j]   (j + e < i always holds there)
                v = w0[i * ld + j];
#pragma unroll
                for (int e = 1; e <= N; ++e) v = fmaf(w0[i * ld + j + e], X[(j + e) * ld + j], v);
            }
            ev[r][s] = v;
        }
    }
    sync();
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int s = 0; s <= r; ++s) {
            w0[(ti + G * r) * ld + tj + G * s] = ev[r][s];
            Et[(tj + G * s) * ld + ti + G * r] = ev[r][s];
        }
    sync();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = ti + G * r;
#pragma unroll
        for (int s = 0; s <= r; ++s) {
            const int j = tj + G * s;
            if (i - j > N) {
                float v = ev[r][s];
#pragma unroll
                for (int e = 1; e <= N; ++e) v = fmaf(X[i * ld + i - e], w0[(i - e) * ld + j], v);
                X[i * ld + j] = v;  // (no thread reads X beyond its band here)
            }
        }
    }
}

struct SimtParams {
    const void *K, *V;
    const float *beta, *g;
    void *W, *U, *Tinv;
    int H_k, H_v, T, C, d_k, d_v, N, S, mode, split, again;
    unsigned flags;
};

// Shared memory in floats: X of every diagonal block, two work matrices per block (a slice of V overlays them once T is
// complete), for two blocks the lower-left one, tables, the slice of K. With `again` that slice lies over the work matrices too,
// which come into use when the Gram product has read it; it is read again for W.
template <int G, int R, int NB>
struct SimtSmem {
    static constexpr int M = G * R, ld = M + 4, mat = M * ld;
    static constexpr int tile = NB * M * kLdk;
    static constexpr int work = 2 * NB * mat > tile ? 2 * NB * mat : tile;
    static constexpr int offX = 0, offW = NB * mat, offX21 = offW + work, offTab = offX21 + (NB - 1) * mat;
    static constexpr int offK = offTab + 4 * NB * M, total = offK + tile;
    static constexpr bool can_read_again = G == 8 && R >= 3;  // (elsewhere it gives no further CTA, or one at registers that spill)
};

// CTAs per SM that the registers are cut to, as far as nothing is spilled. What the other warps of an SM hide is the latency of
// shared memory and of the barriers of a chunk; 64 threads per CTA need many of them (us before and now, d = 128, 16384 chunks):
// 8 rows 8 -> 14 CTAs 80 -> 65, 16 rows 7 -> 8 152 -> 135, 24 rows 7 -> 8 238 -> 226, 32 rows (K read again) 5 -> 8 358 -> 326.
// (256 threads and three CTAs: 24 to 60 bytes spilled; chunks of 64 113 -> 114 with 1024 chunks.)
template <int G, int R, int NB>
constexpr int ctas_per_sm() {
    return G == 8 ? (R == 1 ? 14 : 8) : NB == 1 ? 2 : 1;
}

// G x G threads per diagonal block of G R rows (the chunk is padded to them with tokens that write nothing), NB blocks.
template <typename IO, int G, int R, int NB>
__global__ void __launch_bounds__(G* G* NB, (ctas_per_sm<G, R, NB>())) chunk_simt_kernel(const SimtParams p) {
    using L = SimtSmem<G, R, NB>;
    constexpr int M = L::M, ld = L::ld, NG = G * G, NT = NG * NB;
    extern __shared__ __align__(16) float sm[];
    __shared__ float swt[4];
    const int grp = threadIdx.x / NG;  // diagonal block this thread works on
    const int tl = threadIdx.x % NG, lane = threadIdx.x & 31, wp = tl >> 5;
    // A warp is 4 x 8 threads of the grid: the reads of a left operand touch 4 rows, of a right operand 8. A 16-byte read
    // takes 2 cycles where lanes i and i ^ 1 (or i and i ^ 2) read the same address and 4 otherwise (measured), so the row
    // leaves lane bit 0 out and the column lane bit 1.
    const int ti = (G == 16 ? (wp & 3) * 4 : wp * 4) + ((lane >> 1) & 1) + ((lane >> 4) << 1);
    const int tj = (G == 16 ? (wp >> 2) * 8 : 0) + (lane & 1) + (((lane >> 2) & 3) << 1);
    float* X = sm + L::offX + grp * L::mat;        // row-major, lower blocks
    float* w0 = sm + L::offW + grp * 2 * L::mat;   // Abar, then E, row-major
    float* Et = w0 + L::mat;                       // E transposed
    float* A21 = sm + L::offX21;                   // -A21, finally T21 (row-major)
    const bool again = L::can_read_again && p.again;
    float* Ks = sm + (again ? L::offW : L::offK);
    float* Vs = sm + L::offW;
    float* sbeta = sm + L::offTab;
    float* sg = sbeta + NB * M;
    float* srn = sg + NB * M;   // 1 / ||K_row|| (1 unless the keys are normalised here)
    float* swsc = srn + NB * M; // scale of the rows of K in W besides beta (1 / ||K||, times exp(g) for the gated W)

    const int C = p.C, d_k = p.d_k, d_v = p.d_v, N = p.N;
    const long long chunk = blockIdx.x / p.split;
    const int share = static_cast<int>(blockIdx.x - chunk * p.split);
    const int n_c = p.T / C;
    const long long bh = chunk / n_c;
    const long long tok = bh * (long long)p.T + (chunk - bh * n_c) * C;  // first row of the value-head tensors
    const long long ktok = ((bh / p.H_v) * p.H_k + (bh % p.H_v) / (p.H_v / p.H_k)) * (long long)p.T + (chunk - bh * n_c) * C;
    const IO* Kc = static_cast<const IO*>(p.K) + ktok * d_k;
    const IO* Vc = static_cast<const IO*>(p.V) + tok * d_v;
    auto group_sync = [&]() {
        if (NB == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(NG) : "memory");
    };

    load_tile<NT, 4 * G>(Ks, Kc, C, NB * M, d_k, min(kSliceW, d_k));
    for (int i = threadIdx.x; i < NB * M; i += NT) {
        sbeta[i] = (i < C) ? p.beta[tok + i] : 0.f;
        sg[i] = (i < C) ? p.g[tok + i] : 0.f;
    }
    // ---- Gram matrix: the lower blocks of this group's diagonal block and, of two, half of the rows of the lower-left one
    f2 acc[R][R], acc21[R / 2 > 0 ? R / 2 : 1][R];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int s = 0; s < R; ++s) acc[r][s] = 0ull;
    if (NB == 2) {
#pragma unroll
        for (int r = 0; r < R / 2; ++r)
#pragma unroll
            for (int s = 0; s < R; ++s) acc21[r][s] = 0ull;
    }
    for (int d0 = 0; d0 < d_k; d0 += kSliceW) {
        const int w = min(kSliceW, d_k - d0);
        if (d0 > 0) {
            __syncthreads();
            load_tile<NT, 4 * G>(Ks, Kc + d0, C, NB * M, d_k, w);
        }
        load_wait();
        __syncthreads();
        const float* Kb = Ks + grp * M * kLdk;
#pragma unroll 4
        for (int d = 0; d < w; d += 4) {
            ulonglong2 b[R];
#pragma unroll
            for (int s = 0; s < R; ++s) b[s] = *reinterpret_cast<const ulonglong2*>(Kb + (tj + G * s) * kLdk + d);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(Kb + (ti + G * r) * kLdk + d);
#pragma unroll
                for (int s = 0; s <= r; ++s) {
                    fma2(acc[r][s], a.x, b[s].x);
                    fma2(acc[r][s], a.y, b[s].y);
                }
            }
        }
        if (NB == 2) {
#pragma unroll 2
            for (int d = 0; d < w; d += 4) {
                ulonglong2 b[R];
#pragma unroll
                for (int s = 0; s < R; ++s) b[s] = *reinterpret_cast<const ulonglong2*>(Ks + (tj + G * s) * kLdk + d);
#pragma unroll
                for (int r = 0; r < R / 2; ++r) {
                    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(Ks + (M + ti + G * (r + grp * (R / 2))) * kLdk + d);
#pragma unroll
                    for (int s = 0; s < R; ++s) {
                        fma2(acc21[r][s], a.x, b[s].x);
                        fma2(acc21[r][s], a.y, b[s].y);
                    }
                }
            }
        }
    }
    if (p.flags & GDN_FLAG_G_RAW) {
        // raw log-gates: chunk-local inclusive prefix sum (at most 128 tokens): shuffles inside a warp, then the totals
        // of the warps before it
        const int i = threadIdx.x, w = i >> 5;
        float v = (i < NB * M) ? sg[i] : 0.f;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const float u = __shfl_up_sync(0xFFFFFFFFu, v, off);
            if (lane >= off) v += u;
        }
        if (lane == 31 && w < 4) swt[w] = v;
        __syncthreads();
        if (i < NB * M) {
            for (int k = 0; k < w; ++k) v += swt[k];
            sg[i] = v;
        }
    }
    // row norms from the Gram diagonal
    if (ti == tj) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            srn[grp * M + ti + G * r] = (p.flags & GDN_FLAG_K_L2NORM) ? rsqrtf(fmaxf(sum2(acc[r][r]), 1e-30f)) : 1.f;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < NB * M; i += NT)
        swsc[i] = srn[i] * ((p.flags & GDN_FLAG_W_GATED) ? expf(sg[i]) : 1.f);
    // ---- Abar = -tril(diag(beta) (K K^T o Gamma), -1); rows past the chunk's end are zero; X = I
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = grp * M + ti + G * r;
        const float bi = -sbeta[i] * srn[i], gi = sg[i];
#pragma unroll
        for (int s = 0; s < R; ++s) {
            const int j = grp * M + tj + G * s;
            float v = 0.f;
            if (s <= r && i > j && i < C) v = bi * expf(gi - sg[j]) * sum2(acc[r][s]) * srn[j];
            w0[(ti + G * r) * ld + tj + G * s] = v;
            X[(ti + G * r) * ld + tj + G * s] = (i == j) ? 1.f : 0.f;
        }
    }
    if (NB == 2) {
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
            const int il = ti + G * (r + grp * (R / 2)), i = M + il;
            const float bi = -sbeta[i] * srn[i], gi = sg[i];
#pragma unroll
            for (int s = 0; s < R; ++s) {
                const int j = tj + G * s;
                A21[il * ld + j] = (i < C) ? bi * expf(gi - sg[j]) * sum2(acc21[r][s]) * srn[j] : 0.f;
            }
        }
    }
    __syncthreads();
    const bool k_scaled = (p.flags & (GDN_FLAG_K_L2NORM | GDN_FLAG_W_GATED)) != 0;
    // the rows of K as W reads them (wider keys, and with `again` all, are loaded again, slice by slice)
    if (!again && k_scaled && d_k <= kSliceW) scale_rows<NT>(Ks, swsc, NB * M, d_k);
    if (p.mode == INV_NEUMANN) {
        // ---- band by distance (one row per thread, a barrier per distance: row i needs L_{d-e} of rows i - e)
        const int n = NB == 1 ? C : M;
        for (int d = 1; d <= N && d < n; ++d) {
            const int i = tl;
            if (i >= d && i < n) {
                float v = w0[i * ld + (i - d)];
                for (int e = 1; e < d; ++e) v = fmaf(w0[i * ld + (i - e)], X[(i - e) * ld + (i - d)], v);
                X[i * ld + (i - d)] = v;
            }
            group_sync();
        }
        if (p.S > 0) {
            // (the loops over the band unrolled for the default order)
            if (N == 3) first_term<G, R, 3>(X, w0, Et, ti, tj, N, group_sync);
            else first_term<G, R, 0>(X, w0, Et, ti, tj, N, group_sync);
            // ---- X_{k+1} = T0 + X_k E for 1 <= k < S: block diagonals below `ds` no longer change
            float v[R][R];
            for (int k = 2; k <= p.S; ++k) {
                const int ds = k * (N + 1) / G;
                if (ds >= R) break;
                group_sync();
                switch (ds) {
                    case 0: prod_tri<G, R, 0>(v, X, Et, ti, tj); break;
                    case 1: prod_tri<G, R, (R > 1 ? 1 : 0)>(v, X, Et, ti, tj); break;
                    case 2: prod_tri<G, R, (R > 2 ? 2 : 0)>(v, X, Et, ti, tj); break;
                    default: prod_tri<G, R, (R > 3 ? 3 : 0)>(v, X, Et, ti, tj); break;
                }
                group_sync();
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int s = 0; s <= r; ++s)
                        if (r - s >= ds && ti + G * r - tj - G * s > N) X[(ti + G * r) * ld + tj + G * s] = v[r][s];
            }
        }
        // The products above run over whole blocks, zeros included: a chunk with an entry that is not finite is done again
        // with every sum over its own terms only, so that a token does not reach the tokens before it.
        float bad = 0.f;
        group_sync();
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int s = 0; s <= r; ++s) bad = fmaf(X[(ti + G * r) * ld + tj + G * s], 0.f, bad);
        if (__syncthreads_or(bad != 0.f) && p.S > 0) {
            for (int idx = tl; idx < M * M; idx += NG)
                if (idx / M - idx % M > N) X[(idx / M) * ld + idx % M] = 0.f;
            group_sync();
            for (int k0 = 0; k0 < p.S; ++k0) {  // X_{k+1} = T0 + X_k E
                for (int idx = tl; idx < M * M; idx += NG) {
                    const int i = idx / M, j = idx % M;
                    float v = 0.f;
                    for (int k = j + N + 1; k <= i; ++k) v = fmaf(X[i * ld + k], Et[j * ld + k], v);
                    w0[i * ld + j] = v;
                }
                group_sync();
                for (int idx = tl; idx < M * M; idx += NG)
                    if (idx / M - idx % M > N) X[(idx / M) * ld + idx % M] = w0[(idx / M) * ld + idx % M];
                group_sync();
            }
        }
        if (NB == 2) {
            // ---- T21 = T22 Abar21 T11 (App. E, Eq. 28 with Abar21 = -A21); T11 and the first product transposed
            if (grp == 0) {
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int s = 0; s < R; ++s) Et[(tj + G * s) * ld + ti + G * r] = X[(ti + G * r) * ld + tj + G * s];
            }
            __syncthreads();
            const float* T11t = sm + L::offW + L::mat;
            float* Yt = sm + L::offW;
            // block rows {0, 3} and {1, 2} of the four: as many triangle blocks for either group
#pragma unroll 1
            for (int step = 0; step < 2; ++step) {
                const float* Lm = step == 0 ? A21 : sm + L::offX + L::mat;
                const float* Rm = step == 0 ? T11t : Yt;
                f2 a[R / 2 > 0 ? R / 2 : 1][R];
#pragma unroll
                for (int rr = 0; rr < R / 2; ++rr) {
                    const int r = rr == 0 ? grp : R - 1 - grp;
#pragma unroll
                    for (int s = 0; s < R; ++s) a[rr][s] = 0ull;
                    const int kend = step == 0 ? M : G * (r + 1);
#pragma unroll 2
                    for (int k = 0; k < kend; k += 4) {
                        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(Lm + (ti + G * r) * ld + k);
#pragma unroll
                        for (int s = 0; s < R; ++s) {
                            const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(Rm + (tj + G * s) * ld + k);
                            fma2(a[rr][s], x.x, y.x);
                            fma2(a[rr][s], x.y, y.y);
                        }
                    }
                }
                float nonfinite = 0.f;
#pragma unroll
                for (int rr = 0; rr < R / 2; ++rr) {
#pragma unroll
                    for (int s = 0; s < R; ++s) nonfinite = fmaf(sum2(a[rr][s]), 0.f, nonfinite);
                }
                const bool again = __syncthreads_or(nonfinite != 0.f);
#pragma unroll
                for (int rr = 0; rr < R / 2; ++rr) {
                    const int i = ti + G * (rr == 0 ? grp : R - 1 - grp);
#pragma unroll
                    for (int s = 0; s < R; ++s) {
                        if (step == 0) Yt[(tj + G * s) * ld + i] = sum2(a[rr][s]);
                        else A21[i * ld + tj + G * s] = sum2(a[rr][s]);
                    }
                }
                if (again) {  // (as above: every sum over its own terms only, T11 from the diagonal on and T22 up to it)
#pragma unroll 1
                    for (int e = 0; e < R / 2 * R; ++e) {
                        const int i = ti + G * (e < R ? grp : R - 1 - grp), j = tj + G * (e % R);
                        float v = 0.f;
                        for (int k = step == 0 ? j : 0; k < (step == 0 ? M : i + 1); ++k) v = fmaf(Lm[i * ld + k], Rm[j * ld + k], v);
                        if (step == 0) Yt[j * ld + i] = v;
                        else A21[i * ld + j] = v;
                    }
                }
                __syncthreads();
            }
        }
    } else {
        // ---- forward substitution: thread j owns column j of T. Of two blocks, the sums below run first over the rows of the
        // upper one, then over the lower one's, each with pointers and one stride of its own.
        float* T21 = sm + L::offW + L::mat;
        const int j = threadIdx.x;
        const bool up = NB == 1 || j < M;                                                         // column j in the left blocks
        float* Tu = sm + L::offX + j;                                                             // T(k, j), k < M (left columns)
        float* Tl = up ? T21 + j : sm + L::offX + L::mat + j - M;                                 // T(M + k, j)
        const float* Al = sm + L::offW + 2 * L::mat;                                              // A(M + i, M + k)
        auto row = [&](int i) { return (NB == 1 || i < M) ? sm + L::offW + i * ld : A21 + (i - M) * ld; };  // A(i, k), k < M
        // v + the terms k0 <= k < k1 of row i of A with column j of T, in that order
        auto dot = [&](int i, int k0, int k1, float v) {
            if (up) {
                const float* a = row(i);
                const int end = NB == 1 ? k1 : min(k1, M);
                for (int k = k0; k < end; ++k) v = fmaf(a[k], Tu[k * ld], v);
            }
            if (NB == 2 && k1 > M) {
                const float* a = Al + (i - M) * ld;
                for (int k = max(k0, M) - M; k < k1 - M; ++k) v = fmaf(a[k], Tl[k * ld], v);
            }
            return v;
        };
        auto A = [&](int i) { return up ? row(i)[j] : Al[(i - M) * ld + j - M]; };  // A(i, j)
        auto T = [&](int i) -> float& { return (NB == 1 || i < M) ? Tu[i * ld] : Tl[(i - M) * ld]; };  // T(i, j)
        if (p.mode == INV_FWDSUBST_BLOCKED) {
            // Blocked form (App. E): 16 x 16 diagonal blocks by substitution (Eq. 25), then block rows from
            // S_ij = S_ii sum_{k<i} Abar_ik S_kj (Eq. 27 with T_ik = -Abar_ik).
            if (j < C) {
                const int bend = (j / 16 + 1) * 16;
                for (int i = j + 1; i < bend; ++i) T(i) = dot(i, j + 1, i, A(i));
            }
            __syncthreads();
            if (j < C) {
                for (int bi = j / 16 + 1; bi < C / 16; ++bi) {
                    float tmp[16];
                    for (int r = 0; r < 16; ++r) tmp[r] = dot(bi * 16 + r, j, bi * 16, 0.f);
                    // the diagonal block of these rows (16 divides M: it lies in one of the two)
                    const float* S = (NB == 1 || bi * 16 < M) ? sm + L::offX + bi * 16 * (ld + 1) : sm + L::offX + L::mat + (bi * 16 - M) * (ld + 1);
                    for (int r = 0; r < 16; ++r) {
                        float v = 0.f;
                        for (int q = 0; q <= r; ++q) v = fmaf(S[r * ld + q], tmp[q], v);
                        T(bi * 16 + r) = v;
                    }
                }
            }
        } else if (j < C) {
            // Rows in order (Eq. 2-3): row i of X = Abar_i + Abar_{i,0:i} X_{0:i,:}
            for (int i = j + 1; i < C; ++i) T(i) = dot(i, j + 1, i, A(i));
        }
        __syncthreads();
        if (NB == 2) {
            for (int idx = threadIdx.x; idx < M * M; idx += NT) A21[(idx / M) * ld + idx % M] = T21[(idx / M) * ld + idx % M];
        }
        __syncthreads();
    }

    // ---- W = T diag(w) K, U = T diag(beta) V: units of 4 G columns, this CTA's share of them; two at a time where the
    // second one lies in the same tile. A slice of V comes in (over the work matrices, all read by now) while W is formed.
    constexpr int UW = 4 * G, per_slice = kSliceW / UW;
    const int nk = (d_k + UW - 1) / UW, nv = (d_v + UW - 1) / UW;
    const int u0 = (nk + nv) * share / p.split, u1 = (nk + nv) * (share + 1) / p.split;
    int in_v = -1;  // slice in Vs: index of its first unit
    if (again) {    // (one CTA has all of a chunk: it begins with the first slice of K)
        in_v = 0;
        load_tile<NT, 4 * G>(Ks, Kc, C, NB * M, d_k, min(kSliceW, d_k));
    } else if (u1 > nk) {
        in_v = nk + (max(u0, nk) - nk) / per_slice * per_slice;
        const int col = (in_v - nk) * UW;
        load_tile<NT, 4 * G>(Vs, Vc + col, C, NB * M, d_v, min(kSliceW, d_v - col));
    }
    // T leaves, X <- T diag(beta)
    IO* Tc = (share == 0 && p.Tinv != nullptr) ? static_cast<IO*>(p.Tinv) + chunk * (long long)C * C : nullptr;
    auto take = [&](float* m, int nbi, int nbj, int r, int s) {  // entry (ti + G r, tj + G s) of block (nbi, nbj)
        const int i = nbi * M + ti + G * r, j = nbj * M + tj + G * s;
        float* x = m + (ti + G * r) * ld + tj + G * s;
        const float v = *x;
        *x = v * sbeta[j];
        if (Tc != nullptr && i < C && j < C) st(Tc + i * C + j, v);
    };
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int s = 0; s < R; ++s) take(X, grp, grp, r, s);
    if (NB == 2) {
#pragma unroll
        for (int rr = 0; rr < R / 2; ++rr) {
            const int r = rr + grp * (R / 2);
#pragma unroll
            for (int s = 0; s < R; ++s) {
                take(A21, 1, 0, r, s);
                if (Tc != nullptr) st(Tc + (ti + G * r) * C + M + tj + G * s, 0.f);
            }
        }
    }
    __syncthreads();
    const float* X0 = sm + L::offX;
    const float* X22 = X0 + (NB - 1) * L::mat;
    bool v_ready = false;
    for (int u = u0; u < u1;) {
        const bool is_v = u >= nk;
        const int first = is_v ? nk + (u - nk) / per_slice * per_slice : u / per_slice * per_slice;  // first unit of u's slice
        const int end = min(min(first + per_slice, u1), is_v ? nk + nv : nk);
        const int d = is_v ? d_v : d_k, s0 = (first - (is_v ? nk : 0)) * UW;
        float* B = is_v ? Vs : Ks;
        if (is_v || again ? in_v != first : d_k > kSliceW) {
            __syncthreads();
            load_tile<NT, 4 * G>(B, (is_v ? Vc : Kc) + s0, C, NB * M, d, min(kSliceW, d - s0));
            v_ready = false;
        }
        if (is_v ? !v_ready : again || d_k > kSliceW) {
            load_wait();
            __syncthreads();
            if (is_v) {
                in_v = first;
                v_ready = true;
            } else if (k_scaled) {
                scale_rows<NT>(B, swsc, NB * M, min(kSliceW, d - s0));
                __syncthreads();
            }
        }
        IO* out = (is_v ? static_cast<IO*>(p.U) + tok * d_v : static_cast<IO*>(p.W) + tok * d_k);
        f2 bad = 0ull;
        const int begin = u;
        while (u < end) {
            const int c0 = s0 + (u - first) * UW;
            if (NB == 1 && u + 1 < end) {
                out_columns<IO, G, R, NB, 2>(out, X0, X22, A21, B, C, d, s0, c0, ti, tj, 0, 1, bad);
                u += 2;
            } else if (NB == 2 && u + 1 < end) {  // one unit per group
                out_columns<IO, G, R, NB, 1>(out, X0, X22, A21, B, C, d, s0, c0 + grp * UW, ti, tj, 0, 2, bad);
                u += 2;
            } else {  // a single unit: of two groups, each its own block rows
                out_columns<IO, G, R, NB, 1>(out, X0, X22, A21, B, C, d, s0, c0, ti, tj, NB == 1 ? 0 : grp, NB == 1 ? 1 : grp + 1, bad);
                u += 1;
            }
        }
        if (__syncthreads_or(sum2(bad) != 0.f)) {  // (as above: every sum over its own terms only)
            const int w = (end - begin) * UW;
            for (int idx = threadIdx.x; idx < C * w; idx += NT) {
                const int i = idx / w, c = s0 + (begin - first) * UW + idx % w;
                if (c >= d) continue;
                float v = 0.f;
                for (int j = 0; j <= i; ++j) {
                    const float t = NB == 1 || i < M ? X0[i * ld + j] : j < M ? A21[(i - M) * ld + j] : X22[(i - M) * ld + j - M];
                    v = fmaf(t, B[j * kLdk + c - s0], v);
                }
                st(out + (long long)i * d + c, v);
            }
        }
    }
}

template <typename IO, int G, int R, int NB>
int launch_one(SimtParams p, long long n_chunks, cudaStream_t stream) {
    auto kern = chunk_simt_kernel<IO, G, R, NB>;
    using L = SimtSmem<G, R, NB>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::total * 4) != cudaSuccess) return GDN_ERR_LAUNCH;
    // Fewer chunks than SMs: two or four CTAs share a chunk (each forms the inverse, its part of the columns of W and U), as
    // long as every CTA still has an SM of its own: 8 chunks of 64 take 21 us in four parts, where W and U are half the
    // work of a chunk; with more CTAs than SMs the repeated Gram product and rounds would be paid for twice.
    p.split = n_chunks * 4 <= kSMs ? 4 : n_chunks * 2 <= kSMs ? 2 : 1;
    if (n_chunks * p.split >= (1LL << 31)) return GDN_ERR_UNSUPPORTED;
    // K read again instead of kept from the Gram product to W makes room for more CTAs per SM: from the number of chunks on that no
    // longer fits at once with K kept (7 CTAs per SM up to 24 rows, 5 up to 32; 741 chunks of 32 27 -> 23 us, 1190 of 24 25 -> 23).
    p.again = L::can_read_again && n_chunks > (R == 3 ? 7 : 5) * kSMs;
    const int smem = (p.again ? L::offK : L::total) * 4;
    kern<<<static_cast<int>(n_chunks * p.split), G * G * NB, smem, stream>>>(p);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? GDN_OK : GDN_ERR_LAUNCH;
}

// Thread grid of a diagonal block by its size: 8 x 8 threads (64 per chunk) up to 32 rows, 16 x 16 above; R rows per thread.
template <typename IO>
int launch_size(const SimtParams& p, long long n_chunks, cudaStream_t stream) {
    const int C = p.C;
    if (C <= 8) return launch_one<IO, 8, 1, 1>(p, n_chunks, stream);
    if (C <= 16) return launch_one<IO, 8, 2, 1>(p, n_chunks, stream);
    if (C <= 24) return launch_one<IO, 8, 3, 1>(p, n_chunks, stream);
    if (C <= 32) return launch_one<IO, 8, 4, 1>(p, n_chunks, stream);
    if (C <= 48) return launch_one<IO, 16, 3, 1>(p, n_chunks, stream);
    if (C <= 64) return launch_one<IO, 16, 4, 1>(p, n_chunks, stream);
    return launch_one<IO, 16, 4, 2>(p, n_chunks, stream);
}

}  // namespace

int launch_simt(const Problem& p, InverseMode mode, cudaStream_t stream) {
    const int C = p.C;
    if (!(C >= 2 && (C <= 64 || C == 128))) return GDN_ERR_UNSUPPORTED;
    if (p.d_k > 256 || p.d_v > 256) return GDN_ERR_UNSUPPORTED;
    if (mode == INV_FWDSUBST_BLOCKED && C % 16 != 0) return GDN_ERR_UNSUPPORTED;
    if (p.flags & GDN_FLAG_OUT_FP32) {
        if (p.dtype != GDN_DTYPE_FP32) return GDN_ERR_UNSUPPORTED;  // this kernel writes the element type it reads
    }
    const long long n_chunks = (long long)p.B * p.H_v * (p.T / C);
    if (n_chunks == 0) return GDN_OK;
    const SimtParams q{p.K, p.V, p.beta, p.g, p.W, p.U, p.Tinv, p.H_k, p.H_v, p.T, C, p.d_k, p.d_v, p.order, p.steps, (int)mode, 1, 0, p.flags};
    return p.dtype == GDN_DTYPE_FP32 ? launch_size<float>(q, n_chunks, stream) : launch_size<__nv_bfloat16>(q, n_chunks, stream);
}

}  // namespace gdn
