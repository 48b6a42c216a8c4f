// sf_pp.cuh -- shared device code of the prime-power rings M = t^alpha
// (Sec. 2.1-2.3, Table 2): the ring and modulus constants, the generic
// and the compile-time length-M radix-t transforms, and the dispatch over
// the compiled rings.  Used by the ring arithmetic and RNS RLWE (sf_pp.cu)
// and by the torus scheme (sf_tq.cu).
#pragma once
#include <utility>
#include <vector>

#include "sf_arith.cuh"
#include "sf_internal.h"

#define SF_PP_THREADS 256
#define SF_PP_MAX_T 7
#define SF_PP_MAX_M 4096

struct SfPpMod {
    u64 q, one_p;            // modulus, floor(2^64 / q)
    u64 qinv_neg, r2;        // -q^-1 mod 2^64, 2^128 mod q (Montgomery products of two residues)
    u64 minv, minv_p;        // M^-1 mod q (Shoup)
    u64 h2, h2_p;            // 2^-1 mod q (Shoup)
    u64 c3, c3_p;            // t = 3: (zeta - zeta^2) / 2, zeta = omega^(M/3) (Shoup)
    u64 qh_inv, qh_inv_p;    // (Q / q_i)^-1 mod q_i (Shoup): the RNS digits of key switching
    u64 rm, rm_p;            // 2^64 mod q (Shoup): companions computed on the device
    unsigned binv;           // floor(2^(32 + sh) / q), sh = floor(log2 q): pp_red3
    int sh;
};

typedef ulonglong2 pp_pair;   // (w, floor(w 2^64 / q))

struct SfPpRing {
    int t, alpha, M, N, m, L;
    const u64 *w;            // [L][M] omega_i^e
    const u64 *w_p;          // [L][M] Shoup companions
    const u64 *iw;           // [L][M] omega_i^-e
    const u64 *iw_p;
    const u64 *qhat;         // [L][L][2]: (Q / q_i) mod q_j and its Shoup companion
    const u64 *dftc;         // [L][H][H][4], H = (t-1)/2: C_rk, C_rk', S_rk, S_rk' of the paired t-point DFT
    const pp_pair *tw;       // [L][2][M]: twiddles of the lazy stages (pp_twiddles), forward and inverse
    const pp_pair *dftl;     // [L][SfPpDft::N]: constants of the lazy t-point DFT
    int lazy;                // every prime below 2^50: the compiled transforms run their lazy stages
    SfPpMod mod[SF_MAX_MODULI];
};

struct sf_pp_ring {
    int device;
    SfPpRing R;
    std::vector<u64> q;
    u64 *d_tables = nullptr;     // w, w_p, iw, iw_p
    u64 *d_scratch = nullptr;    // trace work buffers
    size_t scratch_words = 0;
    u64 *d_ks = nullptr;         // key-switch and ciphertext work buffers
    size_t ks_words = 0;
};

// a * b mod q for two residues below q (two Montgomery reductions: a b 2^-64,
// then times 2^128 2^-64)
__device__ __forceinline__ u64 pp_mulmod(u64 a, u64 b, const SfPpMod &P)
{
    return sf_mul_mont(sf_mul_mont(a, b, P.q, P.qinv_neg), P.r2, P.q, P.qinv_neg);
}

// one forward (DIF) stage of span len over the block's vector s
__device__ __forceinline__ void pp_stage_fwd(u64 *s, const SfPpRing &R, int i, int len)
{
    const int t = R.t, third = len / t, stride = R.M / len;
    const u64 q = R.mod[i].q, one_p = R.mod[i].one_p;
    const u64 *w = R.w + (size_t)i * R.M, *wp = R.w_p + (size_t)i * R.M;
    const int root_t = R.M / t;   // omega^(M/t): a primitive t-th root
    for (int idx = threadIdx.x; idx < R.M / t; idx += blockDim.x) {
        const int blk = idx / third, j = idx - blk * third;
        const int base = blk * len + j;
        u64 x[SF_PP_MAX_T];
        for (int r = 0; r < t; ++r) x[r] = s[base + r * third];
        for (int k = 0; k < t; ++k) {
            // y_k = sum_r x_r zeta^(r k), zeta = omega^(M/t); lazily below 2 t q
            u64 acc = x[0];
            for (int r = 1; r < t; ++r) {
                const int e = (root_t * ((r * k) % t)) % R.M;
                acc += sf_mul_shoup_lazy(x[r], w[e], wp[e], q);
            }
            u64 y = sf_reduce(acc, q, one_p);
            // twiddle omega_len^(j k) = omega^(stride j k)
            const int e = (int)(((long long)stride * j * k) % R.M);
            if (e) y = sf_mul_shoup(y, w[e], wp[e], q);
            s[base + k * third] = y;
        }
    }
}

// one inverse (DIT) stage of span len: untwiddle, then the inverse t-point DFT
__device__ __forceinline__ void pp_stage_inv(u64 *s, const SfPpRing &R, int i, int len)
{
    const int t = R.t, third = len / t, stride = R.M / len;
    const u64 q = R.mod[i].q, one_p = R.mod[i].one_p;
    const u64 *iw = R.iw + (size_t)i * R.M, *iwp = R.iw_p + (size_t)i * R.M;
    const int root_t = R.M / t;
    for (int idx = threadIdx.x; idx < R.M / t; idx += blockDim.x) {
        const int blk = idx / third, j = idx - blk * third;
        const int base = blk * len + j;
        u64 x[SF_PP_MAX_T];
        for (int k = 0; k < t; ++k) {
            u64 v = s[base + k * third];
            const int e = (int)(((long long)stride * j * k) % R.M);
            x[k] = e ? sf_mul_shoup(v, iw[e], iwp[e], q) : v;
        }
        for (int r = 0; r < t; ++r) {
            u64 acc = x[0];
            for (int k = 1; k < t; ++k) {
                const int e = (root_t * ((r * k) % t)) % R.M;
                acc += sf_mul_shoup_lazy(x[k], iw[e], iwp[e], q);
            }
            s[base + r * third] = sf_reduce(acc, q, one_p);
        }
    }
}

__device__ __forceinline__ void pp_forward(u64 *s, const SfPpRing &R, int i)
{
    for (int len = R.M; len >= R.t; len /= R.t) {
        pp_stage_fwd(s, R, i, len);
        __syncthreads();
    }
}

__device__ __forceinline__ void pp_inverse(u64 *s, const SfPpRing &R, int i)
{
    for (int len = R.t; len <= R.M; len *= R.t) {
        pp_stage_inv(s, R, i, len);
        __syncthreads();
    }
    const SfPpMod &P = R.mod[i];
    for (int e = threadIdx.x; e < R.M; e += blockDim.x) s[e] = sf_mul_shoup(s[e], P.minv, P.minv_p, P.q);
    __syncthreads();
}

// X^(N + e) = -sum_{k < t-1} X^(e + k m): fold positions N .. M-1 into 0 .. N-1
__device__ __forceinline__ void pp_reduce_phi(u64 *s, const SfPpRing &R, int i)
{
    const u64 q = R.mod[i].q;
    for (int e = threadIdx.x; e < R.m; e += blockDim.x) {
        const u64 v = s[R.N + e];
        for (int k = 0; k < R.t - 1; ++k) s[e + k * R.m] = sf_sub(s[e + k * R.m], v, q);
    }
    __syncthreads();
}

// ---- compile-time rings (Table 2: 3^7, 7^4, 5^5, and the smaller test rings)
// The same stages with t and alpha as template parameters: every span, stride
// and root index is a constant, the t values of a butterfly stay in
// registers, and one thread runs one butterfly per stage (M / t threads,
// rounded up to whole warps).  Twiddle exponents need no reduction: for span
// len, j < len / t and k < t give (M / len) j k < M.

// Radix of a phase of the lazy transforms: two radix-3 stages in one (9 points a
// thread) while that leaves a block two warps of work; 3^4 with radix 9 in 9 threads
// took 149 us for 20000 x 5 transforms, 75 with a butterfly a thread.
__host__ __device__ constexpr int ppt_radix(int t, int M) { return t == 3 && M / 9 >= 64 ? 9 : t; }
// Threads of a block: one group of points each.  Two groups a thread (5^5: 320
// threads of 96 registers instead of 640 of 48) ran the torus key switch of 4096
// ciphertexts in 2727 us against 2428.
__host__ __device__ constexpr int ppt_threads(int t, int M) { return (M / ppt_radix(t, M) + 31) / 32 * 32; }

template <int T, int ALPHA>
struct SfPpT {
    static constexpr int M = T == 3 ? (ALPHA == 2 ? 9 : ALPHA == 3 ? 27 : ALPHA == 4 ? 81 : ALPHA == 5 ? 243 : ALPHA == 6 ? 729 : 2187)
                           : T == 5 ? (ALPHA == 2 ? 25 : ALPHA == 3 ? 125 : ALPHA == 4 ? 625 : 3125)
                                    : (ALPHA == 2 ? 49 : ALPHA == 3 ? 343 : 2401);
    static constexpr int THREADS = ppt_threads(T, M);
    static constexpr int WIDE = (M / T + 31) / 32 * 32;   // k_ppt_ntt_wide: one butterfly a thread and stage
};

// the 3-point DFT with two products: with zeta + zeta^2 = -1,
// y1, y2 = x0 - (x1 + x2) / 2 +- c (x1 - x2), c = (zeta - zeta^2) / 2
// (the inverse transform's root zeta^-1 flips the sign of c)
template <bool INV>
__device__ __forceinline__ void ppt_dft3(u64 &x0, u64 &x1, u64 &x2, const SfPpMod &P)
{
    const u64 q = P.q;
    const u64 sm = sf_add(x1, x2, q), df = sf_sub(x1, x2, q);
    const u64 u = sf_sub(x0, sf_mul_shoup(sm, P.h2, P.h2_p, q), q);
    const u64 v = sf_mul_shoup(df, P.c3, P.c3_p, q);
    x0 = sf_add(x0, sm, q);
    x1 = INV ? sf_sub(u, v, q) : sf_add(u, v, q);
    x2 = INV ? sf_add(u, v, q) : sf_sub(u, v, q);
}

// The t-point DFT for odd t >= 5 by conjugate pairs: with A_r = x_r + x_(t-r),
// B_r = x_r - x_(t-r) (r = 1 .. H, H = (t-1)/2),
//   y_k, y_(t-k) = x_0 + sum_r A_r C_rk +- sum_r B_r S_rk,
// C_rk = (zeta^(rk) + zeta^(-rk)) / 2, S_rk = (zeta^(rk) - zeta^(-rk)) / 2, so
// (t-1)^2 / 2 products instead of t (t-1); the inverse (root zeta^-1) flips S.
template <int T, bool INV>
__device__ __forceinline__ void ppt_dft_pairs(u64 *x, const u64 *dc, u64 q, u64 one_p)
{
    constexpr int H = (T - 1) / 2;
    u64 A[H], B[H];
    u64 y0 = x[0];
#pragma unroll
    for (int r = 1; r <= H; ++r) {
        A[r - 1] = sf_add(x[r], x[T - r], q);
        B[r - 1] = sf_sub(x[r], x[T - r], q);
        y0 = sf_add(y0, A[r - 1], q);
    }
    u64 y[T];
    y[0] = y0;
#pragma unroll
    for (int k = 1; k <= H; ++k) {
        u64 U = 0, V = 0;   // lazy: H terms below 2q each
#pragma unroll
        for (int r = 1; r <= H; ++r) {
            const u64 *c = dc + 4 * ((r - 1) * H + (k - 1));
            U += sf_mul_shoup_lazy(A[r - 1], __ldg(c), __ldg(c + 1), q);
            V += sf_mul_shoup_lazy(B[r - 1], __ldg(c + 2), __ldg(c + 3), q);
        }
        const u64 base = sf_add(x[0], sf_reduce(U, q, one_p), q);
        V = sf_reduce(V, q, one_p);
        y[k] = INV ? sf_sub(base, V, q) : sf_add(base, V, q);
        y[T - k] = INV ? sf_add(base, V, q) : sf_sub(base, V, q);
    }
#pragma unroll
    for (int k = 0; k < T; ++k) x[k] = y[k];
}

// NT: the block's threads.  One forward stage reading its inputs through ld(index) (the block's vector
// itself, or a producer for the first stage) and writing them to s
template <int T, int M, int LEN, int NT, class LD>
__device__ __forceinline__ void ppt_stage_fwd_ld(u64 *s, LD ld, const u64 *w, const u64 *wp, const u64 *dc, u64 q,
                                                 u64 one_p, const SfPpMod &P)
{
    static_assert(T >= 3 && (T & 1), "compiled rings have an odd prime t");
    constexpr int THIRD = LEN / T, STRIDE = M / LEN;
#pragma unroll 1
    for (int g0 = 0; g0 < M / T; g0 += NT) {
        const int idx = g0 + threadIdx.x;
        if (idx >= M / T) break;
        const int blk = idx / THIRD, j = idx - blk * THIRD;
        const int base = blk * LEN + j;
        u64 x[T];
#pragma unroll
        for (int r = 0; r < T; ++r) x[r] = ld(base + r * THIRD);
        if constexpr (T == 3) {
            ppt_dft3<false>(x[0], x[1], x[2], P);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int e = STRIDE * j * k;
                s[base + k * THIRD] = e ? sf_mul_shoup(x[k], __ldg(w + e), __ldg(wp + e), q) : x[k];
            }
        } else {
            ppt_dft_pairs<T, false>(x, dc, q, one_p);
#pragma unroll
            for (int k = 0; k < T; ++k) {
                const int e = STRIDE * j * k;
                s[base + k * THIRD] = e ? sf_mul_shoup(x[k], __ldg(w + e), __ldg(wp + e), q) : x[k];
            }
        }
    }
}

template <int T, int M, int LEN, int NT>
__device__ __forceinline__ void ppt_stage_fwd(u64 *s, const u64 *w, const u64 *wp, const u64 *dc, u64 q, u64 one_p,
                                              const SfPpMod &P)
{
    ppt_stage_fwd_ld<T, M, LEN, NT>(s, [s](int i) { return s[i]; }, w, wp, dc, q, one_p, P);
}

template <int T, int M, int LEN, int NT>
__device__ __forceinline__ void ppt_stage_inv(u64 *s, const u64 *iw, const u64 *iwp, const u64 *dc, u64 q, u64 one_p,
                                              const SfPpMod &P)
{
    static_assert(T >= 3 && (T & 1), "compiled rings have an odd prime t");
    constexpr int THIRD = LEN / T, STRIDE = M / LEN;
#pragma unroll 1
    for (int g0 = 0; g0 < M / T; g0 += NT) {
        const int idx = g0 + threadIdx.x;
        if (idx >= M / T) break;
        const int blk = idx / THIRD, j = idx - blk * THIRD;
        const int base = blk * LEN + j;
        u64 x[T];
#pragma unroll
        for (int k = 0; k < T; ++k) {
            const u64 v = s[base + k * THIRD];
            const int e = STRIDE * j * k;
            x[k] = e ? sf_mul_shoup(v, __ldg(iw + e), __ldg(iwp + e), q) : v;
        }
        if constexpr (T == 3) {
            ppt_dft3<true>(x[0], x[1], x[2], P);
#pragma unroll
            for (int r = 0; r < 3; ++r) s[base + r * THIRD] = x[r];
        } else {
            ppt_dft_pairs<T, true>(x, dc, q, one_p);
#pragma unroll
            for (int r = 0; r < T; ++r) s[base + r * THIRD] = x[r];
        }
    }
}

template <int T, int M, int LEN, int NT>
__device__ __forceinline__ void ppt_forward(u64 *s, const u64 *w, const u64 *wp, const u64 *dc, u64 q, u64 one_p,
                                            const SfPpMod &P)
{
    ppt_stage_fwd<T, M, LEN, NT>(s, w, wp, dc, q, one_p, P);
    __syncthreads();
    if constexpr (LEN / T >= T) ppt_forward<T, M, LEN / T, NT>(s, w, wp, dc, q, one_p, P);
}

// the whole forward transform with the first stage's inputs read through
// ld(index), index < M (each read once), e.g. straight from global memory
template <int T, int M, int NT, class LD>
__device__ __forceinline__ void ppt_forward_ld(u64 *s, LD ld, const u64 *w, const u64 *wp, const u64 *dc, u64 q,
                                               u64 one_p, const SfPpMod &P)
{
    ppt_stage_fwd_ld<T, M, M, NT>(s, ld, w, wp, dc, q, one_p, P);
    __syncthreads();
    if constexpr (M / T >= T) ppt_forward<T, M, M / T, NT>(s, w, wp, dc, q, one_p, P);
}

template <int T, int M, int LEN, int NT>
__device__ __forceinline__ void ppt_inverse(u64 *s, const u64 *iw, const u64 *iwp, const u64 *dc, u64 q, u64 one_p,
                                            const SfPpMod &P)
{
    ppt_stage_inv<T, M, LEN, NT>(s, iw, iwp, dc, q, one_p, P);
    __syncthreads();
    if constexpr (LEN * T <= M) ppt_inverse<T, M, LEN * T, NT>(s, iw, iwp, dc, q, one_p, P);
}

// ---- lazy stages --------------------------------------------------------------
// The stages above keep every value canonical: a comparison and a select after
// each sum and each product.  With primes below 2^50 nothing has to be reduced
// inside a transform: products land below 4q whatever their input (pp_mad), an
// untwiddled sum of t values grows the bound by t per forward stage, to
// max(M, 4 M / 3) q < 2^63 after the last one, and by 4 (t - 1) q per inverse
// stage.  The accumulator rides through the wide multiplies, the sums of a t-point
// DFT with them.  Bound by the integer multiplier; twiddles (w, companion) lie
// stage by stage in the order the threads read them, 16 bytes a load.  4096 x 5
// transforms: 756 us canonical and 466 us lazy at 3^7, 1363 and 745 us at 5^5, 1152
// and 723 us at 7^4.

// acc + r with r = x w (mod q), 0 <= r < 4q for any x < 2^64 (truncated quotient)
__device__ __forceinline__ u64 pp_mad(u64 acc, u64 x, const pp_pair w, u64 q)
{
    return acc + x * w.x + sf_mulhi_trunc(x, w.y) * (0 - q);
}
// v (below 2^32 q) brought below 3q, and to [0, q)
__device__ __forceinline__ u64 pp_red3(u64 v, const SfPpMod &P)
{
    return v + (u64)__umulhi((unsigned)(v >> P.sh), P.binv) * (0 - P.q);
}
__device__ __forceinline__ u64 pp_canon(u64 v, const SfPpMod &P) { return sf_csub(sf_csub(pp_red3(v, P), P.q), P.q); }

// Constants of the lazy t-point DFTs, zeta = omega^(M/t), z_k = zeta^k:
//   t = 3: -1/2, (z_1 - z_2) / 2
//   t = 5: -1/4, (c_1 - c_2) / 2, s_2, s_1 - s_2, -(s_1 + s_2)
//   t = 7: C_rk, S_rk for r, k = 1 .. 3, as in ppt_dft_pairs
// with c_k, s_k = (z_k +- z_-k) / 2.
template <int T>
struct SfPpDft {
    static constexpr int H = (T - 1) / 2, N = T == 3 ? 2 : T == 5 ? 5 : 2 * H * H;
};

// x (below bnd q) replaced by its t-point DFT, forward or inverse, below
// max(t bnd, bnd + 8 H) q.  t = 5 is Winograd's 5-point DFT (5 products, where the
// pairs take 8): c_1 + c_2 = -1/2 makes the even part -1/4 (A_1 + A_2) +- d (A_1 -
// A_2), and the odd part s_1 B_1 + s_2 B_2, s_2 B_1 - s_1 B_2 shares s_2 (B_1 + B_2).
template <int T, bool INV>
__device__ __forceinline__ void ppt_dft_lazy(u64 (&x)[T], const pp_pair *c, u64 q, u64 bnd)
{
    constexpr int H = (T - 1) / 2;
    const u64 bq = bnd * q;
    u64 A[H], B[H], y0 = x[0], y[T];
#pragma unroll
    for (int r = 1; r <= H; ++r) {
        A[r - 1] = x[r] + x[T - r];
        B[r - 1] = x[r] + bq - x[T - r];
        y0 += A[r - 1];
    }
    if constexpr (T == 3) {   // zeta + zeta^2 = -1
        const u64 U = pp_mad(x[0], A[0], __ldg(c + 0), q);
        y[1] = pp_mad(U, B[0], __ldg(c + 1), q);
        y[2] = U + U + 4 * q - y[1];
    } else if constexpr (T == 5) {
        const u64 a = pp_mad(x[0], A[0] + A[1], __ldg(c + 0), q);
        const u64 U1 = pp_mad(a, A[0] + 2 * bq - A[1], __ldg(c + 1), q), U2 = a + a + 4 * q - U1;
        const u64 p = pp_mad(0, B[0] + B[1], __ldg(c + 2), q);
        const u64 V1 = pp_mad(p, B[0], __ldg(c + 3), q), V2 = pp_mad(p, B[1], __ldg(c + 4), q);
        y[1] = U1 + V1;
        y[4] = U1 + 8 * q - V1;
        y[2] = U2 + V2;
        y[3] = U2 + 8 * q - V2;
    } else {
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            u64 U = x[0];
#pragma unroll
            for (int r = 0; r < H; ++r) U = pp_mad(U, A[r], __ldg(c + 2 * (r * H + k - 1)), q);
            y[k] = U;
#pragma unroll
            for (int r = 0; r < H; ++r) y[k] = pp_mad(y[k], B[r], __ldg(c + 2 * (r * H + k - 1) + 1), q);
            y[T - k] = U + U + 4 * H * q - y[k];
        }
    }
    x[0] = y0;
#pragma unroll
    for (int k = 1; k < T; ++k) x[k] = INV ? y[T - k] : y[k];
}

// bound, as a multiple of q, of the inputs of the forward stage of span LEN:
// canonical, then sums of t values or products below 4q
template <int T, int M, int LEN>
__host__ __device__ constexpr int ppt_bound()
{
    return LEN == M ? 1 : T == 3 ? 4 * (M / LEN / 3) : M / LEN;
}

// Twiddles of span LEN: tw[M - LEN + (k - 1) LEN / t + j], j < LEN / t.

// value k of the butterfly at point j of a block of span LEN, (un)twiddled
template <int T, int M, int LEN>
__device__ __forceinline__ void ppt_twiddle(u64 &x, int k, int j, const pp_pair *tw, u64 q)
{
    if (LEN > T && k > 0) x = pp_mad(0, x, __ldg(tw + (M - LEN) + (k - 1) * (LEN / T) + j), q);
}
// forward: the DFT, then the twiddles; inverse: untwiddle, then the DFT with zeta^-1
template <int T, int M, int LEN, bool INV>
__device__ __forceinline__ void ppt_bfly(u64 (&x)[T], int j, const pp_pair *tw, const pp_pair *c, u64 q)
{
#pragma unroll
    for (int k = 0; INV && k < T; ++k) ppt_twiddle<T, M, LEN>(x[k], k, j, tw, q);
    ppt_dft_lazy<T, INV>(x, c, q, INV ? 4 : ppt_bound<T, M, LEN>());
#pragma unroll
    for (int k = 0; !INV && k < T; ++k) ppt_twiddle<T, M, LEN>(x[k], k, j, tw, q);
}

// A phase: the stages of span LEN and, with radix 9, LEN / 3 as well (half the
// exchanges, and the second stage's twiddles serve three butterflies).  idx: the
// thread's group of points, M / radix of them; ld and st read and write point e, all
// inputs before all outputs.
template <int T, int M, int LEN, bool INV, class LD, class ST>
__device__ __forceinline__ void ppt_phase(int idx, LD ld, ST st, const pp_pair *tw, const pp_pair *c, u64 q)
{
    if constexpr (ppt_radix(T, M) == 9 && LEN >= 9) {
        constexpr int D = LEN / 9;
        const int blk = idx / D, j = idx - blk * D, base = blk * LEN + j;
        u64 v[9];
#pragma unroll
        for (int r = 0; r < 9; ++r) v[r] = ld(base + r * D);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if ((h == 0) != INV) {   // span LEN: points r, r + 3, r + 6
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    u64 x[3] = {v[r], v[r + 3], v[r + 6]};
                    ppt_bfly<3, M, LEN, INV>(x, j + r * D, tw, c, q);
                    v[r] = x[0], v[r + 3] = x[1], v[r + 6] = x[2];
                }
            } else {   // span LEN / 3: points 3 k, 3 k + 1, 3 k + 2
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    u64 x[3] = {v[3 * k], v[3 * k + 1], v[3 * k + 2]};
                    ppt_bfly<3, M, LEN / 3, INV>(x, j, tw, c, q);
                    v[3 * k] = x[0], v[3 * k + 1] = x[1], v[3 * k + 2] = x[2];
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 9; ++r) st(base + r * D, v[r]);
    } else {
        // radix 9: span 3 alone, 3 butterflies of neighbouring blocks
        constexpr int D = LEN / T, W = ppt_radix(T, M) / T;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const int g = idx * W + w, blk = g / D, j = g - blk * D, base = blk * LEN + j;
            u64 x[T];
#pragma unroll
            for (int r = 0; r < T; ++r) {
                x[r] = ld(base + r * D);
                if (INV) ppt_twiddle<T, M, LEN>(x[r], r, j, tw, q);
            }
            ppt_dft_lazy<T, INV>(x, c, q, INV ? 4 : ppt_bound<T, M, LEN>());
#pragma unroll
            for (int r = 0; r < T; ++r) {
                if (!INV) ppt_twiddle<T, M, LEN>(x[r], r, j, tw, q);
                st(base + r * D, x[r]);
            }
        }
    }
}

// the block's whole transform from span LEN on; ld reads the first phase's inputs
template <int T, int M, int LEN, class LD>
__device__ __forceinline__ void ppt_lazy_fwd(u64 *s, LD ld, const pp_pair *tw, const pp_pair *c, u64 q)
{
    constexpr int RX = ppt_radix(T, M), NEXT = LEN >= RX ? LEN / RX : LEN / T;
    if (threadIdx.x < M / RX)
        ppt_phase<T, M, LEN, false>(threadIdx.x, ld, [s](int e, u64 v) { s[e] = v; }, tw, c, q);
    __syncthreads();
    if constexpr (NEXT >= T) ppt_lazy_fwd<T, M, NEXT>(s, [s](int e) { return s[e]; }, tw, c, q);
}

// inputs below 3q; the last phase applies M^-1 and leaves canonical values
template <int T, int M, int LEN>
__device__ __forceinline__ void ppt_lazy_inv(u64 *s, const pp_pair *tw, const pp_pair *c, u64 q, const pp_pair minv)
{
    constexpr int RX = ppt_radix(T, M);
    if (threadIdx.x < M / RX)
        ppt_phase<T, M, LEN, true>(
            threadIdx.x, [s](int e) { return s[e]; },
            [&](int e, u64 v) { s[e] = LEN == M ? sf_csub(sf_csub(pp_mad(0, v, minv, q), 2 * q), q) : v; }, tw, c, q);
    __syncthreads();
    if constexpr (LEN < M) ppt_lazy_inv<T, M, LEN * RX>(s, tw, c, q, minv);
}

// first span of the inverse phases: radix 9 takes span 3 alone if alpha is odd
template <int T, int ALPHA>
__host__ __device__ constexpr int ppt_first() { return ppt_radix(T, SfPpT<T, ALPHA>::M) == T || ALPHA % 2 ? T : 9; }

// ---- one interface over the compiled and the generic transforms -------------
// T = 0 stands for the generic ring (runtime t and alpha).  The fused key
// switches of compiled rings are bounded to two blocks per SM (three at t = 3,
// whose blocks are smaller): at M = 5^5 that caps the torus kernel's registers at 48,
// with a few spilled words.  Torus key switch of 4096 ciphertexts, 5 digits: 2423 us
// at 5^5, 1631 us at 3^7 (1709 with two blocks); 4852 and 2747 us with the canonical
// stages.  k_pp_ks spills 248 bytes a thread at 5^5 and 292 at 3^7 under the same
// bounds and still gains by them: 2000 ciphertexts of 3 limbs take 1400 us at 5^5
// (1 block 1690, 3 blocks 1518), 1391 at 7^4 (1853, 1385) and 899 at 3^7 (1 block
// 1323, 2 blocks 958); 30 ciphertexts 56.1 (54.0, 64.4), 58.1 (58.3, 62.3) and
// 55.9 us (47.7, 47.7).
template <int T, int ALPHA>
struct SfPpShape {
    static constexpr int NT = SfPpT<T, ALPHA>::THREADS, MMAX = SfPpT<T, ALPHA>::M, MINB = T == 3 ? 3 : 2;
};
template <int ALPHA>
struct SfPpShape<0, ALPHA> {
    static constexpr int NT = SF_PP_THREADS, MMAX = SF_PP_MAX_M, MINB = 1;
};

// M, N, m of the ring, constants in the compiled ones
template <int T, int ALPHA>
__device__ __forceinline__ int pp_len(const SfPpRing &R) { return T ? SfPpShape<T, ALPHA>::MMAX : R.M; }
template <int T, int ALPHA>
__device__ __forceinline__ int pp_fold(const SfPpRing &R) { return T ? SfPpShape<T, ALPHA>::MMAX / (T ? T : 1) : R.m; }
template <int T, int ALPHA>
__device__ __forceinline__ int pp_deg(const SfPpRing &R) { return pp_len<T, ALPHA>(R) - pp_fold<T, ALPHA>(R); }

// forward transform of the block's length-M vector modulo prime j, the first
// stage reading its inputs through ld(index), index < M (each read once).  LZ
// (compiled rings with R.lazy): the outputs are left below 2^63, see pp_canon.
template <int T, int ALPHA, bool LZ, class LD>
__device__ __forceinline__ void pp_block_forward_ld(u64 *s, LD ld, const SfPpRing &R, int j)
{
    if constexpr (T == 0) {
        for (int e = threadIdx.x; e < R.M; e += blockDim.x) s[e] = ld(e);
        __syncthreads();
        pp_forward(s, R, j);
    } else if constexpr (LZ) {
        constexpr int M = SfPpT<T, ALPHA>::M, C = SfPpDft<T>::N;
        ppt_lazy_fwd<T, M, M>(s, ld, R.tw + (size_t)2 * j * M, R.dftl + (size_t)j * C, R.mod[j].q);
    } else {
        constexpr int M = SfPpT<T, ALPHA>::M, H = (T - 1) / 2;
        const SfPpMod &P = R.mod[j];
        ppt_forward_ld<T, M, SfPpT<T, ALPHA>::THREADS>(s, ld, R.w + (size_t)j * M, R.w_p + (size_t)j * M, R.dftc + (size_t)j * H * H * 4, P.q,
                             P.one_p, P);
    }
}

// inverse transform, scaled by M^-1; inputs canonical, below 3q if LZ
template <int T, int ALPHA, bool LZ>
__device__ __forceinline__ void pp_block_inverse(u64 *s, const SfPpRing &R, int j)
{
    if constexpr (T == 0) {
        pp_inverse(s, R, j);
    } else if constexpr (LZ) {
        constexpr int M = SfPpT<T, ALPHA>::M, C = SfPpDft<T>::N;
        const SfPpMod &P = R.mod[j];
        ppt_lazy_inv<T, M, ppt_first<T, ALPHA>()>(s, R.tw + (size_t)(2 * j + 1) * M, R.dftl + (size_t)j * C, P.q,
                                                                            make_ulonglong2(P.minv, P.minv_p));
    } else {
        constexpr int M = SfPpT<T, ALPHA>::M, H = (T - 1) / 2, NT = SfPpT<T, ALPHA>::THREADS;
        const SfPpMod &P = R.mod[j];
        ppt_inverse<T, M, T, NT>(s, R.iw + (size_t)j * M, R.iw_p + (size_t)j * M, R.dftc + (size_t)j * H * H * 4, P.q,
                             P.one_p, P);
        for (int e = threadIdx.x; e < M; e += NT) s[e] = sf_mul_shoup(s[e], P.minv, P.minv_p, P.q);
        __syncthreads();
    }
}

// floor(x 2^64 / q) for x < q: 2^64 = one_p q + rm, and floor(x rm / q) by
// Shoup's product with at most one correction
__device__ __forceinline__ u64 pp_companion(u64 x, const SfPpMod &P)
{
    u64 h = sf_mulhi(x, P.rm_p);
    const u64 rem = x * P.rm - h * P.q;
    if (rem >= P.q) ++h;
    return x * P.one_p + h;
}

// runs the statements with constexpr T, ALPHA when (t, alpha) is one of the
// compiled rings; `done` tells whether it did
#define SF_PPT_DISPATCH(t, alpha, done, ...)                                                 \
    do {                                                                                       \
        done = true;                                                                           \
        if ((t) == 3 && (alpha) == 7) { constexpr int T = 3, ALPHA = 7; __VA_ARGS__ }          \
        else if ((t) == 3 && (alpha) == 4) { constexpr int T = 3, ALPHA = 4; __VA_ARGS__ }     \
        else if ((t) == 3 && (alpha) == 3) { constexpr int T = 3, ALPHA = 3; __VA_ARGS__ }     \
        else if ((t) == 5 && (alpha) == 5) { constexpr int T = 5, ALPHA = 5; __VA_ARGS__ }     \
        else if ((t) == 5 && (alpha) == 3) { constexpr int T = 5, ALPHA = 3; __VA_ARGS__ }     \
        else if ((t) == 5 && (alpha) == 2) { constexpr int T = 5, ALPHA = 2; __VA_ARGS__ }     \
        else if ((t) == 7 && (alpha) == 4) { constexpr int T = 7, ALPHA = 4; __VA_ARGS__ }     \
        else if ((t) == 7 && (alpha) == 2) { constexpr int T = 7, ALPHA = 2; __VA_ARGS__ }     \
        else done = false;                                                                     \
    } while (0)

// the same with constexpr LZ as well, with T = 0 for every other ring
#define SF_PP_DISPATCH_ANY(R, ...)                                                          \
    do {                                                                                    \
        bool done_ = false;                                                                 \
        if ((R).lazy)                                                                       \
            SF_PPT_DISPATCH((R).t, (R).alpha, done_, [[maybe_unused]] constexpr bool LZ = true; __VA_ARGS__); \
        else                                                                                \
            SF_PPT_DISPATCH((R).t, (R).alpha, done_, [[maybe_unused]] constexpr bool LZ = false; __VA_ARGS__); \
        if (!done_) {                                                                       \
            constexpr int T = 0, ALPHA = 0;                                                 \
            [[maybe_unused]] constexpr bool LZ = false;                                     \
            __VA_ARGS__                                                                     \
        }                                                                                   \
    } while (0)

// the automorphisms of the tower of Sec. 2.3: per step (h, length), the step
// maps x to sum_{k < length} tau_h^k(x)
void sf_pp_tower_steps(const SfPpRing &R, int gamma, std::vector<std::pair<int, int>> &steps);
