// sf_ks_up.cu -- first kernel of a key switch: ModUp of tau_d(u.a).
//
// Groups: (column tile, digit j, part of the moduli); items: merges.  A block
// reads the digit's limbs of tau_d(u.a) -- coefficients that k_ks_gather left, or,
// for NTT-domain operands, the inverse column pass of the rows that k_ks1 left --
// scales them to y_i = [x_i Qhat_i^-1]_{q_i} (canonical: the base conversion
// depends on the representative) and keeps them in registers.  For each modulus
// it converts (lazy sums), runs the forward column pass and stores the
// half-transformed extension x2.
//
// Bound by the integer multiplier (nm forward column passes per digit against
// nd reads and nm writes).  When a launch has fewer units than one resident
// wave the moduli are split over several blocks, which convert again: a single
// rotation at N = 2^16 has 96 (tile, digit) units for 456 block slots.  Digits of
// three and four limbs hold 64 registers of y beside x and spill up to 356 bytes a
// thread of 80 registers; 32 rotations at N = 2^16, 8 + 4 primes of 50 bits take
// 1718 us all the same, 3425 with tile sweeps in shared memory.
#include <algorithm>

#include "sf_async.cuh"
#include "sf_kernels.cuh"
#include "sf_ks.h"
#include "sf_reg.cuh"

template <int LR, int LC, int ND, bool PM>
__global__ void __launch_bounds__(SfShape<LR>::NT, SfShape<LR>::BPS) k_ks2(SfRing R, SfKsBatch B, int ng, int nsplit)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SfColT<LR, PM> T;
    sf_pair *tab = (sf_pair *)smem_raw;                   // [nm][R]
    // two exchange buffers, by turns
    u64 *buf = (u64 *)(tab + (size_t)R.nm * SfShape<LR>::S), *other = buf + SfShape<LR>::WORDS;
    auto turn = [&] {
        u64 *used = buf;
        buf = other;
        other = used;
    };
    sf_pdl_next(B);
    sf_stage_cols<LR>(tab, R.colP, 0, R.nm);
    __syncthreads();
    sf_pdl_wait(B);
    const SfUnitRange U = sf_unit_range(ng * B.count);
    const size_t per = sf_ks_scratch_words(R);
    // item-major: the blocks in flight work on the tiles of a few merges
    SfCursor C(U.u0, ng);   // C.grp: merge, C.item: group
    for (int u = U.u0; u < U.u1; ++u, C.next()) {
        const int grp = C.item, b = C.grp;
        const int part = grp % nsplit, j = (grp / nsplit) % R.dnum, col = (grp / nsplit / R.dnum) * SfShape<LR>::NB + T.b;
        const int lo = j * R.K, nd = min(lo + R.K, R.L) - lo;
        u64 y[ND][8];
        const u64 *src = B.scratch + per * b + ((size_t)((B.ntt ? sf_ks_x1(R) : sf_ks_ta(R)) + lo) << (LR + LC)) + col;
#pragma unroll
        for (int t = 0; t < ND; ++t) {
            if (t >= nd) break;
#pragma unroll
            for (int r = 0; r < 8; ++r) y[t][r] = src[((size_t)t << (LR + LC)) + ((size_t)(B.ntt ? T.kl(r) : T.k1(r)) << LC)];
        }
#pragma unroll
        for (int t = 0; t < ND; ++t) {
            if (t >= nd) break;
            const SfMod &M = R.m[lo + t];
            sf_pair w = make_ulonglong2(R.mu_hinv[j * R.K + t], R.mu_hinv_c[j * R.K + t]);
            if (B.ntt) {
                // NTT-domain operands: TA's rows are inverse transformed, N^-1 rides on the scaling
                T.inverse(y[t], tab + (size_t)(lo + t) * SfShape<LR>::S, buf, M);
                turn();
                w = make_ulonglong2(R.mu_inv[j * R.K + t], R.mu_inv_c[j * R.K + t]);
            }
            if (B.ntt || nd > 1) {
#pragma unroll
                for (int r = 0; r < 8; ++r) y[t][r] = sf_canon(sf_mad<PM>(0, y[t][r], w, M), M);
            }
        }
        // the next unit's points on their way into L2
        if (u + 1 < U.u1) {
            const int ngrp = grp + 1 == ng ? 0 : grp + 1, nb = grp + 1 == ng ? b + 1 : b, nlo = ((ngrp / nsplit) % R.dnum) * R.K;
            const u64 *nsrc = B.scratch + per * nb + ((size_t)((B.ntt ? sf_ks_x1(R) : sf_ks_ta(R)) + nlo) << (LR + LC)) +
                              (ngrp / nsplit / R.dnum) * SfShape<LR>::NB + T.b;
            for (int t = 0; t < min(R.K, R.L - nlo); ++t)
                for (int r = 0; r < 8; ++r)
                    if (T.b % 4 == 0) sf_prefetch_l2(nsrc + ((size_t)t << (LR + LC)) + ((size_t)T.k1(r) << LC));
        }
        for (int m = part * R.nm / nsplit; m < (part + 1) * R.nm / nsplit; ++m) {
            const bool own = m >= lo && m < lo + nd;
            if (own && B.ntt) continue;   // the inner product reads tau_d(u.a) itself
            const SfMod &M = R.m[m];
            u64 x[8];
            if (nd == 1 && (R.modup_copy || own)) {
                // one-limb digit: Qhat = 1, so the conversion is the canonical
                // residue itself, below 4 q_m and taken as it is by the transform
#pragma unroll
                for (int r = 0; r < 8; ++r) x[r] = y[0][r];
            } else {
                // base conversion, lazy: each pair of terms below 4 off
#pragma unroll
                for (int r = 0; r < 8; ++r) x[r] = 0;
#pragma unroll
                for (int t = 0; t < ND; t += 2) {
                    if (t >= nd) break;
                    const size_t ci = ((size_t)(j * R.K + t)) * R.nm + m;
                    const sf_pair w = make_ulonglong2(R.mu_qhat[ci], R.mu_qhat_c[ci]);
                    if (t + 1 < ND && t + 1 < nd) {
                        const sf_pair z = make_ulonglong2(R.mu_qhat[ci + R.nm], R.mu_qhat_c[ci + R.nm]);
#pragma unroll
                        for (int r = 0; r < 8; ++r) x[r] = sf_mad2<PM>(x[r], y[t][r], w, y[t + 1 < ND ? t + 1 : 0][r], z, M);
                    } else {
#pragma unroll
                        for (int r = 0; r < 8; ++r) x[r] = sf_mad<PM>(x[r], y[t][r], w, M);
                    }
                }
            }
            T.forward(x, tab + (size_t)m * SfShape<LR>::S, buf, M);
            turn();
            u64 *dst = B.scratch + per * b + ((size_t)(j * R.nm + m) << (LR + LC)) + col;
#pragma unroll
            for (int t = 0; t < 8; ++t) dst[(size_t)T.kl(t) << LC] = x[t];
        }
    }
}

template <int LR>
static size_t up_smem(const SfRing &R)
{
    return sizeof(sf_pair) * R.nm * SfShape<LR>::S + sizeof(u64) * 2 * SfShape<LR>::WORDS;
}

template <int LR, int LC, int ND, bool PM>
static void up_launch(sf_ctx *ctx, const SfKsBatch &b, cudaStream_t st)
{
    const SfRing &R = ctx->ring;
    const size_t sm = up_smem<LR>(R);
    const int occ = sf_occupancy(k_ks2<LR, LC, ND, PM>, SfShape<LR>::NT, sm);
    const int g0 = ((1 << LC) / SfShape<LR>::NB) * R.dnum;
    // split the moduli only while the launch does not fill one wave
    const int nsplit = (int)std::max<long long>(1, std::min<long long>(R.nm, (long long)ctx->num_sms * occ / ((long long)g0 * b.count)));
    const int ng = g0 * nsplit;
    sf_pdl_launch(k_ks2<LR, LC, ND, PM>, ks_wave_blocks(ctx, occ, ng * b.count, 2), SfShape<LR>::NT, sm, st, R, b, ng, nsplit);
}

sf_status sf_ks_up_launch(sf_ctx *ctx, const SfKsBatch &b, cudaStream_t st)
{
    const int nd = std::min(ctx->ring.K, ctx->ring.L);
    cudaEvent_t ev;
    sf_launch_begin(ctx, SFK_KS2_MODUP_COL, st, &ev);
    SF_RING_DISPATCH(ctx->ring, {
        if (nd == 1) up_launch<LR, LC, 1, PM>(ctx, b, st);
        else if (nd == 2) up_launch<LR, LC, 2, PM>(ctx, b, st);
        else up_launch<LR, LC, 4, PM>(ctx, b, st);
    });
    sf_launch_end(ctx, SFK_KS2_MODUP_COL, st, ev);
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

sf_status sf_ks_up_init()
{
    const int mx = 227 * 1024;
#define SF_ATTR(K) SF_CUDA_TRY(cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
    SF_FOR_RINGS({ SF_ATTR((k_ks2<LR, LC, 1, PM>)) SF_ATTR((k_ks2<LR, LC, 2, PM>)) SF_ATTR((k_ks2<LR, LC, 4, PM>)) });
#undef SF_ATTR
    return SF_OK;
}
