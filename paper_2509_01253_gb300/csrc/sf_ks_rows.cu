// sf_ks_rows.cu -- the row passes of a key switch.
//
// k_ks1 (NTT-domain operands only): inverse row pass of tau_d(u.a).
// k_ks3: groups (row tile, modulus m); items merges.  Per digit the forward
// row pass of its extension (or tau_d(u.a) itself on the digit's own limbs of
// NTT-domain operands) and the product with the key, whose pairs are
// stored in the order the registers hold the values; then the inverse row pass
// of both accumulators, the rows that the ModDown columns read.  The key's data
// limbs carry P^-1 N^-1, so those become ACC P^-1; for NTT-domain operands
// v (+ tau_d(u.b) on the b part), which k_ks_gather left in `out`, is added
// here, so that it rides through the inverse transform.
//
// Bound by the integer multiplier: per point and digit 4 butterflies and two
// multiply-accumulates, plus 8 butterflies for the two inverse passes, against
// 8 bytes read and 16/dnum written.  Every exchange stays inside a warp, so the
// loop over the items has no block barrier; the next digit's points arrive by
// cp.async while this one is transformed.  At 256-point rows a block of 256 threads
// has 32 KB of staged twiddles, an 18 KB exchange buffer and 16 KB of points ahead;
// three blocks per SM for k_ks1, two of 128 registers for k_ks3.
#include <algorithm>

#include "sf_async.cuh"
#include "sf_kernels.cuh"
#include "sf_ks.h"
#include "sf_reg.cuh"

template <int LR, int LC, bool PM>
__global__ void __launch_bounds__(SfShape<LC>::NT, SfShape<LC>::BPS) k_ks1(SfRing R, SfKsBatch B, int ng)
{
    constexpr int NT = SfShape<LC>::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SfRowT<LC, PM> T;
    sf_pair *tw = (sf_pair *)smem_raw;
    u64 *buf = (u64 *)(tw + SfShape<LC>::PAIRS), *pre = buf + SfShape<LC>::WORDS + threadIdx.x;
    sf_pdl_next(B);
    sf_pdl_wait(B);
    const SfUnitRange U = sf_unit_range(ng * B.count);
    const size_t per = sf_ks_scratch_words(R);
    SfCursor C(U.u0, B.count);
    // group = (row tile, limb i), item = merge; each thread copies its own points ahead
    auto prefetch = [&]() {
        const u64 *src = B.scratch + per * C.item + ((size_t)(sf_ks_ta(R) + C.grp % R.L) << (LR + LC)) + T.store_at(C.grp / R.L, 0);
#pragma unroll
        for (int t = 0; t < 8; ++t) sf_cp8(pre + t * NT, src + t * NT);
        sf_cp_commit();
    };
    if (U.u0 < U.u1) prefetch();
    int staged = -1, i = 0;
    size_t off = 0;
    for (int u = U.u0; u < U.u1; ++u) {
        if (C.grp != staged) {
            i = C.grp % R.L;
            off = ((size_t)(sf_ks_x1(R) + i) << (LR + LC)) + ((size_t)T.row(C.grp / R.L, 1 << LR) << LC);
            __syncthreads();   // the previous group's readers are done
            sf_stage_row<LR, LC>(tw, R.rowP, i, C.grp / R.L);
            staged = C.grp;
            __syncthreads();
        }
        const SfMod &M = R.m[i];
        u64 *dst = B.scratch + per * C.item + off;
        u64 x[8];
        sf_cp_wait<0>();
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = pre[t * NT];
        T.template phase_inv<SfRowT<LC, PM>::LAST>(x, tw, M);
        C.next();
        if (u + 1 < U.u1) prefetch();   // this unit's points are in registers
        T.inverse_rest(x, tw, buf, M);
        sf_inv_rows_out(x, M);
#pragma unroll
        for (int t = 0; t < 8; ++t) dst[T.k1(t)] = x[t];
    }
}

template <int LR, int LC, bool PM>
__global__ void __launch_bounds__(SfShape<LC>::NT, SfShape<LC>::BPS_ACC) k_ks3(SfRing R, SfKsBatch B, int ng)
{
    constexpr int NT = SfShape<LC>::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SfRowT<LC, PM> T;
    sf_pair *tw = (sf_pair *)smem_raw;
    u64 *buf = (u64 *)(tw + SfShape<LC>::PAIRS), *pre = buf + SfShape<LC>::WORDS + threadIdx.x;
    sf_pdl_next(B);
    sf_pdl_wait(B);
    const SfUnitRange U = sf_unit_range(ng * B.count);
    const sf_pair *key = (const sf_pair *)B.key;
    // limbs of scratch per merge; as a word count it costs this kernel registers, and 2.7 %
    // (26.1 ms per resnet20-sized convolution at N = 2^14 against 25.4)
    const int per = sf_ks_ta(R) + R.L;
    // group = (row tile, modulus m), item = merge; the digit's own limbs of
    // NTT-domain operands are tau_d(u.a) itself, already transformed
    struct Group {
        int m, tile;
        size_t row;   // this thread's row in a limb
    };
    auto group = [&](int grp) -> Group {
        const int tile = grp / R.nm;
        return {grp - tile * R.nm, tile, (size_t)T.row(tile, 1 << LR) << LC};
    };
    auto own_limb = [&](int m, int j) { return B.ntt && m >= j * R.K && m < min((j + 1) * R.K, R.L); };
    // each thread copies its own points of a digit ahead
    auto prefetch = [&](const Group &G, int item, int j) {
        const u64 *base = B.scratch + ((size_t)(per * item) << (LR + LC));
        if (own_limb(G.m, j)) {
            const u64 *src = base + ((size_t)(sf_ks_ta(R) + G.m) << (LR + LC));
#pragma unroll
            for (int t = 0; t < 8; ++t) sf_cp8(pre + t * NT, src + T.store_at(G.tile, t));
        } else {
            const u64 *src = base + ((size_t)(j * R.nm + G.m) << (LR + LC)) + G.row;
#pragma unroll
            for (int t = 0; t < 8; ++t) sf_cp8(pre + t * NT, src + T.k1(t));
        }
        sf_cp_commit();
    };
    SfCursor C(U.u0, B.count);
    Group G = group(C.grp), N = G;
    if (U.u0 < U.u1) prefetch(G, C.item, 0);
    int staged = -1;
    for (int u = U.u0; u < U.u1; ++u) {
        const int b = C.item;
        if (C.grp != staged) {
            __syncthreads();   // the previous group's readers are done
            sf_stage_row<LR, LC>(tw, R.rowP, G.m, G.tile);
            staged = C.grp;
            __syncthreads();
        }
        const SfMod &M = R.m[G.m];
        C.next();
        if (C.grp != staged) N = group(C.grp);
        SfAcc<PM> acc_a[8], acc_b[8];
        u64 x[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) acc_a[t] = acc_b[t] = {0, 0};
        const sf_pair *ka = key + ((size_t)G.m << (LR + LC)) + T.store_at(G.tile, 0);
#pragma unroll 1
        for (int j = 0; j < R.dnum; ++j) {
            auto ahead = [&]() {   // once the points of this digit are in registers
                if (j + 1 < R.dnum) prefetch(G, b, j + 1);
                else if (u + 1 < U.u1) prefetch(N, C.item, 0);
            };
            sf_cp_wait<0>();
#pragma unroll
            for (int t = 0; t < 8; ++t) x[t] = pre[t * NT];
            if (own_limb(G.m, j)) {
                __syncwarp();
                ahead();
            } else {
                T.template phase_fwd<0>(x, tw, M);
                ahead();
                T.forward_rest(x, tw, buf, M);
            }
            const sf_pair *kb = ka + ((size_t)R.nm << (LR + LC));
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const sf_pair a = __ldg(ka + t * NT), c = __ldg(kb + t * NT);
                sf_acc_add<PM>(acc_a[t], x[t], a, M);
                sf_acc_add<PM>(acc_b[t], x[t], c, M);
            }
            if (j % SF_ACC_TERMS == SF_ACC_TERMS - 1 && j + 1 < R.dnum) {
#pragma unroll
                for (int t = 0; t < 8; ++t) sf_acc_close<PM>(acc_a[t], M), sf_acc_close<PM>(acc_b[t], M);
            }
            ka = kb + ((size_t)R.nm << (LR + LC));
        }
        const u64 *add = B.ntt && G.m < R.L ? merge_out(B, b) + ((size_t)G.m << (LR + LC)) + T.store_at(G.tile, 0) : nullptr;
        u64 *dst = B.scratch + ((size_t)(per * b + sf_ks_acc(R) + G.m) << (LR + LC)) + G.row;
        // one copy of the inverse pass for both parts: the code stays within the
        // instruction cache
#pragma unroll 1
        for (int part = 0; part < 2; ++part) {
            // below 3q, 4q with v
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                SfAcc<PM> a = part ? acc_b[t] : acc_a[t];
                x[t] = sf_acc_close<PM>(a, M);
            }
            if (add) {
#pragma unroll
                for (int t = 0; t < 8; ++t) x[t] += add[t * NT];
                add += (size_t)R.L << (LR + LC);
            }
            T.inverse(x, tw, buf, M);
            sf_inv_rows_out(x, M);
#pragma unroll
            for (int t = 0; t < 8; ++t) dst[T.k1(t)] = x[t];
            dst += (size_t)R.nm << (LR + LC);
        }
        G = N;
    }
}

template <int LC>
static constexpr size_t rows_smem()
{
    return sizeof(sf_pair) * SfShape<LC>::PAIRS + sizeof(u64) * (SfShape<LC>::WORDS + SfShape<LC>::TILE);
}

sf_status sf_ks_rows_launch(sf_ctx *ctx, const SfKsBatch &b, cudaStream_t st)
{
    const SfRing &R = ctx->ring;
    cudaEvent_t ev;
    SF_RING_DISPATCH(R, {
        constexpr int NT = SfShape<LC>::NT;
        constexpr size_t sm = rows_smem<LC>();
        const int ng = ((1 << LR) / SfShape<LC>::NB) * R.nm;
        sf_launch_begin(ctx, SFK_KS3_INNER_ROW, st, &ev);
        sf_pdl_launch(k_ks3<LR, LC, PM>, ks_wave_blocks(ctx, sf_occupancy(k_ks3<LR, LC, PM>, NT, sm), ng * b.count, 8), NT, sm, st, R, b, ng);
        sf_launch_end(ctx, SFK_KS3_INNER_ROW, st, ev);
    });
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

sf_status sf_ks_inv_rows_launch(sf_ctx *ctx, const SfKsBatch &b, cudaStream_t st)
{
    const SfRing &R = ctx->ring;
    cudaEvent_t ev;
    SF_RING_DISPATCH(R, {
        constexpr int NT = SfShape<LC>::NT;
        constexpr size_t sm = rows_smem<LC>();
        const int ng = ((1 << LR) / SfShape<LC>::NB) * R.L;
        sf_launch_begin(ctx, SFK_KS1_INV_ROW, st, &ev);
        sf_pdl_launch(k_ks1<LR, LC, PM>, ks_wave_blocks(ctx, sf_occupancy(k_ks1<LR, LC, PM>, NT, sm), ng * b.count, 8), NT, sm, st, R, b, ng);
        sf_launch_end(ctx, SFK_KS1_INV_ROW, st, ev);
    });
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

sf_status sf_ks_rows_init()
{
    const int mx = 227 * 1024;
#define SF_ATTR(K) SF_CUDA_TRY(cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
    SF_FOR_RINGS({ SF_ATTR((k_ks1<LR, LC, PM>)) SF_ATTR((k_ks3<LR, LC, PM>)) });
#undef SF_ATTR
    return SF_OK;
}
