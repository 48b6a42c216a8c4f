// sf_ks_down.cu -- last kernel of a key switch: ModDown and the merge.
//
// Groups: (column tile, ciphertext part p, share of the data limbs); items:
// merges.  A block runs the inverse column pass of the K special limbs'
// accumulators, scales them to y_k = [x_k Phat_k^-1]_{p_k} (canonical) and keeps
// them in registers; for each data limb it runs the inverse column pass,
// subtracts the base conversion (constants Phat_k P^-1 mod q_i; the
// accumulators carry P^-1 N^-1 already) and adds what k_ks_gather left in `out` (for
// NTT-domain operands the accumulators hold it).  The result is canonical, in the
// coefficient domain, with no forward transform after ModDown.
//
// Bound by the integer multiplier: K + L inverse column passes per part, the
// points of each copied ahead by cp.async while the one before runs.  As in the
// ModUp, a launch that does not fill one wave splits the data limbs.
//
// Three blocks of 80 registers hold x, y and what was in `out` (64 registers at
// K = 2) with 52 to 92 bytes of spills a thread, 180 to 224 at K = 3 and 4.
#include <algorithm>

#include "sf_async.cuh"
#include "sf_kernels.cuh"
#include "sf_ks.h"
#include "sf_reg.cuh"

template <int LR, int LC, int KT, bool PM>
__global__ void __launch_bounds__(SfShape<LR>::NT, SfShape<LR>::BPS) k_ks4(SfRing R, SfKsBatch B, int ng, int nsplit)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SfColT<LR, PM> T;
    sf_pair *tab = (sf_pair *)smem_raw;   // [nm][R], two buffers: points ahead and exchanges by turns
    u64 *buf = (u64 *)(tab + (size_t)R.nm * SfShape<LR>::S), *ahead = buf + SfShape<LR>::WORDS;
    sf_pdl_next(B);
    sf_stage_cols<LR>(tab, R.colP, 0, R.nm);
    __syncthreads();
    sf_pdl_wait(B);
    const SfUnitRange U = sf_unit_range(ng * B.count);
    const size_t per = sf_ks_scratch_words(R);
    // A unit's transforms: the K special limbs, then its share of the data limbs.
    // item-major: the blocks in flight work on the tiles of a few merges.
    struct Unit {
        int lo, steps, col, part;
        const u64 *acc;   // this part's accumulators at this thread's column
    };
    auto unit = [&](const SfCursor &C) -> Unit {   // C.grp: merge, C.item: group
        const int share = C.item % nsplit, g = C.item / nsplit, p = g & 1, col = (g >> 1) * SfShape<LR>::NB + T.b;
        const int lo = share * R.L / nsplit;
        return {lo, R.K + (share + 1) * R.L / nsplit - lo, col, p,
                B.scratch + per * C.grp + ((size_t)(sf_ks_acc(R) + p * R.nm) << (LR + LC)) + col};
    };
    // modulus of step s of a unit; each thread copies its own points of a step ahead
    auto step_mod = [&](const Unit &V, int s) { return s < R.K ? R.L + s : V.lo + s - R.K; };
    constexpr int LAST = SfColT<LR, PM>::LAST;
    auto prefetch = [&](const Unit &V, int s, u64 *to) {
        const u64 *src = V.acc + ((size_t)step_mod(V, s) << (LR + LC));
#pragma unroll
        for (int t = 0; t < 8; ++t) sf_cp8(T.template mine<LAST>(to) + SfShape<LR>::step(LAST, t) * SfShape<LR>::NB, src + ((size_t)T.kl(t) << LC));
        sf_cp_commit();
    };
    SfCursor C(U.u0, ng);
    Unit V = unit(C), N = V;
    if (U.u0 < U.u1) prefetch(V, 0, buf);
    for (int u = U.u0; u < U.u1; ++u) {
        u64 *out0 = merge_out(B, C.grp) + ((size_t)(V.part * R.L) << (LR + LC)) + V.col;
        // `out` holds v (+ tau_d(u.b)) of coefficient-domain operands; a plain
        // rotation has nothing to add on the a part
        const bool add = !B.ntt && (B.add_v || V.part);
        C.next();
        if (u + 1 < U.u1) N = unit(C);
        u64 y[KT][8];
#pragma unroll 1
        for (int s = 0; s < V.steps; ++s) {
            // inverse column pass of step s
            const int m = step_mod(V, s);
            const SfMod &M = R.m[m];
            u64 *out = out0 + ((size_t)m << (LR + LC));
            u64 x[8], o[8];
            sf_cp_wait<0>();
            T.template get<LAST>(x, buf);
            T.inverse(x, tab + (size_t)m * SfShape<LR>::S, buf, M, [&] {
                if (s + 1 < V.steps) prefetch(V, s + 1, ahead);
                else if (u + 1 < U.u1) prefetch(N, 0, ahead);
#pragma unroll
                for (int t = 0; t < 8; ++t) o[t] = add && s >= R.K ? out[(size_t)T.k1(t) << LC] : 0;
            });
            u64 *used = buf;
            buf = ahead;
            ahead = used;
            if (s < R.K) {
                const sf_pair w = make_ulonglong2(R.md_inv[s], R.md_inv_c[s]);
#pragma unroll
                for (int k = 0; k < KT; ++k)
                    if (k == s) {
#pragma unroll
                        for (int r = 0; r < 8; ++r) y[k][r] = sf_canon(sf_mad<PM>(0, x[r], w, M), M);
                    }
                continue;
            }
            // x + out - conv, x below 4 off once x[0] is reduced, a pair of products
            // below 4 off: the sum stays below (5 + 2 KT) off < 2^62
            x[0] = sf_red3(x[0], M);
#pragma unroll
            for (int r = 0; r < 8; ++r) x[r] += o[r] + 2 * KT * M.off;
#pragma unroll
            for (int k = 0; k < KT; k += 2) {
                if (k >= R.K) break;
                const sf_pair w = make_ulonglong2(R.md_phat[(size_t)k * R.L + m], R.md_phat_c[(size_t)k * R.L + m]);
                if (k + 1 < KT && k + 1 < R.K) {
                    const sf_pair z = make_ulonglong2(R.md_phat[(size_t)(k + 1) * R.L + m], R.md_phat_c[(size_t)(k + 1) * R.L + m]);
#pragma unroll
                    for (int r = 0; r < 8; ++r) x[r] -= sf_mad2<PM>(0, y[k][r], w, y[k + 1 < KT ? k + 1 : 0][r], z, M);
                } else {
#pragma unroll
                    for (int r = 0; r < 8; ++r) x[r] -= sf_mad<PM>(0, y[k][r], w, M);
                }
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) out[(size_t)T.k1(r) << LC] = sf_canon(x[r], M);
        }
        V = N;
    }
}

template <int LR>
static size_t down_smem(const SfRing &R)
{
    return sizeof(sf_pair) * R.nm * SfShape<LR>::S + sizeof(u64) * 2 * SfShape<LR>::WORDS;
}

template <int LR, int LC, int KT, bool PM>
static void down_launch(sf_ctx *ctx, const SfKsBatch &b, cudaStream_t st)
{
    const SfRing &R = ctx->ring;
    const size_t sm = down_smem<LR>(R);
    const int occ = sf_occupancy(k_ks4<LR, LC, KT, PM>, SfShape<LR>::NT, sm);
    const int g0 = ((1 << LC) / SfShape<LR>::NB) * 2;
    const int nsplit = (int)std::max<long long>(1, std::min<long long>(R.L, (long long)ctx->num_sms * occ / ((long long)g0 * b.count)));
    const int ng = g0 * nsplit;
    sf_pdl_launch(k_ks4<LR, LC, KT, PM>, ks_wave_blocks(ctx, occ, ng * b.count, 2), SfShape<LR>::NT, sm, st, R, b, ng, nsplit);
}

sf_status sf_ks_down_launch(sf_ctx *ctx, const SfKsBatch &b, cudaStream_t st)
{
    cudaEvent_t ev;
    sf_launch_begin(ctx, SFK_KS4_MODDOWN_COL, st, &ev);
    SF_RING_DISPATCH(ctx->ring, {
        if (ctx->ring.K == 1) down_launch<LR, LC, 1, PM>(ctx, b, st);
        else if (ctx->ring.K == 2) down_launch<LR, LC, 2, PM>(ctx, b, st);
        else down_launch<LR, LC, 4, PM>(ctx, b, st);
    });
    sf_launch_end(ctx, SFK_KS4_MODDOWN_COL, st, ev);
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

sf_status sf_ks_down_init()
{
    const int mx = 227 * 1024;
#define SF_ATTR(K) SF_CUDA_TRY(cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
    SF_FOR_RINGS({ SF_ATTR((k_ks4<LR, LC, 1, PM>)) SF_ATTR((k_ks4<LR, LC, 2, PM>)) SF_ATTR((k_ks4<LR, LC, 4, PM>)) });
#undef SF_ATTR
    return SF_OK;
}
