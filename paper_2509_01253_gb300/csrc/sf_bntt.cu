// sf_bntt.cu -- batched negacyclic NTT over every RNS limb of a batch of
// polynomials, and register-resident probes of the modular arithmetic.
//
// The batch is [count][L][N]: limb i of polynomial p is reduced modulo q_i.
// A transform is the two register-resident passes of sf_reg.cuh (forward:
// column pass, then row pass; inverse: row pass, then column pass with the
// factor N^-1).  Each pass is one launch over the units (group,
// polynomial), several waves of blocks with even shares (ks_wave_blocks), a group being a column or row tile position
// and a limb: a block takes an equal range of units (sf_unit_range), stages a
// group's twiddles when its range enters the group, and copies the next unit's
// points ahead with cp.async while it transforms the current one (loads into
// registers sank behind the transform: the column pass waited on memory).
//
// Bound by the integer multiplier: at N = 2^16 the fmaheavy pipe is busy 57 to
// 70 % of the cycles.  512 x 5 limbs of 2^16, forward: 1961 us with tile sweeps in
// shared memory, 1543 us here; 37 x 3 inverse limbs of 2^14: 32.8 and 26.6 us.
#include <algorithm>

#include "sf_async.cuh"
#include "sf_internal.h"
#include "sf_kernels.cuh"
#include "sf_ks.h"
#include "sf_reg.cuh"
#include "sf_round.h"

// sf_stage_row with every copy of a thread in flight at once: a short batch waits for
// its table, not for throughput.  Calls of 4 x 3 limbs at N = 2^10 to 2^12 back to
// back: 10.3 us with loads through registers, 8.2 so (5.2 to 5.9 and 4.7 to 5.4 us
// apart from the launches); 512 x 5 limbs of 2^16: 1555 and 1543 us.
template <int LR, int LC>
__device__ __forceinline__ void stage_row_async(sf_pair *dst, const sf_pair *__restrict__ table, int mod, int tile)
{
    constexpr int W = SfShape<LC>::PAIRS;
    const sf_pair *src = table + ((size_t)mod * ((1 << LR) / SfShape<LC>::NB) + tile) * W;
    for (int k = threadIdx.x; k < W; k += SfShape<LC>::NT) sf_cp16(dst + k, src + k);
    sf_cp_commit();
}

template <bool INV, int LR, int LC, bool PM>
__global__ void __launch_bounds__(SfShape<LC>::NT, SfShape<LC>::BPS)
    k_bntt_row(SfRing R, const u64 *src, u64 *dst, int count, int ng)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using T_ = SfRowT<LC, PM>;
    const T_ T;
    sf_pair *tw = (sf_pair *)smem_raw;
    u64 *buf = (u64 *)(tw + SfShape<LC>::PAIRS), *ahead = buf + SfShape<LC>::WORDS;
    const SfUnitRange U = sf_unit_range(ng * count);
    const size_t per = (size_t)R.L << (LR + LC);
    // group = (row tile, limb i), item = polynomial; offset of this thread's row
    auto group_off = [&](int grp) -> size_t {
        return ((size_t)(grp % R.L) << (LR + LC)) + ((size_t)T.row(grp / R.L, 1 << LR) << LC) + T.k1(0);
    };
    SfCursor C(U.u0, count);
    size_t off = group_off(C.grp) + per * C.item;
    // each thread copies its own points of the next unit ahead
    auto prefetch = [&]() {
#pragma unroll
        for (int t = 0; t < 8; ++t) sf_cp8(T.template mine<0>(ahead) + SfShape<LC>::step(0, t), src + off + (T.k1(t) - T.k1(0)));
        sf_cp_commit();
    };
    if (U.u0 < U.u1) prefetch();
    int staged = -1, mod = 0;
    for (int u = U.u0; u < U.u1; ++u) {
        if (C.grp != staged) {
            mod = C.grp % R.L;
            __syncthreads();   // the previous group's readers are done
            stage_row_async<LR, LC>(tw, R.rowP, mod, C.grp / R.L);
            staged = C.grp;
            sf_cp_wait<0>();
            __syncthreads();
        }
        const SfMod &M = R.m[mod];
        u64 x[8];
        sf_cp_wait<0>();
        if (INV) __syncwarp();   // the last phase's points lie among the row's threads
        T.template get<INV ? T_::LAST : 0>(x, ahead);
        u64 *d = dst + off;
        // the next unit's copy overtakes this unit's stores: in place, the two units
        // touch different rows or polynomials
        C.next();
        off = C.grp == staged ? off + per : group_off(C.grp);
        if (INV) {
            T.template phase_inv<T_::LAST>(x, tw, M);
            __syncwarp();
            if (u + 1 < U.u1) prefetch();
            T.inverse_rest(x, tw, buf, M);
            sf_inv_rows_out(x, M);
#pragma unroll
            for (int t = 0; t < 8; ++t) d[T.k1(t) - T.k1(0)] = x[t];
        } else {
            T.template phase_fwd<0>(x, tw, M);
            if (u + 1 < U.u1) prefetch();
            T.forward_rest(x, tw, buf, M);
            T.template exchange<T_::LAST, T_::FIRST>(x, buf);   // back to coalesced positions
#pragma unroll
            for (int t = 0; t < 8; ++t) d[T.k1(t) - T.k1(0)] = sf_canon(x[t], M);
        }
    }
}

template <bool INV, int LR, int LC, bool PM>
__global__ void __launch_bounds__(SfShape<LR>::NT, SfShape<LR>::BPS)
    k_bntt_col(SfRing R, const u64 *src, u64 *dst, int count, int ng)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SfColT<LR, PM> T;
    sf_pair *tab = (sf_pair *)smem_raw;
    // two buffers: points ahead and exchanges by turns
    u64 *buf = (u64 *)(tab + SfShape<LR>::S), *ahead = buf + SfShape<LR>::WORDS;
    const SfUnitRange U = sf_unit_range(ng * count);
    const size_t per = (size_t)R.L << (LR + LC);
    // group = (column tile, limb i), item = polynomial; offset of this thread's column
    auto group_off = [&](int grp) -> size_t {
        return ((size_t)(grp % R.L) << (LR + LC)) + (grp / R.L) * SfShape<LR>::NB + T.b;
    };
    SfCursor C(U.u0, count);
    size_t off = group_off(C.grp) + per * C.item;
    // each thread copies its own points of the next unit ahead
    constexpr int PH = INV ? SfColT<LR, PM>::LAST : 0;
    auto prefetch = [&](u64 *to) {
#pragma unroll
        for (int t = 0; t < 8; ++t) sf_cp8(T.template mine<PH>(to) + SfShape<LR>::step(PH, t) * SfShape<LR>::NB, src + off + ((size_t)T.template k<PH>(t) << LC));
        sf_cp_commit();
    };
    if (U.u0 < U.u1) prefetch(buf);
    int staged = -1, mod = 0;
    for (int u = U.u0; u < U.u1; ++u) {
        if (C.grp != staged) {
            mod = C.grp % R.L;
            __syncthreads();   // the previous group's readers are done
            sf_stage_cols<LR>(tab, R.colP, mod, 1);
            staged = C.grp;
            __syncthreads();
        }
        const SfMod &M = R.m[mod];
        u64 x[8];
        sf_cp_wait<0>();
        T.template get<PH>(x, buf);
        u64 *d = dst + off;
        C.next();
        off = C.grp == staged ? off + per : group_off(C.grp);
        auto next = [&] {
            if (u + 1 < U.u1) prefetch(ahead);
        };
        if (INV) {
            T.inverse(x, tab, buf, M, next);
#pragma unroll
            for (int t = 0; t < 8; ++t) d[(size_t)T.k1(t) << LC] = sf_canon(sf_mad<PM>(0, x[t], make_ulonglong2(M.ninv, M.ninv_c), M), M);
        } else {
            T.forward(x, tab, buf, M, next);
#pragma unroll
            for (int t = 0; t < 8; ++t) d[(size_t)T.kl(t) << LC] = x[t];
        }
        u64 *used = buf;
        buf = ahead;
        ahead = used;
    }
}

template <int LC>
static constexpr size_t bntt_smem_row() { return sizeof(sf_pair) * SfShape<LC>::PAIRS + sizeof(u64) * 2 * SfShape<LC>::WORDS; }
template <int LR>
static constexpr size_t bntt_smem_col() { return sizeof(sf_pair) * SfShape<LR>::S + sizeof(u64) * 2 * SfShape<LR>::WORDS; }

template <bool INV, int LR, int LC, bool PM>
static void bntt_row(sf_ctx *ctx, const u64 *src, u64 *dst, int count, cudaStream_t st)
{
    const int ng = ((1 << LR) / SfShape<LC>::NB) * ctx->ring.L;
    const size_t sm = bntt_smem_row<LC>();
    cudaEvent_t ev;
    const int nb = ks_wave_blocks(ctx, sf_occupancy(k_bntt_row<INV, LR, LC, PM>, SfShape<LC>::NT, sm), ng * count, 8);
    sf_launch_begin(ctx, SFK_BNTT_ROW, st, &ev);
    k_bntt_row<INV, LR, LC, PM><<<nb, SfShape<LC>::NT, sm, st>>>(ctx->ring, src, dst, count, ng);
    sf_launch_end(ctx, SFK_BNTT_ROW, st, ev);
}

template <bool INV, int LR, int LC, bool PM>
static void bntt_col(sf_ctx *ctx, const u64 *src, u64 *dst, int count, cudaStream_t st)
{
    const int ng = ((1 << LC) / SfShape<LR>::NB) * ctx->ring.L;
    const size_t sm = bntt_smem_col<LR>();
    cudaEvent_t ev;
    const int nb = ks_wave_blocks(ctx, sf_occupancy(k_bntt_col<INV, LR, LC, PM>, SfShape<LR>::NT, sm), ng * count, 8);
    sf_launch_begin(ctx, SFK_BNTT_COL, st, &ev);
    k_bntt_col<INV, LR, LC, PM><<<nb, SfShape<LR>::NT, sm, st>>>(ctx->ring, src, dst, count, ng);
    sf_launch_end(ctx, SFK_BNTT_COL, st, ev);
}

extern "C" sf_status sf_ntt_batch(sf_ctx *ctx, const uint64_t *d_in, uint64_t *d_out, int32_t count, int32_t inverse,
                                  void *stream)
{
    SF_CHECK_CTX(ctx);
    if (!d_in || !d_out || count < 1 || (inverse != 0 && inverse != 1))
        return sf_set_error(SF_EINVAL, "sf_ntt_batch: bad arguments");
    const SfRing &R = ctx->ring;
    cudaStream_t st = (cudaStream_t)stream;
    // tiles of a limb: R or C over 16, or 8 for 256-point sub-transforms
    if ((long long)count * R.L * (R.log_c == 8 ? std::max(R.r / 8, R.c / (R.log_r == 8 ? 8 : 16)) : R.c / 16) > INT32_MAX)
        return sf_set_error(SF_EINVAL, "sf_ntt_batch: count too large");
    SF_RING_DISPATCH(R, {
        if (!inverse) {
            bntt_col<false, LR, LC, PM>(ctx, d_in, d_out, count, st);
            bntt_row<false, LR, LC, PM>(ctx, d_out, d_out, count, st);
        } else {
            bntt_row<true, LR, LC, PM>(ctx, d_in, d_out, count, st);
            bntt_col<true, LR, LC, PM>(ctx, d_out, d_out, count, st);
        }
    });
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

sf_status sf_bntt_init_attributes()
{
    const int mx = 227 * 1024;
#define SF_ATTR(K) SF_CUDA_TRY(cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
    SF_FOR_RINGS({
        SF_ATTR((k_bntt_row<false, LR, LC, PM>)) SF_ATTR((k_bntt_row<true, LR, LC, PM>))
        SF_ATTR((k_bntt_col<false, LR, LC, PM>)) SF_ATTR((k_bntt_col<true, LR, LC, PM>))
    });
#undef SF_ATTR
    return SF_OK;
}

// ---------------------------------------------------------------- probes ----
// Each thread keeps 8 residues in registers and applies PROBE_ITERS rounds of
// 12 operations to them (a radix-8 unit: 3 stages of 4 butterflies, or 12
// multiply-accumulates), then stores them.  Nothing else is read or written,
// so the rate is the arithmetic ceiling of these operations on this GPU.
#define PROBE_ITERS 1024
#define PROBE_OPS (12 * PROBE_ITERS)

template <int KIND, bool PM>
__global__ void __launch_bounds__(256, 2) k_probe(u64 *buf, SfMod M, sf_pair t0, sf_pair t1, sf_pair t2, sf_pair t3)
{
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    u64 x[8], acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        x[i] = buf[i * stride + t];
        acc[i] = 0;
    }
#pragma unroll 1
    for (int it = 0; it < PROBE_ITERS; ++it) {
        if (KIND == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) sf_fwd<PM>(x[i], x[i + 4], t0, M);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                sf_fwd<PM>(x[i], x[i + 2], t1, M);
                sf_fwd<PM>(x[i + 4], x[i + 6], t2, M);
            }
#pragma unroll
            for (int i = 0; i < 8; i += 2) sf_fwd<PM>(x[i], x[i + 1], t3, M);
        } else if (KIND == 1) {
#pragma unroll
            for (int i = 0; i < 8; i += 2) sf_inv<PM>(x[i], x[i + 1], t3, M, M.off);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                sf_inv<PM>(x[i], x[i + 2], t1, M, M.off);
                sf_inv<PM>(x[i + 4], x[i + 6], t2, M, M.off);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) sf_inv<PM>(x[i], x[i + 4], t0, M, M.off);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                acc[i] = sf_mad<PM>(acc[i], x[i], (i & 3) == 0 ? t0 : (i & 3) == 1 ? t1 : (i & 3) == 2 ? t2 : t3, M);
                x[i] ^= acc[i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[i] = sf_mad<PM>(acc[i], x[i + 4], i == 0 ? t0 : i == 1 ? t1 : i == 2 ? t2 : t3, M);
                x[i] += acc[i + 4];
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) buf[i * stride + t] = x[i] + acc[i];
}

extern "C" sf_status sf_modmul_probe(sf_ctx *ctx, int32_t kind, double *gmodmul_per_s)
{
    SF_CHECK_CTX(ctx);
    if (!gmodmul_per_s || kind < 0 || kind > 2) return sf_set_error(SF_EINVAL, "sf_modmul_probe: bad arguments");
    const SfMod &M = ctx->ring.m[0];
    const int pm = ctx->ring.pm;
    using Kernel = void (*)(u64 *, SfMod, sf_pair, sf_pair, sf_pair, sf_pair);
    static const Kernel kernels[2][3] = {{k_probe<0, false>, k_probe<1, false>, k_probe<2, false>},
                                         {k_probe<0, true>, k_probe<1, true>, k_probe<2, true>}};
    const Kernel kernel = kernels[pm][kind];
    const int grid = ctx->num_sms * sf_occupancy(kernel, 256, 0);
    const size_t words = (size_t)8 * grid * 256;
    SF_CUDA_TRY(cudaDeviceSynchronize());
    void *w = nullptr;
    SF_TRY(sf_scratch(ctx, words * sizeof(u64), &w));
    u64 *buf = (u64 *)w;
    SF_CUDA_TRY(cudaMemset(buf, 0x5a, words * sizeof(u64)));
    // four fixed twiddles modulo q_0 with their companions (sf_mad)
    sf_pair tw[4];
    for (int i = 0; i < 4; ++i) {
        const u64 v = (M.q / 3 + 7919 * (u64)i) % M.q;
        tw[i] = make_ulonglong2(v, pm ? sf_host_mulmod(v, ((u64)1 << 32) % M.q, M.q) : sf_shoup_companion(v, M.q));
    }
    auto launch = [&]() { kernel<<<grid, 256>>>(buf, M, tw[0], tw[1], tw[2], tw[3]); };
    cudaEvent_t a = nullptr, b = nullptr;
    SF_CUDA_TRY(cudaEventCreate(&a));
    if (cudaEventCreate(&b) != cudaSuccess) {
        cudaEventDestroy(a);
        return sf_set_error(SF_ECUDA, "sf_modmul_probe: event creation failed");
    }
    const int reps = 5;
    for (int r = 0; r < 2; ++r) launch();
    cudaEventRecord(a);
    for (int r = 0; r < reps; ++r) launch();
    cudaEventRecord(b);
    cudaError_t e = cudaEventSynchronize(b);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (e != cudaSuccess) return sf_set_error(SF_ECUDA, "sf_modmul_probe: %s", cudaGetErrorString(e));
    SF_CUDA_TRY(cudaGetLastError());
    const double ops = (double)PROBE_OPS * grid * 256 * reps;
    *gmodmul_per_s = ms > 0.f ? ops / (ms * 1e-3) / 1e9 : 0.0;
    return SF_OK;
}
