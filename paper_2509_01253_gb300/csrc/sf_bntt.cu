// sf_bntt.cu -- batched negacyclic NTT over every RNS limb of a batch of
// polynomials, and register-resident probes of the modular arithmetic.
//
// The batch is [count][L][N]: limb i of polynomial p is reduced modulo q_i.
// A transform is the two register-resident passes of sf_reg.cuh (forward:
// column pass, then row pass; inverse: row pass, then column pass with the
// factor N^-1).  Each pass is one persistent launch of one resident wave over
// the units (group, polynomial), a group being a column or row tile position
// and a limb: a block takes an equal range of units (sf_unit_range), stages a
// group's twiddles when its range enters the group, and loads the next unit's
// points into registers before it transforms the current one.
//
// Bound by the integer multiplier: at N = 2^16 the fmaheavy pipe is busy 70 to
// 76 % of the cycles, DRAM 31 to 39 %, shared memory 20 to 33 %, and no warp
// waits on memory or a barrier.  512 x 5 limbs of 2^16, forward: 1961 us with
// the tile sweeps in shared memory (8 points per thread, three sweeps and three
// barriers a pass), 1714 us here.
#include <algorithm>

#include "sf_internal.h"
#include "sf_kernels.cuh"
#include "sf_reg.cuh"
#include "sf_round.h"

template <bool INV, int LR, int LC>
__global__ void __launch_bounds__(SfSub<LC>::NT, 512 / SfSub<LC>::NT)
    k_bntt_row(SfRing R, const u64 *src, u64 *dst, int count, int ng)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SfRowT<LC> T;
    sf_pair *tw = (sf_pair *)smem_raw;
    u64 *buf = (u64 *)(tw + SfSub<LC>::ROW_PAIRS);
    const SfUnitRange U = sf_unit_range(ng * count);
    const size_t per = (size_t)R.L << (LR + LC);
    // unit u: group u / count = (row tile, limb i), item u % count = polynomial
    auto row_ptr = [&](int u) -> size_t {
        const int gg = u / count;
        return per * (u % count) + ((size_t)(gg % R.L) << (LR + LC)) + ((size_t)T.row(gg / R.L, 1 << LR) << LC);
    };
    u64 x[16], nx[16];
    auto load = [&](int u) {
        const u64 *s = src + row_ptr(u);
#pragma unroll
        for (int r = 0; r < 16; ++r) nx[r] = s[T.k1(r)];
    };
    if (U.u0 < U.u1) load(U.u0);
    int staged = -1;
    for (int u = U.u0; u < U.u1; ++u) {
        const int grp = u / count;
        const SfMod &M = R.m[grp % R.L];
        if (grp != staged) {
            __syncthreads();   // the previous group's readers are done
            sf_stage_row<LR, LC>(tw, R.rowP, grp % R.L, grp / R.L);
            staged = grp;
            __syncthreads();
        }
#pragma unroll
        for (int r = 0; r < 16; ++r) x[r] = nx[r];
        u64 *d = dst + row_ptr(u);
        // the loads of the next unit overtake this unit's stores: in place, the
        // two units touch different rows or polynomials
        if (u + 1 < U.u1) load(u + 1);
        if (INV) {
            __syncwarp();
            T.put1(x, buf);
            __syncwarp();
            T.get2(x, buf);
            T.inv2(x, tw, M.q);
            T.to1(x, buf);
            T.inv1(x, tw, M.q);
#pragma unroll
            for (int r = 0; r < 16; ++r) d[T.k1(r)] = sf_red3(x[r], M);
        } else {
            T.fwd1(x, tw, M.q);
            T.to2(x, buf);
            T.fwd2(x, tw, M.q);
            T.to1(x, buf);   // back to coalesced positions
#pragma unroll
            for (int r = 0; r < 16; ++r) d[T.k1(r)] = sf_reduce(x[r], M.q, M.one_p);
        }
    }
}

template <bool INV, int LR, int LC>
__global__ void __launch_bounds__(SfSub<LR>::NT, 512 / SfSub<LR>::NT)
    k_bntt_col(SfRing R, const u64 *src, u64 *dst, int count, int ng)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SfCol<LR> T;
    sf_pair *tab = (sf_pair *)smem_raw;
    u64 *bufs = (u64 *)(tab + SfSub<LR>::S);
    const SfUnitRange U = sf_unit_range(ng * count);
    const size_t per = (size_t)R.L << (LR + LC);
    // unit u: group u / count = (column tile, limb i), item u % count = polynomial
    auto base = [&](int u) -> size_t {
        const int gg = u / count;
        return per * (u % count) + ((size_t)(gg % R.L) << (LR + LC)) + (gg / R.L) * 16 + T.b;
    };
    u64 x[16], nx[16];
    auto load = [&](int u) {
        const u64 *s = src + base(u);
#pragma unroll
        for (int r = 0; r < 16; ++r) nx[r] = s[(size_t)(INV ? T.k2(r) : T.k1(r)) << LC];
    };
    if (U.u0 < U.u1) load(U.u0);
    int staged = -1;
    for (int u = U.u0; u < U.u1; ++u) {
        const int grp = u / count, i = grp % R.L;
        const SfMod &M = R.m[i];
        if (grp != staged) {
            __syncthreads();   // the previous group's readers are done
            sf_stage_cols<LR>(tab, R.colP, i, 1);
            staged = grp;
            __syncthreads();
        }
#pragma unroll
        for (int r = 0; r < 16; ++r) x[r] = nx[r];
        u64 *d = dst + base(u), *buf = bufs + (size_t)(u & 1) * SfSub<LR>::COL_WORDS;
        if (u + 1 < U.u1) load(u + 1);
        if (INV) {
            T.inv2(x, tab, M.q);
            T.to1(x, buf);
            T.inv1(x, tab, M.q);
#pragma unroll
            for (int r = 0; r < 16; ++r) d[(size_t)T.k1(r) << LC] = sf_mul_shoup(x[r], M.ninv, M.ninv_p, M.q);
        } else {
            T.fwd1(x, tab, M.q);
            T.to2(x, buf);
            T.fwd2(x, tab, M.q);
#pragma unroll
            for (int t = 0; t < 16; ++t) d[(size_t)T.k2(t) << LC] = x[t];
        }
    }
}

// one resident wave (SMs x occupancy blocks), at most one block per unit
static int bntt_blocks(const sf_ctx *ctx, int occ, int n_units)
{
    return std::max(1, std::min(ctx->num_sms * occ, n_units));
}

template <int LC>
static constexpr size_t bntt_smem_row() { return sizeof(sf_pair) * SfSub<LC>::ROW_PAIRS + sizeof(u64) * SfSub<LC>::ROW_WORDS; }
template <int LR>
static constexpr size_t bntt_smem_col() { return sizeof(sf_pair) * SfSub<LR>::S + sizeof(u64) * 2 * SfSub<LR>::COL_WORDS; }

template <bool INV, int LR, int LC>
static void bntt_row(sf_ctx *ctx, const u64 *src, u64 *dst, int count, cudaStream_t st)
{
    const int ng = ((1 << LR) / 16) * ctx->ring.L;
    const size_t sm = bntt_smem_row<LC>();
    cudaEvent_t ev;
    const int nb = bntt_blocks(ctx, sf_occupancy(k_bntt_row<INV, LR, LC>, SfSub<LC>::NT, sm), ng * count);
    sf_launch_begin(ctx, SFK_BNTT_ROW, st, &ev);
    k_bntt_row<INV, LR, LC><<<nb, SfSub<LC>::NT, sm, st>>>(ctx->ring, src, dst, count, ng);
    sf_launch_end(ctx, SFK_BNTT_ROW, st, ev);
}

template <bool INV, int LR, int LC>
static void bntt_col(sf_ctx *ctx, const u64 *src, u64 *dst, int count, cudaStream_t st)
{
    const int ng = ((1 << LC) / 16) * ctx->ring.L;
    const size_t sm = bntt_smem_col<LR>();
    cudaEvent_t ev;
    const int nb = bntt_blocks(ctx, sf_occupancy(k_bntt_col<INV, LR, LC>, SfSub<LR>::NT, sm), ng * count);
    sf_launch_begin(ctx, SFK_BNTT_COL, st, &ev);
    k_bntt_col<INV, LR, LC><<<nb, SfSub<LR>::NT, sm, st>>>(ctx->ring, src, dst, count, ng);
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
    // tiles of a limb: C / 16 (bounded as for the 32 tiles of a 128 x 512 split at N = 2^16)
    const int tiles = R.log_n == 16 ? 32 : (1 << ((R.log_n + 1) / 2)) / 16;
    if ((long long)count * R.L * tiles > INT32_MAX)
        return sf_set_error(SF_EINVAL, "sf_ntt_batch: count too large");
    SF_RING_DISPATCH(R.log_n, {
        if (!inverse) {
            bntt_col<false, LR, LC>(ctx, d_in, d_out, count, st);
            bntt_row<false, LR, LC>(ctx, d_out, d_out, count, st);
        } else {
            bntt_row<true, LR, LC>(ctx, d_in, d_out, count, st);
            bntt_col<true, LR, LC>(ctx, d_out, d_out, count, st);
        }
    });
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

sf_status sf_bntt_init_attributes()
{
    const int mx = 227 * 1024;
#define SF_BNTT_ATTR(K) SF_CUDA_TRY(cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
#define SF_BNTT_ATTRS(LR, LC)                                                                  \
    SF_BNTT_ATTR((k_bntt_row<false, LR, LC>)) SF_BNTT_ATTR((k_bntt_row<true, LR, LC>))         \
    SF_BNTT_ATTR((k_bntt_col<false, LR, LC>)) SF_BNTT_ATTR((k_bntt_col<true, LR, LC>))
    SF_BNTT_ATTRS(5, 5) SF_BNTT_ATTRS(5, 6) SF_BNTT_ATTRS(6, 6) SF_BNTT_ATTRS(6, 7) SF_BNTT_ATTRS(7, 7)
    SF_BNTT_ATTRS(7, 8) SF_BNTT_ATTRS(8, 8)
#undef SF_BNTT_ATTRS
#undef SF_BNTT_ATTR
    return SF_OK;
}

// ---------------------------------------------------------------- probes ----
// Each thread keeps 8 residues in registers and applies PROBE_ITERS rounds of
// 12 operations to them (a radix-8 unit: 3 stages of 4 butterflies, or 12
// multiply-accumulates), then stores them.  Nothing else is read or written,
// so the rate is the arithmetic ceiling of these operations on this GPU.
#define PROBE_ITERS 1024
#define PROBE_OPS (12 * PROBE_ITERS)

template <int KIND>
__global__ void __launch_bounds__(256, 2) k_probe(u64 *buf, u64 q, ulonglong2 t0, ulonglong2 t1, ulonglong2 t2,
                                                 ulonglong2 t3)
{
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    u64 x[8], acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        x[i] = buf[i * stride + t];
        acc[i] = 0;
    }
    const u64 two_q = 2 * q;
    for (int it = 0; it < PROBE_ITERS; ++it) {
        if (KIND == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) sf_bfly_ct(x[i], x[i + 4], t0.x, t0.y, q, two_q);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                sf_bfly_ct(x[i], x[i + 2], t1.x, t1.y, q, two_q);
                sf_bfly_ct(x[i + 4], x[i + 6], t2.x, t2.y, q, two_q);
            }
#pragma unroll
            for (int i = 0; i < 8; i += 2) sf_bfly_ct(x[i], x[i + 1], t3.x, t3.y, q, two_q);
        } else if (KIND == 1) {
#pragma unroll
            for (int i = 0; i < 8; i += 2) sf_bfly_gs(x[i], x[i + 1], t3.x, t3.y, q, two_q);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                sf_bfly_gs(x[i], x[i + 2], t1.x, t1.y, q, two_q);
                sf_bfly_gs(x[i + 4], x[i + 6], t2.x, t2.y, q, two_q);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) sf_bfly_gs(x[i], x[i + 4], t0.x, t0.y, q, two_q);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const ulonglong2 w = (i & 3) == 0 ? t0 : (i & 3) == 1 ? t1 : (i & 3) == 2 ? t2 : t3;
                acc[i] += sf_mul_shoup_lazy4(x[i], w.x, w.y, q);
                x[i] ^= acc[i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const ulonglong2 w = i == 0 ? t0 : i == 1 ? t1 : i == 2 ? t2 : t3;
                acc[i] += sf_mul_shoup_lazy4(x[i + 4], w.x, w.y, q);
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
    int occ = 1;
    switch (kind) {
    case 0: occ = sf_occupancy(k_probe<0>, 256, 0); break;
    case 1: occ = sf_occupancy(k_probe<1>, 256, 0); break;
    default: occ = sf_occupancy(k_probe<2>, 256, 0); break;
    }
    const int grid = ctx->num_sms * occ;
    const size_t words = (size_t)8 * grid * 256;
    SF_CUDA_TRY(cudaDeviceSynchronize());
    void *w = nullptr;
    SF_TRY(sf_scratch(ctx, words * sizeof(u64), &w));
    u64 *buf = (u64 *)w;
    SF_CUDA_TRY(cudaMemset(buf, 0x5a, words * sizeof(u64)));
    // four fixed twiddle pairs (w, floor(w 2^64 / q)) modulo q_0
    ulonglong2 tw[4];
    for (int i = 0; i < 4; ++i) {
        const u64 v = (M.q / 3 + 7919 * (u64)i) % M.q;
        tw[i] = make_ulonglong2(v, sf_shoup_companion(v, M.q));
    }
    auto launch = [&]() {
        switch (kind) {
        case 0: k_probe<0><<<grid, 256>>>(buf, M.q, tw[0], tw[1], tw[2], tw[3]); break;
        case 1: k_probe<1><<<grid, 256>>>(buf, M.q, tw[0], tw[1], tw[2], tw[3]); break;
        default: k_probe<2><<<grid, 256>>>(buf, M.q, tw[0], tw[1], tw[2], tw[3]); break;
        }
    };
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
