// sf_ks.cu -- automorphism + hybrid key switching for batches of "merges".
//
// A merge (Sec. 2.4 packing step, Sec. 2.2 key switching) takes E, O
// ([2][L][N]), a shift s and an automorphism index d:
//     u = E - X^s O,  v = E + X^s O
//     (A', B') = KS(tau_d(u.a))        (hybrid: ModUp, <., ksk_d>, ModDown)
//     out = (v.a + A',  v.b + tau_d(u.b) + B')          [add_v = 1]
//     out = (A',        tau_d(u.b) + B')                [add_v = 0: plain rotate]
// Without O, u = v = E (the trace step ct + tau_d(ct), or a rotation).
//
// Ciphertexts between merges are in the coefficient domain: there tau_d and X^s
// are signed index maps, and the result needs no forward transform after
// ModDown.  One merge takes four launches:
//   k_ks_gather : TA = tau_d(u.a); out = v, plus tau_d(u.b) on the b part
//   k_ks2 : ModUp of TA, forward columns                    (sf_ks_up.cu)
//   k_ks3 : forward rows, inner product, inverse rows       (sf_ks_rows.cu)
//   k_ks4 : inverse columns, ModDown, added to out          (sf_ks_down.cu)
// Both forms run (dnum + 2)(L + K) limb transforms per merge; kept in the NTT
// domain throughout, a merge took seven kernels.  The leaves arrive in the NTT
// domain and the first level reads them there: k_ks_gather permutes slots, k_ks1
// runs the inverse rows of TA for k_ks2's inverse columns, and k_ks3 adds `out`
// to its accumulators, so that its result is in the coefficient domain like
// every later one.
#include "sf_ks.h"

#include "sf_kernels.cuh"
#include "sf_reg.cuh"

// Elementwise, one pass over E and O per merge:
//   TA[i][p] = tau_d(u.a)[p],  u = E - X^s O
//   out.a[p] = v.a[p]                      (0 for a plain rotation)
//   out.b[p] = v.b[p] + tau_d(u.b)[p],     v = E + X^s O
// Coefficient-domain operands: tau_d and X^s are signed index maps.  NTT-domain
// operands (storage order): a slot permutation and monomial products, and out
// times N^-1.
// grid (N / (256 SF_EW), L, merges): each thread does SF_EW points, so the
// per-merge pointers are set up once per thread.  Bound by HBM (0.89 of the
// copy bandwidth at N = 2^16): 3.0 us per merge there.  Done inside k_ks2 and
// k_ks4 instead, the gathers' latency cost those kernels 9 us more per merge.
// UNREDUCED (B.unreduced) is an instance of its own: with the test at run time a
// 64 x 64 layer at N = 2^12 took 321.9 us, 320.3 without, a rotation at N = 2^16
// 73.8 and 73.6.
#define SF_EW 8
template <bool UNREDUCED>
__global__ void __launch_bounds__(256) k_ks_gather(SfRing R, SfKsBatch B)
{
    sf_pdl_next(B);
    sf_pdl_wait(B);
    const int b = blockIdx.z, i = blockIdx.y;
    const u64 *E = merge_E(B, b), *O = merge_O(B, b);
    u64 *ta = ks_limb(R, B, b, sf_ks_ta(R) + i);
    u64 *out = merge_out(B, b);
    u64 *oa = out + ((size_t)i << R.log_n), *ob = out + ((size_t)(R.L + i) << R.log_n);
    const SfMod &M = R.m[i];
    const u64 q = M.q;
    const int p0 = blockIdx.x * (256 * SF_EW) + threadIdx.x;
    const size_t ea = (size_t)i << R.log_n, eb = (size_t)(R.L + i) << R.log_n;
    const size_t pb = (size_t)i << (R.log_n + 1);
    if (!B.ntt) {
        const unsigned n = R.n, mask = n - 1;
        const u64 *Ea = E + ea, *Eb = E + eb, *Oa = O ? O + ea : nullptr, *Ob = O ? O + eb : nullptr;
#pragma unroll
        for (int x = 0; x < SF_EW; ++x) {
            const unsigned p = p0 + x * 256;
            if (p >= n) break;
            // p receives index e = p d^-1 mod 2N of u, negated when e >= N
            const unsigned e = (p * B.dinv) & (2 * n - 1), src = e & mask;
            u64 ua = Ea[src], ub = Eb[src], va = 0, vb = 0;
            if (UNREDUCED) {
                ua = sf_reduce(ua, q, M.one_p);
                ub = sf_reduce(ub, q, M.one_p);
            }
            if (B.add_v) {
                va = Ea[p];
                vb = Eb[p];
            }
            if (O) {
                // X^s O has coefficient O[p - s], or -O[p - s + N] below s
                const u64 oas = Oa[(src - B.s) & mask], obs = Ob[(src - B.s) & mask];
                const u64 oap = Oa[(p - B.s) & mask], obp = Ob[(p - B.s) & mask];
                ua = src < B.s ? sf_add(ua, oas, q) : sf_sub(ua, oas, q);
                ub = src < B.s ? sf_add(ub, obs, q) : sf_sub(ub, obs, q);
                va = p < B.s ? sf_sub(va, oap, q) : sf_add(va, oap, q);
                vb = p < B.s ? sf_sub(vb, obp, q) : sf_add(vb, obp, q);
            }
            ta[p] = e >= n ? sf_sub(0, ua, q) : ua;
            if (B.add_v) oa[p] = va;
            ob[p] = e >= n ? sf_sub(vb, ub, q) : sf_add(vb, ub, q);
        }
        return;
    }
#pragma unroll
    for (int x = 0; x < SF_EW; ++x) {
        const int p = p0 + x * 256;
        if (p >= R.n) break;   // rings smaller than one block's 256 SF_EW slots
        const int j = sf_natural_index(p, R.log_r, R.log_c), jsrc = auto_src(j, B.d, R.log_n);
        const int src = sf_storage_index(jsrc, R.log_r, R.log_c);
        // every load before any store (the stores could alias nothing, but the
        // compiler cannot know): 4 coalesced, 4 gathered, 2 monomial pairs
        u64 Eaj = E[ea + p], Ebj = E[eb + p], Eas = E[ea + src], Ebs = E[eb + src];
        if (O) {
            const unsigned kj = mono_index(j, B.s, R.log_n), ks = mono_index(jsrc, B.s, R.log_n);
            const u64 wj = R.pw[pb + kj], wjp = R.pw_p[pb + kj], ws = R.pw[pb + ks], wsp = R.pw_p[pb + ks];
            const u64 Oaj = O[ea + p], Obj = O[eb + p], Oas = O[ea + src], Obs = O[eb + src];
            const u64 xaj = sf_mul_shoup(Oaj, wj, wjp, q), xbj = sf_mul_shoup(Obj, wj, wjp, q);
            const u64 xas = sf_mul_shoup(Oas, ws, wsp, q), xbs = sf_mul_shoup(Obs, ws, wsp, q);
            ta[p] = sf_sub(Eas, xas, q);
            const u64 ub = sf_sub(Ebs, xbs, q);
            Eaj = sf_add(Eaj, xaj, q);
            Ebj = sf_add(sf_add(Ebj, xbj, q), ub, q);
        } else {
            ta[p] = Eas;
            Ebj = sf_add(Ebj, Ebs, q);
        }
        // joins accumulators that carry N^-1
        oa[p] = sf_mul_shoup(Eaj, M.ninv, M.ninv_p, q);
        ob[p] = sf_mul_shoup(Ebj, M.ninv, M.ninv_p, q);
    }
}

sf_status sf_ks_inv_rows_launch(sf_ctx *ctx, const SfKsBatch &b, cudaStream_t st);

sf_status sf_ks_launch(sf_ctx *ctx, const SfKsBatch &B0, cudaStream_t st)
{
    const SfRing &R = ctx->ring;
    if (B0.count <= 0) return SF_OK;
    // d^-1 mod 2^32 by Newton iteration (d odd), then mod 2N
    unsigned inv = (unsigned)B0.d;
    for (int it = 0; it < 5; ++it) inv *= 2u - (unsigned)B0.d * inv;
    cudaEvent_t ev;
    for (int off = 0; off < B0.count; off += 32768) {
        SfKsBatch b = B0;
        b.count = std::min(32768, B0.count - off);
        b.first = B0.first + off;
        b.dinv = inv & (2u * R.n - 1u);
        b.pdl = ks_overlap(b.count);
        b.scratch += sf_ks_scratch_words(R) * off;
        sf_launch_begin(ctx, SFK_KS_GATHER, st, &ev);
        sf_pdl_launch(b.unreduced ? k_ks_gather<true> : k_ks_gather<false>, dim3((R.n + 256 * SF_EW - 1) / (256 * SF_EW), R.L, b.count), 256, 0, st, R, b);
        sf_launch_end(ctx, SFK_KS_GATHER, st, ev);
        if (b.ntt) SF_TRY(sf_ks_inv_rows_launch(ctx, b, st));
        SF_TRY(sf_ks_up_launch(ctx, b, st));
        SF_TRY(sf_ks_rows_launch(ctx, b, st));
        SF_TRY(sf_ks_down_launch(ctx, b, st));
    }
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

// Runs `count` merges sharing (d, s, add_v, key) in launch batches.
sf_status sf_ks_run(sf_ctx *ctx, SfKsBatch B, u64 *scratch, int batch, cudaStream_t st)
{
    batch = std::max(1, batch);
    const int total = B.count;
    for (int off = 0; off < total; off += batch) {
        SfKsBatch b = B;
        b.count = std::min(batch, total - off);
        b.first = B.first + off;
        b.scratch = scratch;
        SF_TRY(sf_ks_launch(ctx, b, st));
    }
    return SF_OK;
}

// Opt the kernels into the full shared-memory carve-out.
sf_status sf_ks_init_attributes()
{
    SF_TRY(sf_ks_up_init());
    SF_TRY(sf_ks_rows_init());
    return sf_ks_down_init();
}
