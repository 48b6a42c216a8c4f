// sf_ks.h -- batched automorphism + key switching (see sf_ks.cu).
#pragma once
#include <algorithm>

#include "sf_internal.h"

// `count` merges sharing d, s, add_v and the key.  Merge number
// x = first + i (i < count) splits into (g, t) = (x / inner, x % inner):
//   E_x = E + g*E_outer + t*E_stride, likewise O_x (O may be null) and out_x;
// every operand [2][L][N].  out must not alias E or O.  Results are in the
// coefficient domain; the operands too, or, with `ntt`, in the NTT domain
// (storage order, canonical): the first key-switched level above the leaves.
struct SfKsBatch {
    const u64 *E;
    size_t E_stride, E_outer;
    const u64 *O;
    size_t O_stride, O_outer;
    u64 *out;
    size_t out_stride, out_outer;
    int first;
    int inner;
    int count;
    int ntt;        // operands in the NTT domain
    int unreduced;  // plain rotation of residues that nothing has checked: brought to [0, q) as they are read
    int d;          // automorphism X -> X^d
    unsigned dinv;  // d^-1 mod 2N (set by sf_ks_launch)
    int pdl;             // launches overlap (sf_pdl_launch)
    unsigned s;     // O is multiplied by X^s
    int add_v;      // 1: out = v + KS(...), 0: plain rotation
    const u64 *key; // [dnum][2][nm][N] pairs of the NTT-domain values, storage order
    u64 *scratch;   // sf_ks_scratch_words(R) words per merge of one launch batch
};

// Scratch of a merge, in limbs: the ModUp extensions [dnum][nm] from limb 0,
// accumulators, tau_d(u.a).  The inverse rows of NTT-domain operands (x1) lie where
// the accumulators go: k_ks2 has read them before k_ks3 writes there.
SF_HD int sf_ks_acc(const SfRing &R) { return R.dnum * R.nm; }
SF_HD int sf_ks_x1(const SfRing &R) { return sf_ks_acc(R); }
SF_HD int sf_ks_ta(const SfRing &R) { return sf_ks_acc(R) + 2 * R.nm; }

// words per merge
SF_HD size_t sf_ks_scratch_words(const SfRing &R) { return (size_t)(sf_ks_ta(R) + R.L) << R.log_n; }
// One launch sequence for B.count merges, scratch for all of them.
sf_status sf_ks_launch(sf_ctx *ctx, const SfKsBatch &B, cudaStream_t st);
// Splits B into launch batches of `batch` merges reusing `scratch`
// (batch * sf_ks_scratch_words words).
sf_status sf_ks_run(sf_ctx *ctx, SfKsBatch B, u64 *scratch, int batch, cudaStream_t st);

// The kernels of one launch sequence, each in its own translation unit:
// ModUp columns (sf_ks_up.cu), rows with the inner product (sf_ks_rows.cu),
// ModDown columns (sf_ks_down.cu).
sf_status sf_ks_up_launch(sf_ctx *ctx, const SfKsBatch &B, cudaStream_t st);
sf_status sf_ks_rows_launch(sf_ctx *ctx, const SfKsBatch &B, cudaStream_t st);
sf_status sf_ks_down_launch(sf_ctx *ctx, const SfKsBatch &B, cudaStream_t st);
sf_status sf_ks_up_init();
sf_status sf_ks_rows_init();
sf_status sf_ks_down_init();

#if defined(__CUDACC__)
__device__ __forceinline__ void merge_gt(const SfKsBatch &B, int b, int &g, int &t)
{
    const int x = B.first + b;
    g = x / B.inner;
    t = x - g * B.inner;
}
__device__ __forceinline__ const u64 *merge_E(const SfKsBatch &B, int b)
{
    int g, t;
    merge_gt(B, b, g, t);
    return B.E + B.E_outer * g + B.E_stride * t;
}
__device__ __forceinline__ const u64 *merge_O(const SfKsBatch &B, int b)
{
    if (!B.O) return nullptr;
    int g, t;
    merge_gt(B, b, g, t);
    return B.O + B.O_outer * g + B.O_stride * t;
}
__device__ __forceinline__ u64 *merge_out(const SfKsBatch &B, int b)
{
    int g, t;
    merge_gt(B, b, g, t);
    return B.out + B.out_outer * g + B.out_stride * t;
}
// this merge's scratch, limb `limb` of it
__device__ __forceinline__ u64 *ks_limb(const SfRing &R, const SfKsBatch &B, int b, int limb)
{
    return B.scratch + sf_ks_scratch_words(R) * b + ((size_t)limb << R.log_n);
}

// coefficient p of E + X^s O of one limb, canonical; e, o: the limb's N
// coefficients (o may be null)
__device__ __forceinline__ u64 merge_coef(const u64 *e, const u64 *o, int p, unsigned s, int n, u64 q)
{
    const u64 v = e[p];
    if (!o) return v;
    const int k = p - (int)s;
    const u64 w = o[k & (n - 1)];
    // X^s O has coefficient O[p - s], or -O[p - s + N] below s
    return k < 0 ? sf_sub(v, w, q) : sf_add(v, w, q);
}
#endif

// Blocks of a launch over n_units (group, item) units, split evenly
// (sf_unit_range): as many waves of num_sms x occupancy blocks as leave a block
// `per_block` units for the tables it stages.  One wave of equal shares lost: the
// warps of an SM's blocks are not served evenly, so that one block ends early and
// leaves the others fewer warps to hide latency with (512 x 5 limbs of 2^16: 1779
// us with one wave, 1550 us with 8 units a block; the key-switch rows 418 and 392
// ms per 32768 at N = 2^16).
static inline int ks_wave_blocks(const sf_ctx *ctx, int occ, int n_units, int per_block)
{
    const int w = ctx->num_sms * occ;
    const int waves = std::max(1, std::min(32, n_units / (w * per_block)));
    return std::max(1, std::min(w * waves, n_units));
}

// The launches of a single rotation or merge overlap (programmatic dependent launch):
// a kernel starts once the blocks of the one before have all started, the column
// kernels stage their twiddle tables, and every kernel waits for the completion of the
// one before (sf_pdl_wait) before its first access to data, so that completion carries
// along the chain; nothing but the tables, written when the context was made, is read
// before.  One rotation at N = 2^16: 83 us launched in order, 73 us so.  (70 us with
// the row kernels' tables staged ahead as well, but the code for it slowed the inner
// product of every batch by up to 2.7 %.)  Batches lose by it, as waiting blocks hold
// room and crowd SMs (64 outputs at N = 2^13, tree levels of 32 .. 1 merges: 326 us in
// order, 345 with every level overlapped that leaves SMs idle, 321 with single merges
// only; a ResNet-20 convolution with every launch overlapped 70.7 and 79.4 ms).
static inline int ks_overlap(int count) { return count == 1; }
#ifdef __CUDACC__
__device__ __forceinline__ void sf_pdl_next(const SfKsBatch &B)
{
    if (B.pdl) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void sf_pdl_wait(const SfKsBatch &B)
{
    if (B.pdl) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// kernel(R, b, args...)
template <class... P, class... A>
static inline void sf_pdl_launch(void (*kernel)(SfRing, SfKsBatch, P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                                 const SfRing &R, const SfKsBatch &b, A... args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = a;
    c.numAttrs = b.pdl ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, R, b, P(args)...);
}
#endif
