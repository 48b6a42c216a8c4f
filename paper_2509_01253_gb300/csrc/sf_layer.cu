// sf_layer.cu -- the linear-layer round (Sec. 4.4, steps 6-10) on the GPU.
//
// Steps 6-8 (extraction at gamma = 0, unshuffle, linear layer): the row
// extracted for stream position p = jN + k is N^-1 X^-k ct_j, so output o is
//     y_o = sum_j w_{o,j}(X) * ct_j,   w_{o,j} = N^-1 sum_{taps i in ct j} Wq[o,i] X^-k(i)
// with k(i) the in-ciphertext position of input i after unshuffling
// (p = sigma_prev^-1(i)).  Three kernels per batch of outputs:
//   leaf_prep: walks each output's receptive field once and buckets its taps
//              by (input ciphertext, column tile: 16 columns, 8 at N = 2^16),
//   leaf_col : scatters its bucket into a zeroed column tile in shared memory
//              and runs the forward column pass,
//   leaf_row : forward row pass, then the product with every input ciphertext
//              (pairs in storage order, sf_reg.cuh), lazy sums -> leaf (NTT
//              domain, storage order).
// Step 9 (shuffle) is the slot -> output map sigma_out; step 10 (packing) is
// the PackLWEs tree plus field trace driven by sf_pack_tree below.
#include "sf_internal.h"
#include "sf_kernels.cuh"
#include "sf_ks.h"
#include "sf_layer.h"
#include "sf_async.cuh"
#include "sf_reg.cuh"

__device__ __forceinline__ int leaf_output(const SfLeafParams &P, int slot)
{
    return P.sig_out ? P.sig_out[slot] : slot;
}

// Calls f(j, row, column, signed Wq) for every tap of output o: input
// ciphertext j, and the coefficient N - k (or 0) of w_{o,j} it lands on as
// (row, column) of the R x C split; the sign carries the X^-k = -X^(N-k) of
// the extraction.  Threads split the taps.
template <class F>
__device__ __forceinline__ void leaf_taps_all(const SfRing &R, const SfLeafParams &P, int o, F f)
{
    const int co = o % P.C_out, hw = o / P.C_out;
    const int ho = hw / P.W_out, wo = hw % P.W_out;
    for (int ti = 0; ti < P.n_terms; ++ti) {
        const SfTermDev &T = P.t[ti];
        const int ntap = T.kh * T.kw * T.C_in;
        const int h0 = ho * T.stride - T.pad, w0 = wo * T.stride - T.pad;
        const int base = T.in_offset + (h0 * T.W + w0) * T.C_in;
        const int64_t *wrow = P.wq + T.w_off + (size_t)co * ntap;
        for (int tt = threadIdx.x; tt < ntap; tt += blockDim.x) {
            const int4 tp = P.taps[T.tap_off + tt];
            const int h = h0 + tp.x, w = w0 + tp.y;
            if (h < 0 || h >= T.H || w < 0 || w >= T.W) continue;
            const int idx = base + tp.z;
            const int p = P.pos_of ? P.pos_of[idx] : idx;
            const int k = p & (R.n - 1);
            const int cidx = k ? R.n - k : 0;
            const int64_t wq = P.gamma2 ? 2 * wrow[tp.w] : wrow[tp.w];
            f(p >> R.log_n, cidx >> R.log_c, cidx & (R.c - 1), k ? -wq : wq);
            if (P.gamma2) {
                // gamma = 2 (Lemma 1 at t = 2): the row is (N/2)^-1 (X^-k ct_j + X^-3k ct3_j), so
                // the tap also lands at X^-3k of the power ct3_j.  With e = 3k mod 2N,
                // X^-e = 1 (e = 0), -X^(N - e) (0 < e <= N), X^(2N - e) (N < e < 2N).
                const int e = (3 * k) & (2 * R.n - 1);
                const int c3 = e == 0 ? 0 : (e <= R.n ? R.n - e : 2 * R.n - e);
                const bool neg = e != 0 && e <= R.n;
                f(P.k_src + (p >> R.log_n), c3 >> R.log_c, c3 & (R.c - 1), neg ? -wq : wq);
            }
        }
    }
}

size_t sf_leaf_tap_words(const SfRing &R, int k_in, int max_taps, int slots)
{
    const size_t nb = (size_t)k_in * sf_leaf_tiles(R) + 1;
    return (size_t)slots * max_taps * 2 + (slots * nb + 1) / 2;
}

// leaf_prep: grid (slots).  Buckets the taps of each slot's output by
// (input ciphertext, column tile) with a counting sort, so that a column
// block reads its own taps instead of scanning the whole receptive field.
#define SF_MAX_BUCKETS 4096
__global__ void __launch_bounds__(256) k_leaf_prep(SfRing R, SfLeafParams P)
{
    __shared__ int cnt[SF_MAX_BUCKETS + 1];
    const int z = blockIdx.x;
    const int o = leaf_output(P, P.s0 + z * P.s_stride);
    const int nb = P.n_buckets, tiles = sf_leaf_tiles(R), wl = sf_leaf_width_log(R);
    int *off = P.tap_off + (size_t)z * (nb + 1);
    for (int b = threadIdx.x; b <= nb; b += blockDim.x) cnt[b] = 0;
    __syncthreads();
    leaf_taps_all(R, P, o, [&](int j, int row, int col, int64_t) { atomicAdd(&cnt[j * tiles + (col >> wl)], 1); });
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int b = 0; b < nb; ++b) {
            const int c = cnt[b];
            cnt[b] = acc;
            off[b] = acc;
            acc += c;
        }
        off[nb] = acc;
    }
    __syncthreads();
    longlong2 *dst = P.tap_buf + (size_t)z * P.max_taps;
    leaf_taps_all(R, P, o, [&](int j, int row, int col, int64_t wq) {
        const int pos = atomicAdd(&cnt[j * tiles + (col >> wl)], 1);
        // the word of the padded column tile it lands on (SfColT)
        dst[pos] = make_longlong2(((row + (row >> 3)) << wl) + (col & ((1 << wl) - 1)), wq);
    });
}

// N^-1 * wq mod q, canonical (|wq| < 2^63)
__device__ __forceinline__ u64 leaf_coeff(const SfMod &M, int64_t wq)
{
    const u64 a = sf_reduce((u64)(wq < 0 ? -wq : wq), M.q, M.one_p);
    const u64 v = sf_mul_shoup(a, M.ninv, M.ninv_p, M.q);
    return (wq < 0 && v) ? M.q - v : v;
}

// leaf_col: grid (column tiles, k_in * L, slots).  Bound by the integer
// multiplier (one forward column pass per tile; the bucket holds a few taps to
// a few hundred).
template <int LR, int LC, bool PM>
__global__ void __launch_bounds__(SfShape<LR>::NT, SfShape<LR>::BPS) k_leaf_col(SfRing R, SfLeafParams P)
{
    constexpr int NT = SfShape<LR>::NT, NB = SfShape<LR>::NB;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SfColT<LR, PM> T;
    const int j = blockIdx.y / R.L, i = blockIdx.y % R.L;
    const SfMod &M = R.m[i];
    sf_pair *tab = (sf_pair *)smem_raw;
    u64 *tile = (u64 *)(tab + SfShape<LR>::S);
    sf_stage_cols<LR>(tab, R.colP, i, 1);
#pragma unroll
    for (int e = 0; e < 9; ++e) tile[threadIdx.x + e * NT] = 0;
    __syncthreads();
    // this block's bucket of taps (built by leaf_prep)
    const int *off = P.tap_off + (size_t)blockIdx.z * (P.n_buckets + 1);
    const int bk = j * ((1 << LC) / NB) + blockIdx.x;
    const int t0 = off[bk], nt = off[bk + 1] - t0;
    const longlong2 *src = P.tap_buf + (size_t)blockIdx.z * P.max_taps + t0;
    for (int t = threadIdx.x; t < nt; t += NT) {
        const longlong2 e = src[t];
        tile[e.x] = leaf_coeff(M, e.y);
    }
    __syncthreads();
    u64 x[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) x[t] = tile[T.at(T.k1(t))];
    T.forward(x, tab, tile, M);
    u64 *dst = P.w1 + ((((size_t)blockIdx.z * P.k_in + j) * R.L + i) << (LR + LC)) + blockIdx.x * NB + T.b;
#pragma unroll
    for (int t = 0; t < 8; ++t) dst[(size_t)T.kl(t) << LC] = x[t];
}

// leaf_row: groups (row tile, limb i), items slots.  Per input
// ciphertext a forward row pass and two multiply-accumulates per point, the
// accumulators in registers.  Bound by the integer multiplier; the staged
// twiddles (32 KB at 256-point rows) serve every slot of the group.
template <int LR, int LC, bool PM>
__global__ void __launch_bounds__(SfShape<LC>::NT, SfShape<LC>::BPS_ACC) k_leaf_row(SfRing R, SfLeafParams P, int ng, int cnt)
{
    constexpr int NT = SfShape<LC>::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SfRowT<LC, PM> T;
    sf_pair *tw = (sf_pair *)smem_raw;
    u64 *buf = (u64 *)(tw + SfShape<LC>::PAIRS), *pre = buf + SfShape<LC>::WORDS + threadIdx.x;
    const SfUnitRange U = sf_unit_range(ng * cnt);
    const sf_pair *ct = (const sf_pair *)P.ct;
    // group = (row tile, limb), item = slot; each thread copies its own points of
    // an input ciphertext ahead
    struct Group {
        int i, tile;
        size_t off;   // this thread's row in the limb, from a ciphertext's first limb
    };
    auto group = [&](int grp) -> Group {
        const int tile = grp / R.L, i = grp - tile * R.L;
        return {i, tile, ((size_t)i << (LR + LC)) + ((size_t)T.row(tile, 1 << LR) << LC)};
    };
    const size_t per = (size_t)R.L << (LR + LC);
    auto prefetch = [&](const Group &G, int z, int j) {
        const u64 *src = P.w1 + ((size_t)z * P.k_in + j) * per + G.off;
#pragma unroll
        for (int t = 0; t < 8; ++t) sf_cp8(pre + t * NT, src + T.k1(t));
        sf_cp_commit();
    };
    SfCursor C(U.u0, cnt);
    Group G = group(C.grp), N = G;
    if (U.u0 < U.u1) prefetch(G, C.item, 0);
    int staged = -1;
    for (int u = U.u0; u < U.u1; ++u) {
        const int z = C.item;
        if (C.grp != staged) {
            __syncthreads();   // the previous group's readers are done
            sf_stage_row<LR, LC>(tw, R.rowP, G.i, G.tile);
            staged = C.grp;
            __syncthreads();
        }
        const SfMod &M = R.m[G.i];
        C.next();
        if (C.grp != staged) N = group(C.grp);
        SfAcc<PM> acc_a[8], acc_b[8];
        u64 x[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) acc_a[t] = acc_b[t] = {0, 0};
        const sf_pair *ca = ct + ((size_t)G.i << (LR + LC)) + T.store_at(G.tile, 0);
#pragma unroll 1
        for (int j = 0; j < P.k_in; ++j) {
            sf_cp_wait<0>();
#pragma unroll
            for (int t = 0; t < 8; ++t) x[t] = pre[t * NT];
            T.template phase_fwd<0>(x, tw, M);
            if (j + 1 < P.k_in) prefetch(G, z, j + 1);   // the points of this one are in registers
            else if (u + 1 < U.u1) prefetch(N, C.item, 0);
            T.forward_rest(x, tw, buf, M);
            const sf_pair *cb = ca + per;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const sf_pair a = __ldg(ca + t * NT), b = __ldg(cb + t * NT);
                sf_acc_add<PM>(acc_a[t], x[t], a, M);
                sf_acc_add<PM>(acc_b[t], x[t], b, M);
            }
            ca = cb + per;
            if (j % SF_ACC_TERMS == SF_ACC_TERMS - 1 && j + 1 < P.k_in) {
#pragma unroll
                for (int t = 0; t < 8; ++t) sf_acc_close<PM>(acc_a[t], M), sf_acc_close<PM>(acc_b[t], M);
            }
        }
        u64 *da = P.leaves + P.leaf_stride * z + ((size_t)G.i << (LR + LC)) + T.store_at(G.tile, 0), *db = da + per;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            da[t * NT] = sf_csub3(sf_acc_close<PM>(acc_a[t], M), M);
            db[t * NT] = sf_csub3(sf_acc_close<PM>(acc_b[t], M), M);
        }
        G = N;
    }
}

template <int LR>
static constexpr size_t leaf_smem_col() { return sizeof(sf_pair) * SfShape<LR>::S + sizeof(u64) * SfShape<LR>::WORDS; }
template <int LC>
static constexpr size_t leaf_smem_row()
{
    return sizeof(sf_pair) * SfShape<LC>::PAIRS + sizeof(u64) * (SfShape<LC>::WORDS + SfShape<LC>::TILE);
}

sf_status sf_leaves_launch(sf_ctx *ctx, const SfLeafParams &P, int cnt, cudaStream_t st)
{
    const SfRing &R = ctx->ring;
    if (cnt <= 0) return SF_OK;
    if (P.s0 + (cnt - 1) * P.s_stride >= P.n_slots_valid) return sf_set_error(SF_EINVAL, "leaf slot without an output");
    cudaEvent_t ev;
    for (int off = 0; off < cnt; off += 65535) {
        SfLeafParams p = P;
        const int c = std::min(65535, cnt - off);
        p.s0 = P.s0 + off * P.s_stride;
        p.w1 = P.w1;    // w1 holds `cnt` slots; reuse from its start for each sub-launch
        p.leaves = P.leaves + P.leaf_stride * off;
        if (P.k_in * sf_leaf_tiles(R) > SF_MAX_BUCKETS) return sf_set_error(SF_EINVAL, "too many input ciphertexts for one round");
        sf_launch_begin(ctx, SFK_LEAF_PREP, st, &ev);
        k_leaf_prep<<<c, 256, 0, st>>>(R, p);
        sf_launch_end(ctx, SFK_LEAF_PREP, st, ev);
        SF_RING_DISPATCH(R, {
            sf_launch_begin(ctx, SFK_LEAF_COL, st, &ev);
            k_leaf_col<LR, LC, PM><<<dim3((1 << LC) / SfShape<LR>::NB, P.k_in * R.L, c), SfShape<LR>::NT, leaf_smem_col<LR>(), st>>>(R, p);
            sf_launch_end(ctx, SFK_LEAF_COL, st, ev);
            sf_launch_begin(ctx, SFK_LEAF_ROW, st, &ev);
            const int ng = ((1 << LR) / SfShape<LC>::NB) * R.L;
            const int occ = sf_occupancy(k_leaf_row<LR, LC, PM>, SfShape<LC>::NT, leaf_smem_row<LC>());
            k_leaf_row<LR, LC, PM><<<ks_wave_blocks(ctx, occ, ng * c, 8), SfShape<LC>::NT, leaf_smem_row<LC>(), st>>>(R, p, ng, c);
            sf_launch_end(ctx, SFK_LEAF_ROW, st, ev);
        });
    }
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

// ------------------------------------------------------------ pack tree --

// Level-1 merge at gamma = 2: out = E + X^s O (out = E without O), in the NTT
// domain (storage order) or the coefficient domain as B.ntt says.
// grid (N / (256 SF_EW), L, merges), SfKsBatch indexing as in the key switch.
#define SF_EW2 8
__global__ void __launch_bounds__(256) k_merge_plain(SfRing R, SfKsBatch B)
{
    const int b = blockIdx.z, i = blockIdx.y;
    const u64 *E = merge_E(B, b), *O = merge_O(B, b);
    u64 *out = merge_out(B, b);
    const SfMod &M = R.m[i];
    const size_t pb = (size_t)i << (R.log_n + 1);
    const int j0 = blockIdx.x * (256 * SF_EW2) + threadIdx.x;
#pragma unroll
    for (int x = 0; x < SF_EW2; ++x) {
        const int j = j0 + x * 256;
        if (j >= R.n) break;
        const unsigned kk = B.ntt ? mono_index(sf_natural_index(j, R.log_r, R.log_c), B.s, R.log_n) : 0;
        for (int part = 0; part < 2; ++part) {
            const size_t limb = (size_t)(part * R.L + i) << R.log_n;
            u64 v;
            if (B.ntt) {
                v = E[limb + j];
                if (O) v = sf_add(v, sf_mul_shoup(O[limb + j], R.pw[pb + kk], R.pw_p[pb + kk], M.q), M.q);
            } else {
                v = merge_coef(E + limb, O ? O + limb : nullptr, j, B.s, R.n, M.q);
            }
            out[limb + j] = v;
        }
    }
}

static sf_status merge_plain_run(sf_ctx *ctx, const SfKsBatch &B, cudaStream_t st)
{
    const SfRing &R = ctx->ring;
    cudaEvent_t ev;
    for (int off = 0; off < B.count; off += 32768) {
        SfKsBatch b = B;
        b.count = std::min(32768, B.count - off);
        b.first = B.first + off;
        sf_launch_begin(ctx, SFK_ELEMWISE, st, &ev);
        k_merge_plain<<<dim3((R.n + 256 * SF_EW2 - 1) / (256 * SF_EW2), R.L, b.count), 256, 0, st>>>(R, b);
        sf_launch_end(ctx, SFK_ELEMWISE, st, ev);
    }
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

// Pack-tree levels level0+1 .. level1 (see sf_layer.h).  Node i of a level
// is zero iff i >= valid[g]; a merge whose O-node is zero runs without O
// (identical result, X^s * 0 = 0), and merges producing zero nodes are
// skipped.  Level lvl merges node t with node t + n_lvl/2 (n_lvl = nodes at
// level lvl-1) using s = N / 2^lvl and d = 2^lvl + 1.
sf_status sf_pack_tree(sf_ctx *ctx, const u64 *keys_base, const std::vector<int32_t> &key_d, size_t key_words,
                       u64 *A, u64 *B, int G, int n_nodes, int level0, const std::vector<int> &valid, bool trace,
                       u64 *ks_scratch, int batch, u64 **res, size_t *res_stride, bool *ntt, cudaStream_t st,
                       bool tau3_done)
{
    const SfRing &R = ctx->ring;
    const size_t ct = (size_t)2 * R.L * R.n;
    auto key_for = [&](int d, const u64 **k) -> sf_status {
        for (size_t t = 0; t < key_d.size(); ++t)
            if (key_d[t] == d) {
                *k = keys_base + key_words * t;
                return SF_OK;
            }
        return sf_set_error(SF_EINVAL, "no rotation key for d = %d", d);
    };
    int levels = 0;
    while ((1 << levels) < n_nodes) ++levels;
    const int level1 = level0 + levels;
    u64 *cur = A, *nxt = B;
    size_t cur_gs = (size_t)n_nodes * ct, nxt_gs = (size_t)(n_nodes / 2 > 0 ? n_nodes / 2 : 1) * ct;
    for (int lvl = level0 + 1; lvl <= level1; ++lvl) {
        const int half = n_nodes >> (lvl - level0);
        const int d = (1 << lvl) + 1;
        // gamma = 2: the tau_3 level is a plain merge (no key, no key switch)
        const bool plain = tau3_done && lvl == 1;
        auto run = [&](const SfKsBatch &b) -> sf_status {
            return plain ? merge_plain_run(ctx, b, st) : sf_ks_run(ctx, b, ks_scratch, batch, st);
        };
        const u64 *key = nullptr;
        if (!plain) SF_TRY(key_for(d, &key));
        SfKsBatch kb;
        memset(&kb, 0, sizeof(kb));
        kb.E_stride = ct;
        kb.O_stride = ct;
        kb.out_stride = ct;
        kb.E_outer = cur_gs;
        kb.O_outer = cur_gs;
        kb.out_outer = nxt_gs;
        kb.d = d;
        kb.s = (unsigned)(R.n >> lvl);
        kb.add_v = 1;
        kb.ntt = *ntt;
        kb.key = key;
        int gi = 0;
        while (gi < G) {
            if (valid[gi] >= n_nodes) {
                // a run of full groups: one batch with (group, merge) indexing
                int g1 = gi;
                while (g1 < G && valid[g1] >= n_nodes) ++g1;
                SfKsBatch b = kb;
                b.E = cur + gi * cur_gs;
                b.O = b.E + (size_t)half * ct;
                b.out = nxt + gi * nxt_gs;
                b.inner = half;
                b.count = (g1 - gi) * half;
                SF_TRY(run(b));
                gi = g1;
                continue;
            }
            const int V = std::min(valid[gi], 2 * half);
            const int active = std::min(V, half);
            const int with_o = std::max(0, std::min(active, V - half));
            SfKsBatch b = kb;
            b.E = cur + gi * cur_gs;
            b.out = nxt + gi * nxt_gs;
            b.inner = 1 << 30;
            if (with_o > 0) {
                SfKsBatch b1 = b;
                b1.O = b.E + (size_t)half * ct;
                b1.count = with_o;
                SF_TRY(run(b1));
            }
            if (active > with_o) {
                SfKsBatch b2 = b;
                b2.O = nullptr;
                b2.first = with_o;
                b2.count = active - with_o;
                SF_TRY(run(b2));
            }
            ++gi;
        }
        std::swap(cur, nxt);
        std::swap(cur_gs, nxt_gs);
        if (!plain) *ntt = false;   // a key switch leaves coefficients
    }
    // field trace: for k = level1+1 .. log2(N): ct <- ct + tau_{2^k+1}(ct)
    // (from k = 2 at gamma = 2: the client's power supplied the tau_3 term)
    for (int k = std::max(level1 + 1, tau3_done ? 2 : 1); trace && k <= R.log_n; ++k) {
        const int d = (1 << k) + 1;
        const u64 *key;
        SF_TRY(key_for(d, &key));
        SfKsBatch b;
        memset(&b, 0, sizeof(b));
        b.E = cur;
        b.E_stride = cur_gs;
        b.out = nxt;
        b.out_stride = nxt_gs;
        b.inner = 1 << 30;
        b.count = G;
        b.d = d;
        b.add_v = 1;
        b.ntt = *ntt;
        b.key = key;
        SF_TRY(sf_ks_run(ctx, b, ks_scratch, batch, st));
        std::swap(cur, nxt);
        std::swap(cur_gs, nxt_gs);
        *ntt = false;
    }
    *res = cur;
    *res_stride = cur_gs;
    return SF_OK;
}

// ------------------------------------------------------------- small ops --

// Bias (the affine part b of f(x) = Ax + b): b-part coefficient l*N/n of
// group g gets bq[channel(sigma_out(g n + l))].
__global__ void k_add_bias(SfRing R, u64 *out, int G, int n, int E_out, const int *sig_out, const int64_t *bq,
                           int C_out, int scale)
{
    const size_t ct = (size_t)2 * R.L * R.n;
    const int stride = R.n / n;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < G * n; x += gridDim.x * blockDim.x) {
        if (x >= E_out) continue;
        int g = x / n, l = x % n;
        int o = sig_out ? sig_out[x] : x;
        int64_t v = bq[o % C_out];
        for (int i = 0; i < R.L; ++i) {
            int64_t q = (int64_t)R.m[i].q;
            int64_t r = v % q;
            if (r < 0) r += q;
            const u64 r1 = (u64)r;
            for (int k = 1; k < scale; ++k) r = (int64_t)sf_add((u64)r, r1, (u64)q);
            u64 *p = out + g * ct + ((size_t)(R.L + i) << R.log_n) + (size_t)l * stride;
            *p = sf_add(*p, (u64)r, (u64)q);
        }
    }
}

sf_status sf_add_bias(sf_ctx *ctx, u64 *out, int G, int n, int E_out, const int *d_sig_out, const int64_t *d_bq,
                      int C_out, cudaStream_t st, int scale)
{
    cudaEvent_t ev;
    sf_launch_begin(ctx, SFK_ELEMWISE, st, &ev);
    int total = G * n;
    k_add_bias<<<std::max(1, std::min((total + 255) / 256, 1024)), 256, 0, st>>>(ctx->ring, out, G, n, E_out, d_sig_out,
                                                                                 d_bq, C_out, scale);
    sf_launch_end(ctx, SFK_ELEMWISE, st, ev);
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

// Whole-ciphertext gather: out[k] = in[perm[k]].
__global__ void k_shuffle_cts(const u64 *in, u64 *out, const int *perm, int count, size_t ct_words)
{
    size_t total = (size_t)count * ct_words;
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < total; x += (size_t)gridDim.x * blockDim.x) {
        size_t k = x / ct_words, w = x % ct_words;
        out[x] = in[(size_t)perm[k] * ct_words + w];
    }
}

sf_status sf_shuffle_launch(sf_ctx *ctx, const u64 *in, u64 *out, const int *d_perm, int count, cudaStream_t st)
{
    const size_t ct = (size_t)2 * ctx->ring.L * ctx->ring.n;
    cudaEvent_t ev;
    sf_launch_begin(ctx, SFK_SHUFFLE, st, &ev);
    size_t total = (size_t)count * ct;
    k_shuffle_cts<<<(int)std::min<size_t>((total + 255) / 256, (size_t)ctx->num_sms * 32), 256, 0, st>>>(in, out, d_perm, count, ct);
    sf_launch_end(ctx, SFK_SHUFFLE, st, ev);
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

// Extraction at gamma = 0 (Lemma 1 with t = 2): out = N^-1 X^-i ct, coefficient domain.
__global__ void k_extract(SfRing R, const u64 *ct, u64 *out, int i)
{
    const size_t total = (size_t)2 * R.L * R.n;
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < total; x += (size_t)gridDim.x * blockDim.x) {
        int limb = (int)((x >> R.log_n) % R.L);
        int k = (int)(x & (R.n - 1));
        size_t base = x - k;
        const SfMod &M = R.m[limb];
        // coefficient k of X^-i a = coefficient k + i of a, negated when k + i >= N
        int src = k + i;
        u64 v = ct[base + (src & (R.n - 1))];
        if (src >= R.n && v) v = M.q - v;
        out[x] = sf_mul_shoup(v, M.ninv, M.ninv_p, M.q);
    }
}

// Extraction at gamma = 2 (Lemma 1 at t = 2, scaled by [K_2 : K_0] = 2):
// out = (N/2)^-1 (X^-i ct + X^-3i ct3), coefficient domain.
__global__ void k_extract2(SfRing R, const u64 *ct, const u64 *ct3, u64 *out, int i)
{
    const size_t total = (size_t)2 * R.L * R.n;
    const int two_n = 2 * R.n;
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < total; x += (size_t)gridDim.x * blockDim.x) {
        int limb = (int)((x >> R.log_n) % R.L);
        int k = (int)(x & (R.n - 1));
        size_t base = x - k;
        const SfMod &M = R.m[limb];
        // coefficient k of X^-e a is a[(k + e) mod 2N] folded by X^N = -1
        auto coef = [&](const u64 *a, int e) -> u64 {
            const int src = (k + e) % two_n;
            u64 v = a[base + (src & (R.n - 1))];
            return (src >= R.n && v) ? M.q - v : v;
        };
        const u64 v = sf_add(coef(ct, i), coef(ct3, (3 * i) % two_n), M.q);
        // (N/2)^-1 = 2 N^-1
        out[x] = sf_add(sf_mul_shoup(v, M.ninv, M.ninv_p, M.q), sf_mul_shoup(v, M.ninv, M.ninv_p, M.q), M.q);
    }
}

sf_status sf_extract2_launch(sf_ctx *ctx, const u64 *ct, const u64 *ct3, u64 *out, int i, cudaStream_t st)
{
    cudaEvent_t ev;
    sf_launch_begin(ctx, SFK_ELEMWISE, st, &ev);
    size_t total = (size_t)2 * ctx->ring.L * ctx->ring.n;
    k_extract2<<<(int)((total + 255) / 256), 256, 0, st>>>(ctx->ring, ct, ct3, out, i);
    sf_launch_end(ctx, SFK_ELEMWISE, st, ev);
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

sf_status sf_extract_launch(sf_ctx *ctx, const u64 *ct, u64 *out, int i, cudaStream_t st)
{
    cudaEvent_t ev;
    sf_launch_begin(ctx, SFK_ELEMWISE, st, &ev);
    size_t total = (size_t)2 * ctx->ring.L * ctx->ring.n;
    k_extract<<<(int)((total + 255) / 256), 256, 0, st>>>(ctx->ring, ct, out, i);
    sf_launch_end(ctx, SFK_ELEMWISE, st, ev);
    SF_CUDA_TRY(cudaGetLastError());
    return SF_OK;
}

sf_status sf_layer_init_attributes()
{
    const int mx = 227 * 1024;
#define SF_ATTR(K) SF_CUDA_TRY(cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
    SF_FOR_RINGS({ SF_ATTR((k_leaf_col<LR, LC, PM>)) SF_ATTR((k_leaf_row<LR, LC, PM>)) });
#undef SF_ATTR
    return SF_OK;
}
