// sf_reg.cuh -- register-resident passes of the negacyclic NTT.
//
// A ring of N = R x C points is transformed as R-point columns and C-point
// rows (R, C between 32 and 256; see sf_tile.cuh for the transform itself).  A
// block of S threads runs 16 sub-transforms of S points, 16 points per thread,
// in two register phases with one exchange through shared memory between them:
//   phase 1: thread i of a sub-transform holds k = i + u S/16 + 16 t
//            (t < S/16, u < 256/S), the stages of distance S/2 .. 16;
//   phase 2: it holds k = 16 i + t, the stages of distance 8, 4, 2, 1.
// The inverse runs them in the opposite order.  Global memory is read and
// written straight from registers, so a pass costs one shared-memory round
// trip (16 bytes per point) against four to six of the sweeps that keep the
// tile in shared memory.  Row passes put the S/16 threads of a row in one warp:
// their exchange needs no block barrier.
//
// Twiddles are Shoup pairs (w, floor(w 2^64 / q)).  psi^-brev(m + g) =
// -psi^brev(m + (m - 1 - g)) for m = 2^a: the inverse twiddle of a group is
// minus the forward twiddle of the mirrored group of its level, so one table
// serves both directions (the inverse butterfly multiplies Y - X instead of
// X - Y).  The mirror of row r is row R - 1 - r; a row tile therefore holds
// eight rows and their mirrors, and the inverse pass reads the same staged
// table at thread index tid ^ (9 S/16 - 1).
//
// NTT-domain polynomials that stay inside the library (leaves, prepared
// inputs, rotation keys) are stored in "storage order", [tile][t][thread] of a
// row pass's phase 2, so that every kernel reads and writes them coalesced
// from registers (sf_storage_index).
#pragma once
#include "sf_arith.cuh"
#include "sf_internal.h"

typedef ulonglong2 sf_pair;   // (w, w')

// shape of the sub-transforms of 2^LS points
template <int LS>
struct SfSub {
    static constexpr int S = 1 << LS, R1 = LS - 4, NI = S / 16, U = 256 / S, NT = S;
    static constexpr int COL_WORDS = 16 * S;              // exchange buffer of a column tile, [k][b]
    static constexpr int PITCH = 17 * NI;                 // row of a row tile: k + k / 16, conflict-free in both phases
    static constexpr int ROW_WORDS = 16 * PITCH;
    static constexpr int ROW_PAIRS = 16 * (S - 1);        // twiddles of a row tile
};

// ---- butterflies -----------------------------------------------------------

// acc + (x*w mod q), the added term in [0, 4q): Shoup's product with the
// truncated quotient (sf_mulhi_trunc); the accumulator rides through the wide
// multiplies, which add it for free
SF_HD u64 sf_mad_shoup_lazy4(u64 acc, u64 x, u64 w, u64 wp, u64 q)
{
    return acc + x * w + sf_mulhi_trunc(x, wp) * (0 - q);
}

// forward: X + wY, X - wY + 4q; bounds grow by 4q per stage (below 72q < 2^57
// after 16 stages from 8q)
__device__ __forceinline__ void sf_fwd(u64 &X, u64 &Y, const sf_pair w, u64 q)
{
    const u64 x = X;
    X = sf_mad_shoup_lazy4(x, Y, w.x, w.y, q);
    Y = x + x + 4 * q - X;
}

// inverse with the mirrored twiddle: X + Y, (Y - X) w.  At stage k of a pass
// (k = 0 .. 7) inputs are below 4q 2^k and off = 4q 2^k, so the difference is
// positive and below 2^(k+3) q <= 2^10 q < 2^60; no conditional subtraction.
__device__ __forceinline__ void sf_inv(u64 &X, u64 &Y, const sf_pair w, u64 q, u64 off)
{
    const u64 d = Y - X + off;
    X = X + Y;
    Y = sf_mad_shoup_lazy4(0, d, w.x, w.y, q);
}

// v < 2^63 (and below 2^32 q) brought below 3q: q̂ = floor((v >> sh) binv / 2^32)
// is floor(v / q) minus at most 2
__device__ __forceinline__ u64 sf_red3(u64 v, const SfMod &M)
{
    return v + (u64)__umulhi((unsigned)(v >> M.sh), M.binv) * (0 - M.q);
}

// ---- phases ------------------------------------------------------------------
// x holds phase-1 element (t, u) at t U + u, phase-2 element t at t.  tw(k)
// returns the twiddle of local index k (level 2^a: k = 2^a + group).

template <int LS, class TW>
__device__ __forceinline__ void sf_p1_fwd(u64 (&x)[16], TW tw, u64 q)
{
    constexpr int R1 = SfSub<LS>::R1, U = SfSub<LS>::U;
#pragma unroll
    for (int s = 0; s < R1; ++s) {
        const int d = 1 << (R1 - 1 - s);
#pragma unroll
        for (int g = 0; g < (1 << s); ++g) {
            const sf_pair w = tw((1 << s) + g);
#pragma unroll
            for (int a = 0; a < d; ++a)
#pragma unroll
                for (int u = 0; u < U; ++u) sf_fwd(x[(2 * d * g + a) * U + u], x[(2 * d * g + a + d) * U + u], w, q);
        }
    }
}

// tw(e): twiddle e = 2^s - 1 + g of the thread's 16 points (stage s, group g)
template <class TW>
__device__ __forceinline__ void sf_p2_fwd(u64 (&x)[16], TW tw, u64 q)
{
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const int d = 8 >> s;
#pragma unroll
        for (int g = 0; g < (1 << s); ++g) {
            const sf_pair w = tw((1 << s) - 1 + g);
#pragma unroll
            for (int a = 0; a < d; ++a) sf_fwd(x[2 * d * g + a], x[2 * d * g + a + d], w, q);
        }
    }
}

// inverse phase 2 (stages 0 .. 3 of the pass); tw(e) as above, mirrored
template <class TW>
__device__ __forceinline__ void sf_p2_inv(u64 (&x)[16], TW tw, u64 q)
{
#pragma unroll
    for (int s = 3; s >= 0; --s) {
        const int d = 8 >> s;
        const u64 off = q << (2 + (3 - s));
#pragma unroll
        for (int g = 0; g < (1 << s); ++g) {
            const sf_pair w = tw((1 << s) - 1 + g);
#pragma unroll
            for (int a = 0; a < d; ++a) sf_inv(x[2 * d * g + a], x[2 * d * g + a + d], w, q, off);
        }
    }
}

// inverse phase 1 (stages 4 .. 4 + R1 - 1 of the pass)
template <int LS, class TW>
__device__ __forceinline__ void sf_p1_inv(u64 (&x)[16], TW tw, u64 q)
{
    constexpr int R1 = SfSub<LS>::R1, U = SfSub<LS>::U;
#pragma unroll
    for (int s = R1 - 1; s >= 0; --s) {
        const int d = 1 << (R1 - 1 - s);
        const u64 off = q << (2 + 4 + (R1 - 1 - s));
#pragma unroll
        for (int g = 0; g < (1 << s); ++g) {
            const sf_pair w = tw((1 << s) + g);
#pragma unroll
            for (int a = 0; a < d; ++a)
#pragma unroll
                for (int u = 0; u < U; ++u) sf_inv(x[(2 * d * g + a) * U + u], x[(2 * d * g + a + d) * U + u], w, q, off);
        }
    }
}

// ---- column tiles --------------------------------------------------------------
// 16 columns of 2^LR points; thread: column b = tid & 15, i = tid >> 4, so a
// half-warp touches 16 consecutive words of one row of the polynomial.  The
// column table is colT[k], k < R, staged once; buf is an exchange buffer.

template <int LR>
struct SfCol {
    using Sub = SfSub<LR>;
    int b, i;
    __device__ __forceinline__ SfCol() : b(threadIdx.x & 15), i(threadIdx.x >> 4) {}
    // row of phase-1 element r = t U + u, of phase-2 element t
    __device__ __forceinline__ int k1(int r) const { return i + (r % Sub::U) * Sub::NI + 16 * (r / Sub::U); }
    __device__ __forceinline__ int k2(int t) const { return 16 * i + t; }

    __device__ __forceinline__ void fwd1(u64 (&x)[16], const sf_pair *tab, u64 q) const
    {
        sf_p1_fwd<LR>(x, [&](int k) { return tab[k]; }, q);
    }
    __device__ __forceinline__ void fwd2(u64 (&x)[16], const sf_pair *tab, u64 q) const
    {
        sf_p2_fwd(x, [&](int e) {
            const int s = e >= 7 ? 3 : e >= 3 ? 2 : e >= 1 ? 1 : 0, g = e - ((1 << s) - 1);
            return tab[(Sub::NI << s) + (i << s) + g];
        }, q);
    }
    __device__ __forceinline__ void inv2(u64 (&x)[16], const sf_pair *tab, u64 q) const
    {
        sf_p2_inv(x, [&](int e) {
            const int s = e >= 7 ? 3 : e >= 3 ? 2 : e >= 1 ? 1 : 0, g = e - ((1 << s) - 1);
            return tab[(Sub::NI << s) + ((Sub::NI - 1 - i) << s) + (1 << s) - 1 - g];
        }, q);
    }
    __device__ __forceinline__ void inv1(u64 (&x)[16], const sf_pair *tab, u64 q) const
    {
        sf_p1_inv<LR>(x, [&](int k) {
            const int m = k >= 8 ? 8 : k >= 4 ? 4 : k >= 2 ? 2 : 1;
            return tab[3 * m - 1 - k];
        }, q);
    }
    // phase 1 -> phase 2 and back through buf; one block barrier each.  Passes
    // that follow one another alternate between two buffers, so the barrier of
    // one also orders the reads of the one before against the next writes.
    __device__ __forceinline__ void to2(u64 (&x)[16], u64 *buf) const
    {
#pragma unroll
        for (int r = 0; r < 16; ++r) buf[k1(r) * 16 + b] = x[r];
        __syncthreads();
#pragma unroll
        for (int t = 0; t < 16; ++t) x[t] = buf[k2(t) * 16 + b];
    }
    __device__ __forceinline__ void to1(u64 (&x)[16], u64 *buf) const
    {
#pragma unroll
        for (int t = 0; t < 16; ++t) buf[k2(t) * 16 + b] = x[t];
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 16; ++r) x[r] = buf[k1(r) * 16 + b];
    }
};

// ---- row tiles -------------------------------------------------------------------
// 8 rows and their mirrors; thread: row b = tid / NI, i = tid % NI (the threads
// of a row share a warp).  Staged table tw: phase-1 twiddles (k, b) at
// (k - 1) 16 + b, k < NI; phase-2 twiddles (e, thread) at P2 + e NT + tid.

template <int LC>
struct SfRowT {
    using Sub = SfSub<LC>;
    static constexpr int P2 = 16 * (Sub::NI - 1), MIR = 9 * Sub::NI - 1;
    int b, i;
    __device__ __forceinline__ SfRowT() : b(threadIdx.x / Sub::NI), i(threadIdx.x % Sub::NI) {}
    // row of the polynomial that row b of tile `tile` is (R rows in all)
    __device__ __forceinline__ int row(int tile, int R) const { return b < 8 ? 8 * tile + b : R - 1 - 8 * tile - (b - 8); }
    __device__ __forceinline__ int k1(int r) const { return i + (r % Sub::U) * Sub::NI + 16 * (r / Sub::U); }

    __device__ __forceinline__ void fwd1(u64 (&x)[16], const sf_pair *tw, u64 q) const
    {
        sf_p1_fwd<LC>(x, [&](int k) { return tw[(k - 1) * 16 + b]; }, q);
    }
    __device__ __forceinline__ void fwd2(u64 (&x)[16], const sf_pair *tw, u64 q) const
    {
        sf_p2_fwd(x, [&](int e) { return tw[P2 + e * Sub::NT + threadIdx.x]; }, q);
    }
    __device__ __forceinline__ void inv2(u64 (&x)[16], const sf_pair *tw, u64 q) const
    {
        const int tid = threadIdx.x ^ MIR;
        sf_p2_inv(x, [&](int e) {
            const int s = e >= 7 ? 3 : e >= 3 ? 2 : e >= 1 ? 1 : 0, g = e - ((1 << s) - 1);
            return tw[P2 + ((2 << s) - 2 - g) * Sub::NT + tid];
        }, q);
    }
    __device__ __forceinline__ void inv1(u64 (&x)[16], const sf_pair *tw, u64 q) const
    {
        sf_p1_inv<LC>(x, [&](int k) {
            const int m = k >= 8 ? 8 : k >= 4 ? 4 : k >= 2 ? 2 : 1;
            return tw[(3 * m - 2 - k) * 16 + (b ^ 8)];
        }, q);
    }
    __device__ __forceinline__ void put1(const u64 (&x)[16], u64 *buf) const
    {
#pragma unroll
        for (int r = 0; r < 16; ++r) buf[b * Sub::PITCH + k1(r) + (k1(r) >> 4)] = x[r];
    }
    __device__ __forceinline__ void put2(const u64 (&x)[16], u64 *buf) const
    {
#pragma unroll
        for (int t = 0; t < 16; ++t) buf[b * Sub::PITCH + 17 * i + t] = x[t];
    }
    __device__ __forceinline__ void get1(u64 (&x)[16], const u64 *buf) const
    {
#pragma unroll
        for (int r = 0; r < 16; ++r) x[r] = buf[b * Sub::PITCH + k1(r) + (k1(r) >> 4)];
    }
    __device__ __forceinline__ void get2(u64 (&x)[16], const u64 *buf) const
    {
#pragma unroll
        for (int t = 0; t < 16; ++t) x[t] = buf[b * Sub::PITCH + 17 * i + t];
    }
    // exchanges inside the warp: the leading barrier orders the previous
    // exchange's reads before these writes
    __device__ __forceinline__ void to2(u64 (&x)[16], u64 *buf) const
    {
        __syncwarp();
        put1(x, buf);
        __syncwarp();
        get2(x, buf);
    }
    __device__ __forceinline__ void to1(u64 (&x)[16], u64 *buf) const
    {
        __syncwarp();
        put2(x, buf);
        __syncwarp();
        get1(x, buf);
    }
    // storage order: element t of this thread in tile `tile`
    __device__ __forceinline__ static size_t store_at(int tile, int t)
    {
        return (size_t)tile * 16 * Sub::S + (size_t)t * Sub::NT + threadIdx.x;
    }
};

// stages the column tables of moduli m0 .. m0 + n - 1, or one row tile's table
template <int LR>
__device__ __forceinline__ void sf_stage_cols(sf_pair *dst, const sf_pair *__restrict__ table, int m0, int n)
{
    for (int k = threadIdx.x; k < (n << LR); k += SfSub<LR>::NT) dst[k] = table[((size_t)m0 << LR) + k];
}
template <int LR, int LC>
__device__ __forceinline__ void sf_stage_row(sf_pair *dst, const sf_pair *__restrict__ table, int mod, int tile)
{
    constexpr int W = SfSub<LC>::ROW_PAIRS;
    const sf_pair *src = table + ((size_t)mod * ((1 << LR) / 16) + tile) * W;
    for (int k = threadIdx.x; k < W; k += SfSub<LC>::NT) dst[k] = src[k];
}

// storage index of NTT slot j (natural bit-reversed order) and back
__host__ __device__ __forceinline__ int sf_storage_index(int j, int log_r, int log_c)
{
    const int R = 1 << log_r, ni = 1 << (log_c - 4);
    const int row = j >> log_c, col = j & ((1 << log_c) - 1);
    const bool mir = row >= R / 2;
    const int rr = mir ? R - 1 - row : row;
    return (((rr >> 3) << 4) << log_c) + ((col & 15) << log_c) + ((rr & 7) + (mir ? 8 : 0)) * ni + (col >> 4);
}
__host__ __device__ __forceinline__ int sf_natural_index(int p, int log_r, int log_c)
{
    const int R = 1 << log_r, ni_l = log_c - 4;
    const int tile = p >> (log_c + 4), t = (p >> log_c) & 15, b = (p >> ni_l) & 15, i = p & ((1 << ni_l) - 1);
    const int row = b < 8 ? 8 * tile + b : R - 1 - 8 * tile - (b - 8);
    return (row << log_c) + 16 * i + t;
}

// ---- balanced persistent partition ----------------------------------------
// A persistent launch of gridDim.x blocks over n_units work units numbered
// group-major (u = group * n_items + item) gives block x the units
// [x n / grid, (x + 1) n / grid): every block the floor or the ceiling of the
// mean, whatever the group count, and a block restages tables only where its
// range crosses into a new group.
struct SfUnitRange {
    int u0, u1;
};
__device__ __forceinline__ SfUnitRange sf_unit_range(int n_units)
{
    return {(int)((long long)blockIdx.x * n_units / gridDim.x),
            (int)(((long long)blockIdx.x + 1) * n_units / gridDim.x)};
}

// runs the statements with constexpr LR, LC for the ring size log_n (10..16)
#define SF_RING_DISPATCH(log_n, ...)                                  \
    do {                                                              \
        switch (log_n) {                                              \
        case 10: { constexpr int LR = 5, LC = 5; __VA_ARGS__ } break; \
        case 11: { constexpr int LR = 5, LC = 6; __VA_ARGS__ } break; \
        case 12: { constexpr int LR = 6, LC = 6; __VA_ARGS__ } break; \
        case 13: { constexpr int LR = 6, LC = 7; __VA_ARGS__ } break; \
        case 14: { constexpr int LR = 7, LC = 7; __VA_ARGS__ } break; \
        case 15: { constexpr int LR = 7, LC = 8; __VA_ARGS__ } break; \
        default: { constexpr int LR = 8, LC = 8; __VA_ARGS__ } break; \
        }                                                             \
    } while (0)

// resident blocks per SM of a kernel, at least 1
template <class K>
static int sf_occupancy(K kernel, int threads, size_t smem)
{
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        b = 1;
    }
    return b > 1 ? b : 1;
}
