// sf_reg.cuh -- register-resident passes of the negacyclic NTT.
//
// Transform (Longa-Naehrig 2016 merged form): forward Cooley-Tukey with the
// table psi_brev[k] = psi^brev(k) (psi a primitive 2N-th root), natural-order
// input, bit-reversed output: out[j] = a(psi^(2 brev(j) + 1)).  Inverse:
// Gentleman-Sande with psi^-brev(k), then a factor N^-1.  Index j = r C + c with
// N = R C (R, C between 32 and 256): the forward stages of distance >= C mix
// elements of one column ("column pass"), the others stay inside one row.
// Local stage of m groups, group g: global table index m + g for every column,
// m (R + r) + g for row r.
//
// A pass keeps its points in registers and exchanges them through shared memory
// between phases; global memory is read and written straight from registers.
//
// Every thread holds 8 points and runs up to three stages per phase, in two
// (32, 64 points) or three phases (128, 256 points).  A tile is 2048 points at
// 128 and 256 points (16 or 8 sub-transforms, 256 threads): with three blocks
// per SM a kernel has 24 warps and 80 registers a thread; the kernels that hold
// the accumulators of inner products beside the points run two blocks of 128
// registers (SfShape::BPS_ACC).  The C/8 threads of a row share a warp, so row
// exchanges need no block barrier and the warps of a block run independently;
// columns take one block barrier a transform (SfColT).  16 points a thread (one
// exchange less, 128 registers, 16 warps) lost: the inner product ran 25.6 us
// per key switch at N = 2^16, waiting on memory and on instruction fetches.
//
// Twiddles are pairs (w, companion), see sf_mad.  psi^-brev(m + g) =
// -psi^brev(m + (m - 1 - g)) for m = 2^a: the inverse twiddle of a group is
// minus the forward twiddle of the mirrored group of its level, so one table
// serves both directions (the inverse butterfly multiplies Y - X instead of
// X - Y).  The mirror of row r is row R - 1 - r; a row tile therefore holds
// rows and their mirrors, and the inverse pass reads the same staged table at
// mirrored positions.
//
// NTT-domain polynomials that stay inside the library (leaves, prepared
// inputs, rotation keys) are stored in "storage order", [tile][t][thread] of a
// row pass's last phase, so that every kernel reads and writes them coalesced
// from registers (sf_storage_index).
#pragma once
#include "sf_arith.cuh"
#include "sf_internal.h"

typedef ulonglong2 sf_pair;   // (w, companion)

// Shape of a tile: NB sub-transforms of 2^LS points (for rows NB / 2 rows and
// their mirrors), LP threads each.  Phase ph holds index bits P .. P + 2 of a
// point's position k in the registers and runs the stages of distance
// 2^HI .. 2^LO.
template <int LS>
struct SfShape {
    static constexpr int LS_ = LS, S = 1 << LS, NB = LS == 8 ? 8 : 16, HALF = NB / 2, LP = S / 8, NT = NB * LP, TILE = NB * S;
    // exchange buffers: a row k + k / 8 of [b], a column tile [k + k / 8][b]
    static constexpr int PITCH = 9 * LP, WORDS = NB * PITCH;
    static constexpr int PAIRS = NB * (S - 1);   // twiddles of a row tile
    static constexpr int NP = LS >= 7 ? 3 : 2;
    // blocks per SM: 24 warps of 80 registers; 16 of 128 for the kernels with the
    // inner products' accumulators, which otherwise spill and hold back the key's
    // loads (per round of 32768 key switches at N = 2^16, 5 + 2 primes: 548 ms at
    // 24 warps, 490 at 16; the leaf rows 117 and 102 ms)
    static constexpr int BPS = 768 / NT, BPS_ACC = 512 / NT;
    SF_HD static constexpr int P(int ph) { return ph == 0 ? LS - 3 : (ph == 1 && LS >= 7) ? 2 : 0; }
    SF_HD static constexpr int LO(int ph) { return P(ph); }
    SF_HD static constexpr int HI(int ph) { return ph == 0 ? LS - 1 : P(ph - 1) - 1; }
    // padded position k + k / 8 of register t of thread i in phase ph: pos(ph, i) + step(ph, t)
    SF_HD static constexpr int pos(int ph, int i)
    {
        const int p = P(ph), hi = i >> p, lo = i & ((1 << p) - 1);
        return (hi << (p + 3)) + lo + (hi << p) + (p >= 3 ? lo >> 3 : 0);
    }
    SF_HD static constexpr int step(int ph, int t)
    {
        const int p = P(ph);
        return (t << p) + (p >= 3 ? t << (p - 3) : p == 2 ? t >> 1 : 0);
    }
    // groups of threads that share a phase's twiddles, in one row
    SF_HD static constexpr int H(int ph) { return S >> (P(ph) + 3); }
    // first entry of stage q (q <= HI) of phase ph among the phase's entries: 2^(P+2-q') per stage q'
    SF_HD static constexpr int E(int ph, int q) { return (1 << (P(ph) + 2 - q)) - (1 << (P(ph) + 2 - HI(ph))); }
    // first entry of phase ph in a row tile's table
    SF_HD static constexpr int OFF(int ph)
    {
        return ph == 0 ? 0 : (ph == 1 ? 0 : E(1, LO(1) - 1) * NB * H(1)) + E(0, LO(0) - 1) * NB * H(0);
    }
};

// ---- products and butterflies -----------------------------------------------

// v (below 2^32 q) brought below 3q: floor((v >> sh) binv / 2^32) is floor(v / q)
// minus at most 2
__device__ __forceinline__ u64 sf_red3(u64 v, const SfMod &M)
{
    return v + (u64)__umulhi((unsigned)(v >> M.sh), M.binv) * (0 - M.q);
}

// Two forms of a product by a fixed operand w < q, both with a stored companion
// and both returning acc + r with r = x w (mod q), 0 <= r < off for any x < 2^64;
// the accumulator rides through the wide multiplies, which add it for free.
//
// PM = false, any q < 2^51: Shoup's product, companion floor(w 2^64 / q), with
// the truncated quotient (sf_mulhi_trunc): r < 4q.  9 multiplies, 19 instructions
// a butterfly.
//
// PM = true, q = 2^50 - delta with small delta (the largest NTT primes of 50
// bits): with x = x0 + 2^32 x1 and the companion v = 2^32 w mod q,
//     x w = x0 w + x1 v = T (mod q),   T < 2^83,
// and since q is almost 2^50 the high parts of w and v are the quotients
// themselves: qh = floor(x0 floor(w / 2^19) / 2^32) + floor(x1 floor(v / 2^19) /
// 2^32) is T / 2^51 less at most 4 (four floors), and below 2^32, so r = T - qh 2q
// = (T - qh 2^51) + qh 2 delta lies in [0, 2^53 + 2^33 delta).  8 multiplies, 15
// instructions: register-resident forward butterflies run at 1289 G/s against
// 1164, inverse ones at 1272 against 1145.
template <bool PM>
__device__ __forceinline__ u64 sf_mad(u64 acc, u64 x, const sf_pair w, const SfMod &M)
{
    if constexpr (PM) {
        const unsigned x0 = (unsigned)x, x1 = (unsigned)(x >> 32);
        const unsigned qh = __umulhi(x0, (unsigned)(w.x >> 19)) + __umulhi(x1, (unsigned)(w.y >> 19));
        return acc + x0 * w.x + x1 * w.y + qh * M.n2q;
    } else {
        return acc + x * w.x + sf_mulhi_trunc(x, w.y) * (0 - M.q);
    }
}

// acc + x w + y z (mod q) for canonical x, y, the added part below 4 off; with PM
// the two products share the last multiply: 4q times the sum of their quotients
// by 2^52, each below 2^30 + 2^17 and short by less than 4, so the rest is below
// 8 2^52 + 2^33 delta
template <bool PM>
__device__ __forceinline__ u64 sf_mad2(u64 acc, u64 x, const sf_pair w, u64 y, const sf_pair z, const SfMod &M)
{
    if constexpr (PM) {
        const unsigned x0 = (unsigned)x, x1 = (unsigned)(x >> 32), y0 = (unsigned)y, y1 = (unsigned)(y >> 32);
        const unsigned qh = __umulhi(x0, (unsigned)(w.x >> 20)) + __umulhi(x1, (unsigned)(w.y >> 20)) +
                            __umulhi(y0, (unsigned)(z.x >> 20)) + __umulhi(y1, (unsigned)(z.y >> 20));
        return acc + x0 * w.x + x1 * w.y + y0 * z.x + y1 * z.y + qh * (2 * M.n2q);
    } else {
        return sf_mad<PM>(sf_mad<PM>(acc, x, w, M), y, z, M);
    }
}

// Inner products: acc.s + sum of x_j w_j, canonical w_j, closed by sf_acc_close.
// With PM the quotients of all terms are summed and multiplied once; by 2^53 each
// is below 2^30 (x < 2^64), so a sum holds 4 terms (SF_ACC_TERMS) between closes.
#define SF_ACC_TERMS 4
template <bool PM>
struct SfAcc {
    u64 s;
    unsigned qh;
};
template <bool PM>
__device__ __forceinline__ void sf_acc_add(SfAcc<PM> &a, u64 x, const sf_pair w, const SfMod &M)
{
    if constexpr (PM) {
        const unsigned x0 = (unsigned)x, x1 = (unsigned)(x >> 32);
        a.s = a.s + x0 * w.x + x1 * w.y;
        a.qh += __umulhi(x0, (unsigned)(w.x >> 21)) + __umulhi(x1, (unsigned)(w.y >> 21));
    } else {
        a.s = sf_mad<PM>(a.s, x, w, M);
    }
}
// the sum below 3q; the accumulator goes on from it.  Before: per term
// T - qh 2^53 < 4 2^53 and qh 8 delta < 2^33 delta, so four terms stay below
// 2^57 + 2^35 delta <= 4 off + 2^57 < 2^61.
template <bool PM>
__device__ __forceinline__ u64 sf_acc_close(SfAcc<PM> &a, const SfMod &M)
{
    if constexpr (PM) a.s = a.s + a.qh * (4 * M.n2q);
    a.s = sf_red3(a.s, M);
    a.qh = 0;
    return a.s;
}

// forward: X + wY, X - wY + off; bounds grow by off per stage, from at most
// 8 off to 24 off < 2^63 after 16 stages (checked when the context is made)
template <bool PM>
__device__ __forceinline__ void sf_fwd(u64 &X, u64 &Y, const sf_pair w, const SfMod &M)
{
    const u64 x = X;
    X = sf_mad<PM>(x, Y, w, M);
    Y = x + x + M.off - X;
}

// inverse with the mirrored twiddle: X + Y, (Y - X) w.  `off` is a multiple of q
// above every input (sf_inv_off), so the difference is positive.
template <bool PM>
__device__ __forceinline__ void sf_inv(u64 &X, u64 &Y, const sf_pair w, const SfMod &M, u64 off)
{
    const u64 d = Y - X + off;
    X = X + Y;
    Y = sf_mad<PM>(0, d, w, M);
}

// v (below 2^32 q) brought to [0, q)
__device__ __forceinline__ u64 sf_csub3(u64 v, const SfMod &M) { return sf_csub(sf_csub(v, M.q), M.q); }   // v < 3q
__device__ __forceinline__ u64 sf_canon(u64 v, const SfMod &M) { return sf_csub3(sf_red3(v, M), M); }

// ---- column tiles --------------------------------------------------------------
// NB columns of 2^LR points; thread: column b = tid % NB, i = tid / NB, so NB
// consecutive threads touch NB consecutive words of one row of the polynomial.
// Register t of phase ph holds k = (i >> P) 2^(P+3) + t 2^P + (i mod 2^P).  The
// column table is tab[k], k < R; buf is the exchange buffer.

// Bounds of an inverse pass (multiples of q, off1 = max(8q, off) <= 2^58).  Its
// inputs are below off1; a product stays below off and the bound of a sum doubles.
// Before the last phase (three stages) the registers that were sums in three
// stages of the phase before, or in two after two others, are reduced
// (sf_inv_fold), so that its inputs are below 4 off1 and every value stays below
// 2^63.  After the last phase x[4 .. 7] are products, below off, x[2], x[3] below
// 2 off and x[1] below 4 off; x[0] is below 32 off1.
template <int LS>
__device__ __forceinline__ u64 sf_inv_off(int st, const SfMod &M)
{
    return M.off1 << (st < LS - 3 ? st : st - (LS - 3) + 2);
}
template <int LS>
__device__ __forceinline__ void sf_inv_fold(u64 (&x)[8], const SfMod &M)
{
    if (LS >= 6) x[0] = sf_red3(x[0], M);
    if (LS == 7) x[4] = sf_red3(x[4], M);
}

// rows of an inverse pass handed to its columns: below off again
__device__ __forceinline__ void sf_inv_rows_out(u64 (&x)[8], const SfMod &M)
{
#pragma unroll
    for (int t = 0; t < 4; ++t) x[t] = sf_red3(x[t], M);
}

template <int LR, bool PM>
struct SfColT {
    using Sh = SfShape<LR>;
    static constexpr int LAST = Sh::NP - 1;
    int b, i;
    __device__ __forceinline__ SfColT() : b(threadIdx.x % Sh::NB), i(threadIdx.x / Sh::NB) {}
    template <int PH>
    __device__ __forceinline__ int k(int t) const
    {
        constexpr int P = Sh::P(PH);
        return ((i >> P) << (P + 3)) + (t << P) + (i & ((1 << P) - 1));
    }
    __device__ __forceinline__ int k1(int t) const { return k<0>(t); }
    __device__ __forceinline__ int kl(int t) const { return k<LAST>(t); }
    __device__ __forceinline__ int at(int kk) const { return (kk + (kk >> 3)) * Sh::NB + b; }

    template <int PH>
    __device__ __forceinline__ void phase_fwd(u64 (&x)[8], const sf_pair *tab, const SfMod &M) const
    {
        constexpr int P = Sh::P(PH), HI = Sh::HI(PH), LO = Sh::LO(PH);
#pragma unroll
        for (int st = HI; st >= LO; --st) {
            const int d = 1 << (st - P), lc = P + 2 - st;
#pragma unroll
            for (int sub = 0; sub < (1 << lc); ++sub) {
                const sf_pair w = tab[(Sh::S >> (st + 1)) + ((i >> P) << lc) + sub];
#pragma unroll
                for (int a = 0; a < d; ++a) sf_fwd<PM>(x[2 * d * sub + a], x[2 * d * sub + a + d], w, M);
            }
        }
    }
    // stages of the inverse pass (bounds: sf_inv_off)
    template <int PH>
    __device__ __forceinline__ void phase_inv(u64 (&x)[8], const sf_pair *tab, const SfMod &M) const
    {
        constexpr int P = Sh::P(PH), HI = Sh::HI(PH), LO = Sh::LO(PH);
#pragma unroll
        for (int st = LO; st <= HI; ++st) {
            const int d = 1 << (st - P), lc = P + 2 - st;
            const u64 off = sf_inv_off<Sh::LS_>(st, M);
#pragma unroll
            for (int sub = 0; sub < (1 << lc); ++sub) {
                // group g mirrored: 2 m - 1 - g with m = S >> (st + 1)
                const sf_pair w = tab[(Sh::S >> st) - 1 - ((i >> P) << lc) - sub];
#pragma unroll
                for (int a = 0; a < d; ++a) sf_inv<PM>(x[2 * d * sub + a], x[2 * d * sub + a + d], w, M, off);
            }
        }
        if (PH == 1) sf_inv_fold<Sh::LS_>(x, M);
    }
    // The first of the two exchanges (last of an inverse pass) crosses the block;
    // the other one stays among the threads that hold one 32-point stretch of every
    // column: a warp at 256 points, two at 128.  A thread overwrites only the words
    // it read last, so an exchange takes one barrier, and a transform one block
    // barrier, if a block's consecutive transforms alternate between two buffers:
    // a thread past that barrier of one transform has all threads past their reads
    // of the other buffer (`after` may then copy points into this thread's words of
    // it).  With four block barriers a transform, 512 x 5 limbs of 2^16 took 1550 us
    // against 1515 and the ModDown 228 ms against 222 per 32768 key switches.
    template <int PH>
    __device__ __forceinline__ u64 *mine(u64 *buf) const { return buf + Sh::pos(PH, i) * Sh::NB + b; }
    template <int PH>
    __device__ __forceinline__ void put(const u64 (&x)[8], u64 *buf) const
    {
#pragma unroll
        for (int t = 0; t < 8; ++t) mine<PH>(buf)[Sh::step(PH, t) * Sh::NB] = x[t];
    }
    template <int PH>
    __device__ __forceinline__ void get(u64 (&x)[8], u64 *buf) const
    {
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = mine<PH>(buf)[Sh::step(PH, t) * Sh::NB];
    }
    __device__ __forceinline__ static void stretch_sync()
    {
        if constexpr (4 * Sh::NB == 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + threadIdx.x / (4 * Sh::NB)), "n"(4 * Sh::NB) : "memory");
    }
    template <class F>
    __device__ __forceinline__ void forward(u64 (&x)[8], const sf_pair *tab, u64 *buf, const SfMod &M, F after) const
    {
        phase_fwd<0>(x, tab, M);
        put<0>(x, buf);
        __syncthreads();
        after();
        get<1>(x, buf);
        phase_fwd<1>(x, tab, M);
        if constexpr (Sh::NP == 3) {
            put<1>(x, buf);
            stretch_sync();
            get<2>(x, buf);
            phase_fwd<2>(x, tab, M);
        }
    }
    template <class F>
    __device__ __forceinline__ void inverse(u64 (&x)[8], const sf_pair *tab, u64 *buf, const SfMod &M, F after) const
    {
        phase_inv<LAST>(x, tab, M);
        put<LAST>(x, buf);
        if constexpr (Sh::NP == 3) {
            stretch_sync();
            get<1>(x, buf);
            phase_inv<1>(x, tab, M);
            put<1>(x, buf);
        }
        __syncthreads();
        after();
        get<0>(x, buf);
        phase_inv<0>(x, tab, M);
    }
    __device__ __forceinline__ void forward(u64 (&x)[8], const sf_pair *tab, u64 *buf, const SfMod &M) const
    {
        forward(x, tab, buf, M, [] {});
    }
    __device__ __forceinline__ void inverse(u64 (&x)[8], const sf_pair *tab, u64 *buf, const SfMod &M) const
    {
        inverse(x, tab, buf, M, [] {});
    }
};

// ---- row tiles -------------------------------------------------------------------
// Thread: row b = tid / LP, i = tid % LP.  Register t of phase ph holds element
// k = (i >> P) 2^(P+3) + t 2^P + (i mod 2^P).  The staged table holds, per
// phase and stage, [sub][b][high]: the twiddle of group (high, sub) of row b.

template <int LC, bool PM>
struct SfRowT {
    using Sh = SfShape<LC>;
    static constexpr int FIRST = 0, LAST = Sh::NP - 1;
    int b, i;
    __device__ __forceinline__ SfRowT() : b(threadIdx.x / Sh::LP), i(threadIdx.x % Sh::LP) {}
    // row of the polynomial that row b of tile `tile` is (R rows in all)
    __device__ __forceinline__ int row(int tile, int R) const
    {
        return b < Sh::HALF ? Sh::HALF * tile + b : R - 1 - Sh::HALF * tile - (b - Sh::HALF);
    }
    template <int PH>
    __device__ __forceinline__ int k(int t) const
    {
        constexpr int P = Sh::P(PH);
        return ((i >> P) << (P + 3)) + (t << P) + (i & ((1 << P) - 1));
    }
    // element of the first phase: t LP + i, consecutive over the threads of a row
    __device__ __forceinline__ int k1(int t) const { return k<0>(t); }

    template <int PH>
    __device__ __forceinline__ void phase_fwd(u64 (&x)[8], const sf_pair *tw, const SfMod &M) const
    {
        constexpr int P = Sh::P(PH), HI = Sh::HI(PH), LO = Sh::LO(PH), H = Sh::H(PH);
        const sf_pair *tp = tw + Sh::OFF(PH) + b * H + (i >> P);
#pragma unroll
        for (int st = HI; st >= LO; --st) {
            const int d = 1 << (st - P);
#pragma unroll
            for (int sub = 0; sub < (8 >> (st - P + 1)); ++sub) {
                const sf_pair w = tp[(Sh::E(PH, st) + sub) * Sh::NB * H];
#pragma unroll
                for (int a = 0; a < d; ++a) sf_fwd<PM>(x[2 * d * sub + a], x[2 * d * sub + a + d], w, M);
            }
        }
    }
    // stages of the inverse pass (bounds: sf_inv_off)
    template <int PH>
    __device__ __forceinline__ void phase_inv(u64 (&x)[8], const sf_pair *tw, const SfMod &M) const
    {
        constexpr int P = Sh::P(PH), HI = Sh::HI(PH), LO = Sh::LO(PH), H = Sh::H(PH);
        const sf_pair *tp = tw + Sh::OFF(PH) + (b ^ Sh::HALF) * H + (H - 1 - (i >> P));
#pragma unroll
        for (int st = LO; st <= HI; ++st) {
            const int d = 1 << (st - P), subs = 8 >> (st - P + 1);
            const u64 off = sf_inv_off<Sh::LS_>(st, M);
#pragma unroll
            for (int sub = 0; sub < subs; ++sub) {
                const sf_pair w = tp[(Sh::E(PH, st) + subs - 1 - sub) * Sh::NB * H];
#pragma unroll
                for (int a = 0; a < d; ++a) sf_inv<PM>(x[2 * d * sub + a], x[2 * d * sub + a + d], w, M, off);
            }
        }
        if (PH == 1) sf_inv_fold<Sh::LS_>(x, M);
    }
    template <int PH>
    __device__ __forceinline__ u64 *mine(u64 *buf) const { return buf + b * Sh::PITCH + Sh::pos(PH, i); }
    template <int PH>
    __device__ __forceinline__ void put(const u64 (&x)[8], u64 *buf) const
    {
#pragma unroll
        for (int t = 0; t < 8; ++t) mine<PH>(buf)[Sh::step(PH, t)] = x[t];
    }
    template <int PH>
    __device__ __forceinline__ void get(u64 (&x)[8], u64 *buf) const
    {
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = mine<PH>(buf)[Sh::step(PH, t)];
    }
    // exchange inside the warp; the leading barrier orders the reads of the
    // previous exchange before these writes
    template <int FROM, int TO>
    __device__ __forceinline__ void exchange(u64 (&x)[8], u64 *buf) const
    {
        __syncwarp();
        exchange_on<FROM, TO>(x, buf);
    }
    // the same where this thread read the words it writes last
    template <int FROM, int TO>
    __device__ __forceinline__ void exchange_on(u64 (&x)[8], u64 *buf) const
    {
        put<FROM>(x, buf);
        __syncwarp();
        get<TO>(x, buf);
    }
    // forward pass: first-phase elements in, last-phase elements out (storage order)
    __device__ __forceinline__ void forward(u64 (&x)[8], const sf_pair *tw, u64 *buf, const SfMod &M) const
    {
        phase_fwd<0>(x, tw, M);
        forward_rest(x, tw, buf, M);
    }
    __device__ __forceinline__ void forward_rest(u64 (&x)[8], const sf_pair *tw, u64 *buf, const SfMod &M) const
    {
        exchange<0, 1>(x, buf);
        phase_fwd<1>(x, tw, M);
        if constexpr (Sh::NP == 3) {
            exchange_on<1, 2>(x, buf);
            phase_fwd<2>(x, tw, M);
        }
    }
    // inverse pass: the other way round
    __device__ __forceinline__ void inverse(u64 (&x)[8], const sf_pair *tw, u64 *buf, const SfMod &M) const
    {
        phase_inv<LAST>(x, tw, M);
        inverse_rest(x, tw, buf, M);
    }
    __device__ __forceinline__ void inverse_rest(u64 (&x)[8], const sf_pair *tw, u64 *buf, const SfMod &M) const
    {
        if constexpr (Sh::NP == 3) {
            exchange<2, 1>(x, buf);
            phase_inv<1>(x, tw, M);
            exchange_on<1, 0>(x, buf);
        } else {
            exchange<1, 0>(x, buf);
        }
        phase_inv<0>(x, tw, M);
    }
    // storage order: last-phase element t of this thread in tile `tile`
    __device__ __forceinline__ static size_t store_at(int tile, int t)
    {
        return (size_t)tile * Sh::TILE + (size_t)t * Sh::NT + threadIdx.x;
    }
};

// stages the column tables of moduli m0 .. m0 + n - 1, or one row tile's table
template <int LR>
__device__ __forceinline__ void sf_stage_cols(sf_pair *dst, const sf_pair *__restrict__ table, int m0, int n)
{
    for (int k = threadIdx.x; k < (n << LR); k += SfShape<LR>::NT) dst[k] = table[((size_t)m0 << LR) + k];
}
template <int LR, int LC>
__device__ __forceinline__ void sf_stage_row(sf_pair *dst, const sf_pair *__restrict__ table, int mod, int tile)
{
    constexpr int W = SfShape<LC>::PAIRS;
    const sf_pair *src = table + ((size_t)mod * ((1 << LR) / SfShape<LC>::NB) + tile) * W;
    for (int k = threadIdx.x; k < W; k += SfShape<LC>::NT) dst[k] = src[k];
}

// storage index of NTT slot j (natural bit-reversed order) and back
SF_HD int sf_storage_index(int j, int log_r, int log_c)
{
    const int R = 1 << log_r, hl = log_c == 8 ? 2 : 3, lp = log_c - 3;
    const int row = j >> log_c, col = j & ((1 << log_c) - 1);
    const int mir = row >= R / 2, rr = mir ? R - 1 - row : row;
    const int b = (rr & ((1 << hl) - 1)) + (mir << hl);
    return ((rr >> hl) << (hl + 1 + log_c)) + ((col & 7) << (hl + 1 + lp)) + (b << lp) + (col >> 3);
}
SF_HD int sf_natural_index(int p, int log_r, int log_c)
{
    const int R = 1 << log_r, hl = log_c == 8 ? 2 : 3, lp = log_c - 3;
    const int tile = p >> (hl + 1 + log_c), t = (p >> (hl + 1 + lp)) & 7, b = (p >> lp) & ((2 << hl) - 1), i = p & ((1 << lp) - 1);
    const int rr = (tile << hl) + (b & ((1 << hl) - 1));
    return (((b >> hl) ? R - 1 - rr : rr) << log_c) + 8 * i + t;
}

// ---- balanced partition ----------------------------------------
// A launch of gridDim.x blocks over n_units work units numbered
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

// Walks a block's units (group, item) without a division per unit.
struct SfCursor {
    int grp, item, n_items;
    __device__ __forceinline__ SfCursor(int u, int n) : grp(u / n), item(u % n), n_items(n) {}
    __device__ __forceinline__ void next()
    {
        if (++item == n_items) {
            item = 0;
            ++grp;
        }
    }
};

// runs the statements with constexpr LR, LC, PM for the ring R
#define SF_RING_DISPATCH(R, ...)                              \
    do {                                                      \
        if ((R).pm) {                                         \
            constexpr bool PM = true;                         \
            SF_SIZE_DISPATCH((R).log_n, __VA_ARGS__);         \
        } else {                                              \
            constexpr bool PM = false;                        \
            SF_SIZE_DISPATCH((R).log_n, __VA_ARGS__);         \
        }                                                     \
    } while (0)

// the same for every ring size and either product (kernel attributes)
#define SF_FOR_RINGS(...)                                                          \
    do {                                                                           \
        for (int ln_ = 10; ln_ <= 16; ++ln_) {                                     \
            { constexpr bool PM = true; SF_SIZE_DISPATCH(ln_, __VA_ARGS__); }      \
            { constexpr bool PM = false; SF_SIZE_DISPATCH(ln_, __VA_ARGS__); }     \
        }                                                                          \
    } while (0)

// runs the statements with constexpr LR, LC for the ring size log_n (10..16)
#define SF_SIZE_DISPATCH(log_n, ...)                                  \
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
