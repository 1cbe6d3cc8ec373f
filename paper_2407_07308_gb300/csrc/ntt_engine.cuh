// ntt_engine.cuh -- the NTT engine: negacyclic NTT / inverse NTT over batches of RNS
// limbs, with the key-switching and modulus-switching steps fused into their
// loads and stores.
//
// Transform (BoostCom Sec. 2.2: radix-2 NTT, Cooley-Tukey forward and
// Gentleman-Sande inverse, for power-of-two N):
//   forward  A[k] = a(psi^(2 brv(k) + 1)), natural-order input, bit-reversed
//            output; stage s (s = 0..logN-1) pairs j, j + N/2^(s+1) with the
//            twiddle psi^brv(2^s + (j >> (logN - s)));
//   inverse  the stages undone in reverse order with psi^-brv(.), then N^-1.
//
// GB300 mapping.  N = 2^n is split as 2^n1 x 2^n2 (n1 = ceil(n/2)).  The
// forward transform is two passes: "columns" runs global stages 0..n1-1,
// which only combine residues j = e 2^n2 + lo of one column lo, and "rows"
// runs stages n1..n-1 inside contiguous rows of 2^n2 residues.  Each pass is
// made of sub-transforms of size 2^M (M = n1 or n2) whose twiddles are
// entries of the full table: at local stage u, element e of a sub-transform
// with block index hi uses psi^brv(2^(S+u) + hi 2^u + (e >> (M-u))), S its
// first global stage.  The inverse runs rows first, then columns.  The
// half-transformed limb between the passes lives in the job's output limb.
//
// Units.  Every CTA has 128 threads holding 16 residues each, so a unit of
// work is 2048 residues in shared memory: NS = 2^(11-M) sub-transforms of 2^M
// points.  A sub-transform runs as one radix-16 round (4 stages on strided
// residues) and one round of the remaining M-4 stages (contiguous blocks).
// Column passes read and write global memory straight from the rounds'
// registers, with one exchange in shared memory between them (two where the
// load converts several limbs); row passes exchange twice.  A column unit is
// NC adjacent columns of each of NS/NC jobs (one job, but two at n = 10 and
// where two targets share their sources); a row unit is either one row of each
// of 16 jobs that share a prime times NS/16 adjacent rows (the batched case:
// the CTA stages those rows' twiddles once), or NS adjacent rows of one job
// (small batches; twiddles read through the cache).
// Global memory is read and written in coalesced runs of at least 64 bytes
// (32 in paired column units at N = 2^15).
//
// What bounds the passes: the multiplier pipe before all else (72 to 87% of
// its slots in the row passes and in columns of one word; the columns that
// convert several limbs are at 62 to 65% and wait on loads and barriers
// besides).  Register-resident probes: a 32-bit multiply-add takes one slot of
// it, a 32 x 32 -> 64 or high product two, and a 64-bit accumulation puts one
// of its two additions there, so a butterfly's chained product takes about 15
// slots; the other pipes and the shared memory run beside it as long as they
// stay well below their peaks.
// Measured on the comparison of 16 pairs (N = 2^14, 10 + 3 primes, one
// replay) and on 7 pairs at N = 2^15 (p = 257, 3 digits, level 17): 12.0 and
// 59.8 ms with conversions in 128-bit arithmetic, normalised inverse
// butterflies and three conflicting exchanges a pass; 12.1 and 57.6 ms with
// the arithmetic below alone; 11.2 and 50.0 ms with the layouts too; 9.7 and
// 41.1 ms with joined segments and sums of two products a statement.
//
// Segments and persistence.  A launch carries a table of up to FHE_SEGS
// segments; a segment is the limb jobs of one or more batches of a context and
// level, with their ring degree, twiddle and constant tables.  One launch can
// therefore serve ciphertexts of different level and origin: the units of all
// segments are numbered in order and every CTA walks them with a grid stride
// (segments of different ring degree: one launch each).
// The grid is either one CTA per unit or a fixed number of resident CTAs per
// SM (the autotuner's choice per context).  Launches of a few units per SM run
// both passes in one kernel, a cluster of CTAs per limb (k_fwd_small).
//
// Load/store functors let one kernel body serve the plain transform and the
// fused variants: ModUp (basis conversion of a key-switching digit computed
// while loading, then NTT), ModDown and modulus switching (correction
// computed while loading, subtract-and-scale applied while storing).
// Butterflies are Harvey's lazy ones (values below (4s+7)q after s forward
// stages, below 4q 2^s inverse) with Shoup twiddles.
//
// The kernels and functors are templates instantiated by ntt.cu (limb maps,
// the plain and scaled transforms, the autotuner), ntt_ks.cu (key switching:
// ModUp, ModDown, relinearise + switch) and ntt_ms.cu (modulus switching),
// which compile in parallel.
#pragma once
#include <string.h>

#include <algorithm>

#include "fhe_internal.h"

namespace {

// The butterflies' twiddle product: shoup_lazy4_chain.
// Measured on the GB300 (16-pair comparison at N = 2^14, identical results):
// the C form 2454 slot-comparisons/s, the chain with its quotient's two high
// products summed by an add-with-carry 2563, by a wide multiply-add 2606
// (register-resident forward butterflies: 1015 -> 1173 G/s for the first
// chain).  Also measured and not kept: X + t by multiply-adds as well (2606,
// no gain on its own: 2570), and the inverse's 4q reduction as an unsigned
// minimum (2554).
FHE_HD u64 bfly_mul(u64 a, const ulonglong2 w, u64 q)
{
    return shoup_lazy4_chain(a, w.x, w.y, 0 - q);
}

// Forward butterfly without normalisation: t = [Y w] in [0, 4q) for any
// 64-bit Y (bfly_mul), so if X, Y < B then X + t and X - t + 4q lie in
// [0, B + 4q).  Inputs below 7q (canonical residues, or the lazy results of
// the fused conversions) stay below (4s + 7) q <= 67 q < 2^64 after s <= 15
// stages for primes below 2^57; one reduction at the end brings every value
// to [0, q).  q4 = 4q.
FHE_HD void ct_bfly(u64 &X, u64 &Y, const ulonglong2 w, u64 q, u64 q4)
{
    const u64 t = bfly_mul(Y, w, q);
    const u64 x = X;
    X = x + t;
    Y = x - t + q4;
}

// Inverse butterfly without normalisation: for X, Y < B, B a multiple of q,
// X + Y < 2B and [(X - Y + B) w] in [0, 4q) (bfly_mul takes any 64-bit
// operand, and X - Y + B < 2B).  Sums double from stage to stage, so the
// stages' bounds are 4q 2^j; reduce_few brings the sums back at the end of a
// row pass (and, for primes above 54 bits, between its two rounds), where a
// compare and subtract in every butterfly took 5 of its 22 instructions.
FHE_HD void gs_bfly(u64 &X, u64 &Y, const ulonglong2 w, u64 q, u64 B)
{
    const u64 d = X - Y + B;
    X = X + Y;
    Y = bfly_mul(d, w, q);
}

// Stages s0 .. s0+R-1 of the forward transform on one group x[0..2^R) whose
// block index is hi.
template <int R, class TW>
FHE_HD void fwd_round(u64 (&x)[1 << R], int s0, int hi, const TW &W, u64 q, u64 q4)
{
#pragma unroll
    for (int u = 0; u < R; u++) {
        const int half = 1 << (R - 1 - u);
#pragma unroll
        for (int t = 0; t < (1 << u); t++) {
            const ulonglong2 w = W.get(s0 + u, (hi << u) + t);
#pragma unroll
            for (int k = 0; k < half; k++) {
                const int e = t * 2 * half + k;
                ct_bfly(x[e], x[e + half], w, q, q4);
            }
        }
    }
}

// One stage of the inverse on x[0..2^R): local stage U, butterflies of
// half-distance 2^(R-1-U).  A template per stage keeps every index a
// compile-time constant, so x stays in registers.
template <int R, int U, class TW>
FHE_HD void inv_stage(u64 (&x)[1 << R], int s0, int hi, const TW &W, u64 q, u64 B)
{
    constexpr int half = 1 << (R - 1 - U);
#pragma unroll
    for (int t = 0; t < (1 << U); t++) {
        const ulonglong2 w = W.get(s0 + U, (hi << U) + t);
#pragma unroll
        for (int k = 0; k < half; k++) gs_bfly(x[t * 2 * half + k], x[t * 2 * half + k + half], w, q, B);
    }
    if constexpr (U > 0) inv_stage<R, U - 1>(x, s0, hi, W, q, 2 * B);
}

// Inputs below B; outputs below 2^R B, the upper half of x below 4q.
template <int R, class TW>
FHE_HD void inv_round(u64 (&x)[1 << R], int s0, int hi, const TW &W, u64 q, u64 B)
{
    inv_stage<R, R - 1>(x, s0, hi, W, q, B);
}

// ---------------------------------------------------------------------------
// unit geometry
// ---------------------------------------------------------------------------

constexpr int T = 128;  // threads per CTA, 16 residues each

// Register cap: FHE_NTT_MINB resident CTAs of 128 threads per SM (8: 64
// registers a thread).  Measured as above (16 pairs at N = 2^14 / 7 pairs at
// 2^15): 9 CTAs 11.6 / 53.1 ms (spills), 8 CTAs 11.2 / 50.7, 7 CTAs 11.25 /
// 49.9; 8 with the paired column kernels at 7 11.2 / 50.0.
#ifndef FHE_NTT_MINB
#define FHE_NTT_MINB 8
#endif
// The same for the column kernels of paired units (two targets per load).
#ifndef FHE_NTT_MINB_PAIRED
#define FHE_NTT_MINB_PAIRED 7
#endif
// The maps and layouts below also run on the host (selftest.cu).  Their inlining
// is left to the compiler: forced, it cost the fused row kernels 16 bytes of
// spills at N = 2^14 and 2^15.
// Shared-memory twiddle tables: entry k at k + k / 8 (one 16-byte pad per 8
// entries), so that the second round's strided twiddle reads (stride up to 8
// entries across threads) hit distinct banks.
__host__ __device__ constexpr int twp(int k) { return k + (k >> 3); }
__host__ __device__ constexpr int twp_size(int n) { return n + n / 8 + 1; }

// Sub-transforms of 2^M points, 16 residues a thread.
template <int M>
struct Sub {
    static constexpr int SZ = 1 << M;  // elements per sub-transform
    static constexpr int G = SZ / 16;  // threads per sub-transform
    static constexpr int NS = T / G;   // sub-transforms per unit
    static constexpr int R2 = M - 4;   // stages of the second round
    static_assert(M >= 5 && M <= 8, "sub-transform size");
    static_assert(NS * SZ == 16 * T, "16 residues a thread");
};

// Shared-memory layouts of a unit: element e of sub-transform c at
// c P + slot(c) + e + (e >> 4), in u64 words.  A 64-bit access is served
// conflict-free when the 16 lanes of a half-warp hit 16 distinct words mod
// 16.  Column passes put neighbouring sub-transforms in neighbouring lanes
// (c = t % NS): 16 columns of one element want P odd; 8 columns x 2 elements
// (M = 8) P = 2 mod 16; paired units also store 8 columns x 2 (M = 7: P = 2,
// the second job's columns one word further) or 4 columns x 4 elements (M =
// 8: P = 4, two words further).  Row passes put a sub-transform's own threads
// side by side (c = t / G), so that their global reads are runs of G words:
// P = G mod 16 spreads 16 / G sub-transforms x G words.  (Before, one layout
// with P odd served all of them, with two-way conflicts in the second round
// and three exchanges a pass instead of one or two; ncu: L1 at 59-68% of its
// peak in the column and row passes.)
constexpr int at_least_mod16(int n, int r) { return n + ((r - n) % 16 + 16) % 16; }

template <int M, bool PAIRED>
struct ColLay {
    using C = Sub<M>;
    static constexpr int BASE = C::SZ + C::SZ / 16;
    static constexpr int P = M == 8 ? at_least_mod16(BASE, PAIRED ? 4 : 2)
                             : M == 7 && PAIRED ? at_least_mod16(BASE, 2) : at_least_mod16(BASE, 1 + 2 * (BASE % 16 / 2));
    static constexpr int SLOT = !PAIRED ? 0 : M == 8 ? 2 : M == 7 ? 1 : 0;  // the second job's shift
    static constexpr int WORDS = C::NS * P + SLOT;
    __host__ __device__ static int base(int c) { return c * P + (SLOT && c >= C::NS / 2 ? SLOT : 0); }
    __host__ __device__ static int at(int c, int e) { return base(c) + e + (e >> 4); }
};

template <int M>
struct RowLay {
    using C = Sub<M>;
    static constexpr int P = at_least_mod16(C::SZ + C::SZ / 16, C::G % 16);
    static constexpr int WORDS = C::NS * P;
    __host__ __device__ static int base(int c) { return c * P; }
    __host__ __device__ static int at(int c, int e) { return c * P + e + (e >> 4); }
};

// staged twiddles (ulonglong2) of a row unit: one table of up to 255 entries,
// or two of 127
constexpr int TW_ROWS = twp_size(255) > 2 * twp_size(127) ? twp_size(255) : 2 * twp_size(127);
constexpr int ROW_J = 16;                    // jobs per grouped row unit

// Twiddle accessors: get(s, j) = psi^brv(2^s + j), the twiddle of global
// stage s with in-stage index j < 2^s.
struct GTw {  // the full table in global memory, read-only path
    const ulonglong2 *__restrict__ p;
    __host__ __device__ ulonglong2 get(int s, int j) const
    {
#ifdef __CUDA_ARCH__
        return __ldg(p + (1 << s) + j);
#else
        return p[(1 << s) + j];
#endif
    }
};

struct PrefixTw {  // the first entries of the table, copied to shared memory
    const ulonglong2 *sm;
    __host__ __device__ ulonglong2 get(int s, int j) const { return sm[twp((1 << s) + j)]; }
};

// Row twiddles of one row hi (stages N1.., in-stage index hi 2^u + t) staged
// at offset 2^u - 1 + t.
struct RowTw {
    const ulonglong2 *sm;
    int N1, hi;
    __host__ __device__ ulonglong2 get(int s, int j) const
    {
        const int u = s - N1;
        return sm[twp((1 << u) - 1 + j - (hi << u))];
    }
};

// The two rounds of a sub-transform c on a thread's 16 residues.  First
// round (local stages 0..3): thread g of G holds elements e = k G + g, k < 16.
// Second round (stages 4..M-1): thread g' holds e = 16 g' .. 16 g' + 15, as
// 16 / G blocks of G.  geo gives each sub-transform's twiddle accessor, block
// index and prime.
//
// Inverse (second round first): inputs below 4q.  With primes of at most
// INV_WIDE_BITS bits the values of the other round start below 4q 2^(M-4) and
// end below 4q 2^M <= 2^64; for larger primes reduce_few brings them below 2q
// first.
constexpr int INV_WIDE_BITS = 54;

template <int M, bool FWD, class Geo>
FHE_HD void round1(u64 (&x)[16], const Geo &geo, int c)
{
    const auto W = geo.tw(c);
    const u64 q = geo.q(c), q4 = 4 * q;  // lazy bound of the butterflies
    if constexpr (FWD) {
        fwd_round<4>(x, geo.S, geo.hi(c), W, q, q4);
    } else {
        const ModQ &m = geo.mq(c);
        u64 B = q4 << Sub<M>::R2;
        if (m.bshift > INV_WIDE_BITS - 2) {
#pragma unroll
            for (int k = 0; k < 16; k++) x[k] = reduce_few(x[k], m);
            B = q4;
        }
        inv_round<4>(x, geo.S, geo.hi(c), W, q, B);
    }
}

template <int M, bool FWD, class Geo>
FHE_HD void round2(u64 (&x)[16], const Geo &geo, int c, int gp)
{
    constexpr int G = Sub<M>::G, R2 = Sub<M>::R2, NB = 16 / G;
    const auto W = geo.tw(c);
    const u64 q = geo.q(c), q4 = 4 * q;
#pragma unroll
    for (int i = 0; i < NB; i++) {
        u64 y[G];
#pragma unroll
        for (int f = 0; f < G; f++) y[f] = x[i * G + f];
        if constexpr (FWD)
            fwd_round<R2>(y, geo.S + 4, geo.hi(c) * 16 + gp * NB + i, W, q, q4);
        else
            inv_round<R2>(y, geo.S + 4, geo.hi(c) * 16 + gp * NB + i, W, q, q4);
#pragma unroll
        for (int f = 0; f < G; f++) x[i * G + f] = y[f];
    }
}

// A thread's residues in shared memory: at the first round's elements (base
// b + g, elements k G apart) or the second's (base b + 17 g', contiguous).
template <int G>
FHE_HD void put1(u64 *b, const u64 (&x)[16])
{
#pragma unroll
    for (int k = 0; k < 16; k++) b[k * G + ((k * G) >> 4)] = x[k];
}
template <int G>
FHE_HD void get1(const u64 *b, u64 (&x)[16])
{
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = b[k * G + ((k * G) >> 4)];
}
FHE_HD void put2(u64 *b, const u64 (&x)[16])
{
#pragma unroll
    for (int k = 0; k < 16; k++) b[k] = x[k];
}
FHE_HD void get2(const u64 *b, u64 (&x)[16])
{
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = b[k];
}

// Column pass of ring degree 2^(N1+N2): NC adjacent columns of NJ jobs.
// XJ = 2 asks for two jobs per unit where one would hold all NS columns
// (half as many columns each): functors whose loads convert several source
// limbs pair jobs that read the same sources (fwd_cols_unit).  At N = 2^15 a
// paired unit holds 4 columns (32-byte runs, one sector each) and a larger
// twiddle table.
__host__ __device__ constexpr bool col_paired(int xj, int ns, int nc1) { return xj == 2 && nc1 == ns; }

template <int N1, int N2, int XJ = 1>
struct ColGeo {
    using C = Sub<N1>;
    static constexpr int NS = C::NS, SZ = C::SZ, NN = 1 << (N1 + N2);
    static constexpr int NC1 = NS < (1 << N2) ? NS : (1 << N2);
    static constexpr bool PAIRED = col_paired(XJ, NS, NC1);
    using Lay = ColLay<N1, PAIRED>;
    static constexpr int NC = PAIRED ? NC1 / 2 : NC1;                  // columns per job
    static constexpr int NJ = NS / NC;                                 // jobs per unit
    static constexpr int BLK = (1 << N2) / NC;                         // column blocks per job
    static constexpr int TWC = twp_size(1 << N1);                      // staged twiddles per job
    static constexpr int TW = NJ * TWC;
    static_assert(NJ <= 2, "jobs per column unit");
    // a unit's first job and its first column
    __host__ __device__ static int job0(int lu) { return lu / BLK * NJ; }
    __host__ __device__ static int lo0(int lu) { return lu % BLK * NC; }
};

template <int N1, int N2, int XJ = 1>
struct ColTw {
    using Gm = ColGeo<N1, N2, XJ>;
    const ulonglong2 *W;
    u64 q0, q1;
    const ModQ *m0, *m1;
    static constexpr int S = 0;
    __host__ __device__ PrefixTw tw(int c) const { return PrefixTw{W + (c / Gm::NC) * Gm::TWC}; }
    __host__ __device__ int hi(int) const { return 0; }
    __host__ __device__ u64 q(int c) const { return c / Gm::NC == 0 ? q0 : q1; }
    __host__ __device__ const ModQ &mq(int c) const { return c / Gm::NC == 0 ? *m0 : *m1; }
};

// Row pass: grouped (16 jobs of one prime x R adjacent rows) or single (NS
// adjacent rows of one job).
template <int N1, int N2>
struct RowGeo {
    using C = Sub<N2>;
    static constexpr int NS = C::NS, SZ = C::SZ, NN = 1 << (N1 + N2);
    using Lay = RowLay<N2>;
    static constexpr int R = NS / ROW_J;         // rows per grouped unit
    static constexpr int CH = (1 << N1) / R;     // row chunks per limb (grouped)
    // row chunks per limb (single; a limb with fewer than NS rows, n = 10,
    // always takes the grouped form)
    static constexpr int CHS = (1 << N1) >= NS ? (1 << N1) / NS : 1;
    static constexpr int TWR = twp_size(SZ - 1); // staged twiddles per row
    static_assert(NS >= ROW_J && NS % ROW_J == 0, "row units");
    static_assert(R * TWR <= TW_ROWS, "twiddle staging");
};

template <int N1, int N2>
struct RowGrpTw {
    const ulonglong2 *W;
    int hi0;
    const ModQ &m;
    int S;
    __host__ __device__ RowTw tw(int c) const
    {
        constexpr int R = RowGeo<N1, N2>::R;
        return RowTw{W + (c % R) * RowGeo<N1, N2>::TWR, N1, hi0 + c % R};
    }
    __host__ __device__ int hi(int c) const { return hi0 + c % RowGeo<N1, N2>::R; }
    __host__ __device__ u64 q(int) const { return m.q; }
    __host__ __device__ const ModQ &mq(int) const { return m; }
};

struct RowOneTw {
    GTw g;
    int hi0;
    const ModQ &m;
    int S;
    __host__ __device__ GTw tw(int) const { return g; }
    __host__ __device__ int hi(int c) const { return hi0 + c; }
    __host__ __device__ u64 q(int) const { return m.q; }
    __host__ __device__ const ModQ &mq(int) const { return m; }
};

// ---------------------------------------------------------------------------
// segment tables
// ---------------------------------------------------------------------------

// Per segment: jobs = outer * nl, job = o * nl + l, and the prime of a job
// depends on l only (so the jobs l, nl + l, 2 nl + l ... can share a CTA).  A
// segment joins the batches of one context, level and count (the products of
// a wave): outer item o belongs to payload first + o / per, as its item o %
// per, so that small batches fill the grouped row units together.  Row units
// of 16 jobs serve the first gouter outer items, units of one job the rest.
struct SegHdr {
    int logN, outer, nl, gouter;
    int u_cols, u_rows, xj, g_units;  // xj: the functor's XJ (0 read as 1); g_units: grouped row units
    int first, per;
    const ModQ *mq;
    const ulonglong2 *tw;    // forward or inverse table of the segment's context
    const ulonglong2 *ninv;  // N^-1 per prime (Shoup pairs)
};

constexpr int DIR_FWD = 1, DIR_INV = 2;

template <class S>
struct SegIO {
    using Payload = S;
    int nseg, ucols, urows, pad;  // segments (headers); payloads may be more
    SegHdr h[FHE_SEGS];
    S s[FHE_SEGS];
    // the payload of a job, with the job's place in it
    __host__ __device__ const S &payload(int sg, int &job) const
    {
        const SegHdr &H = h[sg];
        const int k = H.outer == H.per ? 0 : job / (H.nl * H.per);
        job -= k * H.nl * H.per;
        return s[H.first + k];
    }
    // jobs per column unit asked for (2: functors whose loads convert, with same_src)
    static constexpr int XJ = 1;
    static constexpr bool PLAIN = false;
    static constexpr int DIRS = DIR_FWD;  // the directions a functor serves
};

template <class IO>
__device__ __forceinline__ int seg_of(const IO &io, int u, bool rows)
{
    int sg = 0;
    while (sg + 1 < io.nseg && (rows ? io.h[sg + 1].u_rows : io.h[sg + 1].u_cols) <= u) sg++;
    return sg;
}

// ---------------------------------------------------------------------------
// conversions computed by the loads of a forward transform (ModUp, ModDown,
// the switch corrections): sum_a t_a c_a mod r over n source limbs
// ---------------------------------------------------------------------------

// n source limbs one after the other from src, the target's constants, the
// target limb and its prime
struct Conv {
    const u64 *src;
    u64 *dst;
    int n, prime;
    DotC c[FHE_MAXK];
};

// positions converted together by a thread of a paired unit
#ifndef FHE_NTT_CONV_P
#define FHE_NTT_CONV_P 2
#endif
constexpr int CONV_P = FHE_NTT_CONV_P;

// Two targets of the same sources at P positions n, n + STEP, ..: each source
// word is loaded once and split into half words once; four wide
// multiply-adds per source and target, one 32-bit Montgomery step per target
// (DotAcc).  Results in [q, 7q): the forward butterflies take any input whose
// lazy bound stays below 2^64 ((4 s + 7) q after s stages), and the
// transform's last step reduces.  With 128-bit multiply-adds and a Barrett
// reduction a converted residue took 112 instructions for 3 sources (ncu,
// ModUp at N = 2^14), here about 30.
template <int P, int STEP, int NN>
__device__ __forceinline__ void conv_pair(const Conv &a, const Conv &b, const ModQ &ma, const ModQ &mb, int n,
                                          u64 (&v0)[P], u64 (&v1)[P])
{
    DotAcc s0[P], s1[P];
#pragma unroll
    for (int p = 0; p < P; p++) {
        s0[p] = DotAcc{0, (int64_t)(2 * ma.q2)};
        s1[p] = DotAcc{0, (int64_t)(2 * mb.q2)};
    }
    const int h = ma.half, ns = a.n;
    const u64 *src = a.src + n;
#pragma unroll 1
    for (int i0 = 0; i0 < ns; i0 += 4) {
        u64 x[4][P];  // up to four sources' words in flight
#pragma unroll
        for (int i = 0; i < 4; i++)
            if (i0 + i < ns) {
#pragma unroll
                for (int p = 0; p < P; p++) x[i][p] = src[(size_t)i * NN + p * STEP];
            }
#pragma unroll
        for (int i = 0; i < 4; i++)
            if (i0 + i < ns) {
                const DotC c0 = a.c[i0 + i], c1 = b.c[i0 + i];
#pragma unroll
                for (int p = 0; p < P; p++) {
                    const uint32_t xl = (uint32_t)x[i][p] & (((uint32_t)1 << h) - 1), xh = (uint32_t)(x[i][p] >> h);
                    dot_mac(s0[p], xl, xh, c0);
                    dot_mac(s1[p], xl, xh, c1);
                }
                if (h > 27 && (i & 1)) {  // primes above 54 bits: two sources a sum
#pragma unroll
                    for (int p = 0; p < P; p++) {
                        s0[p] = DotAcc{0, dot_fold(s0[p], ma)};
                        s1[p] = DotAcc{0, dot_fold(s1[p], mb)};
                    }
                }
            }
        src += (size_t)4 * NN;
    }
#pragma unroll
    for (int p = 0; p < P; p++) {
        v0[p] = (u64)dot_fold(s0[p], ma);
        v1[p] = (u64)dot_fold(s1[p], mb);
    }
}

// One target at position n.
template <int NN>
__device__ __forceinline__ u64 conv_one(const Conv &a, const ModQ &m, int n)
{
    DotAcc s{0, (int64_t)(2 * m.q2)};
    const u64 *src = a.src + n;
#pragma unroll 1
    for (int i0 = 0; i0 < a.n; i0 += 4) {
        u64 x[4];
#pragma unroll
        for (int i = 0; i < 4; i++) x[i] = i0 + i < a.n ? src[(size_t)i * NN] : 0;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            if (i0 + i < a.n) dot_mac(s, x[i], a.c[i0 + i], m.half);
            if (m.half > 27 && (i & 1)) s = DotAcc{0, dot_fold(s, m)};
        }
        src += (size_t)4 * NN;
    }
    return (u64)dot_fold(s, m);
}

// One target at P positions n, n + STEP, ..
template <int P, int STEP, int NN>
__device__ __forceinline__ void conv_single(const Conv &a, const ModQ &m, int n, u64 *v)
{
    DotAcc s[P];
#pragma unroll
    for (int p = 0; p < P; p++) s[p] = DotAcc{0, (int64_t)(2 * m.q2)};
    const int ns = a.n;
    const u64 *src = a.src + n;
#pragma unroll 1
    for (int i0 = 0; i0 < ns; i0 += 4) {
        u64 x[4][P];
#pragma unroll
        for (int i = 0; i < 4; i++)
            if (i0 + i < ns) {
#pragma unroll
                for (int p = 0; p < P; p++) x[i][p] = src[(size_t)i * NN + p * STEP];
            }
#pragma unroll
        for (int i = 0; i < 4; i++)
            if (i0 + i < ns) {
                const DotC c = a.c[i0 + i];
#pragma unroll
                for (int p = 0; p < P; p++) {
                    dot_mac(s[p], x[i][p], c, m.half);
                    if (m.half > 27 && (i & 1)) s[p] = DotAcc{0, dot_fold(s[p], m)};
                }
            }
        src += (size_t)4 * NN;
    }
#pragma unroll
    for (int p = 0; p < P; p++) v[p] = (u64)dot_fold(s[p], m);
}

// ---------------------------------------------------------------------------
// kernels' stores: out = x A + d B mod q with constants, d = y - v for the
// transform's lazy value v (below 71 q), x and y below 2q
// ---------------------------------------------------------------------------

// y + 2q - v (mod q) for y below 2q, in (0, 4q); canonical for primes above 56 bits, whose
// half words leave no room for the multiple (DotAcc)
__device__ __forceinline__ u64 lazy_diff(u64 y, u64 v, const ModQ &m)
{
    u64 d = y + m.q2 - reduce_few(v, m);
    if (m.half > 28) d = reduce4q(d, m.q2, m.q);
    return d;
}

// d B, canonical
__device__ __forceinline__ u64 scaled1(u64 d, const DotC &B, const ModQ &m)
{
    DotAcc s{0, 0};
    dot_mac(s, d, B, m.half);
    return centred_mod(dot_fold(s, m), m.q);
}

// x A + d B, canonical
__device__ __forceinline__ u64 scaled2(u64 x, const DotC &A, u64 d, const DotC &B, const ModQ &m)
{
    DotAcc s{0, 0};
    dot_mac(s, x, A, m.half);
    dot_mac(s, d, B, m.half);
    return centred_mod(dot_fold(s, m), m.q);
}

// ---------------------------------------------------------------------------
// the unit bodies
// ---------------------------------------------------------------------------

// Asynchronous copies global -> shared memory (16 and 8 bytes): tiles and
// twiddle tables go there without passing through registers, all of a
// thread's copies in flight at once; async_wait before the barrier that
// publishes them.
__device__ __forceinline__ void async16(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Stores of a forward row pass: word r goes to index idx(r) of state st(r)
// with value val(r) (the transform's lazy value, below 71 q) when ok(r).
// Staged: the operands the store reads (IO::NPRE per word) are loaded for a
// chunk of words before any of the chunk's writes, so those loads overlap.
template <class IO, class StF, class Ok, class Idx, class Val>
__device__ __forceinline__ void tile_out(const IO &io, const typename IO::RowK &rk, const ModQ &m, int tid, StF st,
                                         Ok ok, Idx idx, Val val)
{
    constexpr int IT = 16;
    if constexpr (IO::NPRE > 0) {
        constexpr int CH = IT / 2;
#pragma unroll
        for (int k0 = 0; k0 < IT; k0 += CH) {
            u64 a[CH][IO::NPRE];
#pragma unroll
            for (int k = 0; k < CH; k++) {
                const int r = tid + (k0 + k) * T;
#pragma unroll
                for (int w = 0; w < IO::NPRE; w++) a[k][w] = ok(r) ? io.pre(st(r), idx(r), w) : 0;
            }
#pragma unroll
            for (int k = 0; k < CH; k++) {
                const int r = tid + (k0 + k) * T;
                if (ok(r)) io.store_pre(rk, m, st(r), idx(r), val(r), a[k]);
            }
        }
    } else {
#pragma unroll 4
        for (int k = 0; k < IT; k++) {
            const int r = tid + k * T;
            if (ok(r)) io.store_pre(rk, m, st(r), idx(r), val(r), nullptr);
        }
    }
}

// The jobs of a column unit: slot j (j < NJ) holds job0 + j.
template <int N1, int N2, class IO>
__device__ __forceinline__ int col_jobs(const IO &io, int sg, int lu, typename IO::CSt *sts, int *lo0)
{
    using Gm = ColGeo<N1, N2, IO::XJ>;
    const SegHdr &H = io.h[sg];
    const int njobs = H.outer * H.nl;
    const int job0 = Gm::job0(lu);
    *lo0 = Gm::lo0(lu);
    if (threadIdx.x < Gm::NJ && job0 + (int)threadIdx.x < njobs) io.begin_c(sg, job0 + threadIdx.x, sts[threadIdx.x]);
    __syncthreads();
    return njobs - job0;  // valid job slots (>= 1)
}

// Stages the first 2^N1 twiddles of a job's prime (the column stages).
template <int N1>
__device__ __forceinline__ void col_twiddles(ulonglong2 *W, const ulonglong2 *tw)
{
#pragma unroll
    for (int i = threadIdx.x; i < (1 << N1); i += T) async16(W + twp(i), tw + i);
}

struct PdlWait {
    __device__ void operator()() const { pdl_wait(); }
};

// Column units of one job.  Thread (c, g) reads and writes column lo0 + c in
// global memory straight from its rounds' registers (neighbouring lanes,
// neighbouring columns); shared memory carries the one exchange between the
// rounds.
template <int N1, int N2, class IO>
__device__ __forceinline__ void fwd_cols_unit1(const IO &io, int sg, int lu, u64 *sm, ulonglong2 *W,
                                               const typename IO::CSt &st)
{
    using Gm = ColGeo<N1, N2, 1>;
    using C = typename Gm::C;
    const int c = threadIdx.x % C::NS, g = threadIdx.x / C::NS;
    const SegHdr &H = io.h[sg];
    const int lo = Gm::lo0(lu) + c;
    col_twiddles<N1>(W, H.tw + (size_t)st.prime * Gm::NN);
    const ModQ &m = H.mq[st.prime];
    const ColTw<N1, N2, 1> geo{W, m.q, m.q, &m, &m};
    pdl_wait();
    u64 x[16];
    if constexpr (IO::XJ == 2) {
#pragma unroll
        for (int k = 0; k < 16; k += 4)
            conv_single<4, (C::G << N2), Gm::NN>(st.cv, m, ((k * C::G + g) << N2) + lo, x + k);
    } else {
        const u64 *src = io.src(st) + (g << N2) + lo;
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = src[(k * C::G) << N2];
        if constexpr (!IO::PLAIN) {
#pragma unroll
            for (int k = 0; k < 16; k++) x[k] = io.conv(st, x[k]);
        }
    }
    async_wait();
    __syncthreads();  // the twiddles
    round1<N1, true>(x, geo, c);
    u64 *b = sm + Gm::Lay::base(c);
    put1<C::G>(b + g, x);
    __syncthreads();
    get2(b + 17 * g, x);
    round2<N1, true>(x, geo, c, g);
    u64 *mid = io.inter(st) + (g << (N2 + 4)) + lo;
#pragma unroll
    for (int k = 0; k < 16; k++) mid[k << N2] = x[k];
}

// The last product of an inverse transform: a value anywhere in 64 bits times
// N^-1 (and the entry's constant), canonical.
FHE_HD u64 inv_scaled(u64 v, const ulonglong2 ni, const ModQ &m)
{
    return reduce4q(shoup_lazy4_chain(v, ni.x, ni.y, 0 - m.q), m.q2, m.q);
}

template <int N1, int N2, class IO, class Wait = PdlWait>
__device__ __forceinline__ void inv_cols_unit1(const IO &io, int sg, int lu, u64 *sm, ulonglong2 *W, Wait wait = {})
{
    using Gm = ColGeo<N1, N2, 1>;
    using C = typename Gm::C;
    const int c = threadIdx.x % C::NS, g = threadIdx.x / C::NS;
    const SegHdr &H = io.h[sg];
    const int lo = Gm::lo0(lu) + c;
    typename IO::CSt st;
    io.begin_c(sg, Gm::job0(lu), st);
    col_twiddles<N1>(W, H.tw + (size_t)st.prime * Gm::NN);
    const ModQ &m = H.mq[st.prime];
    const ColTw<N1, N2, 1> geo{W, m.q, m.q, &m, &m};
    wait();
    u64 x[16];
    const u64 *mid = io.inter(st) + (g << (N2 + 4)) + lo;
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = mid[k << N2];
    async_wait();
    __syncthreads();  // the twiddles
    round2<N1, false>(x, geo, c, g);
    u64 *b = sm + Gm::Lay::base(c);
    put2(b + 17 * g, x);
    __syncthreads();
    get1<C::G>(b + g, x);
    round1<N1, false>(x, geo, c);
    const ulonglong2 ni = io.final_scale(st);
#pragma unroll
    for (int k = 0; k < 16; k++) io.store(st, ((k * C::G + g) << N2) + lo, inv_scaled(x[k], ni, m));
}

// Forward, columns: global stages 0..N1-1.
template <int N1, int N2, class IO>
__device__ __forceinline__ void fwd_cols_unit(const IO &io, int sg, int lu, u64 *sm, ulonglong2 *W,
                                              typename IO::CSt *sts)
{
    using Gm = ColGeo<N1, N2, IO::XJ>;
    using C = typename Gm::C;
    if constexpr (Gm::NJ == 1) {
        typename IO::CSt st;  // computed by every thread, in registers
        io.begin_c(sg, Gm::job0(lu), st);
        fwd_cols_unit1<N1, N2>(io, sg, lu, sm, W, st);
        return;
    }
    const int tid = threadIdx.x, c = tid % C::NS, g = tid / C::NS;
    int lo0;
    const int nvalid = col_jobs<N1, N2>(io, sg, lu, sts, &lo0);
    const SegHdr &H = io.h[sg];
    const ModQ &m0 = H.mq[sts[0].prime], &m1 = H.mq[sts[nvalid > 1 ? Gm::NJ - 1 : 0].prime];
    for (int j = 0; j < Gm::NJ && j < nvalid; j++)
        col_twiddles<N1>(W + j * Gm::TWC, H.tw + (size_t)sts[j].prime * Gm::NN);
    pdl_wait();
    bool paired = false;
    if constexpr (Gm::PAIRED) {
        // both slots at once: column col of slot 0 and of slot 1 at the same
        // element, so each source word is loaded once
        static_assert(Gm::NJ == 2 && 2 * Gm::NC * Gm::SZ == 16 * T, "paired column unit");
        paired = nvalid >= 2 && io.same_src(sts[0], sts[1]);  // uniform in the CTA
        if (paired) {
            constexpr int ES = T / Gm::NC;  // elements between a thread's words
            const int col = tid % Gm::NC, e0 = tid / Gm::NC;
#pragma unroll 1
            for (int k = 0; k < 8; k += CONV_P) {
                u64 v0[CONV_P], v1[CONV_P];
                conv_pair<CONV_P, (ES << N2), Gm::NN>(sts[0].cv, sts[1].cv, m0, m1, ((e0 + k * ES) << N2) + lo0 + col,
                                                      v0, v1);
#pragma unroll
                for (int p = 0; p < CONV_P; p++) {
                    sm[Gm::Lay::at(col, e0 + (k + p) * ES)] = v0[p];
                    sm[Gm::Lay::at(Gm::NC + col, e0 + (k + p) * ES)] = v1[p];
                }
            }
        }
    }
    if constexpr (Gm::PAIRED) {
        // a unit whose jobs read different sources, or with one job left (a
        // slot without a job transforms what is there and stores nothing):
        // rolled loops, small code beside the paired path.  (As an else-branch
        // of that path it slowed the paired units: 7 pairs at N = 2^15 39.79
        // -> 39.91 ms, 16 products 2042 -> 2051 us.)
        if (!paired) {
            constexpr int ES = T / Gm::NC;
            const int col = tid % Gm::NC, e0 = tid / Gm::NC;
#pragma unroll 1
            for (int j = 0; j < 2 && j < nvalid; j++)
#pragma unroll 1
                for (int k = 0; k < 8; k++)
                    sm[Gm::Lay::at(j * Gm::NC + col, e0 + k * ES)] =
                        conv_one<Gm::NN>(sts[j].cv, j == 0 ? m0 : m1, ((e0 + k * ES) << N2) + lo0 + col);
        }
    }
    u64 x[16];
    if constexpr (!Gm::PAIRED) {
        // n = 10: thread (c, g) takes its first round's words as in
        // fwd_cols_unit1; a slot without a job transforms the first job's and
        // stores nothing
        const int jv = c / Gm::NC < nvalid ? c / Gm::NC : 0, lo = lo0 + c % Gm::NC;
        const typename IO::CSt &st = sts[jv];
        if constexpr (IO::XJ == 2) {
            // conversions in a rolled loop, by way of the thread's own places
            // in shared memory (unrolled into registers they spilled)
            const ModQ &m = jv == 0 ? m0 : m1;
#pragma unroll 1
            for (int k = 0; k < 16; k += CONV_P) {
                u64 v[CONV_P];
                conv_single<CONV_P, (C::G << N2), Gm::NN>(st.cv, m, ((k * C::G + g) << N2) + lo, v);
#pragma unroll
                for (int p = 0; p < CONV_P; p++) sm[Gm::Lay::at(c, (k + p) * C::G + g)] = v[p];
            }
        } else {
            // all loads in flight (one after the other, a transform of 288
            // plain limbs took 18.5 us among others and 30 alone; 15 and 19)
            const u64 *src = io.src(st) + (g << N2) + lo;
#pragma unroll
            for (int k = 0; k < 16; k++) x[k] = src[(k * C::G) << N2];
            if constexpr (!IO::PLAIN) {
#pragma unroll
                for (int k = 0; k < 16; k++) x[k] = io.conv(st, x[k]);
            }
        }
    }
    async_wait();
    __syncthreads();
    const ColTw<N1, N2, IO::XJ> geo{W, m0.q, m1.q, &m0, &m1};
    u64 *b = sm + Gm::Lay::base(c);
    if constexpr (IO::XJ == 2) get1<C::G>(b + g, x);
    round1<N1, true>(x, geo, c);
    put1<C::G>(b + g, x);
    __syncthreads();
    get2(b + 17 * g, x);
    round2<N1, true>(x, geo, c, g);
    const int j = c / Gm::NC;
    if (j < nvalid) {
        u64 *mid = io.inter(sts[j]) + (g << (N2 + 4)) + lo0 + c % Gm::NC;
#pragma unroll
        for (int k = 0; k < 16; k++) mid[k << N2] = x[k];
    }
}

// Inverse, columns: undoes global stages N1-1..0, then scales (N^-1 times the
// job's constant) and stores.
template <int N1, int N2, class IO>
__device__ __forceinline__ void inv_cols_unit(const IO &io, int sg, int lu, u64 *sm, ulonglong2 *W,
                                              typename IO::CSt *sts)
{
    using Gm = ColGeo<N1, N2, IO::XJ>;
    using C = typename Gm::C;
    if constexpr (Gm::NJ == 1) {
        inv_cols_unit1<N1, N2>(io, sg, lu, sm, W);
        return;
    }
    const int c = threadIdx.x % C::NS, g = threadIdx.x / C::NS;
    int lo0;
    const int nvalid = col_jobs<N1, N2>(io, sg, lu, sts, &lo0);
    const SegHdr &H = io.h[sg];
    const ModQ &m0 = H.mq[sts[0].prime], &m1 = H.mq[sts[nvalid > 1 ? Gm::NJ - 1 : 0].prime];
    for (int j = 0; j < Gm::NJ && j < nvalid; j++)
        col_twiddles<N1>(W + j * Gm::TWC, H.tw + (size_t)sts[j].prime * Gm::NN);
    const ColTw<N1, N2, IO::XJ> geo{W, m0.q, m1.q, &m0, &m1};
    // a slot without a job transforms the first job's words and stores nothing
    const int j = c / Gm::NC, lo = lo0 + c % Gm::NC, jv = j < nvalid ? j : 0;
    pdl_wait();
    u64 x[16];
    const u64 *mid = io.inter(sts[jv]) + (g << (N2 + 4)) + lo;
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = mid[k << N2];
    async_wait();
    __syncthreads();
    round2<N1, false>(x, geo, c, g);
    u64 *b = sm + Gm::Lay::base(c);
    put2(b + 17 * g, x);
    __syncthreads();
    get1<C::G>(b + g, x);
    round1<N1, false>(x, geo, c);
    if (j < nvalid) {
        const ulonglong2 ni = io.final_scale(sts[j]);
        const ModQ &m = j == 0 ? m0 : m1;
#pragma unroll
        for (int k = 0; k < 16; k++) io.store(sts[j], ((k * C::G + g) << N2) + lo, inv_scaled(x[k], ni, m));
    }
}

// The jobs of a row unit: slots jj < nvalid, rows hi0 on.  Grouped: jobs
// (o0 + jj) nl + l, R rows; single: one job, l, NS rows.
template <int N1, int N2, bool GRP>
struct RowUnit {
    using Gm = RowGeo<N1, N2>;
    int hi0, nvalid, o0, l;
    __host__ __device__ RowUnit(const SegHdr &H, int lu)
    {
        if (GRP) {
            const int OC = (H.gouter + ROW_J - 1) / ROW_J;
            const int hc = lu % Gm::CH, t = lu / Gm::CH;
            const int oc = t % OC;
            l = t / OC;
            hi0 = hc * Gm::R;
            o0 = oc * ROW_J;
            nvalid = H.gouter - o0 < ROW_J ? H.gouter - o0 : ROW_J;
        } else {
            const int v = lu - H.g_units;
            hi0 = (v % Gm::CHS) * Gm::NS;
            nvalid = 1;
            o0 = 0;
            l = H.gouter * H.nl + v / Gm::CHS;
        }
    }
    __host__ __device__ int job(const SegHdr &H, int jj) const { return GRP ? (o0 + jj) * H.nl + l : l; }
};

// The same, with the jobs' states begun; returns the number of valid slots.
template <int N1, int N2, bool GRP, class IO>
__device__ __forceinline__ int row_jobs(const IO &io, int sg, int lu, typename IO::RSt *sts, int *hi0)
{
    const RowUnit<N1, N2, GRP> u(io.h[sg], lu);
    *hi0 = u.hi0;
    if ((int)threadIdx.x < u.nvalid) io.begin_r(sg, u.job(io.h[sg], threadIdx.x), sts[threadIdx.x]);
    __syncthreads();
    return u.nvalid;
}

// Grouped rows stage the R rows' twiddles: entry k of row r is the stage
// u = floor(log2(k+1)) twiddle with in-stage index (hi0 + r) 2^u + k+1-2^u.
template <int N1, int N2>
__device__ __forceinline__ void row_twiddles(ulonglong2 *W, const ulonglong2 *tw, int hi0)
{
    using Gm = RowGeo<N1, N2>;
    constexpr int NW = Gm::R * (Gm::SZ - 1);
#pragma unroll
    for (int i = threadIdx.x; i < NW; i += T) {
        const int r = i / (Gm::SZ - 1), e = i % (Gm::SZ - 1);
        const int u = 31 - __clz(e + 1);
        async16(W + r * Gm::TWR + twp(e), tw + (1 << (N1 + u)) + ((hi0 + r) << u) + (e + 1 - (1 << u)));
    }
}

// word r of a row unit -> (sub-transform c = r >> N2, element f); the job
// slot and row of c
template <int N1, int N2, bool GRP>
struct RowMap {
    using Gm = RowGeo<N1, N2>;
    int hi0;
    __host__ __device__ int c(int r) const { return r >> N2; }
    __host__ __device__ int f(int r) const { return r & (Gm::SZ - 1); }
    __host__ __device__ int cslot(int c) const { return GRP ? c / Gm::R : 0; }
    __host__ __device__ int crow(int c) const { return hi0 + (GRP ? c % Gm::R : c); }
    __host__ __device__ int slot(int r) const { return cslot(c(r)); }
    __host__ __device__ int row(int r) const { return crow(c(r)); }
};

// Forward, rows: global stages N1..N1+N2-1, then the functor's store.
template <int N1, int N2, bool GRP, class IO, class Wait = PdlWait>
__device__ __forceinline__ void fwd_rows_unit(const IO &io, int sg, int lu, u64 *sm, ulonglong2 *W,
                                          typename IO::RSt *sts, Wait wait = {})
{
    using Gm = RowGeo<N1, N2>;
    using C = typename Gm::C;
    using Lay = typename Gm::Lay;
    const int tid = threadIdx.x;
    const SegHdr &H = io.h[sg];
    int hi0;
    const int nvalid = row_jobs<N1, N2, GRP>(io, sg, lu, sts, &hi0);
    const RowMap<N1, N2, GRP> mp{hi0};
    const int prime = sts[0].prime;
    const ModQ &m = H.mq[prime];
    const ulonglong2 *tw = H.tw + (size_t)prime * Gm::NN;
    if (GRP) row_twiddles<N1, N2>(W, tw, hi0);
    wait();
    // thread (c, g) reads its first round's words: runs of G words
    const int c = tid / C::G, g = tid % C::G;
    u64 x[16];
    {
        const int j = mp.cslot(c);  // a slot without a job transforms the first job's words and stores nothing
        const u64 *src = io.inter(sts[j < nvalid ? j : 0]) + (mp.crow(c) << N2) + g;
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = src[k * C::G];
    }
    if (GRP) {
        async_wait();
        __syncthreads();  // the twiddles
    }
    u64 *b = sm + Lay::base(c);
    if (GRP) {
        const RowGrpTw<N1, N2> geo{W, hi0, m, N1};
        round1<N2, true>(x, geo, c);
        put1<C::G>(b + g, x);
        __syncthreads();
        get2(b + 17 * g, x);
        round2<N2, true>(x, geo, c, g);
    } else {
        const RowOneTw geo{GTw{tw}, hi0, m, N1};
        round1<N2, true>(x, geo, c);
        put1<C::G>(b + g, x);
        __syncthreads();
        get2(b + 17 * g, x);
        round2<N2, true>(x, geo, c, g);
    }
    put2(b + 17 * g, x);
    __syncthreads();
    const typename IO::RowK rk = io.row_k(sg, prime);
    tile_out(
        io, rk, m, tid, [&](int r) -> const typename IO::RSt & { return sts[mp.slot(r)]; },
        [&](int r) { return mp.slot(r) < nvalid; }, [&](int r) { return (mp.row(r) << N2) + mp.f(r); },
        [&](int r) { return sm[Lay::at(mp.c(r), mp.f(r))]; });
}

// Inverse, rows first: undoes global stages N1+N2-1..N1.
template <int N1, int N2, bool GRP, class IO, class Wait = PdlWait>
__device__ __forceinline__ void inv_rows_unit(const IO &io, int sg, int lu, u64 *sm, ulonglong2 *W,
                                          typename IO::RSt *sts, Wait wait = {})
{
    using Gm = RowGeo<N1, N2>;
    using C = typename Gm::C;
    using Lay = typename Gm::Lay;
    const int tid = threadIdx.x;
    const SegHdr &H = io.h[sg];
    int hi0;
    const int nvalid = row_jobs<N1, N2, GRP>(io, sg, lu, sts, &hi0);
    const RowMap<N1, N2, GRP> mp{hi0};
    const int prime = sts[0].prime;
    const ModQ &m = H.mq[prime];
    const ulonglong2 *tw = H.tw + (size_t)prime * Gm::NN;
    if (GRP) row_twiddles<N1, N2>(W, tw, hi0);
    wait();
    // a unit's jobs are of one map entry and one mask, so either all or none have an addend
    // per polynomial; its words are computed on the way, eight at a time with
    // all loads before the first store (one at a time, each store held the
    // next loads back: 16 pairs at N = 2^14 1.04 -> 0.83 ms of these passes)
    if (io.adds(sts[0]) || io.adds(sts[nvalid > 1 ? 1 : 0])) {
#pragma unroll 1
        for (int k0 = 0; k0 < 16; k0 += 8) {
            u64 v[8], w[8];
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const int r = tid + (k0 + k) * T, j = mp.slot(r), i = (mp.row(r) << N2) + mp.f(r);
                v[k] = j < nvalid ? sts[j].in[i] : 0;
                w[k] = j < nvalid ? io.addend(sts[j], i) : 0;
            }
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const int r = tid + (k0 + k) * T, j = mp.slot(r);
                if (j < nvalid) sm[Lay::at(mp.c(r), mp.f(r))] = io.sum(sts[j], v[k], w[k]);
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < 16; k++) {
            const int r = tid + k * T, j = mp.slot(r);
            if (j < nvalid) async8(&sm[Lay::at(mp.c(r), mp.f(r))], sts[j].in + (mp.row(r) << N2) + mp.f(r));
        }
    }
    async_wait();
    __syncthreads();
    const int c = tid / C::G, g = tid % C::G;
    u64 *b = sm + Lay::base(c);
    u64 x[16];
    get2(b + 17 * g, x);  // a slot without a job transforms what is there and stores nothing
    if (GRP) {
        const RowGrpTw<N1, N2> geo{W, hi0, m, N1};
        round2<N2, false>(x, geo, c, g);
        put2(b + 17 * g, x);
        __syncthreads();
        get1<C::G>(b + g, x);
        round1<N2, false>(x, geo, c);
    } else {
        const RowOneTw geo{GTw{tw}, hi0, m, N1};
        round2<N2, false>(x, geo, c, g);
        put2(b + 17 * g, x);
        __syncthreads();
        get1<C::G>(b + g, x);
        round1<N2, false>(x, geo, c);
    }
    // the sums (below 4q 2^N2) come down to 2q for the column pass
    const int j = mp.cslot(c);
    if (j < nvalid) {
        u64 *mid = io.inter(sts[j]) + (mp.crow(c) << N2) + g;
#pragma unroll
        for (int k = 0; k < 16; k++) mid[k * C::G] = k < 8 ? reduce_few(x[k], m) : x[k];
    }
}

// ---------------------------------------------------------------------------
// kernels: one per (functor, direction, pass, ring degree).  A launch whose
// segments mix ring degrees runs one kernel per degree: a kernel that
// dispatched every unit on its segment's degree halved the launches of an
// uneven batch but spilled and fetched more instructions (32 requests over
// 2^13..2^15: 55.6 ms a pass with it, 50.8 without; 4 requests 5.13 and 4.33).
// The second pass of a transform takes the units from the last to the first:
// what the first pass wrote last is what the L2 still holds of a launch larger
// than it (7 pairs at N = 2^15 40.03 -> 39.82 ms, tournament of 8 ciphertexts
// 153.7 -> 152.9, plain transforms of 152 MB 532 -> 527 us).
// ---------------------------------------------------------------------------

template <int L>
struct Deg {
    static constexpr int N1 = (L + 1) / 2, N2 = L / 2;
};

constexpr int ROW_WORDS = RowLay<7>::WORDS;
static_assert(RowLay<5>::WORDS <= ROW_WORDS && RowLay<6>::WORDS <= ROW_WORDS, "row units");

template <class IO, int L>
__global__ void __launch_bounds__(T, IO::XJ == 2 ? FHE_NTT_MINB_PAIRED : FHE_NTT_MINB)
    k_fwd_cols(const __grid_constant__ IO io)
{
    pdl_trigger();
    __shared__ u64 sm[ColGeo<Deg<L>::N1, Deg<L>::N2, IO::XJ>::Lay::WORDS];
    __shared__ ulonglong2 W[ColGeo<Deg<L>::N1, Deg<L>::N2, IO::XJ>::TW];
    __shared__ typename IO::CSt sts[ColGeo<Deg<L>::N1, Deg<L>::N2, IO::XJ>::NJ];
    for (int u = blockIdx.x; u < io.ucols; u += gridDim.x) {
        const int sg = seg_of(io, u, false), lu = u - io.h[sg].u_cols;
        fwd_cols_unit<Deg<L>::N1, Deg<L>::N2>(io, sg, lu, sm, W, sts);
        __syncthreads();
    }
}

template <class IO, int L>
__global__ void __launch_bounds__(T, FHE_NTT_MINB)
    k_fwd_rows(const __grid_constant__ IO io)
{
    pdl_trigger();
    __shared__ u64 sm[ROW_WORDS];
    __shared__ ulonglong2 W[TW_ROWS];
    __shared__ typename IO::RSt sts[ROW_J];
    for (int v = blockIdx.x; v < io.urows; v += gridDim.x) {
        const int u = io.urows - 1 - v;
        const int sg = seg_of(io, u, true), lu = u - io.h[sg].u_rows;
        if (lu < io.h[sg].g_units)
            fwd_rows_unit<Deg<L>::N1, Deg<L>::N2, true>(io, sg, lu, sm, W, sts);
        else
            fwd_rows_unit<Deg<L>::N1, Deg<L>::N2, false>(io, sg, lu, sm, W, sts);
        __syncthreads();
    }
}

template <class IO, int L>
__global__ void __launch_bounds__(T, FHE_NTT_MINB) k_inv_rows(const __grid_constant__ IO io)
{
    pdl_trigger();
    __shared__ u64 sm[ROW_WORDS];
    __shared__ ulonglong2 W[TW_ROWS];
    __shared__ typename IO::RSt sts[ROW_J];
    for (int u = blockIdx.x; u < io.urows; u += gridDim.x) {
        const int sg = seg_of(io, u, true), lu = u - io.h[sg].u_rows;
        if (lu < io.h[sg].g_units)
            inv_rows_unit<Deg<L>::N1, Deg<L>::N2, true>(io, sg, lu, sm, W, sts);
        else
            inv_rows_unit<Deg<L>::N1, Deg<L>::N2, false>(io, sg, lu, sm, W, sts);
        __syncthreads();
    }
}

template <class IO, int L>
__global__ void __launch_bounds__(T, FHE_NTT_MINB) k_inv_cols(const __grid_constant__ IO io)
{
    pdl_trigger();
    __shared__ u64 sm[ColGeo<Deg<L>::N1, Deg<L>::N2, IO::XJ>::Lay::WORDS];
    __shared__ ulonglong2 W[ColGeo<Deg<L>::N1, Deg<L>::N2, IO::XJ>::TW];
    __shared__ typename IO::CSt sts[ColGeo<Deg<L>::N1, Deg<L>::N2, IO::XJ>::NJ];
    for (int v = blockIdx.x; v < io.ucols; v += gridDim.x) {
        const int u = io.ucols - 1 - v;
        const int sg = seg_of(io, u, false), lu = u - io.h[sg].u_cols;
        inv_cols_unit<Deg<L>::N1, Deg<L>::N2>(io, sg, lu, sm, W, sts);
        __syncthreads();
    }
}

// Both passes of a small launch in one kernel: a cluster of CTAs per job (a
// limb's 1 .. 16 units), a column unit and a single-job row unit of it each,
// with a cluster barrier (release / acquire) where the kernels' boundary would
// be.  Such a launch is bound by latency: the second pass's state and twiddles
// are fetched before the first pass runs (its wait), and a limb's rows start
// when its own columns are done.  Four CTAs per SM, since six (80 registers) ran 5-7%
// slower.  One LT + EQ at N = 2^14, 10 primes: 2078 -> 1718 us; one less-than
// at N = 2^12 499 -> 425; one rotation at N = 2^15 (9 primes) 297 -> 250.
template <int L>
constexpr int SMALL_CTAS = 1 << (L - 11);  // units of a limb: the cluster
constexpr int SMALL_LO = 11, SMALL_HI = 15;

template <int L>
__device__ __forceinline__ void job_barrier()
{
    if constexpr (SMALL_CTAS<L> == 1)
        __syncthreads();
    else
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

template <int L>
struct SmallGeo {
    using Col = ColGeo<Deg<L>::N1, Deg<L>::N2, 1>;
    using Row = RowGeo<Deg<L>::N1, Deg<L>::N2>;
    static_assert(Col::NJ == 1 && Col::BLK == SMALL_CTAS<L> && Row::CHS == SMALL_CTAS<L>, "units of a limb");
    static constexpr int WORDS = Col::Lay::WORDS > ROW_WORDS ? Col::Lay::WORDS : ROW_WORDS;
};

template <class IO, int L>
__global__ void __launch_bounds__(T, 4) k_fwd_small(const __grid_constant__ IO io)
{
    pdl_trigger();
    constexpr int N1 = Deg<L>::N1, N2 = Deg<L>::N2;
    __shared__ u64 sm[SmallGeo<L>::WORDS];
    __shared__ ulonglong2 W[SmallGeo<L>::Col::TW];
    __shared__ typename IO::RSt rst[1];
    __shared__ typename IO::CSt cst[1];
    const int u = blockIdx.x, sg = seg_of(io, u, false), lu = u - io.h[sg].u_cols;
    if (threadIdx.x == 32) io.begin_c(sg, SmallGeo<L>::Col::job0(lu), cst[0]);  // published by row_jobs' barrier
    fwd_rows_unit<N1, N2, false>(io, sg, lu, sm, W, rst, [&] {
        fwd_cols_unit1<N1, N2>(io, sg, lu, sm, W, cst[0]);
        job_barrier<L>();
    });
}

template <class IO, int L>
__global__ void __launch_bounds__(T, 4) k_inv_small(const __grid_constant__ IO io)
{
    pdl_trigger();
    constexpr int N1 = Deg<L>::N1, N2 = Deg<L>::N2;
    __shared__ u64 sm[SmallGeo<L>::WORDS];
    __shared__ ulonglong2 W[SmallGeo<L>::Col::TW];
    __shared__ typename IO::RSt rst[1];
    const int u = blockIdx.x, sg = seg_of(io, u, false), lu = u - io.h[sg].u_cols;
    inv_cols_unit1<N1, N2>(io, sg, lu, sm, W, [&] {
        inv_rows_unit<N1, N2, false>(io, sg, lu, sm, W, rst);
        job_barrier<L>();
    });
}

// ---------------------------------------------------------------------------
// load/store functors (one payload per segment).  A column pass keeps its
// jobs' states as CSt (begin_c), a row pass as RSt (begin_r); RowK holds the
// constants a row unit's stores share (its jobs have one prime and level).
// ---------------------------------------------------------------------------

struct NoRowK {
};

// A limb map: job (o, l) reads limb in_limb[l] of outer item o and writes
// limb out_limb[l]; prime[l]; the inverse's final scale is N^-1 times the
// map entry's constant (scale[l], device) or plain N^-1.
struct MapSeg {
    const u64 *in;
    u64 *out;
    long long in_outer, out_outer;  // u64 elements
    const ulonglong2 *scale;
    uint8_t in_limb[FHE_MAXP], out_limb[FHE_MAXP], prime[FHE_MAXP];
};

// Whether two payloads' jobs l, nl + l, .. share primes and constants, so that
// one segment may hold both.
inline bool joins(const MapSeg &a, const MapSeg &b) { return !memcmp(a.prime, b.prime, sizeof(a.prime)); }
template <class S>
inline bool joins(const S &a, const S &b)
{
    return a.P == b.P;
}

struct MapSt {
    const u64 *in;
    u64 *out;
    int prime;
};

struct MapCSt : MapSt {
    ulonglong2 fs;
};

template <class Io>
__device__ __forceinline__ const typename Io::Payload &map_begin(const Io &io, int sg, int job, MapSt &t, int *o_,
                                                                 int *l_)
{
    const SegHdr &H = io.h[sg];
    const typename Io::Payload &S = io.payload(sg, job);
    const int N = 1 << H.logN, o = job / H.nl, l = job % H.nl;
    t.in = S.in + o * S.in_outer + (long long)S.in_limb[l] * N;
    t.out = S.out + o * S.out_outer + (long long)S.out_limb[l] * N;
    t.prime = S.prime[l];
    *o_ = o;
    *l_ = l;
    return S;
}

struct IOMap : SegIO<MapSeg> {
    static constexpr int DIRS = DIR_FWD | DIR_INV;
    using CSt = MapCSt;
    using RSt = MapSt;
    using RowK = NoRowK;
    __device__ void begin_c(int sg, int job, CSt &t) const
    {
        int o, l;
        const MapSeg &S = map_begin(*this, sg, job, t, &o, &l);
        t.fs = S.scale ? S.scale[l] : h[sg].ninv[t.prime];
    }
    __device__ void begin_r(int sg, int job, RSt &t) const
    {
        int o, l;
        map_begin(*this, sg, job, t, &o, &l);
    }
    __device__ RowK row_k(int, int) const { return {}; }
    static constexpr bool PLAIN = true;  // a column pass loads src's words as they are
    __device__ const u64 *src(const CSt &t) const { return t.in; }
    // the inverse row pass's word: the limb's alone
    __device__ static constexpr bool adds(const RSt &) { return false; }
    __device__ u64 addend(const RSt &, int) const { return 0; }
    __device__ u64 sum(const RSt &, u64 v, u64) const { return v; }
    __device__ void store(const CSt &t, int i, u64 v) const { t.out[i] = v; }
    static constexpr int NPRE = 0;  // operands the store reads
    __device__ u64 pre(const RSt &, int, int) const { return 0; }
    __device__ void store_pre(const RowK &, const ModQ &m, const RSt &t, int i, u64 v, const u64 *) const
    {
        t.out[i] = reduce2q(reduce_few(v, m), m.q);
    }
    __device__ u64 *inter(const MapSt &t) const { return t.out; }
    __device__ ulonglong2 final_scale(const CSt &t) const { return t.fs; }
};

// A scaled inverse whose last map entry (limb l-1 of the relinearisation
// accumulators) loads y = acc + (P mod q) addend: the first step of the
// relinearisation fused with the modulus switch.  Job = (ct, poly) * nl + entry.
struct YSeg : MapSeg {
    const u64 *abase;
    long long a_outer, a_poly;
    int amask, alimb;
    u64 Pm, Pm_s, qm;
};

inline bool joins(const YSeg &a, const YSeg &b)
{
    // a row unit asks its first two jobs whether there are addends
    return joins(static_cast<const MapSeg &>(a), static_cast<const MapSeg &>(b)) && a.Pm == b.Pm && a.qm == b.qm &&
           a.amask == b.amask;
}

struct YRSt : MapSt {
    const u64 *add;
    u64 Pm, Pm_s, qm;
};

struct IOScaledY : SegIO<YSeg> {
    static constexpr int DIRS = DIR_INV;
    using CSt = MapCSt;
    using RSt = YRSt;
    __device__ void begin_c(int sg, int job, CSt &t) const
    {
        int o, e;
        const YSeg &S = map_begin(*this, sg, job, t, &o, &e);
        t.fs = S.scale[e];
    }
    __device__ void begin_r(int sg, int job, RSt &t) const
    {
        int o, e;
        const YSeg &S = map_begin(*this, sg, job, t, &o, &e);
        const int N = 1 << h[sg].logN, pi = o & 1;
        const long long c = o >> 1;
        t.add = (e == h[sg].nl - 1 && ((S.amask >> pi) & 1))
                    ? S.abase + c * S.a_outer + pi * S.a_poly + (long long)S.alimb * N
                    : nullptr;
        t.Pm = S.Pm;
        t.Pm_s = S.Pm_s;
        t.qm = S.qm;
    }
    // the y entry's word: an accumulator below 2q and a product below q
    __device__ static bool adds(const RSt &t) { return t.add != nullptr; }
    __device__ u64 addend(const RSt &t, int i) const { return t.add ? t.add[i] : 0; }
    __device__ u64 sum(const RSt &t, u64 v, u64 w) const { return t.add ? v + shoup(w, t.Pm, t.Pm_s, t.qm) : v; }
    __device__ void store(const CSt &t, int i, u64 v) const { t.out[i] = v; }
    static constexpr int NPRE = 0;
    __device__ u64 *inter(const MapSt &t) const { return t.out; }
    __device__ ulonglong2 final_scale(const CSt &t) const { return t.fs; }
};

struct ConvCSt {
    Conv cv;
    int prime;
};

// a row pass that reads and writes one limb
struct DstRSt {
    u64 *out;
    int prime;
};

// ModUp: extended limb t of digit j of ct c:  y = sum_a t_a (Q_j/q_a) mod r,
// where the source limbs already hold t_a = [x_a (Q_j/q_a)^-1]_{q_a} (the
// inverse NTT that produced them applied that factor).  Job = c * njobs + e
// (entry e: digit, target limb, prime).
struct ModUpSeg {
    const u64 *d2c;  // [count][l][N] coefficient domain
    u64 *ext;        // [count][dnum][l+K][N]
    const ModUpParams *P;
    int l, K, dnum, pad;
};

struct IOModUp : SegIO<ModUpSeg> {
    using CSt = ConvCSt;
    using RSt = DstRSt;
    using RowK = NoRowK;
    __device__ u64 *target(int sg, int job, int *entry) const
    {
        const SegHdr &H = h[sg];
        const ModUpSeg &S = payload(sg, job);
        const int c = job / H.nl, e = job % H.nl;
        *entry = e;
        return S.ext + (((long long)c * S.dnum + S.P->job_digit[e]) * (S.l + S.K) + S.P->job_tgt[e] << H.logN);
    }
    __device__ void begin_c(int sg, int job, CSt &t) const
    {
        int e;
        t.cv.dst = target(sg, job, &e);
        const ModUpSeg &S = payload(sg, job);
        const ModUpParams *P = S.P;
        const int j = P->job_digit[e], tg = P->job_tgt[e];
        t.cv.n = P->digit_n[j];
        t.cv.src = S.d2c + ((long long)(job / h[sg].nl) * S.l + P->digit_lo[j] << h[sg].logN);
        t.prime = t.cv.prime = P->job_prime[e];
#pragma unroll
        for (int a = 0; a < FHE_MAXK; a++)
            if (a < t.cv.n) t.cv.c[a] = P->hat[j][a][tg];
    }
    __device__ void begin_r(int sg, int job, RSt &t) const
    {
        int e;
        t.out = target(sg, job, &e);
        t.prime = s[h[sg].first].P->job_prime[e];
    }
    __device__ RowK row_k(int, int) const { return {}; }
    // two targets of one digit (same sources): each source word loaded once
    static constexpr int XJ = 2;
    __device__ bool same_src(const CSt &a, const CSt &b) const { return a.cv.src == b.cv.src && a.cv.n == b.cv.n; }
    static constexpr int NPRE = 0;
    __device__ u64 pre(const RSt &, int, int) const { return 0; }
    __device__ void store_pre(const RowK &, const ModQ &m, const RSt &t, int k, u64 v, const u64 *) const
    {
        t.out[k] = reduce2q(reduce_few(v, m), m.q);
    }
    __device__ u64 *inter(const CSt &t) const { return t.cv.dst; }
    __device__ u64 *inter(const RSt &t) const { return t.out; }
};

// a row pass whose store combines the transform with an operand or two
struct DownRSt {
    const u64 *x, *add;
    u64 *out;
    int prime;
};

// ModDown of poly pi of ct c, data limb i:
//   delta_i = sum_k t_k * (p P/p_k mod q_i),  out_i = (acc_i - delta_i) P^-1 + addend_i,
// where the special limbs already hold t_k = [acc_{P,k} p^-1 (P/p_k)^-1]_{p_k}
// (applied by the inverse NTT that produced them).  Job = (c, pi) * l + i.
struct ModDownSeg {
    const u64 *accP;  // [count][2][K][N] coefficient domain
    const u64 *acc;   // [count][2][l+K][N] NTT domain
    const u64 *abase;
    long long a_outer, a_poly;
    u64 *out;         // [count][2][l][N]
    const ModDownParams *P;
    int l, K, amask, pad;
};

struct IOModDown : SegIO<ModDownSeg> {
    using CSt = ConvCSt;
    using RSt = DownRSt;
    struct RowK {
        DotC pinv;
    };
    __device__ void begin_c(int sg, int job, CSt &t) const
    {
        const ModDownSeg &S = payload(sg, job);
        const int logN = h[sg].logN, o = job / S.l, i = job % S.l;
        t.cv.src = S.accP + ((long long)o * S.K << logN);
        t.cv.dst = S.out + ((long long)job << logN);
        t.cv.n = S.K;
        t.prime = t.cv.prime = i;
#pragma unroll
        for (int k = 0; k < FHE_MAXK; k++)
            if (k < S.K) t.cv.c[k] = S.P->phat[k][i];
    }
    __device__ void begin_r(int sg, int job, RSt &t) const
    {
        const ModDownSeg &S = payload(sg, job);
        const int logN = h[sg].logN, o = job / S.l, i = job % S.l, c = o >> 1, pi = o & 1;
        t.x = S.acc + ((long long)o * (S.l + S.K) + i << logN);
        t.add = ((S.amask >> pi) & 1) ? S.abase + c * S.a_outer + pi * S.a_poly + ((long long)i << logN) : nullptr;
        t.out = S.out + ((long long)job << logN);
        t.prime = i;
    }
    __device__ RowK row_k(int sg, int i) const { return RowK{s[h[sg].first].P->pinv[i]}; }
    // two data limbs of one (ct, poly): the special limbs loaded once
    static constexpr int XJ = 2;
    __device__ bool same_src(const CSt &a, const CSt &b) const { return a.cv.src == b.cv.src && a.cv.n == b.cv.n; }
    static constexpr int NPRE = 2;  // accumulator, addend
    __device__ u64 pre(const RSt &t, int k, int w) const { return w == 0 ? t.x[k] : (t.add ? t.add[k] : 0); }
    __device__ void store_pre(const RowK &K, const ModQ &m, const RSt &t, int k, u64 v, const u64 *pv) const
    {
        t.out[k] = addmod(scaled1(lazy_diff(pv[0], v, m), K.pinv, m), pv[1], m.q);
    }
    __device__ u64 *inter(const CSt &t) const { return t.cv.dst; }
    __device__ u64 *inter(const RSt &t) const { return t.out; }
};

// Modulus switch l -> l-1 of poly pi of ct c, limb i < l-1:
//   delta_i = p w mod q_i,  out_i = (x_i - delta_i) q_{l-1}^-1,
// where `last` already holds w = [x_{l-1} p^-1]_{q_{l-1}} in the coefficient
// domain (applied by the inverse NTT that produced it).
// Job = (c, pi) * (l-1) + i.
struct SwitchSeg {
    const u64 *last;  // [count][npoly][N] coefficient domain
    const u64 *in;    // [count][npoly][l][N]
    u64 *out;         // [count][npoly][l-1][N]
    const ModSwitchParams *P;
    int l, npoly;
};

struct SwitchRowK {
    DotC inv;
};

struct IOModSwitch : SegIO<SwitchSeg> {
    struct CSt {
        const u64 *last;
        u64 *out;
        u64 nq, pi, pis;
        int prime;
    };
    using RSt = DownRSt;
    using RowK = SwitchRowK;
    __device__ void begin_c(int sg, int job, CSt &t) const
    {
        const SwitchSeg &S = payload(sg, job);
        const int logN = h[sg].logN, o = job / (S.l - 1), i = job % (S.l - 1);
        t.last = S.last + ((long long)o << logN);
        t.out = S.out + ((long long)job << logN);
        t.prime = i;
        t.nq = 0 - h[sg].mq[i].q;
        t.pi = S.P->p_i[i];
        t.pis = S.P->p_i_s[i];
    }
    __device__ void begin_r(int sg, int job, RSt &t) const
    {
        const SwitchSeg &S = payload(sg, job);
        const int logN = h[sg].logN, o = job / (S.l - 1), i = job % (S.l - 1);
        t.x = S.in + ((long long)o * S.l + i << logN);
        t.add = nullptr;
        t.out = S.out + ((long long)job << logN);
        t.prime = i;
    }
    __device__ RowK row_k(int sg, int i) const { return RowK{s[h[sg].first].P->qinv[i]}; }
    // a column pass's word is p w, in [0, 4q)
    static constexpr bool PLAIN = false;
    __device__ const u64 *src(const CSt &t) const { return t.last; }
    __device__ u64 conv(const CSt &t, u64 v) const { return shoup_lazy4_chain(v, t.pi, t.pis, t.nq); }
    static constexpr int NPRE = 1;  // the limb being switched
    __device__ u64 pre(const RSt &t, int k, int) const { return t.x[k]; }
    __device__ void store_pre(const RowK &K, const ModQ &m, const RSt &t, int k, u64 v, const u64 *pv) const
    {
        t.out[k] = scaled1(lazy_diff(pv[0], v, m), K.inv, m);
    }
    __device__ u64 *inter(const CSt &t) const { return t.out; }
    __device__ u64 *inter(const RSt &t) const { return t.out; }
};

// Relinearisation fused with the modulus switch that follows it (l -> l-1)
// for poly pi of ct c, kept limb i < l-1:
//   correction_i = sum_{k<K} t_k h[k][i] + w h[K][i] (coefficient domain),
//   out_i = (acc_i P^-1 + add_i - NTT(correction)_i) q_{l-1}^-1,
// where src holds t_0..t_{K-1} (the special limbs, already scaled) and w.
// The store is one two-term sum: acc_i (P q_{l-1})^-1 + (add_i -
// NTT(correction)_i) q_{l-1}^-1.  Job = (c, pi) * (l-1) + i.
struct RelinMSSeg {
    const u64 *src;  // [count][2][K+1][N] coefficient domain
    const u64 *acc;  // [count][2][l+K][N] NTT domain
    const u64 *abase;
    long long a_outer, a_poly;
    u64 *out;        // [count][2][l-1][N]
    const RelinMSParams *P;
    int l, K, amask, pad;
};

struct IORelinMS : SegIO<RelinMSSeg> {
    using CSt = ConvCSt;
    using RSt = DownRSt;
    struct RowK {
        DotC a, d;
    };
    __device__ void begin_c(int sg, int job, CSt &t) const
    {
        const RelinMSSeg &S = payload(sg, job);
        const int logN = h[sg].logN, m = S.l - 1, o = job / m, i = job % m;
        t.cv.src = S.src + ((long long)o * (S.K + 1) << logN);
        t.cv.dst = S.out + ((long long)job << logN);
        t.cv.n = S.K + 1;
        t.prime = t.cv.prime = i;
#pragma unroll
        for (int k = 0; k < FHE_MAXK; k++)
            if (k <= S.K) t.cv.c[k] = S.P->h[k][i];
    }
    __device__ void begin_r(int sg, int job, RSt &t) const
    {
        const RelinMSSeg &S = payload(sg, job);
        const int logN = h[sg].logN, m = S.l - 1, o = job / m, i = job % m, c = o >> 1, pi = o & 1;
        t.x = S.acc + ((long long)o * (S.l + S.K) + i << logN);
        t.add = ((S.amask >> pi) & 1) ? S.abase + c * S.a_outer + pi * S.a_poly + ((long long)i << logN) : nullptr;
        t.out = S.out + ((long long)job << logN);
        t.prime = i;
    }
    __device__ RowK row_k(int sg, int i) const { return RowK{s[h[sg].first].P->pqinv[i], s[h[sg].first].P->qminv[i]}; }
    // two data limbs of one (ct, poly): the K + 1 sources loaded once
    static constexpr int XJ = 2;
    __device__ bool same_src(const CSt &a, const CSt &b) const { return a.cv.src == b.cv.src && a.cv.n == b.cv.n; }
    static constexpr int NPRE = 2;  // accumulator, addend
    __device__ u64 pre(const RSt &t, int k, int w) const { return w == 0 ? t.x[k] : (t.add ? t.add[k] : 0); }
    __device__ void store_pre(const RowK &K, const ModQ &m, const RSt &t, int k, u64 v, const u64 *pv) const
    {
        t.out[k] = scaled2(pv[0], K.a, lazy_diff(pv[1], v, m), K.d, m);
    }
    __device__ u64 *inter(const CSt &t) const { return t.cv.dst; }
    __device__ u64 *inter(const RSt &t) const { return t.out; }
};

// k modulus switches at once (l -> l-k), poly pi of ct c, kept limb i < l-k:
//   correction_i = sum_{t<k} w_t G[t][i],  out_i = (x_i - NTT(correction)_i) D_k^-1.
// Job = (c, pi) * (l-k) + i.
struct MultiSeg {
    const u64 *src;  // [count][npoly][k][N] coefficient domain: w_0 .. w_{k-1}
    const u64 *in;   // [count][npoly][l][N]
    u64 *out;        // [count][npoly][l-k][N]
    const MultiSwitchParams *P;
    int l, k, npoly, pad;
};

struct IOMultiSwitch : SegIO<MultiSeg> {
    using CSt = ConvCSt;
    using RSt = DownRSt;
    using RowK = SwitchRowK;
    __device__ void begin_c(int sg, int job, CSt &t) const
    {
        const MultiSeg &S = payload(sg, job);
        const int logN = h[sg].logN, kept = S.l - S.k, o = job / kept, i = job % kept;
        t.cv.src = S.src + ((long long)o * S.k << logN);
        t.cv.dst = S.out + ((long long)job << logN);
        t.cv.n = S.k;
        t.prime = t.cv.prime = i;
#pragma unroll
        for (int j = 0; j < FHE_MAXK; j++)
            if (j < S.k) t.cv.c[j] = S.P->G[j][i];
    }
    __device__ void begin_r(int sg, int job, RSt &t) const
    {
        const MultiSeg &S = payload(sg, job);
        const int logN = h[sg].logN, kept = S.l - S.k, o = job / kept, i = job % kept;
        t.x = S.in + ((long long)o * S.l + i << logN);
        t.add = nullptr;
        t.out = S.out + ((long long)job << logN);
        t.prime = i;
    }
    __device__ RowK row_k(int sg, int i) const { return RowK{s[h[sg].first].P->Dinv[i]}; }
    // two kept limbs of one (ct, poly): the k switch values loaded once
    static constexpr int XJ = 2;
    __device__ bool same_src(const CSt &a, const CSt &b) const { return a.cv.src == b.cv.src && a.cv.n == b.cv.n; }
    static constexpr int NPRE = 1;
    __device__ u64 pre(const RSt &t, int j, int) const { return t.x[j]; }
    __device__ void store_pre(const RowK &K, const ModQ &m, const RSt &t, int j, u64 v, const u64 *pv) const
    {
        t.out[j] = scaled1(lazy_diff(pv[0], v, m), K.inv, m);
    }
    __device__ u64 *inter(const CSt &t) const { return t.cv.dst; }
    __device__ u64 *inter(const RSt &t) const { return t.out; }
};

// ---------------------------------------------------------------------------
// host side: unit counts, grids, launches
// ---------------------------------------------------------------------------

struct Split {
    int n1, n2, ns1, ns2;
};

Split split_of(int logN)
{
    Split s;
    s.n1 = (logN + 1) / 2;
    s.n2 = logN / 2;
    s.ns1 = 2048 >> s.n1;
    s.ns2 = 2048 >> s.n2;
    return s;
}

// Row units are grouped (16 jobs of one prime) as far as the outer items fill
// them; a rest of fewer than GROUP_MIN_OUTER items takes units of adjacent
// rows of one job, whose twiddles are read through the cache (twice the data's
// bytes at N2 = 7).
constexpr int GROUP_MIN_OUTER = 12;

// Unit counts of a segment (column and row passes) from its geometry.
void unit_counts(SegHdr &H)
{
    const Split sp = split_of(H.logN);
    const int njobs = H.outer * H.nl;
    int nc = std::min(sp.ns1, 1 << sp.n2);
    if (col_paired(H.xj, sp.ns1, nc)) nc /= 2;  // ColGeo's paired units
    const int nj = sp.ns1 / nc, blk = (1 << sp.n2) / nc;
    H.u_cols = ((njobs + nj - 1) / nj) * blk;
    const bool always = (1 << sp.n1) < sp.ns2;  // a limb has fewer rows than a unit
    const int rest = H.outer % ROW_J;
    H.gouter = always || rest >= GROUP_MIN_OUTER ? H.outer : H.outer - rest;
    H.g_units = H.nl * ((H.gouter + ROW_J - 1) / ROW_J) * ((1 << sp.n1) / (sp.ns2 / ROW_J));
    H.u_rows = H.g_units + (H.outer - H.gouter) * H.nl * ((1 << sp.n1) / sp.ns2);
}

// Fills the header of a segment (jobs = outer * nl) with its unit counts
// (turned into first units by finish()).
void seg_header(SegHdr &H, const fhe_ctx *c, bool fwd, int outer, int nl)
{
    memset(&H, 0, sizeof(H));
    H.logN = c->logN;
    H.outer = outer;
    H.nl = nl;
    H.mq = c->d_mq;
    H.tw = fwd ? c->d_fwd : c->d_inv;
    H.ninv = c->d_ninv;
    H.per = outer;
    unit_counts(H);
}

// Grid of a pass: one CTA per unit (variant 0) or a fixed number of resident
// CTAs per SM that walk the units (variants 1..3: 6, 4 and 2 per SM).
int grid_of(int variant, int sms, int units)
{
    static const int per_sm[FHE_NTT_VARIANTS] = {0, 6, 4, 2};
    if (variant <= 0 || variant >= FHE_NTT_VARIANTS || sms <= 0) return units;
    return std::min(units, per_sm[variant] * sms);
}
int grid_of(const fhe_ctx *c, int units) { return grid_of(c->ntt_variant, c->sms, units); }

// Unit counts per segment (seg_header) -> first unit of each segment.
template <class IO>
void finish(IO &io)
{
    int uc = 0, ur = 0;
    for (int s = 0; s < io.nseg; s++) {
        const int nc = io.h[s].u_cols, nr = io.h[s].u_rows;
        io.h[s].u_cols = uc;
        io.h[s].u_rows = ur;
        uc += nc;
        ur += nr;
    }
    io.ucols = uc;
    io.urows = ur;
}

// The unit counts of a subset's segments, recomputed from their geometry
// (for a launch split by ring degree after finish()).
template <class IO>
void recount(IO &io)
{
    for (int s = 0; s < io.nseg; s++) unit_counts(io.h[s]);
}

// Where both passes run as one kernel: launches of at most this many units per
// SM.  On a context's own stream the one kernel wins to about 6 (LT + EQ of 3
// at N = 2^14: 3020 us without, 2785 at 6, 2798 at 8, 2846 at 12); at N = 2^15,
// whose clusters of 16 take more of the chip at once, to one resident wave (one
// LT + EQ of 12 primes: 2366 without, 2177 at 2, 2075 at 4, 2085 at 6; sixteen
// products 2058 at 4, 2069 at 6).  Under the scheduler other streams fill the
// chip and pairing targets is worth more (32 uneven requests: 46.1 ms without,
// 45.6 at 1, 45.9 at 2, 46.7 at 4).
#ifndef FHE_NTT_SMALL
#define FHE_NTT_SMALL 6
#endif
#ifndef FHE_NTT_SMALL_15
#define FHE_NTT_SMALL_15 4
#endif
#ifndef FHE_NTT_SMALL_BRANCH
#define FHE_NTT_SMALL_BRANCH 1
#endif

// Whether a launch of `limbs` limbs of ring degree 2^logN runs as one kernel.
bool one_kernel(int logN, int sms, bool on_branch, long long limbs)
{
    if (logN < SMALL_LO || logN > SMALL_HI) return false;
    const int own = logN == 15 ? FHE_NTT_SMALL_15 : FHE_NTT_SMALL;
    return (limbs << (logN - 11)) <= (long long)(on_branch ? FHE_NTT_SMALL_BRANCH : own) * sms;
}

// Polynomials of nl limbs that the autotuner times for a request of njobs
// limbs: a multiple of 16 from 16 on, so that the row units take their grouped
// form as in batched use, and raised until both passes have TUNE_UNITS units
// per SM.  Below, the choice would rest on noise: launches of up to 6 units per
// SM run as one kernel, which has no grid policy, and a pass of fewer units
// than a policy's resident CTAs gets the grid of every other (six per SM is the
// most; twice that, so that a CTA walks at least two units).
constexpr int TUNE_UNITS = 12;
static_assert(TUNE_UNITS > FHE_NTT_SMALL && TUNE_UNITS > FHE_NTT_SMALL_15, "timed in two passes");

int tune_outer(int logN, int nl, int sms, int njobs)
{
    int outer = std::max(1, njobs / nl);
    if (outer >= 16) outer -= outer % 16;
    const int need = TUNE_UNITS * sms;
    SegHdr H;
    memset(&H, 0, sizeof(H));
    H.logN = logN;
    H.nl = nl;
    for (; (long long)outer * nl < 2LL * need; outer = outer / 16 * 16 + 16) {  // a limb is half a unit or more
        H.outer = outer;
        unit_counts(H);
        if (std::min(H.u_cols, H.u_rows) >= need) break;
    }
    return outer;
}

// The segment's units of the one-kernel form from unit u on (a limb's units, one
// limb after the other, in both passes); the unit after them.
int one_kernel_units(SegHdr &H, int u)
{
    H.gouter = H.g_units = 0;
    H.u_cols = H.u_rows = u;
    return u + (H.outer * H.nl << (H.logN - SMALL_LO));
}

template <class IO, int L>
void launch_passes(fhe_ctx *c, IO &io, bool fwd)
{
    if constexpr (L >= SMALL_LO && L <= SMALL_HI) {
        constexpr int C = SMALL_CTAS<L>;
        long long limbs = 0;
        for (int s = 0; s < io.nseg; s++) limbs += (long long)io.h[s].outer * io.h[s].nl;
        if (one_kernel(L, c->sms, c->on_branch, limbs)) {
            int u = 0;
            for (int s = 0; s < io.nseg; s++) u = one_kernel_units(io.h[s], u);
            const bool pdl = pdl_on(c, u, T);
            if constexpr ((IO::DIRS & DIR_FWD) != 0)
                if (fwd) launch_pdl_cluster(k_fwd_small<IO, L>, pdl, u, T, C, c->stream, io);
            if constexpr ((IO::DIRS & DIR_INV) != 0)
                if (!fwd) launch_pdl_cluster(k_inv_small<IO, L>, pdl, u, T, C, c->stream, io);
            c->launches++;
            return;
        }
    }
    if constexpr ((IO::DIRS & DIR_FWD) != 0)
        if (fwd) {
            launch_pdl(k_fwd_cols<IO, L>, pdl_on(c, grid_of(c, io.ucols), T), grid_of(c, io.ucols), T, c->stream, io);
            launch_pdl(k_fwd_rows<IO, L>, pdl_on(c, grid_of(c, io.urows), T), grid_of(c, io.urows), T, c->stream, io);
        }
    if constexpr ((IO::DIRS & DIR_INV) != 0)
        if (!fwd) {
            launch_pdl(k_inv_rows<IO, L>, pdl_on(c, grid_of(c, io.urows), T), grid_of(c, io.urows), T, c->stream, io);
            launch_pdl(k_inv_cols<IO, L>, pdl_on(c, grid_of(c, io.ucols), T), grid_of(c, io.ucols), T, c->stream, io);
        }
    c->launches += 2;
}

// Segments of one degree take that degree's kernels; a mix is split by degree.
template <class IO>
void launch_segments(fhe_ctx *c, IO &io, bool fwd)
{
    int lo = 99, hi = 0;
    for (int s = 0; s < io.nseg; s++) lo = std::min(lo, io.h[s].logN), hi = std::max(hi, io.h[s].logN);
    finish(io);
    if (io.ucols == 0) return;
    if (lo == hi) {
        switch (lo) {
        case 10: launch_passes<IO, 10>(c, io, fwd); break;
        case 11: launch_passes<IO, 11>(c, io, fwd); break;
        case 12: launch_passes<IO, 12>(c, io, fwd); break;
        case 13: launch_passes<IO, 13>(c, io, fwd); break;
        case 14: launch_passes<IO, 14>(c, io, fwd); break;
        case 15: launch_passes<IO, 15>(c, io, fwd); break;
        default: break;
        }
    } else {
        for (int n = lo; n <= hi; n++) {
            IO sub;
            memset(&sub, 0, sizeof(sub));
            int np = 0;
            for (int s = 0; s < io.nseg; s++)
                if (io.h[s].logN == n) {
                    SegHdr &H = sub.h[sub.nseg++];
                    H = io.h[s];
                    for (int k = 0; k < H.outer / H.per; k++) sub.s[np + k] = io.s[io.h[s].first + k];
                    H.first = np;
                    np += H.outer / H.per;
                }
            if (sub.nseg) {
                recount(sub);
                launch_segments(c, sub, fwd);
            }
        }
    }
}

// Launches both passes of the segments in io on the stream of `c` (the
// first segment's context).  bytes / bfly: algorithmic traffic and butterflies
// of the whole launch, for the per-class timing.
template <class IO>
void run(fhe_ctx *c, IO &io, bool fwd, int cls, double bytes, double bfly)
{
    if (io.nseg == 0) return;
    prof_begin(c, cls, bytes, bfly);
    launch_segments(c, io, fwd);
    prof_end(c);
}

double bfly_of(const fhe_ctx *c, double njobs) { return njobs * (c->N / 2) * c->logN; }

void map_seg(MapSeg &S, const u64 *in, u64 *out, const LimbMap &m, const ulonglong2 *scale)
{
    memset(&S, 0, sizeof(S));
    S.in = in;
    S.out = out;
    S.in_outer = m.in_outer;
    S.out_outer = m.out_outer;
    S.scale = scale;
    for (int i = 0; i < m.nl; i++) {
        S.in_limb[i] = (uint8_t)m.in_limb[i];
        S.out_limb[i] = (uint8_t)m.out_limb[i];
        S.prime[i] = (uint8_t)m.prime[i];
    }
}

// Runs `fill(io, 0, item, ..)` over items: the payloads of one context and
// geometry that join side by side as one segment, in launches of at most
// FHE_SEGS payloads.
template <class IO, class Item, class Fill>
void run_many(const std::vector<Item> &items, bool fwd, int cls, Fill fill)
{
    struct One {
        fhe_ctx *c;
        SegHdr h;
        typename IO::Payload s;
        double bytes, bfly;
        bool taken;
    };
    std::vector<One> all;
    all.reserve(items.size());
    std::unique_ptr<IO> tmp(new IO);
    for (const Item &it : items) {
        One o;
        memset(&o, 0, sizeof(o));
        memset(&tmp->h[0], 0, sizeof(tmp->h[0]));
        memset(&tmp->s[0], 0, sizeof(tmp->s[0]));
        if (!fill(*tmp, 0, it, &o.bytes, &o.bfly)) continue;
        o.c = it.c;
        o.h = tmp->h[0];
        o.s = tmp->s[0];
        all.push_back(o);
    }
    std::vector<One *> order;
    for (size_t i = 0; i < all.size(); i++)
        for (size_t j = i; j < all.size(); j++)
            if (!all[j].taken && (j == i || (!all[i].taken && all[j].c == all[i].c && all[j].h.nl == all[i].h.nl &&
                                             all[j].h.per == all[i].h.per && joins(all[j].s, all[i].s)))) {
                if (j != i) all[j].taken = true;
                order.push_back(&all[j]);
            } else if (j == i) {
                break;
            }
    for (size_t i = 0; i < order.size();) {
        memset(tmp.get(), 0, sizeof(IO));
        IO &io = *tmp;
        fhe_ctx *c0 = order[i]->c;
        double bytes = 0, bfly = 0;
        for (int np = 0; i < order.size() && np < FHE_SEGS; i++, np++) {
            const One &o = *order[i];
            SegHdr *H = io.nseg ? &io.h[io.nseg - 1] : nullptr;
            if (H && o.c == order[i - 1]->c && H->nl == o.h.nl && H->per == o.h.per && joins(io.s[H->first], o.s)) {
                H->outer += o.h.outer;
            } else {
                H = &io.h[io.nseg++];
                *H = o.h;
                H->first = np;
                if (IO::XJ != 1) H->xj = IO::XJ;
            }
            io.s[np] = o.s;
            unit_counts(*H);
            bytes += o.bytes;
            bfly += o.bfly;
        }
        run(c0, io, fwd, cls, bytes, bfly);
    }
}

}  // namespace
