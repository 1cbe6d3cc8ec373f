// many.cu -- the streaming kernels of a product or a switch over several
// batches in one launch: element-wise ciphertext arithmetic, the tensor
// product, the key-switching inner product and the switch folds.
//
// A launch carries a table of up to FHE_SEGS segments (one batch each, of any
// context, level and size on one device); segment s owns a contiguous range
// of blocks, so a block never straddles two segments and every warp still
// reads 256 contiguous bytes.  Single batches run through the same kernels,
// sums and small products with a table of one.
#include <string.h>

#include <algorithm>

#include "fhe_internal.h"

namespace {

constexpr int TPB = 256;
constexpr int EW_ELEMS = TPB * 4;  // elements per block of the element-wise kernels

// |k| < q: k mod q in [0, q)
__device__ __forceinline__ u64 small_mod(int64_t k, u64 q) { return k >= 0 ? (u64)k : q - (u64)(-k); }

// A launch's segments (kernel parameters) and the elements a block of the
// element-wise kernels takes.  A call on one batch takes a table of one: with
// room for FHE_SEGS the parameters of an addition are 4.4 KB, and a small
// fhe_add took 3.7 us among others, 3.3 with one; fhe_mul 3.6 and 3.2.
template <class Seg, int CAP, int ELEMS = EW_ELEMS>
struct Table {
    static constexpr int cap = CAP, elems = ELEMS;
    int nseg, rms;  // rms: the folds' kind
    Seg s[CAP];
};

template <class Seg, int CAP, int ELEMS>
__device__ __forceinline__ int block_seg(const Table<Seg, CAP, ELEMS> &t)
{
    int sg = 0;
    if constexpr (CAP > 1)
        while (sg + 1 < t.nseg && t.s[sg + 1].b0 <= (int)blockIdx.x) sg++;
    return sg;
}

// ---- element-wise: x0 + x1, x0 - x1, -x0, sum_t k_t x_t, k0 x0, x0 + k0 on
// poly 0 of 2-poly ciphertexts (poly 1 copied) ------------------------------

struct EwSeg {
    const u64 *x[8];
    u64 *out;
    const ModQ *mq;
    long long total;  // elements: outer * level * N
    int logN, level, n, op, b0, vec;  // vec: every pointer 16-byte aligned
    int small, pad;   // small: q sum |k_j| < 2^64 for every prime (see small_scaled)
    int64_t k[8];     // centred scalars, |k| < p
};

// V adjacent elements (one limb: N is even) as one load per operand
template <int V>
struct Vec {
    u64 v[V];
};

template <int V>
__device__ __forceinline__ Vec<V> ld_vec(const u64 *p)
{
    Vec<V> r;
    if constexpr (V == 2) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p);
        r.v[0] = t.x;
        r.v[1] = t.y;
    } else {
        r.v[0] = *p;
    }
    return r;
}

template <int V>
__device__ __forceinline__ void st_vec(u64 *p, const Vec<V> &r)
{
    if constexpr (V == 2)
        *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(r.v[0], r.v[1]);
    else
        *p = r.v[0];
}

// A block's EW_ELEMS elements lie in one limb (EW_ELEMS divides N, N >= 2^10),
// so the limb's prime and the polynomial index are per-block constants
// (measured with the tensor's per-block addressing and 16-byte loads, and the
// 64-bit scalar products: tensor 0.83 -> 0.67 ms, element-wise 1.40 -> 1.35 ms
// per step on the 16-pair comparison at N = 2^14).
template <int V>
__device__ __forceinline__ void ew_block(const EwSeg &S)
{
    const long long base = (long long)(blockIdx.x - S.b0) * EW_ELEMS;
    const long long li = base >> S.logN;
    const int i = (int)(li % S.level);
    const u64 q = S.mq[i].q;
#pragma unroll
    for (int e = threadIdx.x * V; e < EW_ELEMS; e += TPB * V) {
        const long long idx = base + e;
        if (idx >= S.total) break;
        Vec<V> r;
        switch (S.op) {
        case FHE_EW_ADD: {
            const Vec<V> a = ld_vec<V>(S.x[0] + idx), b = ld_vec<V>(S.x[1] + idx);
#pragma unroll
            for (int u = 0; u < V; u++) r.v[u] = addmod(a.v[u], b.v[u], q);
            break;
        }
        case FHE_EW_SUB: {
            const Vec<V> a = ld_vec<V>(S.x[0] + idx), b = ld_vec<V>(S.x[1] + idx);
#pragma unroll
            for (int u = 0; u < V; u++) r.v[u] = submod(a.v[u], b.v[u], q);
            break;
        }
        case FHE_EW_NEG: {
            const Vec<V> a = ld_vec<V>(S.x[0] + idx);
#pragma unroll
            for (int u = 0; u < V; u++) r.v[u] = negmod(a.v[u], q);
            break;
        }
        case FHE_EW_CMUL: {
            const Vec<V> a = ld_vec<V>(S.x[0] + idx);
            if (S.small) {
#pragma unroll
                for (int u = 0; u < V; u++) r.v[u] = reduce64(small_scaled(a.v[u], S.k[0], q), S.mq[i]);
                break;
            }
            const u64 k = small_mod(S.k[0], q);
#pragma unroll
            for (int u = 0; u < V; u++) r.v[u] = barrett128((u128)a.v[u] * k, S.mq[i]);
            break;
        }
        case FHE_EW_CADD: {
            const int poly = (int)((li / S.level) % 2);
            const Vec<V> a = ld_vec<V>(S.x[0] + idx);
            const u64 k = small_mod(S.k[0], q);
#pragma unroll
            for (int u = 0; u < V; u++) r.v[u] = poly == 0 ? addmod(a.v[u], k, q) : a.v[u];
            break;
        }
        default: {  // FHE_EW_LINCOMB: at most eight products below the Barrett bound
            if (S.small) {
                u64 acc[V];
#pragma unroll
                for (int u = 0; u < V; u++) acc[u] = 0;
#pragma unroll
                for (int j = 0; j < 8; j++)
                    if (j < S.n) {
                        const Vec<V> a = ld_vec<V>(S.x[j] + idx);
#pragma unroll
                        for (int u = 0; u < V; u++) acc[u] += small_scaled(a.v[u], S.k[j], q);
                    }
#pragma unroll
                for (int u = 0; u < V; u++) r.v[u] = reduce64(acc[u], S.mq[i]);
                break;
            }
            u128 acc[V];
#pragma unroll
            for (int u = 0; u < V; u++) acc[u] = 0;
#pragma unroll
            for (int j = 0; j < 8; j++)
                if (j < S.n) {
                    const Vec<V> a = ld_vec<V>(S.x[j] + idx);
                    const u64 k = small_mod(S.k[j], q);
#pragma unroll
                    for (int u = 0; u < V; u++) acc[u] += (u128)a.v[u] * k;
                }
#pragma unroll
            for (int u = 0; u < V; u++) r.v[u] = barrett128(acc[u], S.mq[i]);
        }
        }
        st_vec<V>(S.out + idx, r);
    }
}

template <class Tb>
__global__ void k_ew_many(const __grid_constant__ Tb t)
{
    pdl_begin();
    const EwSeg &S = t.s[block_seg(t)];
    if (S.vec)
        ew_block<2>(S);
    else
        ew_block<1>(S);
}

// ---- linear combinations of shared operands ---------------------------------
// out[o] = sum_t k[o][t] x[t] for up to eight outputs over the same (up to
// eight) operands: the leaves of a Paterson-Stockmeyer evaluation combine the
// same baby powers with different coefficients.  Bound by HBM: each operand
// word is read once for all outputs, where a launch of single combinations
// read it once per output (the leaves' operands of a batch exceed L2: p = 257
// has 16 leaves over eight powers).  Measured per pass, all element-wise
// launches: 7 pairs at N = 2^15 4.59 -> 2.19 ms, 16 pairs at N = 2^14 0.96 ->
// 0.49 ms.  Sums in 64 bits (small_start, small_add).

constexpr int LC_N = 8;

struct LcSeg {
    const u64 *x[LC_N];
    u64 *out[LC_N];
    const ModQ *mq;
    long long total;  // elements: outer * level * N
    int logN, level, n, nout, b0, vec;
    int32_t k[LC_N][LC_N];  // [output][operand]
    uint32_t neg[LC_N];     // sum of |k| over an output's negative scalars
};

template <int V>
__device__ __forceinline__ void lc_block(const LcSeg &S)
{
    const long long base = (long long)(blockIdx.x - S.b0) * EW_ELEMS;
    const int i = (int)((base >> S.logN) % S.level);  // a block's elements lie in one limb
    const ModQ &m = S.mq[i];
    const u64 q = m.q;
#pragma unroll 1
    for (int e = threadIdx.x * V; e < EW_ELEMS; e += TPB * V) {
        const long long idx = base + e;
        if (idx >= S.total) break;
        Vec<V> a[LC_N];
#pragma unroll
        for (int t = 0; t < LC_N; t++)
            if (t < S.n) a[t] = ld_vec<V>(S.x[t] + idx);
#pragma unroll 1
        for (int o = 0; o < S.nout; o++) {
            u64 acc[V];
#pragma unroll
            for (int u = 0; u < V; u++) acc[u] = small_start(q, S.neg[o]);
#pragma unroll
            for (int t = 0; t < LC_N; t++)
                if (t < S.n) {
                    const int32_t k = S.k[o][t];
#pragma unroll
                    for (int u = 0; u < V; u++) acc[u] = small_add(acc[u], a[t].v[u], k);
                }
            Vec<V> r;
#pragma unroll
            for (int u = 0; u < V; u++) r.v[u] = reduce64(acc[u], m);
            st_vec<V>(S.out[o] + idx, r);
        }
    }
}

template <class Tb>
__global__ void k_lincomb_many(const __grid_constant__ Tb t)
{
    pdl_begin();
    const LcSeg &S = t.s[block_seg(t)];
    if (S.vec)
        lc_block<2>(S);
    else
        lc_block<1>(S);
}

// ---- tensor: (a0,a1) x (b0,b1) -> (a0 b0, a0 b1 + a1 b0, a1 b1) -----------

struct TensorSeg {
    const u64 *a, *b;
    u64 *out;
    const ModQ *mq;
    long long total;  // count * level * N
    int logN, level, b0, vec;  // vec: every pointer 16-byte aligned
};

template <int V, int ELEMS>
__device__ __forceinline__ void tensor_block(const TensorSeg &S)
{
    // one limb of one ciphertext per block (ELEMS divides N)
    const long long LN = (long long)S.level << S.logN;
    const long long base = (long long)(blockIdx.x - S.b0) * ELEMS;
    if (base >= S.total) return;
    const long long c = base / LN, r0 = base % LN;
    const ModQ m = S.mq[(int)(r0 >> S.logN)];
    const u64 *a0 = S.a + 2 * c * LN + r0, *a1 = a0 + LN;
    const u64 *b0 = S.b + 2 * c * LN + r0, *b1 = b0 + LN;
    u64 *o0 = S.out + 3 * c * LN + r0, *o1 = o0 + LN, *o2 = o1 + LN;
#pragma unroll
    for (int e = threadIdx.x * V; e < ELEMS; e += TPB * V) {
        const Vec<V> x0 = ld_vec<V>(a0 + e), x1 = ld_vec<V>(a1 + e), y0 = ld_vec<V>(b0 + e), y1 = ld_vec<V>(b1 + e);
        Vec<V> r0v, r1v, r2v;
#pragma unroll
        for (int u = 0; u < V; u++) {
            r0v.v[u] = barrett128((u128)x0.v[u] * y0.v[u], m);
            r1v.v[u] = barrett128((u128)x0.v[u] * y1.v[u] + (u128)x1.v[u] * y0.v[u], m);
            r2v.v[u] = barrett128((u128)x1.v[u] * y1.v[u], m);
        }
        st_vec<V>(o0 + e, r0v);
        st_vec<V>(o1 + e, r1v);
        st_vec<V>(o2 + e, r2v);
    }
}

template <class Tb>
__global__ void k_tensor_many(const __grid_constant__ Tb t)
{
    pdl_begin();
    const TensorSeg &S = t.s[block_seg(t)];
    if (S.vec)
        tensor_block<2, Tb::elems>(S);
    else
        tensor_block<1, Tb::elems>(S);
}

// ---- key-switching inner product ------------------------------------------
// acc[c][pi][r] = sum_j y_j[r] ksk_j[pi][prime(r)], y_j[r] = x_c[r] for r in
// digit j, else the ModUp limb.  A block covers TPB coefficients of one
// extended limb r for CB ciphertexts; each thread loads its 2 dnum key words
// once for its CB ciphertexts.
//
// Bound by the multiplier pipe, and by the loads' round trips where few
// ciphertexts share a launch.  The key words are stored as packed half words
// times 2^(2h) (see HalfAcc): a product is three wide multiplications, a sum
// is reduced by two half-word Montgomery steps.  All of a thread's words come
// by asynchronous copies into shared memory before its first product.
// Ciphertexts of items that use the same key at the same level (the products
// of a wave, the requests of an uneven batch) form one run: their key words
// are loaded once for CB of them, and a thread multiplies only for the
// ciphertexts it has (single requests used to multiply for four).
//
// Measured per pass (before: 128-bit multiply-adds, one run per item, one
// digit's words ahead in registers): tournament of 8 ciphertexts, N = 2^15,
// 36.5 -> 15.5 ms; 7 pairs at N = 2^15 5.80 -> 4.58 ms; 16 pairs at N = 2^14
// 1.53 -> 1.38 ms (17.7 / 5.24 / 1.55 with one product a statement instead of
// the digits in pairs; 23.6 / 7.6 / 1.84 with the words ahead in registers).
// Ciphertexts a thread and blocks an SM, one product a statement (16 pairs /
// 7 pairs / tournament, ms): 4 and 3 as here; 2 and 4 1.81 / 6.14 / 19.2; 3
// and 3 1.62 / 5.46 / 18.7; 5 and 2 1.68 / 5.58 / 20.5.

#ifndef FHE_KS_CB
#define FHE_KS_CB 4
#endif
#ifndef FHE_KS_MINB
#define FHE_KS_MINB 3
#endif
constexpr int KS_CB = FHE_KS_CB;  // ciphertexts per thread (key words reused across them)

struct KsSeg {
    const u64 *ext, *xbase, *ksk;
    u64 *acc;
    const ModQ *mq;
    long long x_outer;
    int count, l, K, L, dnum, logN, b0, nbx;  // nbx: blocks along n
    int run;  // ciphertexts of the run this item opens (0: the item belongs to an earlier one's)
};

using KsTable = Table<KsSeg, FHE_SEGS>;

// Digit group g of this thread's copies has arrived once at most `left` later
// groups are in flight.
__device__ __forceinline__ void async_wait_left(int left)
{
    switch (left) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
    case 4: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
    case 5: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
    case 6: asm volatile("cp.async.wait_group 6;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 7;" ::: "memory"); break;
    }
}

__device__ __forceinline__ void async8(u64 *dst, const u64 *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// The sums of a thread's ciphertexts (FULL: all KS_CB of them, so that no
// branch stands between the copies).  own(cc): the ciphertext's word of the
// digit that holds limb r itself; ep: its ModUp words, advanced digit by
// digit; out(cc): its two sums.  w: the thread's words in shared memory, TPB
// apart: the two key words, then the ciphertexts', digit by digit.  Every
// digit's words are under way before the first product, in registers they
// would take 12 dnum (one digit ahead, in registers: four round trips to L2
// one after the other for dnum = 4, which bounded the kernel).
template <bool FULL, class Own, class Out>
__device__ __forceinline__ void ks_sum(u64 *w, const u64 *(&ep)[KS_CB], const u64 *kp, long long kstride,
                                       long long dstride, int rdig, int dnum, int ncb, const ModQ &m, Own own, Out out)
{
    const int h = m.half;
    const uint32_t mask = ((uint32_t)1 << h) - 1;
    {
        u64 *d = w;
        for (int j = 0; j < dnum; j++, kp += 2 * kstride, d += (2 + KS_CB) * TPB) {
            async8(d, kp);
            async8(d + TPB, kp + kstride);
        }
        pdl_wait();
        d = w;
        for (int j = 0; j < dnum; j++, d += (2 + KS_CB) * TPB) {
#pragma unroll
            for (int cc = 0; cc < KS_CB; cc++) {
                if (FULL || cc < ncb) async8(d + (2 + cc) * TPB, j == rdig ? own(cc) : ep[cc]);
                ep[cc] += dstride;
            }
            asm volatile("cp.async.commit_group;" ::: "memory");  // the first also holds the key words
        }
    }
    HalfAcc a0[KS_CB], a1[KS_CB];
#pragma unroll
    for (int cc = 0; cc < KS_CB; cc++) a0[cc] = a1[cc] = HalfAcc{0, 0, 0};
    auto split = [&](u64 z) { return halves((uint32_t)z & mask, (uint32_t)(z >> h)); };
    constexpr int DW = (2 + KS_CB) * TPB;  // a digit's words
    int j = 0;
    for (; j + 2 <= dnum; j += 2, w += 2 * DW) {
        async_wait_left(dnum - 2 - j);
        const Halves c0 = halves_of(w[0]), c1 = halves_of(w[TPB]), d0 = halves_of(w[DW]), d1 = halves_of(w[DW + TPB]);
#pragma unroll
        for (int cc = 0; cc < KS_CB; cc++)
            if (FULL || cc < ncb) {
                const Halves z = split(w[(2 + cc) * TPB]), y = split(w[DW + (2 + cc) * TPB]);
                half_mac2(a0[cc], z, c0, y, d0);
                half_mac2(a1[cc], z, c1, y, d1);
            }
    }
    if (j < dnum) {
        async_wait_left(0);
        const Halves c0 = halves_of(w[0]), c1 = halves_of(w[TPB]);
#pragma unroll
        for (int cc = 0; cc < KS_CB; cc++)
            if (FULL || cc < ncb) {
                const Halves z = split(w[(2 + cc) * TPB]);
                half_mac(a0[cc], z, c0);
                half_mac(a1[cc], z, c1);
            }
    }
    // in [0, 2q): what reads the sums (the inverse transforms and the stores
    // of ModDown and of relinearise + switch) takes them
#pragma unroll
    for (int cc = 0; cc < KS_CB; cc++)
        if (FULL || cc < ncb) {
            u64 *o = out(cc);
            o[0] = reduce_few(half_mont(a0[cc], m), m);
            o[dstride] = reduce_few(half_mont(a1[cc], m), m);
        }
}

__global__ void __launch_bounds__(TPB, FHE_KS_MINB) k_ks_inner_many(const __grid_constant__ KsTable t)
{
    pdl_trigger();
    extern __shared__ u64 ks_words[];  // [dnum][2 + KS_CB][TPB]
    const int sg = block_seg(t);
    const KsSeg &S = t.s[sg];
    const int lb = blockIdx.x - S.b0;
    const int lK = S.l + S.K, N = 1 << S.logN;
    const int bx = lb % S.nbx, r = (lb / S.nbx) % lK, cz = lb / (S.nbx * lK);
    const int n = bx * TPB + threadIdx.x;
    if (n >= N) return;
    const int prime = r < S.l ? r : S.L + (r - S.l);
    const ModQ &m = S.mq[prime];
    const int rdig = r < S.l ? r / S.K : -1;
    const int ncb = min(KS_CB, S.run - cz * KS_CB);
    // the block's ciphertexts: item and place in it (the run's ciphertexts in
    // order, over the items from sg on)
    int it[KS_CB], pl[KS_CB];
    {
        int i = sg, c = cz * KS_CB;
#pragma unroll
        for (int cc = 0; cc < KS_CB; cc++) {
            it[cc] = sg;
            pl[cc] = 0;
            if (cc < ncb) {
                while (c >= t.s[i].count) c -= t.s[i].count, i++;
                it[cc] = i;
                pl[cc] = c++;
            }
        }
    }
    const u64 *ep[KS_CB];
#pragma unroll
    for (int cc = 0; cc < KS_CB; cc++)
        ep[cc] = t.s[it[cc]].ext + ((long long)pl[cc] * S.dnum * lK + r) * N + n;
    auto own = [&](int cc) { return t.s[it[cc]].xbase + pl[cc] * t.s[it[cc]].x_outer + (long long)r * N + n; };
    auto out = [&](int cc) { return t.s[it[cc]].acc + ((long long)pl[cc] * 2 * lK + r) * N + n; };
    const u64 *kp = S.ksk + (long long)prime * N + n;
    const long long kstride = (long long)(S.L + S.K) * N, dstride = (long long)lK * N;
    if (ncb == KS_CB)
        ks_sum<true>(ks_words + threadIdx.x, ep, kp, kstride, dstride, rdig, S.dnum, ncb, m, own, out);
    else
        ks_sum<false>(ks_words + threadIdx.x, ep, kp, kstride, dstride, rdig, S.dnum, ncb, m, own, out);
}

// ---- folds of the fused relinearise + switch and of the multi-prime switch

struct FoldSeg {
    u64 *src;
    const ModQ *mq;
    const void *P;    // RelinMSParams (k = 0) or MultiSwitchParams
    long long total;  // outer * N
    int logN, l, k, K, b0, vec;  // vec: src 16-byte aligned
};

// y - s for the folded sum s (within 3q of 0) of constant products
__device__ __forceinline__ u64 fold_sub(u64 y, int64_t s, const ModQ &m)
{
    return reduce2q(reduce_few(y + 2 * m.q2 - (u64)s, m), m.q);
}

// The relinearise + switch fold: src[c][pi] = (t_0 .. t_{K-1}, Y') -> Y' -
// sum_k t_k p_k^-1 mod q_{l-1}.  A block's FOLD_ELEMS words lie in one
// polynomial (FOLD_ELEMS divides N), so polynomial and constants are found
// once; a thread has one pair of adjacent words, all its 16-byte loads in
// flight together (with two pairs in turn, the second's loads behind the
// first's store, the kernel waited on loads 13 of 18 cycles an instruction
// at 46% of HBM; folds of 12 max/min pairs at N = 2^15 0.80 -> 0.68 ms).
constexpr int FOLD_ELEMS = TPB * 2;

__device__ __forceinline__ void fold_rms_block(const FoldSeg &S)
{
    const int N = 1 << S.logN;
    const long long base = (long long)(blockIdx.x - S.b0) * FOLD_ELEMS;
    if (base >= S.total) return;
    const long long o = base >> S.logN;
    const RelinMSParams *P = (const RelinMSParams *)S.P;
    const ModQ &m = S.mq[S.l - 1];
    const int h = m.half;
    u64 *b = S.src + o * (S.K + 1) * N + (base & (N - 1)) + threadIdx.x * 2;
    auto pair = [&](const u64 *p) {
        return S.vec ? *reinterpret_cast<const ulonglong2 *>(p) : make_ulonglong2(p[0], p[1]);
    };
    ulonglong2 v[FHE_MAXK];
    u64 *y = b + (long long)S.K * N;
#pragma unroll
    for (int k = 0; k < FHE_MAXK; k++)
        if (k < S.K) v[k] = pair(b + (long long)k * N);
    const ulonglong2 yv = pair(y);
    DotAcc a0{0, 0}, a1{0, 0};
#pragma unroll
    for (int k = 0; k < FHE_MAXK; k++)
        if (k < S.K) {
            const DotC c = P->pkinv[k];
            dot_mac(a0, v[k].x, c, h);
            dot_mac(a1, v[k].y, c, h);
            if (h > 27 && (k & 1)) a0 = DotAcc{0, dot_fold(a0, m)}, a1 = DotAcc{0, dot_fold(a1, m)};
        }
    const ulonglong2 w = make_ulonglong2(fold_sub(yv.x, dot_fold(a0, m), m), fold_sub(yv.y, dot_fold(a1, m), m));
    if (S.vec)
        *reinterpret_cast<ulonglong2 *>(y) = w;
    else
        y[0] = w.x, y[1] = w.y;
}

// multi-switch: src[o] = (X'_0 .. X'_{k-1}) -> w_j = X'_j - sum_{t<j} w_t F[j][t],
// one word a thread: its words of all k limbs loaded first, then the
// recurrence in registers.
__device__ __forceinline__ void fold_multi_block(const FoldSeg &S)
{
    const int N = 1 << S.logN;
    const MultiSwitchParams *P = (const MultiSwitchParams *)S.P;
    const long long idx = (long long)(blockIdx.x - S.b0) * TPB + threadIdx.x;
    if (idx >= S.total) return;
    u64 *b = S.src + (idx >> S.logN) * S.k * N + (idx & (N - 1));
    u64 w[FHE_MAXK];
#pragma unroll
    for (int j = 0; j < FHE_MAXK; j++)
        if (j < S.k) w[j] = b[(long long)j * N];
#pragma unroll
    for (int j = 1; j < FHE_MAXK; j++)
        if (j < S.k) {
            const ModQ &m = S.mq[S.l - 1 - j];
            DotAcc a{0, 0};
#pragma unroll
            for (int t = 0; t < FHE_MAXK; t++)
                if (t < j) {
                    dot_mac(a, w[t], P->F[j][t], m.half);
                    if (m.half > 27 && (t & 1)) a = DotAcc{0, dot_fold(a, m)};
                }
            w[j] = fold_sub(w[j], dot_fold(a, m), m);
            b[(long long)j * N] = w[j];
        }
}

template <class Tb>
__global__ void __launch_bounds__(TPB) k_fold_many(const __grid_constant__ Tb t)
{
    pdl_begin();
    const FoldSeg &S = t.s[block_seg(t)];
    if (t.rms)
        fold_rms_block(S);
    else
        fold_multi_block(S);
}

int ew_blocks(long long total, int elems) { return (int)((total + elems - 1) / elems); }

// Launches a kernel over items[i ..) as one table Tb; fill sets a segment from
// an item and returns its blocks (0 = nothing to do) and its algorithmic
// bytes.  Returns the first item behind the table.
template <class Tb, class Item, class Fill, class Launch>
size_t launch_table(const std::vector<Item> &items, size_t i, int cls, const Fill &fill, const Launch &launch)
{
    Tb t;
    memset(&t, 0, sizeof(t));
    fhe_ctx *c = items[i].c;
    int blocks = 0;
    double bytes = 0;
    for (; i < items.size() && t.nseg < Tb::cap; i++) {
        double b = 0;
        const int nb = fill(t.s[t.nseg], items[i], Tb::elems, &b);
        if (nb <= 0) continue;
        t.s[t.nseg].b0 = blocks;
        blocks += nb;
        bytes += b;
        t.nseg++;
    }
    if (!t.nseg) return i;
    prof_begin(c, cls, bytes);
    launch(t, pdl_on(c, blocks, TPB), blocks, c->stream);
    prof_end(c);
    c->launches++;
    return i;
}

template <class Seg, class Item, class Fill, class Launch>
void launch_tables(const std::vector<Item> &items, int cls, const Fill &fill, const Launch &launch)
{
    for (size_t i = 0; i < items.size();) i = launch_table<Table<Seg, FHE_SEGS>>(items, i, cls, fill, launch);
}

}  // namespace

// q_max sum |k_j| < 2^64 over the item's scalars: its combination fits 64 bits
static bool fits64(const EwArgs &a)
{
    u64 qmax = 0;
    for (u64 q : a.c->q) qmax = q > qmax ? q : qmax;
    const int nk = a.op == FHE_EW_LINCOMB ? a.n : 1;
    unsigned __int128 ksum = 0;
    for (int j = 0; j < nk && j < 8; j++) ksum += (u64)(a.k[j] < 0 ? -a.k[j] : a.k[j]);
    return small_fits(qmax, ksum);
}

// Linear combinations over the same operands, as many as fit one segment
// (LC_N operands in all, LC_N outputs): at least two items.
struct LcItem {
    fhe_ctx *c;
    std::vector<const EwArgs *> of;
    std::vector<const u64 *> x;
};

// Takes the combinations that share operands out of `items`.
static std::vector<LcItem> shared_lincombs(const std::vector<EwArgs> &items, std::vector<EwArgs> &rest)
{
    std::vector<LcItem> open;
    for (const EwArgs &a : items) {
        if (a.op != FHE_EW_LINCOMB || a.n < 1 || !fits64(a)) {
            rest.push_back(a);
            continue;
        }
        LcItem *to = nullptr;
        for (LcItem &g : open) {
            const EwArgs &b = *g.of[0];
            if (g.c != a.c || b.level != a.level || b.outer != a.outer || (int)g.of.size() == LC_N) continue;
            int fresh = 0;
            for (int j = 0; j < a.n; j++) fresh += std::find(g.x.begin(), g.x.end(), a.x[j]) == g.x.end();
            if (fresh < a.n && (int)g.x.size() + fresh <= LC_N) {
                to = &g;
                break;
            }
        }
        if (!to) {
            open.push_back(LcItem{a.c, {}, {}});
            to = &open.back();
        }
        for (int j = 0; j < a.n; j++)
            if (std::find(to->x.begin(), to->x.end(), a.x[j]) == to->x.end()) to->x.push_back(a.x[j]);
        to->of.push_back(&a);
    }
    std::vector<LcItem> got;
    for (LcItem &g : open)
        if (g.of.size() > 1)
            got.push_back(g);
        else
            rest.push_back(*g.of[0]);
    return got;
}

void launch_ew_many(const std::vector<EwArgs> &all)
{
    std::vector<EwArgs> rest;
    std::vector<LcItem> shared;
    if (all.size() > 1) shared = shared_lincombs(all, rest);
    const std::vector<EwArgs> &items = all.size() > 1 ? rest : all;
    launch_tables<LcSeg>(
        shared, FHE_K_ELEMWISE,
        [](LcSeg &S, const LcItem &g, int elems, double *bytes) {
            const EwArgs &a = *g.of[0];
            S.total = (long long)a.outer * a.level * a.c->N;
            if (S.total <= 0) return 0;
            bool vec = true;
            S.n = (int)g.x.size();
            for (int t = 0; t < S.n; t++) {
                S.x[t] = g.x[t];
                vec = vec && ((uintptr_t)g.x[t] & 15) == 0;
            }
            S.nout = (int)g.of.size();
            for (int o = 0; o < S.nout; o++) {
                const EwArgs &b = *g.of[o];
                S.out[o] = b.out;
                vec = vec && ((uintptr_t)b.out & 15) == 0;
                for (int j = 0; j < b.n; j++) {  // an operand may occur more than once
                    const int t = (int)(std::find(g.x.begin(), g.x.end(), b.x[j]) - g.x.begin());
                    S.k[o][t] += (int32_t)b.k[j];
                }
                for (int t = 0; t < S.n; t++)
                    if (S.k[o][t] < 0) S.neg[o] += (uint32_t)-S.k[o][t];
            }
            S.mq = a.c->d_mq;
            S.logN = a.c->logN;
            S.level = a.level;
            S.vec = vec;
            *bytes = 8.0 * (S.n + S.nout) * S.total;
            return ew_blocks(S.total, elems);
        },
        [](const auto &t, bool pdl, int blocks, cudaStream_t s) {
            launch_pdl(k_lincomb_many<std::decay_t<decltype(t)>>, pdl, blocks, TPB, s, t);
        });
    auto fill = [](EwSeg &S, const EwArgs &a, int elems, double *bytes) {
        S.total = (long long)a.outer * a.level * a.c->N;
        if (S.total <= 0) return 0;
        for (int j = 0; j < 8; j++) S.x[j] = a.x[j], S.k[j] = a.k[j];
        S.out = a.out;
        S.mq = a.c->d_mq;
        S.logN = a.c->logN;
        S.level = a.level;
        S.n = a.n;
        S.op = a.op;
        bool vec = ((uintptr_t)a.out & 15) == 0;
        for (int j = 0; j < 8; j++) vec = vec && ((uintptr_t)a.x[j] & 15) == 0;
        S.vec = vec;
        S.small = (a.op == FHE_EW_LINCOMB || a.op == FHE_EW_CMUL) && fits64(a);
        const int reads = a.op == FHE_EW_LINCOMB ? a.n : (a.op == FHE_EW_ADD || a.op == FHE_EW_SUB) ? 2 : 1;
        *bytes = 8.0 * (reads + 1) * S.total;
        return ew_blocks(S.total, elems);
    };
    auto launch = [](const auto &t, bool pdl, int blocks, cudaStream_t s) {
        launch_pdl(k_ew_many<std::decay_t<decltype(t)>>, pdl, blocks, TPB, s, t);
    };
    if (items.size() == 1)
        launch_table<Table<EwSeg, 1>>(items, 0, FHE_K_ELEMWISE, fill, launch);
    else
        launch_tables<EwSeg>(items, FHE_K_ELEMWISE, fill, launch);
}

void launch_tensor_many(const std::vector<TensorArgs> &items)
{
    auto fill = [](TensorSeg &S, const TensorArgs &a, int elems, double *bytes) {
        S.total = (long long)a.count * a.level * a.c->N;
        if (S.total <= 0) return 0;
        S.a = a.a;
        S.b = a.b;
        S.out = a.out;
        S.mq = a.c->d_mq;
        S.logN = a.c->logN;
        S.level = a.level;
        S.vec = (((uintptr_t)a.a | (uintptr_t)a.b | (uintptr_t)a.out) & 15) == 0;
        *bytes = 8.0 * 7 * S.total;
        return ew_blocks(S.total, elems);
    };
    auto launch = [](const auto &t, bool pdl, int blocks, cudaStream_t s) {
        launch_pdl(k_tensor_many<std::decay_t<decltype(t)>>, pdl, blocks, TPB, s, t);
    };
    // one batch of at most two blocks per SM: blocks of half the elements,
    // whose second step would only wait for the first (one ciphertext at
    // N = 2^10, alone: 12.5 us with whole blocks, 11.5 with halves; larger
    // batches are better off with whole ones, 48 at N = 2^15 262 against 277)
    if (items.size() == 1 &&
        (long long)items[0].count * items[0].level * items[0].c->N <= 2LL * EW_ELEMS * items[0].c->sms)
        launch_table<Table<TensorSeg, 1, EW_ELEMS / 2>>(items, 0, FHE_K_TENSOR, fill, launch);
    else
        launch_tables<TensorSeg>(items, FHE_K_TENSOR, fill, launch);
}

// shared memory of a block for dnum digits
static int ks_bytes(int dnum) { return (int)sizeof(u64) * dnum * (2 + KS_CB) * TPB; }

void launch_ks_inner_many(const std::vector<KsInnerArgs> &items)
{
    // items of one key and level side by side (a run); an item keeps its
    // place otherwise
    std::vector<KsInnerArgs> a;
    std::vector<char> taken(items.size(), 0);
    for (size_t i = 0; i < items.size(); i++) {
        if (taken[i] || items[i].count <= 0) continue;
        for (size_t j = i; j < items.size(); j++)
            if (!taken[j] && items[j].count > 0 && items[j].c == items[i].c && items[j].ksk == items[i].ksk &&
                items[j].level == items[i].level) {
                a.push_back(items[j]);
                taken[j] = 1;
            }
    }
    for (size_t i = 0; i < a.size();) {
        KsTable t;
        memset(&t, 0, sizeof(t));
        fhe_ctx *c0 = a[i].c;
        int blocks = 0, dmax = 0;
        double bytes = 0;
        while (i < a.size() && t.nseg < FHE_SEGS) {
            fhe_ctx *c = a[i].c;
            const int level = a[i].level, dnum = c->modup[level].dnum, lead = t.nseg;
            const u64 *key = a[i].ksk;
            dmax = std::max(dmax, dnum);
            const int b0 = blocks;
            int run = 0;
            for (; i < a.size() && t.nseg < FHE_SEGS && a[i].c == c && a[i].ksk == key && a[i].level == level; i++) {
                KsSeg &S = t.s[t.nseg++];
                S.ext = a[i].ext;
                S.xbase = a[i].xbase;
                S.ksk = key;
                S.acc = a[i].acc;
                S.mq = c->d_mq;
                S.x_outer = a[i].x_outer;
                S.count = a[i].count;
                S.l = level;
                S.K = c->K;
                S.L = c->L;
                S.dnum = dnum;
                S.logN = c->logN;
                S.nbx = (c->N + TPB - 1) / TPB;
                run += a[i].count;
            }
            blocks += t.s[lead].nbx * (level + c->K) * ((run + KS_CB - 1) / KS_CB);
            // the items behind the leader own no blocks
            for (int s = lead; s < t.nseg; s++) t.s[s].b0 = s == lead ? b0 : blocks;
            t.s[lead].run = run;
            // per (r, n): 2 dnum key words once per CB ciphertexts, dnum inputs and 2 outputs per ciphertext
            bytes += 8.0 * (double)(level + c->K) * c->N * (2.0 * dnum + run * (dnum + 2.0));
        }
        prof_begin(c0, FHE_K_KS_INNER, bytes);
        // per device, once: more than 48 KB of dynamic shared memory
        static std::mutex mu;
        static bool allowed[64] = {false};
        {
            std::lock_guard<std::mutex> g(mu);
            const int dev = c0->device >= 0 && c0->device < 64 ? c0->device : 0;
            if (!allowed[dev])
                allowed[dev] = cudaFuncSetAttribute(k_ks_inner_many, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    ks_bytes(FHE_MAXD)) == cudaSuccess;
        }
        launch_pdl_smem(k_ks_inner_many, pdl_on(c0, blocks, TPB), blocks, TPB, ks_bytes(dmax), c0->stream, t);
        prof_end(c0);
        c0->launches++;
    }
}

void launch_ks_inner(fhe_ctx *c, const u64 *ext, const u64 *xbase, long long x_outer, const u64 *ksk, u64 *acc,
                     int count, int level)
{
    launch_ks_inner_many({KsInnerArgs{c, ext, xbase, x_outer, ksk, acc, count, level}});
}

void launch_rms_fold_many(const std::vector<FoldArgs> &items)
{
    launch_tables<FoldSeg>(
        items, FHE_K_ELEMWISE,
        [](FoldSeg &S, const FoldArgs &a, int, double *bytes) {
            fhe_ctx *c = a.c;
            S.total = (long long)a.outer * 2 * c->N;  // (ct, poly) pairs
            if (S.total <= 0) return 0;
            S.src = a.src;
            S.mq = c->d_mq;
            S.P = c->d_rms + a.level;
            S.logN = c->logN;
            S.l = a.level;
            S.K = c->K;
            S.vec = ((uintptr_t)a.src & 15) == 0;
            *bytes = 8.0 * (c->K + 2.0) * S.total;
            return (int)(S.total / FOLD_ELEMS);
        },
        [](auto &t, bool pdl, int blocks, cudaStream_t s) {
            t.rms = 1;
            launch_pdl(k_fold_many<std::decay_t<decltype(t)>>, pdl, blocks, TPB, s, t);
        });
}

void launch_rms_fold(fhe_ctx *c, u64 *src, int count, int level)
{
    launch_rms_fold_many({FoldArgs{c, src, count, level, 0}});
}

void launch_ms_fold(fhe_ctx *c, u64 *src, int outer, int level, int k)
{
    launch_ms_fold_many({FoldArgs{c, src, outer, level, k}});
}

void launch_tensor(fhe_ctx *c, const u64 *a, const u64 *b, u64 *out, int count, int level)
{
    launch_tensor_many({TensorArgs{c, a, b, out, count, level}});
}

void launch_add(fhe_ctx *c, const u64 *a, const u64 *b, u64 *out, int outer, int level, int sub)
{
    launch_ew_many({EwArgs{c, sub ? FHE_EW_SUB : FHE_EW_ADD, 2, {a, b}, {}, out, outer, level}});
}

void launch_ms_fold_many(const std::vector<FoldArgs> &items)
{
    launch_tables<FoldSeg>(
        items, FHE_K_ELEMWISE,
        [](FoldSeg &S, const FoldArgs &a, int, double *bytes) {
            fhe_ctx *c = a.c;
            S.total = (long long)a.outer * c->N;
            if (S.total <= 0 || a.k < 2) return 0;
            S.src = a.src;
            S.mq = c->d_mq;
            S.P = c->d_mss + (size_t)a.level * (FHE_MAXK + 1) + a.k;
            S.logN = c->logN;
            S.l = a.level;
            S.k = a.k;
            *bytes = 8.0 * 2.0 * a.k * S.total;
            return (int)((S.total + TPB - 1) / TPB);
        },
        [](auto &t, bool pdl, int blocks, cudaStream_t s) {
            t.rms = 0;
            launch_pdl(k_fold_many<std::decay_t<decltype(t)>>, pdl, blocks, TPB, s, t);
        });
}
