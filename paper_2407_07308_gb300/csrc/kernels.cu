// kernels.cu -- streaming (HBM-bound) kernels on NTT-domain limbs of one batch:
// neg, scalar and constant terms, plaintext operands, Galois automorphisms as
// index permutations (sums, tensor products, inner products and switch folds
// run through many.cu's kernels, as a table of one batch), and small helpers
// for key generation, encryption and decryption.
//
// Layout: a batch of ciphertexts is u64 [count][npoly][level][N]; an "outer"
// index runs over count*npoly polys, and the limb of element idx is
// (idx >> logN) % level, so one flat grid covers the batch and every warp
// reads 256 contiguous bytes.
#include <string.h>

#include "fhe_internal.h"

namespace {

constexpr int TPB = 256;

inline int grid_for(long long n, int per_thread = 1)
{
    long long b = (n + (long long)TPB * per_thread - 1) / ((long long)TPB * per_thread);
    if (b > (1 << 30)) b = 1 << 30;
    return (int)(b > 0 ? b : 1);
}

__global__ void k_neg(const u64 *__restrict__ a, u64 *__restrict__ out, long long total, int logN, int level,
                      const ModQ *__restrict__ mq)
{
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const u64 q = mq[(int)((idx >> logN) % level)].q;
        out[idx] = negmod(a[idx], q);
    }
}

struct LimbConsts {
    u64 w[FHE_MAXP], ws[FHE_MAXP];
};

__global__ void k_mul_const(const u64 *__restrict__ a, u64 *__restrict__ out, long long total, int logN, int level,
                            const ModQ *__restrict__ mq, const LimbConsts k)
{
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int i = (int)((idx >> logN) % level);
        out[idx] = shoup(a[idx], k.w[i], k.ws[i], mq[i].q);
    }
}

// Adds the constant k_i (mod q_i) at every NTT point of poly 0; copies poly 1.
__global__ void k_add_const(const u64 *__restrict__ a, u64 *__restrict__ out, long long total, int logN, int level,
                            const ModQ *__restrict__ mq, const LimbConsts k)
{
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long li = idx >> logN;
        const int i = (int)(li % level);
        const int poly = (int)((li / level) % 2);
        out[idx] = poly == 0 ? addmod(a[idx], k.w[i], mq[i].q) : a[idx];
    }
}

// c0 of every ciphertext of a batch plus / minus one plaintext m[level][N]
// (NTT domain); c1 and further polynomials are left as they are (the caller
// copied them).  out may equal a.
__global__ void k_add_plain(const u64 *__restrict__ a, const u64 *__restrict__ m, u64 *__restrict__ out,
                            long long total, int logN, int level, long long ct_stride, int sub,
                            const ModQ *__restrict__ mq)
{
    const long long LN = (long long)level << logN;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long c = idx / LN, r = idx % LN;
        const u64 q = mq[(int)(r >> logN)].q;
        const u64 x = a[c * ct_stride + r], y = m[r];
        out[c * ct_stride + r] = sub ? submod(x, y, q) : addmod(x, y, q);
    }
}

// out[o][i][k] = in[o][i][perm[k]]: sigma_g in the NTT domain.
__global__ void k_automorphism(const u64 *__restrict__ in, u64 *__restrict__ out, long long total, int logN,
                               const int *__restrict__ perm)
{
    const int mask = (1 << logN) - 1;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long base = idx & ~(long long)mask;
        out[idx] = in[base + perm[idx & mask]];
    }
}

// out[o][i] = a[o][i] * b[o'][i] pointwise, b's outer stride b_outer (0 = broadcast).
__global__ void k_mul_poly(const u64 *__restrict__ a, const u64 *__restrict__ b, u64 *__restrict__ out,
                           long long total, int logN, int level, long long b_outer, const ModQ *__restrict__ mq)
{
    const long long LN = (long long)level << logN;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long o = idx / LN, r = idx % LN;
        out[idx] = barrett128((u128)a[idx] * b[o * b_outer + r], mq[(int)(r >> logN)]);
    }
}

// out[o][i][n] = scale * x[o][n] mod q_{prime[i]}
__global__ void k_rns_from_i64(const int64_t *__restrict__ x, int64_t scale, u64 *__restrict__ out,
                               long long total, int logN, int nl, const LimbConsts pm, const ModQ *__restrict__ mq)
{
    const int N = 1 << logN;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long li = idx >> logN;
        const int i = (int)(li % nl);
        const long long o = li / nl;
        const int n = (int)(idx & (N - 1));
        const u64 q = mq[(int)pm.w[i]].q;
        const int64_t v = scale * x[o * N + n];
        const int64_t r = v % (int64_t)q;
        out[idx] = (u64)(r < 0 ? r + (int64_t)q : r);
    }
}

// v mod q in [0, q); a sum and a comparison where |v| < q, which all but the
// smallest primes make of p times an error's bound
__device__ __forceinline__ u64 lift(int64_t v, u64 q)
{
    if (v < 0) v += (int64_t)q;
    if ((u64)v < q) return (u64)v;
    const int64_t r = v % (int64_t)q;
    return (u64)(r < 0 ? r + (int64_t)q : r);
}

// The three polynomials of an encryption, out[3][count][L][N]: u, p e0 + m and
// p e1 over the first L primes.  m holds mn coefficients a plaintext, N / mn
// apart.  One launch, and one transform over all three, in place of three of
// each: at one ciphertext every launch is a few microseconds of latency.  A
// client's round trip (encryption of 2 ciphertexts, N = 2^14, 10 primes, in 5
// launches in place of 16; a reply's decryption with M coefficients over the
// bus in place of N) went from 334 to 150 us.
__global__ void k_enc_rns(const int64_t *__restrict__ u, const int64_t *__restrict__ e0, const int64_t *__restrict__ e1,
                          const int64_t *__restrict__ m, int mn, int64_t p, u64 *__restrict__ out, long long total,
                          int logN, int L, const ModQ *__restrict__ mq)
{
    const int N = 1 << logN, gap = N / mn;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long li = idx >> logN, o = li / L;
        const int i = (int)(idx & (N - 1));
        const u64 q = mq[(int)(li - o * L)].q;
        const long long s = o * N + i;
        out[idx] = lift(u[s], q);
        out[total + idx] = lift(p * e0[s] + (i % gap == 0 ? m[o * mn + i / gap] : 0), q);
        out[2 * total + idx] = lift(p * e1[s], q);
    }
}

// ct[o][pi] = t[1 + pi][o] + t[0][o] pk[pi] (NTT domain; t[3][count][L][N]),
// both polynomials written where they belong
__global__ void k_enc_combine(const u64 *__restrict__ t, const u64 *__restrict__ pk, u64 *__restrict__ ct,
                              long long total, int logN, int L, const ModQ *__restrict__ mq)
{
    const long long LN = (long long)L << logN;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long o = idx / LN, r = idx - o * LN;
        const ModQ m = mq[(int)(r >> logN)];
        const u64 u = t[idx];
        u64 *d = ct + 2 * o * LN + r;
        d[0] = addmod(t[total + idx], barrett128((u128)u * pk[r], m), m.q);
        d[LN] = addmod(t[2 * total + idx], barrett128((u128)u * pk[LN + r], m), m.q);
    }
}

// t[o] = c0 + c1 s of two-poly ciphertexts of one limb (NTT domain)
__global__ void k_dec_dot(const u64 *__restrict__ ct, const u64 *__restrict__ s, u64 *__restrict__ t, long long total,
                          int logN, const ModQ *__restrict__ mq)
{
    const int N = 1 << logN;
    const ModQ m = mq[0];
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long o = idx >> logN;
        const int n = (int)(idx & (N - 1));
        t[idx] = addmod(ct[2 * o * N + n], barrett128((u128)ct[(2 * o + 1) * N + n] * s[n], m), m.q);
    }
}

// out = c + a * b (pointwise), b with outer stride b_outer; c may be NULL.
// With neg != 0: out = c - a * b.
__global__ void k_muladd(const u64 *__restrict__ a, const u64 *__restrict__ b, const u64 *__restrict__ cc,
                         u64 *__restrict__ out, long long total, int logN, int level, long long b_outer, int neg,
                         const ModQ *__restrict__ mq)
{
    const long long LN = (long long)level << logN;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long o = idx / LN, r = idx % LN;
        const ModQ m = mq[(int)(r >> logN)];
        const u64 t = barrett128((u128)a[idx] * b[o * b_outer + r], m);
        const u64 base = cc ? cc[idx] : 0;
        out[idx] = neg ? submod(base, t, m.q) : addmod(base, t, m.q);
    }
}

// One digit of a switching key over the L+K primes (NTT domain):
//   k0 = e - a s + [i in D_j] (P mod q_i) s',  k1 = a,
// both stored as the inner product reads them: times 2^(2h) (R) mod q_i, as
// packed half words (half_const).
__global__ void k_ksk_digit(const u64 *__restrict__ a, const u64 *__restrict__ e, const u64 *__restrict__ s,
                            const u64 *__restrict__ sp, u64 *__restrict__ k0, u64 *__restrict__ k1, long long total,
                            int logN, int dlo, int dhi, const LimbConsts Pm, const LimbConsts R,
                            const ModQ *__restrict__ mq)
{
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(idx >> logN);
        const ModQ m = mq[i];
        u64 v = submod(e[idx], barrett128((u128)a[idx] * s[idx], m), m.q);
        if (i >= dlo && i < dhi) v = addmod(v, shoup(sp[idx], Pm.w[i], Pm.ws[i], m.q), m.q);
        k0[idx] = half_pack(shoup(v, R.w[i], R.ws[i], m.q), m.half);
        k1[idx] = half_pack(shoup(a[idx], R.w[i], R.ws[i], m.q), m.half);
    }
}

// Decryption residues (limb 0, canonical mod q0) -> plaintext coefficients:
// the centred representative in (-q0/2, q0/2], reduced mod p into [0, p).
__global__ void k_centre_mod_p(const u64 *__restrict__ x, int64_t *__restrict__ out, long long n, u64 q0, int64_t p)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const u64 v = x[i];
        const int64_t cv = v > q0 / 2 ? -(int64_t)(q0 - v) : (int64_t)v;
        int64_t r = cv % p;
        out[i] = r < 0 ? r + p : r;
    }
}

// The same for plaintexts of a subring (coefficients N / M apart), a block for
// every SUB_RUN coefficients of a ciphertext: out[o][0 .. M) the subring's
// coefficients, then a word a block for whether it met another that is not
// zero.  M words a ciphertext cross the bus in place of N.
constexpr int SUB_RUN = 1024;
__global__ void __launch_bounds__(256)
    k_centre_sub(const u64 *__restrict__ x, int64_t *__restrict__ out, int N, int M, int runs, u64 q0, int64_t p)
{
    const int o = blockIdx.x / runs, b = blockIdx.x % runs;
    const u64 *xo = x + (long long)o * N;
    int64_t *d = out + (long long)o * (M + runs);
    const int gap = N / M, end = min(N, (b + 1) * SUB_RUN);
    int other = 0;
    for (int i = b * SUB_RUN + threadIdx.x; i < end; i += blockDim.x) {
        const u64 v = xo[i];
        const int64_t cv = v > q0 / 2 ? -(int64_t)(q0 - v) : (int64_t)v;
        int64_t r = cv % p;
        if (r < 0) r += p;
        if (i % gap == 0)
            d[i / gap] = r;
        else
            other |= r != 0;
    }
    other = __syncthreads_or(other);
    if (threadIdx.x == 0) d[M + b] = other;
}

// out = sum_t w_t x_t (mod q_i), up to 8 ciphertext batches of one shape;
// w[t][i] is the scalar of term t reduced mod q_i.  Eight products of
// canonical residues stay below the Barrett bound, so one reduction suffices.
struct LinComb {
    const u64 *x[8];
    u64 w[8][FHE_MAXP];
    int n;
};

__global__ void k_lincomb(const LinComb lc, u64 *__restrict__ out, long long total, int logN, int level,
                          const ModQ *__restrict__ mq)
{
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int i = (int)((idx >> logN) % level);
        u128 acc = 0;
#pragma unroll
        for (int t = 0; t < 8; t++)
            if (t < lc.n) acc += (u128)lc.x[t][idx] * lc.w[t][i];
        out[idx] = barrett128(acc, mq[i]);
    }
}

}  // namespace

// words: u64 words read + written per element (algorithmic traffic)
#define LAUNCH_CLS_W(cls, words, kern, total, ...)                                          \
    do {                                                                                    \
        long long _t = (total);                                                             \
        if (_t > 0) {                                                                       \
            prof_begin(c, cls, 8.0 * (words) * (double)_t);                                 \
            kern<<<grid_for(_t), TPB, 0, c->stream>>>(__VA_ARGS__);                         \
            prof_end(c);                                                                    \
            c->launches++;                                                                  \
        }                                                                                   \
    } while (0)
#define LAUNCH_CLS(cls, kern, total, ...) LAUNCH_CLS_W(cls, 2, kern, total, __VA_ARGS__)
#define LAUNCH(kern, total, ...) LAUNCH_CLS_W(FHE_K_ELEMWISE, 2, kern, total, __VA_ARGS__)

void launch_neg(fhe_ctx *c, const u64 *a, u64 *out, int outer, int level)
{
    LAUNCH(k_neg, (long long)outer * level * c->N, a, out, (long long)outer * level * c->N, c->logN, level, c->d_mq);
}

void launch_mul_const(fhe_ctx *c, const u64 *a, u64 *out, int outer, int level, const u64 *w, const u64 *ws)
{
    LimbConsts k;
    for (int i = 0; i < level; i++) k.w[i] = w[i], k.ws[i] = ws[i];
    LAUNCH(k_mul_const, (long long)outer * level * c->N, a, out, (long long)outer * level * c->N, c->logN, level,
           c->d_mq, k);
}

void launch_add_const(fhe_ctx *c, const u64 *a, u64 *out, int count, int level, const u64 *kv)
{
    LimbConsts k;
    for (int i = 0; i < level; i++) k.w[i] = kv[i], k.ws[i] = 0;
    LAUNCH(k_add_const, (long long)count * 2 * level * c->N, a, out, (long long)count * 2 * level * c->N, c->logN,
           level, c->d_mq, k);
}

void launch_automorphism(fhe_ctx *c, const u64 *in, u64 *out, int outer, int level, const int *perm)
{
    LAUNCH_CLS(FHE_K_AUTOMORPHISM, k_automorphism, (long long)outer * level * c->N, in, out, (long long)outer * level * c->N, c->logN, perm);
}

void launch_add_plain(fhe_ctx *c, const u64 *a, const u64 *m, u64 *out, int count, int npoly, int level, int sub)
{
    const long long total = (long long)count * level * c->N;
    LAUNCH_CLS_W(FHE_K_ELEMWISE, 3, k_add_plain, total, a, m, out, total, c->logN, level,
                 (long long)npoly * level * c->N, sub, c->d_mq);
}

void launch_mul_poly(fhe_ctx *c, const u64 *a, const u64 *b, u64 *out, int outer, int level, long long b_outer)
{
    LAUNCH(k_mul_poly, (long long)outer * level * c->N, a, b, out, (long long)outer * level * c->N, c->logN, level,
           b_outer, c->d_mq);
}

void launch_rns_from_i64(fhe_ctx *c, const int64_t *x, int64_t scale, u64 *out, int outer, int nl, const int *primes)
{
    LimbConsts pm;
    for (int i = 0; i < nl; i++) pm.w[i] = (u64)primes[i], pm.ws[i] = 0;
    LAUNCH(k_rns_from_i64, (long long)outer * nl * c->N, x, scale, out, (long long)outer * nl * c->N, c->logN, nl,
           pm, c->d_mq);
}

void launch_muladd(fhe_ctx *c, const u64 *a, const u64 *b, const u64 *cc, u64 *out, int outer, int level,
                   long long b_outer, int neg)
{
    LAUNCH(k_muladd, (long long)outer * level * c->N, a, b, cc, out, (long long)outer * level * c->N, c->logN, level,
           b_outer, neg, c->d_mq);
}

void launch_ksk_digit(fhe_ctx *c, const u64 *a, const u64 *e, const u64 *s, const u64 *sp, u64 *k0, u64 *k1, int dlo,
                      int dhi, const u64 *Pw, const u64 *Pws)
{
    LimbConsts Pm, R;
    for (int i = 0; i < c->np; i++) {
        Pm.w[i] = Pw[i], Pm.ws[i] = Pws[i];
        R.w[i] = (u64)(((u128)1 << (2 * c->mq[i].half)) % c->q[i]);
        R.ws[i] = shoup_const(R.w[i], c->q[i]);
    }
    LAUNCH(k_ksk_digit, (long long)c->np * c->N, a, e, s, sp, k0, k1, (long long)c->np * c->N, c->logN, dlo, dhi, Pm,
           R, c->d_mq);
}

// ---------------------------------------------------------------------------
// per-class event timing
// ---------------------------------------------------------------------------

static cudaEvent_t prof_event(fhe_ctx *c)
{
    if (!c->prof_events.empty()) {
        cudaEvent_t e = c->prof_events.back();
        c->prof_events.pop_back();
        return e;
    }
    cudaEvent_t e;
    cudaEventCreate(&e);
    return e;
}

// Inside a stream capture a plain event record is only a dependency marker;
// recorded as external it becomes an event-record node of the graph.
static void prof_record(fhe_ctx *c, cudaEvent_t e)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(c->stream, &st);
    if (st == cudaStreamCaptureStatusActive)
        cudaEventRecordWithFlags(e, c->stream, cudaEventRecordExternal);
    else
        cudaEventRecord(e, c->stream);
}

void prof_begin(fhe_ctx *c, int cls, double bytes, double bfly)
{
    if (!c->prof_on) return;
    cudaEvent_t a = prof_event(c), b = prof_event(c);
    prof_record(c, a);
    c->prof_rec.push_back({a, b});
    c->prof_rec_cls.push_back(cls);
    c->prof_rec_bytes.push_back(bytes);
    c->prof_rec_bfly.push_back(bfly);
}

void prof_end(fhe_ctx *c)
{
    if (!c->prof_on || c->prof_rec.empty()) return;
    prof_record(c, c->prof_rec.back().second);
}

extern "C" int fhe_ctx_profile(fhe_ctx *c, int on)
{
    if (!c) return FHE_EINVAL;
    c->prof_on = on != 0;
    return 0;
}

extern "C" int fhe_ctx_profile_read(fhe_ctx *c, double *ms, int64_t *count, double *bytes, double *bfly, int ncls)
{
    if (!c || ncls < 0) return FHE_EINVAL;
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) return FHE_ECUDA;
    for (int i = 0; i < ncls; i++) {
        if (ms) ms[i] = 0;
        if (count) count[i] = 0;
        if (bytes) bytes[i] = 0;
        if (bfly) bfly[i] = 0;
    }
    for (size_t r = 0; r < c->prof_rec.size(); r++) {
        float t = 0;
        cudaEventElapsedTime(&t, c->prof_rec[r].first, c->prof_rec[r].second);
        const int k = c->prof_rec_cls[r];
        if (k >= 0 && k < ncls) {
            if (ms) ms[k] += t;
            if (count) count[k] += 1;
            if (bytes) bytes[k] += c->prof_rec_bytes[r];
            if (bfly) bfly[k] += c->prof_rec_bfly[r];
        }
        c->prof_events.push_back(c->prof_rec[r].first);
        c->prof_events.push_back(c->prof_rec[r].second);
    }
    c->prof_rec.clear();
    c->prof_rec_cls.clear();
    c->prof_rec_bytes.clear();
    c->prof_rec_bfly.clear();
    return FHE_K_COUNT;
}

void launch_lincomb(fhe_ctx *c, const u64 *const *x, const u64 (*w)[FHE_MAXP], int n, u64 *out, int outer,
                    int level)
{
    LinComb lc;
    memset(&lc, 0, sizeof(lc));
    lc.n = n;
    for (int t = 0; t < n; t++) {
        lc.x[t] = x[t];
        for (int i = 0; i < level; i++) lc.w[t][i] = w[t][i];
    }
    LAUNCH_CLS_W(FHE_K_ELEMWISE, n + 1, k_lincomb, (long long)outer * level * c->N, lc, out,
                 (long long)outer * level * c->N, c->logN, level, c->d_mq);
}

void launch_centre_mod_p(fhe_ctx *c, const u64 *x, int64_t *out, long long n)
{
    LAUNCH(k_centre_mod_p, n, x, out, n, c->q[0], (int64_t)c->p);
}

void launch_enc_rns(fhe_ctx *c, const int64_t *u, const int64_t *e0, const int64_t *e1, const int64_t *m, int mn,
                    u64 *out, int count, int level)
{
    const long long total = (long long)count * level * c->N;
    LAUNCH_CLS_W(FHE_K_ELEMWISE, 3 + 3.0 / level, k_enc_rns, total, u, e0, e1, m, mn, (int64_t)c->p, out, total,
                 c->logN, level, c->d_mq);
}

void launch_enc_combine(fhe_ctx *c, const u64 *t, const u64 *pk, u64 *ct, int count, int level)
{
    const long long total = (long long)count * level * c->N;
    LAUNCH_CLS_W(FHE_K_ELEMWISE, 5 + 2.0 / count, k_enc_combine, total, t, pk, ct, total, c->logN, level, c->d_mq);
}

void launch_dec_dot(fhe_ctx *c, const u64 *ct, const u64 *s, u64 *t, int count)
{
    const long long total = (long long)count * c->N;
    LAUNCH_CLS_W(FHE_K_ELEMWISE, 3 + 1.0 / count, k_dec_dot, total, ct, s, t, total, c->logN, c->d_mq);
}

int centre_sub_runs(const fhe_ctx *c) { return (c->N + SUB_RUN - 1) / SUB_RUN; }

void launch_centre_sub(fhe_ctx *c, const u64 *x, int64_t *out, int count)
{
    if (count < 1) return;
    const int runs = centre_sub_runs(c);
    prof_begin(c, FHE_K_ELEMWISE, 8.0 * count * (c->N + c->M + runs));
    k_centre_sub<<<count * runs, 256, 0, c->stream>>>(x, out, c->N, c->M, runs, c->q[0], (int64_t)c->p);
    prof_end(c);
    c->launches++;
}
