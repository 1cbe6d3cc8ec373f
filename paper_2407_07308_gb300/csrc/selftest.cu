// selftest.cu -- host checks of the NTT engine, run without a GPU: they call
// the engine's own functions (ntt_engine.cuh), so that they hold for what the
// launches and kernels do.
#include "ntt_engine.cuh"

// Which payloads may stand side by side in one segment: a row unit takes its
// prime, constants and whether there is an addend from its first jobs.
extern "C" int fhe_selftest_ntt_joins(void)
{
    int bad = 0;
    YSeg a;
    memset(&a, 0, sizeof(a));
    a.prime[0] = 7;
    a.prime[1] = 3;
    a.Pm = 11;
    a.qm = 13;
    a.amask = 3;
    YSeg b = a;
    b.in_limb[1] = 5;  // places and buffers may differ
    b.in_outer = 1 << 20;
    b.a_poly = 1 << 10;
    bad += !joins(a, b);
    for (int mask = 0; mask < 3; mask++) {
        b = a;
        b.amask = mask;
        bad += joins(a, b) || joins(b, a);
    }
    b = a, b.prime[1] = 4, bad += joins(a, b);
    b = a, b.Pm = 12, bad += joins(a, b);
    b = a, b.qm = 17, bad += joins(a, b);
    RelinMSSeg x, y;  // the others: one context and level, that is one constant table
    memset(&x, 0, sizeof(x));
    y = x;
    bad += !joins(x, y);
    y.P = reinterpret_cast<const RelinMSParams *>(&y);
    bad += joins(x, y);
    return bad;
}

// The batch the autotuner times and what each grid policy makes of it.
extern "C" int fhe_selftest_ntt_tune(int log_n, int nprimes, int sms, int njobs, int32_t *out)
{
    if (!ntt_supported_logn(log_n) || nprimes < 1 || nprimes > FHE_MAXP || sms < 1 || njobs < 1 || !out)
        return FHE_EINVAL;
    SegHdr H;
    memset(&H, 0, sizeof(H));
    H.logN = log_n;
    H.nl = std::min(nprimes, 10);
    H.outer = tune_outer(log_n, H.nl, sms, njobs);
    unit_counts(H);
    out[0] = H.outer * H.nl;
    out[1] = one_kernel(log_n, sms, false, out[0]);
    for (int v = 0; v < FHE_NTT_VARIANTS; v++) {
        out[2 + v] = grid_of(v, sms, H.u_cols);
        out[2 + FHE_NTT_VARIANTS + v] = grid_of(v, sms, H.u_rows);
    }
    return 0;
}
