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

// ---------------------------------------------------------------------------
// units and layouts
// ---------------------------------------------------------------------------

namespace {

// how often each residue of each limb is touched
struct Cover {
    int logN, limbs;
    std::vector<uint8_t> seen;
    int bad = 0;
    Cover(int n, int l) : logN(n), limbs(l), seen((size_t)l << n, 0) {}
    void touch(int job, int pos)
    {
        if (job < 0 || job >= limbs || pos < 0 || pos >> logN)
            bad++;
        else
            seen[((size_t)job << logN) + pos]++;
    }
    int misses() const
    {
        int n = bad;
        for (uint8_t x : seen) n += x != 1;
        return n;
    }
};

SegHdr header(int logN, int outer, int nl, int xj)
{
    SegHdr H;
    memset(&H, 0, sizeof(H));
    H.logN = logN;
    H.outer = H.per = outer;
    H.nl = nl;
    H.xj = xj;
    unit_counts(H);
    return H;
}

template <int L, int XJ>
int cover_cols(const SegHdr &H)
{
    using Gm = ColGeo<Deg<L>::N1, Deg<L>::N2, XJ>;
    const int njobs = H.outer * H.nl;
    Cover cv(L, njobs);
    for (int lu = 0; lu < H.u_cols; lu++)
        for (int c = 0; c < Gm::NS; c++) {
            const int job = Gm::job0(lu) + c / Gm::NC;
            if (job >= njobs) continue;  // a slot without a job
            for (int e = 0; e < Gm::SZ; e++) cv.touch(job, (e << Deg<L>::N2) + Gm::lo0(lu) + c % Gm::NC);
        }
    return cv.misses();
}

template <int L, bool GRP>
void touch_rows(const SegHdr &H, int lu, Cover &cv)
{
    const RowUnit<Deg<L>::N1, Deg<L>::N2, GRP> u(H, lu);
    const RowMap<Deg<L>::N1, Deg<L>::N2, GRP> mp{u.hi0};
    for (int jj = 0; jj < u.nvalid; jj++) cv.bad += u.job(H, jj) % H.nl != u.job(H, 0) % H.nl;  // one prime
    for (int r = 0; r < 16 * T; r++)
        if (mp.slot(r) < u.nvalid) cv.touch(u.job(H, mp.slot(r)), (mp.row(r) << Deg<L>::N2) + mp.f(r));
}

template <int L>
int check_units(int outer, int nl)
{
    int bad = 0;
    SegHdr H = header(L, outer, nl, 0);
    bad += cover_cols<L, 1>(H);
    Cover rows(L, outer * nl);
    for (int lu = 0; lu < H.u_rows; lu++)
        if (lu < H.g_units)
            touch_rows<L, true>(H, lu, rows);
        else
            touch_rows<L, false>(H, lu, rows);
    bad += rows.misses();
    bad += cover_cols<L, 2>(header(L, outer, nl, 2));
    if constexpr (L >= SMALL_LO && L <= SMALL_HI) {
        // one kernel: a CTA's column unit and row unit belong to one limb, and
        // a limb's units to one cluster
        using Col = typename SmallGeo<L>::Col;
        const int first = 3 * SMALL_CTAS<L>;
        bad += one_kernel_units(H, first) != first + SMALL_CTAS<L> * outer * nl || H.u_cols != first || H.u_rows != first;
        Cover cols(L, outer * nl), small(L, outer * nl);
        for (int lu = 0; lu < SMALL_CTAS<L> * outer * nl; lu++) {
            bad += RowUnit<Deg<L>::N1, Deg<L>::N2, false>(H, lu).job(H, 0) != Col::job0(lu) ||
                   Col::job0(lu) != lu / SMALL_CTAS<L>;
            touch_rows<L, false>(H, lu, small);
            for (int c = 0; c < Col::NS; c++)
                for (int e = 0; e < Col::SZ; e++) cols.touch(Col::job0(lu), (e << Deg<L>::N2) + Col::lo0(lu) + c);
        }
        bad += cols.misses() + small.misses();
    }
    return bad;
}

// A layout of a unit's sub-transforms keeps their elements apart inside its
// words, and a thread's exchanges go to the elements of its rounds.
template <int M, class Lay>
int check_layout()
{
    using C = Sub<M>;
    int bad = 0;
    std::vector<int> at(Lay::WORDS, -1);
    for (int c = 0; c < C::NS; c++)
        for (int e = 0; e < C::SZ; e++) {
            const int w = Lay::at(c, e);
            if (w < 0 || w >= Lay::WORDS || at[w] >= 0) {
                bad++;
                continue;
            }
            at[w] = c * C::SZ + e;
        }
    std::vector<u64> sm(Lay::WORDS);
    for (int c = 0; c < C::NS; c++)
        for (int g = 0; g < C::G; g++) {
            u64 x[16], y[16];
            u64 *b = sm.data() + Lay::base(c);
            for (int k = 0; k < 16; k++) x[k] = 1000 * c + 20 * g + k + 1;
            put1<C::G>(b + g, x);
            get1<C::G>(b + g, y);
            for (int k = 0; k < 16; k++) bad += sm[Lay::at(c, k * C::G + g)] != x[k] || y[k] != x[k];
            put2(b + 17 * g, x);
            get2(b + 17 * g, y);
            for (int k = 0; k < 16; k++) bad += sm[Lay::at(c, 16 * g + k)] != x[k] || y[k] != x[k];
        }
    return bad;
}

template <int M>
int check_layouts()
{
    return check_layout<M, ColLay<M, false>>() + check_layout<M, ColLay<M, true>>() +
           (M < 8 ? check_layout<M, RowLay<(M < 8 ? M : 7)>>() : 0);
}

// Payloads side by side: every job of a joined segment finds its payload and
// its place in it.
int check_payloads()
{
    int bad = 0;
    std::unique_ptr<IOMap> io(new IOMap);
    memset(io.get(), 0, sizeof(IOMap));
    const int nl = 3, per[2] = {4, 1}, parts[2] = {3, 5};
    for (int sg = 0, first = 0; sg < 2; first += parts[sg++]) {
        SegHdr &H = io->h[sg];
        H.nl = nl;
        H.per = per[sg];
        H.outer = per[sg] * parts[sg];
        H.first = first;
        for (int job = 0; job < H.outer * nl; job++) {
            int in = job;
            const MapSeg *p = &io->payload(sg, in);
            const int o = job / nl;
            bad += p != &io->s[first + o / per[sg]] || in != (o % per[sg]) * nl + job % nl;
        }
    }
    return bad;
}

}  // namespace

extern "C" int fhe_selftest_ntt_units(int log_n, int outer, int nl)
{
    if (outer < 1 || nl < 1 || nl > FHE_MAXP || outer > 4096) return FHE_EINVAL;
    switch (log_n) {
    case 10: return check_units<10>(outer, nl);
    case 11: return check_units<11>(outer, nl);
    case 12: return check_units<12>(outer, nl);
    case 13: return check_units<13>(outer, nl);
    case 14: return check_units<14>(outer, nl);
    case 15: return check_units<15>(outer, nl);
    default: return FHE_EINVAL;
    }
}

extern "C" int fhe_selftest_ntt_layouts(void)
{
    return check_layouts<5>() + check_layouts<6>() + check_layouts<7>() + check_layouts<8>() + check_payloads();
}
