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

// ---------------------------------------------------------------------------
// arithmetic: one pass over a limb, thread by thread, with the kernels' rounds,
// twiddle accessors, layouts and closing reductions
// ---------------------------------------------------------------------------

namespace {

struct Limb {
    const u64 *in;
    u64 *out;
    std::vector<char> set;
    int bad = 0;
    Limb(const u64 *i, u64 *o, int N) : in(i), out(o), set(N, 0) {}
    void put(int i, u64 v)  // several slots of a unit hold the same limb
    {
        bad += set[i] && out[i] != v;
        out[i] = v;
        set[i] = 1;
    }
};

template <int L, bool FWD, int XJ>
void pass_cols(Limb &io, const ModQ &m, const ulonglong2 *tw, ulonglong2 ninv)
{
    constexpr int N1 = Deg<L>::N1, N2 = Deg<L>::N2;
    using Gm = ColGeo<N1, N2, XJ>;
    using C = typename Gm::C;
    std::vector<u64> sm(Gm::Lay::WORDS);
    std::vector<ulonglong2> W(Gm::TW);
    for (int j = 0; j < Gm::NJ; j++)
        for (int i = 0; i < (1 << N1); i++) W[j * Gm::TWC + twp(i)] = tw[i];
    const ColTw<N1, N2, XJ> geo{W.data(), m.q, m.q, &m, &m};
    for (int lu = 0; lu < Gm::BLK; lu++)
        for (int half = 0; half < 2; half++)  // before and after the exchange
            for (int t = 0; t < T; t++) {
                const int c = t % C::NS, g = t / C::NS, lo = Gm::lo0(lu) + c % Gm::NC;
                u64 *b = sm.data() + Gm::Lay::base(c), x[16];
                if (FWD && half == 0) {
                    for (int k = 0; k < 16; k++) x[k] = io.in[((k * C::G + g) << N2) + lo];
                    round1<N1, true>(x, geo, c);
                    put1<C::G>(b + g, x);
                } else if (FWD) {
                    get2(b + 17 * g, x);
                    round2<N1, true>(x, geo, c, g);
                    for (int k = 0; k < 16; k++) io.put((((g << 4) + k) << N2) + lo, x[k]);
                } else if (half == 0) {
                    for (int k = 0; k < 16; k++) x[k] = io.in[(((g << 4) + k) << N2) + lo];
                    round2<N1, false>(x, geo, c, g);
                    put2(b + 17 * g, x);
                } else {
                    get1<C::G>(b + g, x);
                    round1<N1, false>(x, geo, c);
                    for (int k = 0; k < 16; k++) io.put(((k * C::G + g) << N2) + lo, inv_scaled(x[k], ninv, m));
                }
            }
}

template <int L, bool FWD, bool GRP>
void pass_rows(Limb &io, const ModQ &m, const ulonglong2 *tw)
{
    constexpr int N1 = Deg<L>::N1, N2 = Deg<L>::N2;
    using Gm = RowGeo<N1, N2>;
    using C = typename Gm::C;
    using Lay = typename Gm::Lay;
    std::vector<u64> sm(Lay::WORDS);
    std::vector<ulonglong2> W(TW_ROWS);
    for (int lu = 0; lu < (GRP ? Gm::CH : Gm::CHS); lu++) {
        const int hi0 = lu * (GRP ? Gm::R : Gm::NS);
        const RowMap<N1, N2, GRP> mp{hi0};
        for (int r = 0; r < (GRP ? Gm::R : 0); r++)
            for (int e = 0; e < Gm::SZ - 1; e++) {
                int u = 0;
                while ((2 << u) <= e + 1) u++;
                W[r * Gm::TWR + twp(e)] = tw[(1 << (N1 + u)) + ((hi0 + r) << u) + (e + 1 - (1 << u))];
            }
        const RowGrpTw<N1, N2> grp{W.data(), hi0, m, N1};
        const RowOneTw one{GTw{tw}, hi0, m, N1};
        auto first = [&](u64(&x)[16], int c) {
            if constexpr (GRP)
                round1<N2, FWD>(x, grp, c);
            else
                round1<N2, FWD>(x, one, c);
        };
        auto second = [&](u64(&x)[16], int c, int g) {
            if constexpr (GRP)
                round2<N2, FWD>(x, grp, c, g);
            else
                round2<N2, FWD>(x, one, c, g);
        };
        for (int half = 0; half < 2; half++)
            for (int t = 0; t < T; t++) {
                const int c = t / C::G, g = t % C::G, row = mp.crow(c) << N2;
                u64 *b = sm.data() + Lay::base(c), x[16];
                if (FWD && half == 0) {
                    for (int k = 0; k < 16; k++) x[k] = io.in[row + k * C::G + g];
                    first(x, c);
                    put1<C::G>(b + g, x);
                } else if (FWD) {
                    get2(b + 17 * g, x);
                    second(x, c, g);
                    for (int k = 0; k < 16; k++) io.put(row + 16 * g + k, reduce2q(reduce_few(x[k], m), m.q));
                } else if (half == 0) {
                    for (int k = 0; k < 16; k++) x[k] = io.in[row + 16 * g + k];
                    second(x, c, g);
                    put2(b + 17 * g, x);
                } else {
                    get1<C::G>(b + g, x);
                    first(x, c);
                    for (int k = 0; k < 16; k++) io.put(row + k * C::G + g, k < 8 ? reduce_few(x[k], m) : x[k]);
                }
            }
    }
}

template <int L>
int run_pass(u64 q, int pass, const u64 *in, u64 *out)
{
    const int N = 1 << L;
    std::vector<ulonglong2> fwd(N), inv(N);
    ulonglong2 ninv;
    limb_tables(q, L, fwd.data(), inv.data(), &ninv);
    const ModQ m = make_modq(q);
    Limb io(in, out, N);
    switch (pass) {
    case 0:
        pass_cols<L, true, 1>(io, m, fwd.data(), ninv);
        pass_cols<L, true, 2>(io, m, fwd.data(), ninv);
        break;
    case 1:
        pass_rows<L, true, true>(io, m, fwd.data());
        if (L > 10) pass_rows<L, true, false>(io, m, fwd.data());  // n = 10 has grouped units only
        break;
    case 2:
        pass_rows<L, false, true>(io, m, inv.data());
        if (L > 10) pass_rows<L, false, false>(io, m, inv.data());
        break;
    default:
        pass_cols<L, false, 1>(io, m, inv.data(), ninv);
        pass_cols<L, false, 2>(io, m, inv.data(), ninv);
    }
    for (char s : io.set) io.bad += !s;
    return io.bad;
}

}  // namespace

extern "C" int fhe_selftest_ntt_pass(int log_n, uint64_t q, int pass, const uint64_t *in, uint64_t *out)
{
    if (!in || !out || pass < 0 || pass > 3 || !ntt_supported_logn(log_n) || q >> 57 || (q - 1) % (2ull << log_n) ||
        !host_is_prime(q))
        return FHE_EINVAL;
    switch (log_n) {
    case 10: return run_pass<10>(q, pass, in, out);
    case 11: return run_pass<11>(q, pass, in, out);
    case 12: return run_pass<12>(q, pass, in, out);
    case 13: return run_pass<13>(q, pass, in, out);
    case 14: return run_pass<14>(q, pass, in, out);
    default: return run_pass<15>(q, pass, in, out);
    }
}
