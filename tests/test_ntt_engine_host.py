"""The NTT engine's own host functions and templates, run on the CPU through the
library's self-tests."""
import numpy as np
import pytest

from oracle.bgv import Oracle


@pytest.fixture(scope="module")
def fhe():
    from paper_2407_07308_gb300 import build

    build.build()
    from paper_2407_07308_gb300 import fhe as f

    return f


def test_segments_join_only_what_shares_a_unit(fhe):
    """Batches of one segment share row units, which look at their first jobs
    only: a batch with an addend and one without (or with it on another
    polynomial) stay apart, as do other primes and constants."""
    assert fhe.fhe_selftest_ntt_joins() == 0


@pytest.mark.parametrize("sms", [148, 152])
@pytest.mark.parametrize("nprimes", [2, 5, 13, 24])
@pytest.mark.parametrize("logN", [10, 11, 12, 13, 14, 15])
def test_autotuner_times_batches_that_tell_the_policies_apart(fhe, logN, nprimes, sms):
    """Whatever is asked for, the timed batch runs in two passes (launches in
    one kernel have no grid policy) and every policy gives it a grid of its
    own; from the default request up, a batch that does so already stays."""
    nl = min(nprimes, 10)
    for njobs in (1, 64, 320, 5000):
        limbs, one, cols, rows = fhe.fhe_selftest_ntt_tune(logN, nprimes, sms, njobs)
        assert not one and limbs % nl == 0
        for grids in (cols, rows):
            assert sorted(set(grids), reverse=True) == grids, (njobs, grids)
            assert grids[1:] == [6 * sms, 4 * sms, 2 * sms]
    if logN >= 14:  # 320 limbs are 2560 units and more
        assert fhe.fhe_selftest_ntt_tune(logN, nprimes, sms, 320)[0] == 320 // nl // 16 * 16 * nl


@pytest.mark.parametrize("outer,nl", [(1, 3), (5, 2), (11, 1), (12, 2), (16, 3), (21, 2), (28, 1), (29, 1), (40, 2)])
@pytest.mark.parametrize("logN", [10, 11, 12, 13, 14, 15])
def test_units_cover_every_residue_once(fhe, logN, outer, nl):
    """Column units of one job and of pairs (an odd number of jobs leaves a
    slot empty), grouped row units with the rest as single ones (fewer than 12
    outer items beyond a multiple of 16), and the one-kernel form."""
    assert fhe.fhe_selftest_ntt_units(logN, outer, nl) == 0


def test_layouts_keep_elements_apart(fhe):
    assert fhe.fhe_selftest_ntt_layouts() == 0


@pytest.mark.parametrize("bits", [24, 36, 50, 53, 54, 55, 56, 57])
@pytest.mark.parametrize("logN", [10, 11, 12, 13, 14, 15])
def test_passes_hold_at_the_top_of_their_ranges(fhe, logN, bits):
    """The passes' arithmetic with the largest primes of a size: canonical
    inputs give the oracle's transforms, and so do the same residues lifted
    to the top of each pass's input range, among them all words at the top
    (whose sums reach the inverse's bound 4q 2^M, at 54 bits all of 64)."""
    n1, N = (logN + 1) // 2, 1 << logN
    lo = 2 ** bits - 2 ** (bits - (1 if bits < 30 else 5))
    o = Oracle(logN, 17, 1, 1, 2 ** (logN + 1), lo, 2 ** bits)
    q = o.primes[-1]
    assert q.bit_length() == bits
    rng = np.random.default_rng(bits * 100 + logN)

    def run(which, x):
        bad, y = fhe.fhe_selftest_ntt_pass(logN, q, which, x)
        assert bad == 0
        return y

    def lifts(x, top):
        """The residues of x as they are, at the top of [0, top q), and anywhere in it."""
        r = x % np.uint64(q)
        yield r
        yield r + np.uint64((top - 1) * q)
        yield r + rng.integers(0, top, size=N, dtype=np.uint64) * np.uint64(q)

    mixed = rng.integers(0, q, size=N, dtype=np.uint64)
    mixed[::5] = q - 1
    for a in (mixed, np.full(N, q - 1, np.uint64)):
        want = o.ntt(1, a)
        for x in lifts(a, 7):
            mid = run(0, x)
            assert int(mid.max()) < (4 * n1 + 7) * q
            assert np.array_equal(run(1, mid), want)
        for x in lifts(mid, 4 * n1 + 7):
            assert np.array_equal(run(1, x), want)
        want = o.intt(1, a)
        for x in lifts(a, 4):
            mid = run(2, x)
            assert int(mid.max()) < 4 * q
            assert np.array_equal(run(3, mid), want)
        for x in lifts(mid, 4):
            assert np.array_equal(run(3, x), want)
    top = np.full(N, q - 1, np.uint64)  # the same for the inverse columns alone: every word 4q - 1
    full = run(3, top + np.uint64(3 * q))
    assert np.array_equal(full, run(3, top)) and int(full.max()) < q


@pytest.mark.parametrize("bits", [24, 36, 54, 55, 56, 57])
def test_modarith_selftest_at_every_prime_size(fhe, bits):
    """The modular arithmetic, among it the linear combinations' sums with the
    largest scalars that fit 64 bits, for the largest primes of a size."""
    lo = 2 ** bits - 2 ** (bits - (1 if bits < 30 else 6))
    assert fhe.fhe_selftest_modarith(2 ** 12, lo, 2 ** bits, 4, 5000) == 0
