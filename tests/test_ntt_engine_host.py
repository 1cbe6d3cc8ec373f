"""The NTT engine's own host functions and templates, run on the CPU through the
library's self-tests."""
import pytest


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
