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
