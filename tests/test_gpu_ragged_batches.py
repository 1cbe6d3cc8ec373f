"""GPU: ragged counts give the bits of each ciphertext on its own.

Batches and jobs of one context are joined into common launches: an NTT
segment spans several jobs, and groups of outer items leave a remainder that
runs as single items, so the counts here lie on both sides of a group (11, 12,
13), leave remainders, and mix in one submission.  Encryption lifts u, p e0 + m
and p e1 in one pass, and decryption returns the subring's coefficients only;
both at ragged counts, with noise larger than a prime, and for plaintexts that
are no slot encoding."""
import random

import numpy as np
import pytest

from tests.params import CHAIN50

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_07308_gb300 import build

    build.build()


def _setup(**kw):
    from tests.gpu_setup import GpuSetup

    return GpuSetup(seed=31, **dict(dict(p=17, L=6, K=2), **kw), **CHAIN50)


@pytest.mark.parametrize("logN", [10, 12, 13, 14, 15])
@pytest.mark.parametrize("counts", [(1, 2), (11, 1), (12, 5), (13,)])
def test_ragged_jobs_match_singles(logN, counts):
    from paper_2407_07308_gb300 import fhe

    g = _setup(logN=logN)
    try:
        rnd = random.Random(logN)
        jobs, rows = [], []
        for i, n in enumerate(counts):
            x, y = ([[rnd.randrange(9) for _ in range(g.ns)] for _ in range(n)] for _ in range(2))
            rows.append((x, y))
            jobs.append(fhe.Job(g.ctx, g.evk, fhe.FHE_JOB_COMPARE, [g.encrypt_slots(x, seed=2 * i)],
                                [g.encrypt_slots(y, seed=2 * i + 1)]))
        batch = fhe.fhe_batch_submit(jobs)
        assert fhe.fhe_batch_wait(batch, 120000) == 0
        fhe.fhe_batch_destroy(batch)
        for i, (job, (x, y)) in enumerate(zip(jobs, rows)):
            lt, eq = g.export(g.own(job.out0[0])), g.export(g.own(job.out1[0]))
            xe, ye = g.encrypt_each(x, seed=2 * i), g.encrypt_each(y, seed=2 * i + 1)
            for k in {0, len(x) // 2, len(x) - 1}:
                a, b = fhe.fhe_compare(g.ctx, g.evk, [xe[k]], [ye[k]])
                assert np.array_equal(g.export(g.own(a))[0], lt[k]), (i, k)
                assert np.array_equal(g.export(g.own(b))[0], eq[k]), (i, k)
    finally:
        g.close()


@pytest.mark.parametrize("logN,count", [(10, 1), (11, 5), (15, 3)])
def test_encryption_lifts_any_noise(logN, count):
    """With u = 0 a ciphertext is (p e0 + m, p e1): its residues against
    integers, for noise up to the range of a signed word, m in the subring."""
    from paper_2407_07308_gb300 import fhe

    g = _setup(logN=logN)
    try:
        rng = np.random.default_rng(logN)
        lim = (2 ** 63 - 1) // g.p - 1
        e = rng.integers(-lim, lim, size=(2, count, g.N), dtype=np.int64)
        e[:, :, ::3] = rng.integers(-20, 21, size=e[:, :, ::3].shape)
        e[:, :, 0], e[:, :, -1] = -lim, lim
        slots = rng.integers(0, g.p, size=(count, g.ns)).astype(np.uint64)
        zero = np.zeros((count, g.N), np.int64)
        m = g.export(g.own(fhe.fhe_encrypt_explicit(g.ctx, g.pk, slots, zero, zero, zero)))[:, 0]
        got = g.export(g.own(fhe.fhe_encrypt_explicit(g.ctx, g.pk, slots, zero, e[0], e[1])))
        for l, q in enumerate(g.primes[: g.L]):
            assert (m[:, l] < g.p).all()
            assert np.array_equal(got[:, 0, l].astype(object), (g.p * e[0].astype(object) + m[:, l].astype(object)) % q)
            assert np.array_equal(got[:, 1, l].astype(object), g.p * e[1].astype(object) % q)
    finally:
        g.close()


@pytest.mark.parametrize("logN", [10, 13])
def test_decrypt_refuses_other_plaintexts(logN):
    """Ciphertexts of one batch at the top level and at one prime: slot
    encodings decrypt, and a plaintext outside the subring is refused."""
    from paper_2407_07308_gb300 import fhe

    g = _setup(logN=logN)
    try:
        d = 2
        digits = np.zeros((3, g.ns, d), np.uint64)
        digits[:, :, 0] = 5
        good = g.encrypt_ext(digits, d, seed=1)
        digits[2, 0, 1] = 1
        bad = g.encrypt_ext(digits, d, seed=1)
        for level in (g.L, 1):
            a, b = (c if level == g.L else g.own(fhe.fhe_mod_switch(g.ctx, c, level)) for c in (good, bad))
            assert (g.decrypt(a) == 5).all()
            with pytest.raises(fhe.FheError, match="slot encoding"):
                g.decrypt(b)
    finally:
        g.close()
