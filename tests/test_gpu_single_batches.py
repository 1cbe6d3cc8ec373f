"""GPU: calls on one batch take a launch table of one, and products of few
ciphertexts smaller blocks: counts on both sides of that line (two blocks of
1024 words per SM) against the oracle and against each ciphertext alone."""
import random

import numpy as np
import pytest

from tests.params import CHAIN50

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("logN", [10, 12, 15])
@pytest.mark.parametrize("above", [0, 1])
def test_one_batch_matches_oracle_and_singles(logN, above):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_07308_gb300 import build

    build.build()
    from paper_2407_07308_gb300 import fhe
    from tests.gpu_setup import GpuSetup
    from tests.oracle_setup import OracleSetup

    params = dict(logN=logN, p=17, L=5, K=1, **CHAIN50)
    o, g = OracleSetup(seed=9, **params), GpuSetup(seed=9, **params)
    try:
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        count = max(1, 2 * sms * 1024 // (5 << logN)) + above
        rnd = random.Random(logN)
        rows = [[[rnd.randrange(17) for _ in range(g.ns)] for _ in range(count)] for _ in range(2)]
        a, b = (g.encrypt_slots(rows[s], seed=s) for s in range(2))
        a1, b1 = (g.encrypt_each(rows[s], seed=s) for s in range(2))
        ops = {
            "mul": (lambda x, y: fhe.fhe_mul(g.ctx, x, y), o.o.tensor),
            "add": (lambda x, y: fhe.fhe_add(g.ctx, x, y), o.o.add),
            "sub": (lambda x, y: fhe.fhe_sub(g.ctx, x, y), o.o.sub),
        }
        for name, (op, ref) in ops.items():
            got = g.export(g.own(op(a, b)))
            for k in range(count):
                assert np.array_equal(got[k], g.export(g.own(op(a1[k], b1[k])))[0]), (name, k)
            k = count - 1
            ca, cb = (o.encrypt_row(rows[s], s, k) for s in range(2))
            assert np.array_equal(got[k], ref(ca, cb).data), name
    finally:
        g.close()
