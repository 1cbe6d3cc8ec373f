"""GPU parity at the prime sizes a context accepts, from 24 bits to the largest
(57): the half-word sums of the conversions and fused stores fold earlier
above 54 bits and take a canonical operand at 57, and the inverse transform
normalises between its rounds above 54 bits.  Products, switches by one and
by several primes, relinearisation and a rotation against the CPU oracle,
bit for bit, at an odd count of source limbs (K = 3, a short last digit)."""
import random

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bits,logN", [(24, 11), (33, 11), (50, 15), (51, 11), (54, 11), (54, 13), (55, 11), (56, 12),
                                       (57, 11), (57, 13)])
def test_operations_bitexact_at_prime_size(bits, logN):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_07308_gb300 import build

    build.build()
    from paper_2407_07308_gb300 import fhe
    from tests.gpu_setup import GpuSetup
    from tests.oracle_setup import OracleSetup

    p, L, K = 17, 7, 3
    params = dict(logN=logN, p=p, L=L, K=K, U=2 ** (logN + 1) * p, lo=2 ** (bits - 1), hi=2 ** bits)
    if bits > 50:  # the largest primes of the size: the tightest case of every bound
        params["lo"] = 2 ** bits - 2 ** (bits - 6)
    o, g = OracleSetup(seed=7, galois=(5,), **params), GpuSetup(seed=7, galois=(5,), **params)
    try:
        assert g.primes == o.o.primes and all(q.bit_length() == bits for q in g.primes)
        rnd = random.Random(bits)
        a, b = ([rnd.randrange(p) for _ in range(g.ns)] for _ in range(2))
        ca, cb = o.encrypt_slots([a, b], seed=3)
        ga, gb = g.encrypt_each([a, b], seed=3)
        oc, X = o.o, g.ctx
        down = ca
        for _ in range(5):
            down = oc.modswitch(down)
        t = g.own(fhe.fhe_mul(X, ga, gb))
        checks = [
            ("modswitch", oc.modswitch(ca), fhe.fhe_mod_switch(X, ga, L - 1)),
            ("modswitch by 5", down, fhe.fhe_mod_switch(X, ga, L - 5)),
            ("relin", oc.relin(oc.tensor(ca, cb), o.rlk), fhe.fhe_relinearize(X, g.evk, t)),
            ("mul_relin", o.evaluator().mul(ca, cb), fhe.fhe_mul_relin(X, g.evk, ga, gb)),
            ("rotate", oc.rotate(ca, 5, o.gks[5]), fhe.fhe_rotate(X, g.evk, ga, 5)),
        ]
        for name, want, got in checks:
            g.own(got)
            assert np.array_equal(g.export(got)[0], want.data), name
    finally:
        g.close()
