"""GPU: both forms of a transform against the oracle, bit for bit.

Launches of a few units per SM run both passes in one kernel; larger ones run
a column and a row kernel, whose CTAs walk the units under the grid policies 1
to 3.  The counts lie on both sides of the line and leave ragged rests of row
groups, and the launch counter says which form ran.  The line itself (6 units
of 2048 residues per SM, 4 at N = 2^15) is asked of the library."""
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


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
@pytest.mark.parametrize("logN", [10, 11, 12, 13, 14, 15])
def test_plain_transforms_match_oracle_in_both_forms(logN, variant):
    from oracle.bgv import Oracle
    from paper_2407_07308_gb300 import fhe

    L, K, N = 3, 2, 1 << logN
    o = Oracle(logN, 131, L, K, **CHAIN50)
    ctx = fhe.fhe_ctx_create(logN, 131, L, K, CHAIN50["U"], CHAIN50["lo"], CHAIN50["hi"])
    try:
        fhe.fhe_ctx_ntt_variant(ctx, variant)
        nl = L + K
        most = ((4 if logN == 15 else 6) * _sms() >> (logN - 11)) // nl if logN > 10 else 0  # in one kernel
        walk = 13 * _sms() * 2 // nl if logN == 10 else (7 * _sms() >> (logN - 11)) // nl  # more units than CTAs
        rng = np.random.default_rng(100 * logN + variant)
        counts = [1, most, most + 1, walk // 16 * 16 + 21, walk // 16 * 16 + 29]
        for count in sorted(set(c for c in counts if c)):
            a = np.stack([rng.integers(0, q, size=(count, N), dtype=np.uint64) for q in o.primes], axis=1)
            for i, q in enumerate(o.primes):
                a[-1, i] = q - 1  # the largest values
            for name, f, ref in (("forward", fhe.fhe_ntt_forward_batch, o.ntt), ("inverse", fhe.fhe_ntt_inverse_batch, o.intt)):
                dev = torch.from_numpy(a.view(np.int64).copy()).cuda()
                before = fhe.fhe_ctx_launches(ctx)
                f(ctx, dev.data_ptr(), count, nl)
                assert fhe.fhe_ctx_launches(ctx) - before == (1 if count <= most else 2), count
                torch.cuda.synchronize()
                got = dev.cpu().numpy().view(np.uint64)
                for c in range(count):
                    for i in range(nl):
                        assert np.array_equal(got[c, i], ref(i, a[c, i])), (name, count, c, i)
    finally:
        fhe.fhe_ctx_destroy(ctx)


@pytest.mark.parametrize("logN", [11, 12, 13, 14, 15])
def test_fused_transforms_match_oracle_in_both_forms(logN):
    """Products, switches by one and by three primes and a rotation of a batch
    whose smallest transform (two limbs a ciphertext) takes two kernels and
    more units than any policy's CTAs, under every policy; and of one
    ciphertext, in one kernel each."""
    from paper_2407_07308_gb300 import fhe
    from tests.gpu_setup import GpuSetup
    from tests.oracle_setup import OracleSetup

    params = dict(logN=logN, p=17, L=5, K=2, **CHAIN50)
    o, g = OracleSetup(seed=5, galois=(5,), **params), GpuSetup(seed=5, galois=(5,), **params)
    try:
        # launches: tensor, inner product and fold one each; a transform one or two
        ops = {
            "mul_relin": (lambda a, b: fhe.fhe_mul_relin(g.ctx, g.evk, a, b), 3, 4),
            "switch by one": (lambda a, b: fhe.fhe_mod_switch(g.ctx, a, 4), 0, 2),
            "switch by three": (lambda a, b: fhe.fhe_mod_switch(g.ctx, a, 2), 1, 2),
            "rotate": (lambda a, b: fhe.fhe_rotate(g.ctx, g.evk, a, 5), 2, 4),
        }
        rnd = random.Random(logN)
        count = (6 * _sms() >> (logN - 10)) + 5
        rows = [[[rnd.randrange(17) for _ in range(g.ns)] for _ in range(count)] for _ in range(2)]
        want = {}
        for k in (0, count // 2, count - 1):
            ca, cb = (o.encrypt_row(rows[s], 3 + s, k) for s in range(2))
            down = o.o.modswitch(ca)
            want[k] = {"mul_relin": o.evaluator().mul(ca, cb), "switch by one": down,
                       "switch by three": o.o.modswitch(o.o.modswitch(down)), "rotate": o.o.rotate(ca, 5, o.gks[5])}
        xa, xb = (g.encrypt_slots(rows[s], seed=3 + s) for s in range(2))
        whole = {}
        for variant in range(4):
            fhe.fhe_ctx_ntt_variant(g.ctx, variant)
            for name, (op, single, transforms) in ops.items():
                before = fhe.fhe_ctx_launches(g.ctx)
                h = op(xa, xb)
                assert fhe.fhe_ctx_launches(g.ctx) - before == single + 2 * transforms, name
                got = g.export(h)
                fhe.fhe_ct_destroy(h)
                if variant == 0:
                    whole[name] = got
                    for k, w in want.items():
                        assert np.array_equal(got[k], w[name].data), (name, k)
                assert np.array_equal(got, whole[name]), (name, variant)
        r = [g.encrypt_each(rows[s], seed=3 + s)[-1] for s in range(2)]
        for name, (op, single, transforms) in ops.items():
            before = fhe.fhe_ctx_launches(g.ctx)
            h = g.own(op(*r))
            assert fhe.fhe_ctx_launches(g.ctx) - before == single + transforms, name
            assert np.array_equal(g.export(h)[0], want[count - 1][name].data), name
    finally:
        g.close()
