"""The work whose time this library is judged by: encrypted comparisons and what surrounds them.

A case names one kind of work and its sizes.  The parameter sets are the ones of the benchmark and
the tests: the 36-bit chain of the small ring (4 + 1 primes), the 50-bit chain with 10 + 3 primes,
and the universal 50-bit chain with 20 + 4 primes over N = 2^13 .. 2^15 and p in {17, 131, 257}.

Every pass starts from ciphertexts (or slot values, or residues) on hand and ends with the result
exported into a reply buffer, as a server that answers a client does; results are switched down to
one prime before that, because a reply is sent at its smallest.
"""
import math
import weakref

import numpy as np
import torch

from paper_2407_07308_gb300 import fhe, synth

CHAIN50 = (2 ** 16 * 17 * 131 * 257, 2 ** 49, 2 ** 50)
CHAIN36 = (8192 * 17, 2 ** 35, 2 ** 36)
CHAINS = {"small": (4, 1, CHAIN36), "mid": (10, 3, CHAIN50), "universal": (20, 4, CHAIN50)}
SLOTS = {17: 8, 131: 2, 257: 128}
SCRATCH_WORDS = 1 << 20  # count * npoly * N of one fhe_mod_switch_noalloc call


def listed():
    return [
        # one less-than on the small ring: the least a caller can ask for; launches and latency
        {"name": "lt_small_ring", "kind": "compare", "chain": "small", "log_n": 12, "p": 17, "d": 1, "level": 4,
         "count": 1, "eq": False},
        # one request of the mid ring answered on its own (LT and EQ), call by call
        {"name": "compare_one", "kind": "compare", "chain": "mid", "log_n": 14, "p": 131, "d": 2, "level": 10,
         "count": 1, "eq": True},
        # the benchmark's batch: 16 pairs, captured once and replayed
        {"name": "compare_plan_16", "kind": "plan", "chain": "mid", "log_n": 14, "p": 131, "d": 2, "level": 10,
         "count": 16},
        # a wide comparison at the largest ring, an odd number of ciphertexts and digits
        {"name": "compare_wide", "kind": "compare", "chain": "universal", "log_n": 15, "p": 257, "d": 3, "level": 17,
         "count": 7, "eq": True},
        # requests of mixed ring, prime, digit count and level in one submission, as a serving queue hands over
        {"name": "uneven_batch", "kind": "batch", "requests": 32, "mix": 3},
        # pairwise maxima and minima of two batches
        {"name": "max_min", "kind": "max_min", "chain": "universal", "log_n": 15, "p": 257, "d": 2, "level": 11,
         "count": 12},
        # the maximum and minimum over all slots of a batch: cross rounds, rotations and refreshes (a whole call)
        {"name": "tournament", "kind": "tournament", "log_n": 15, "p": 257, "d": 2, "count": 8},
        # short rows sorted
        {"name": "sort_rows", "kind": "sort", "log_n": 13, "p": 17, "d": 2, "count": 24},
        # one product per ciphertext at full level: the operation everything above is made of
        {"name": "multiply", "kind": "multiply", "chain": "universal", "log_n": 15, "p": 257, "level": 20,
         "count": 16},
        # sums over rotations, a few ciphertexts
        {"name": "rotate_sum", "kind": "rotate", "chain": "mid", "log_n": 14, "p": 17, "level": 9, "count": 3,
         "rotations": 3},
        # transforms and a modulus switch on the caller's own device buffers
        {"name": "raw_transforms", "kind": "transforms", "log_n": 13, "level": 19, "count": 61},
        # the client's side: slots encrypted and sent, a result decrypted
        {"name": "client", "kind": "client", "chain": "mid", "log_n": 14, "p": 131, "level": 10, "count": 2},
    ]


def _log_int(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm."""
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def _lowest_level(log_n, p, d, maxmin=False):
    lv = max(4, (p - 2).bit_length() + (d - 1).bit_length() + int(maxmin))
    return max(lv, (p - 2).bit_length() + 2) if p == 257 and log_n >= 14 else lv


def draw(rng):
    kind = rng.choice(["compare", "compare", "plan", "batch", "max_min", "tournament", "sort", "multiply", "rotate",
                       "transforms", "client"])
    if kind in ("compare", "plan"):
        chain = rng.choice(["small", "mid", "universal", "universal"])
        if chain == "small":
            # p = 17, d = 1 takes four levels: all that this ring has
            case = {"kind": kind, "chain": chain, "log_n": 12, "p": 17, "d": 1, "level": 4,
                    "count": _log_int(rng, 1, 64)}
        else:
            log_n, p, d = rng.choice([13, 14, 15]), rng.choice([17, 131, 257]), rng.randint(1, 4)
            top = CHAINS[chain][0]
            while _lowest_level(log_n, p, d) > top:
                d -= 1
            case = {"kind": kind, "chain": chain, "log_n": log_n, "p": p, "d": d,
                    "level": rng.randint(_lowest_level(log_n, p, d), top), "count": _log_int(rng, 1, 16)}
        return case if kind == "plan" else dict(case, eq=rng.random() < 0.7)
    if kind == "batch":
        return {"kind": kind, "requests": _log_int(rng, 4, 32), "mix": rng.randrange(1 << 20)}
    if kind == "max_min":
        log_n, p, d = rng.choice([13, 14, 15]), rng.choice([17, 131, 257]), rng.randint(1, 3)
        return {"kind": kind, "chain": "universal", "log_n": log_n, "p": p, "d": d,
                "level": rng.randint(_lowest_level(log_n, p, d, True), 20), "count": _log_int(rng, 1, 16)}
    if kind == "tournament":
        return {"kind": kind, "log_n": rng.choice([13, 14, 15]), "p": rng.choice([17, 257]), "d": rng.randint(1, 2),
                "count": rng.randint(2, 8)}
    if kind == "sort":
        return {"kind": kind, "log_n": rng.choice([13, 14]), "p": 17, "d": rng.randint(1, 2),
                "count": _log_int(rng, 1, 24)}
    if kind in ("multiply", "rotate", "client"):
        chain = rng.choice(["mid", "universal"])
        top = CHAINS[chain][0]
        case = {"kind": kind, "chain": chain, "log_n": rng.choice([13, 14, 15]), "p": rng.choice([17, 257]),
                "level": top if kind == "client" else rng.randint(2, top),
                "count": _log_int(rng, 1, 4 if kind == "client" else 24)}
        return dict(case, rotations=rng.randint(1, 3)) if kind == "rotate" else case
    log_n = rng.choice([12, 13, 14, 15])
    return {"kind": kind, "log_n": log_n, "level": rng.randint(2, 20),
            "count": _log_int(rng, 1, SCRATCH_WORDS // (2 << log_n))}


# ---------------------------------------------------------------------------
# contexts and keys: a program makes them once and keeps them; the states of a
# case share them while any of these lives
# ---------------------------------------------------------------------------

_rings = weakref.WeakValueDictionary()


class Ring:
    def __init__(self, chain, log_n, p, keys):
        L, K, (mod, lo, hi) = CHAINS[chain]
        self.stream = torch.cuda.Stream()
        self.ctx = fhe.fhe_ctx_create(log_n, p, L, K, mod, lo, hi,
                                      allocator=fhe.torch_allocator(torch.cuda.current_device()),
                                      stream=self.stream.cuda_stream)
        self.p, self.N, self.L, self.slots = p, 1 << log_n, L, fhe.fhe_ctx_info(self.ctx).slots
        self.base = (p + 1) // 2
        self.sk, self.pk = fhe.fhe_keygen(self.ctx, 100 * log_n + p)
        self.galois = {"none": lambda _: [], "rotate": lambda c: fhe.fhe_sort_galois(c)[:3],
                       "sort": fhe.fhe_sort_galois, "tournament": fhe.fhe_tournament_galois}[keys](self.ctx)
        self.evk = fhe.fhe_evk_create(self.ctx, self.sk, self.galois, 100 * log_n + p + 1)

    def encrypt(self, values, seed, level=None):
        """Slot values (count, slots) as one batch handle at `level`."""
        h = fhe.fhe_encrypt(self.ctx, self.pk, np.asarray(values, dtype=np.uint64).reshape(-1, self.slots), seed)
        if level is None or level == self.L:
            return h
        low = fhe.fhe_mod_switch(self.ctx, h, level)
        fhe.fhe_ct_destroy(h)
        return low

    def lower(self, h):
        """The ciphertext switched down to one prime; the given handle is given back."""
        if fhe.fhe_ct_shape(h)[2] == 1:
            return h
        low = fhe.fhe_mod_switch(self.ctx, h, 1)
        fhe.fhe_ct_destroy(h)
        return low

    def __del__(self):
        if getattr(self, "evk", None) is not None:
            fhe.fhe_ctx_sync(self.ctx)
            fhe.fhe_evk_destroy(self.evk)
            fhe.fhe_sk_destroy(self.sk)
            fhe.fhe_pk_destroy(self.pk)
            fhe.fhe_ctx_destroy(self.ctx)


class State:
    """The rings, operand handles, plan and reply buffers of one case; given back when dropped."""

    def __init__(self, case):
        self.case, self.rings, self.handles, self.plan, self.replies = case, [], [], None, []

    def reply_buffer(self, ring, count, level=1):
        """Pinned memory for one reply, which a server keeps (int64: every prime is below 2^58)."""
        self.replies.append(torch.empty((count, 2, level, ring.N), dtype=torch.int64, pin_memory=True))

    def reply(self, ring, handles, at=0, keep=False):
        """Exports the handles into the reply buffers from `at` on; gives them back unless they are kept."""
        out = self.replies[at:at + len(handles)]
        for h, buf in zip(handles, out):
            rc = fhe.lib().fhe_ct_export_coeff(ring.ctx, h, buf.data_ptr())
            if rc != 0:
                raise fhe.FheError(rc, "export")
            if not keep:
                fhe.fhe_ct_destroy(h)
        return out

    def ring(self, chain, log_n, p, keys="none"):
        key = (chain, log_n, p, keys)
        r = _rings.get(key)
        if r is None:
            r = _rings[key] = Ring(*key)
        self.rings.append(r)
        return r

    def own(self, handles):
        self.handles += handles
        return handles

    def __del__(self):
        for r in self.rings:
            fhe.fhe_ctx_sync(r.ctx)
        if self.plan is not None:
            fhe.fhe_plan_destroy(self.plan)
        for h in self.handles:
            fhe.fhe_ct_destroy(h)


def _pair(state, ring, g, d, level, count):
    """Two operands of d digits: uniform values in [0, base^d), three of ten equal."""
    hi = ring.base ** d
    x = g.integers(0, hi, size=count * ring.slots)
    y = np.where(g.random(x.size) < 0.3, x, g.integers(0, hi, size=x.size))
    seed = int(g.integers(1 << 40))
    xs = [ring.encrypt(v, seed + k, level) for k, v in enumerate(synth.to_digits(x, ring.base, d))]
    ys = [ring.encrypt(v, seed + 50 + k, level) for k, v in enumerate(synth.to_digits(y, ring.base, d))]
    return state.own(xs), state.own(ys)


def _requests(case):
    """The rings, digit counts and levels of a mixed submission, by its mix alone."""
    g = synth.rng(case["mix"])
    got = []
    for _ in range(case["requests"]):
        log_n, p, d = int(g.choice([13, 14, 15])), int(g.choice([17, 131, 257])), int(g.integers(1, 5))
        got.append((log_n, p, d, int(g.integers(_lowest_level(log_n, p, d), 21))))
    return got


def prepare(case, seed):
    s, kind, g = State(case), case["kind"], synth.rng(seed)
    if kind in ("compare", "plan", "max_min"):
        s.r = s.ring(case["chain"], case["log_n"], case["p"])
        s.xs, s.ys = _pair(s, s.r, g, case["d"], case["level"], case["count"])
        if kind == "plan":
            s.plan = fhe.fhe_compare_plan(s.r.ctx, s.r.evk, s.xs, s.ys)
            s.out = [fhe.fhe_plan_result(s.plan, 0), fhe.fhe_plan_result(s.plan, 1)]
            for h in s.out:
                s.reply_buffer(s.r, case["count"], fhe.fhe_ct_shape(h)[2])
        else:
            for _ in range(2 * case["d"] if kind == "max_min" else 1 + int(case["eq"])):
                s.reply_buffer(s.r, case["count"])
    elif kind == "batch":
        s.jobs = []
        for log_n, p, d, level in _requests(case):
            r = s.ring("universal", log_n, p)
            s.jobs.append((r, *_pair(s, r, g, d, level, 1)))
            for _ in range(2):
                s.reply_buffer(r, 1)
    elif kind in ("tournament", "sort"):
        s.r = s.ring("universal", case["log_n"], case["p"], kind)
        v = synth.values_with_duplicates(g, case["count"] * s.r.slots, s.r.base ** case["d"], 0.1)
        seed_ct = int(g.integers(1 << 40))
        s.xs = s.own([s.r.encrypt(x, seed_ct + k) for k, x in enumerate(synth.to_digits(v, s.r.base, case["d"]))])
        s.refresh_seed = int(g.integers(1 << 40))
        for _ in range(case["d"] * (2 if kind == "tournament" else 1)):
            s.reply_buffer(s.r, 1 if kind == "tournament" else case["count"])
    elif kind in ("multiply", "rotate"):
        s.r = s.ring(case["chain"], case["log_n"], case["p"], "rotate" if kind == "rotate" else "none")
        n = case["count"] * s.r.slots
        seed_ct = int(g.integers(1 << 40))
        s.a, s.b = s.own([s.r.encrypt(g.integers(0, s.r.p, size=n), seed_ct + k, case["level"]) for k in range(2)])
        s.reply_buffer(s.r, case["count"])
    elif kind == "transforms":
        s.r = s.ring("universal", case["log_n"], 17)
        tg = torch.Generator(device="cuda")
        tg.manual_seed(seed)
        n, level = case["count"], case["level"]
        s.x = torch.empty((n, 2, level, s.r.N), dtype=torch.int64, device="cuda")
        for i, q in enumerate(fhe.fhe_ctx_primes(s.r.ctx)[:level]):
            s.x[:, :, i] = torch.randint(0, q, (n, 2, s.r.N), dtype=torch.int64, device="cuda", generator=tg)
        s.y = torch.empty((n, 2, level - 1, s.r.N), dtype=torch.int64, device="cuda")
    else:
        s.r = s.ring(case["chain"], case["log_n"], case["p"])
        s.reply_buffer(s.r, case["count"], case["level"])
        s.slots = g.integers(0, s.r.p, size=(case["count"], s.r.slots)).astype(np.uint64)
        s.seed = int(g.integers(1 << 40))
        s.result = s.own([s.r.encrypt(g.integers(0, s.r.p, size=s.slots.size), s.seed + 1, 1)])[0]
    torch.cuda.synchronize()
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "compare":
        lt, eq = fhe.fhe_compare(s.r.ctx, s.r.evk, s.xs, s.ys, want_lt=True, want_eq=case["eq"])
        return s.reply(s.r, [s.r.lower(h) for h in ([lt, eq] if case["eq"] else [lt])])
    if kind == "plan":
        fhe.fhe_plan_run(s.plan, s.r.ctx)
        return s.reply(s.r, s.out, keep=True)
    if kind == "max_min":
        mx, mn = fhe.fhe_max_min(s.r.ctx, s.r.evk, s.xs, s.ys)
        return s.reply(s.r, [s.r.lower(h) for h in mx + mn])
    if kind == "batch":
        jobs = [fhe.Job(r.ctx, r.evk, fhe.FHE_JOB_COMPARE, xs, ys) for r, xs, ys in s.jobs]
        b = fhe.fhe_batch_submit(jobs, fhe.FHE_BATCH_ALIGN_LEVELS | fhe.FHE_BATCH_FUSE_RINGS)
        if fhe.fhe_batch_wait(b, 60000) != 0:
            raise RuntimeError("batch not done in a minute")
        fhe.fhe_batch_destroy(b)
        return [s.reply(r, [r.lower(h) for h in j.out0 + j.out1], at=2 * i)
                for i, ((r, _, _), j) in enumerate(zip(s.jobs, jobs))]
    if kind == "tournament":
        mx, mn = fhe.fhe_tournament(s.r.ctx, s.r.evk, s.r.sk, s.r.pk, s.xs, s.refresh_seed)
        return s.reply(s.r, [s.r.lower(h) for h in mx + mn])
    if kind == "sort":
        return s.reply(s.r, [s.r.lower(h) for h in fhe.fhe_sort(s.r.ctx, s.r.evk, s.xs)])
    if kind == "multiply":
        return s.reply(s.r, [s.r.lower(fhe.fhe_mul_relin(s.r.ctx, s.r.evk, s.a, s.b))])
    if kind == "rotate":
        acc = fhe.fhe_add(s.r.ctx, s.a, s.b)
        for g in s.r.galois[:case["rotations"]]:
            t = fhe.fhe_rotate(s.r.ctx, s.r.evk, acc, g)
            u = fhe.fhe_add(s.r.ctx, acc, t)
            fhe.fhe_ct_destroy(acc)
            fhe.fhe_ct_destroy(t)
            acc = u
        return s.reply(s.r, [s.r.lower(acc)])
    if kind == "transforms":
        # to evaluation form, one prime dropped, and back: the caller's buffers end as they began
        n, level = case["count"], case["level"]
        fhe.fhe_ntt_forward_batch(s.r.ctx, s.x.data_ptr(), 2 * n, level)
        fhe.fhe_mod_switch_noalloc(s.r.ctx, s.x.data_ptr(), s.y.data_ptr(), n, 2, level)
        fhe.fhe_ntt_inverse_batch(s.r.ctx, s.x.data_ptr(), 2 * n, level)
        return {"x": s.x, "y": s.y}
    sent = s.reply(s.r, [fhe.fhe_encrypt(s.r.ctx, s.r.pk, s.slots, s.seed)])
    return {"sent": sent, "slots": fhe.fhe_decrypt(s.r.ctx, s.r.sk, s.result).view(np.int64)}


def exact(case, seed):
    """Every output is a whole residue modulo a prime, equal to the last bit between two correct
    programs; there is nothing to approximate."""
    return None


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _key_switch(level, K, drop):
    """Limb transforms of one key switch at `level` (drop: the switch to level - 1 in the same step)."""
    dnum = -(-level // K)
    back = level + 2 * K + (2 if drop else 0)
    return back + dnum * (level + K) - level + 2 * (level - 1 if drop else level)


def _products(p, d, maxmin=False):
    """Products of a comparison by depth: the polynomial's (8 / 23 / 30 a digit for p = 17 / 131 / 257,
    evenly over its depths), the digit merge (two a pair) and the selection (one a digit)."""
    depth, each = (p - 2).bit_length(), {17: 8, 131: 23, 257: 30}[p]
    got = [d * each / depth] * depth
    while d > 1:
        got.append(2 * (d // 2))
        d = (d + 1) // 2
    return got + ([2.0] if maxmin else [])


def _flops(log_n, transforms):
    """Three modular operations per butterfly."""
    return 3.0 * transforms * (log_n << (log_n - 1))


def _compare_work(log_n, K, level, p, d, count, outputs, maxmin=False):
    N, prods = 1 << log_n, _products(p, d, maxmin)
    transforms = sum(n * _key_switch(max(1, level - t), K, level - t > 1) for t, n in enumerate(prods))
    key = -(-level // K) * 2 * (level + K) * N
    out = 2 * N
    return {"bytes": 8 * (key + count * (2 * d * 2 * level * N + outputs * out)),
            "flops": _flops(log_n, count * transforms)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [_compare_work(n, 4, level, p, d, 1, 2) for n, p, d, level in _requests(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    log_n, N, count = case["log_n"], 1 << case["log_n"], case["count"]
    L, K, _ = CHAINS[case.get("chain", "universal")]
    if kind in ("compare", "plan"):
        return _compare_work(log_n, K, case["level"], case["p"], case["d"], count, 1 + int(case.get("eq", True)))
    if kind == "max_min":
        return _compare_work(log_n, K, case["level"], case["p"], case["d"], count, 2 * case["d"], True)
    if kind == "tournament":
        # rounds halve the batch down to one ciphertext, then fold its slots; a maximum and a minimum track,
        # each started at the level its refresh gives
        rounds, c = [], count
        while c > 1:
            rounds.append(c // 2)
            c = (c + 1) // 2
        rounds += [1] * (SLOTS[case["p"]].bit_length() - 1)
        each = [_compare_work(log_n, K, 20, case["p"], case["d"], c, 0, True)["flops"] for c in rounds]
        key = 5 * 2 * 24 * N * (1 + SLOTS[case["p"]].bit_length() - 1)
        return {"bytes": 8 * (key + case["d"] * 2 * N * (20 * count + 2)), "flops": 2 * sum(each)}
    if kind == "sort":
        # every value of a row against the others, then its selection by rank
        cols = SLOTS[case["p"]] // 2
        w = _compare_work(log_n, K, 20, case["p"], case["d"], count, case["d"])
        return {"bytes": w["bytes"], "flops": 2 * (cols - 1) * w["flops"]}
    level = case["level"]
    key = -(-level // K) * 2 * (level + K) * N
    if kind == "multiply":
        return {"bytes": 8 * (key + count * N * (4 * level + 2)),
                "flops": _flops(log_n, count * _key_switch(level, K, True))}
    if kind == "rotate":
        return {"bytes": 8 * (case["rotations"] * key + count * N * (4 * level + 2)),
                "flops": _flops(log_n, count * case["rotations"] * _key_switch(level, K, False))}
    if kind == "transforms":
        return {"bytes": 8 * 2 * count * N * (4 * level + (level - 1)),
                "flops": _flops(log_n, 2 * count * (2 * level + 1 + level - 1))}
    # the public key, three samples a ciphertext, the ciphertexts sent; the result and the secret read
    return {"bytes": 8 * N * (2 * level + count * (3 + 2 * level) + 2 * count + 1),
            "flops": _flops(log_n, count * (3 * level + 1))}
