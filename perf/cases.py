"""Timed cases of the CKKS library: the calls a user's program makes, through the Python binding.

A program keeps a context and its evaluation keys for as long as it runs, so both live here once per parameter
set; every state has ciphertexts, plaintexts and output buffers of its own. Ciphertext residues are uniform in
[0, q_i), which is how fresh and computed ciphertexts are distributed; they are torch tensors that the library
borrows, so that the outputs are tensors too. Evaluation keys are uniform residues as well.
"""
import functools
import weakref

import numpy as np
import torch

from paper_2407_13055_gb300 import ckks as K

# Parameter sets by name: (log2 N, ciphertext primes, auxiliary primes, digits). "2530" is the prime system with
# level windows and rational rescaling; the others rescale by one prime. toy1 / toy4 are the small test rings.
SETS = {
    "d3": (16, 40, 14, 3),
    "d5": (16, 40, 8, 5),
    "d1": (16, 40, 40, 1),
    "2530": (16, 15, 5, 3),
    "toy4": (12, 4, 1, 4),
    "toy1": (12, 4, 4, 1),
}
FLAGS = {"none": 0, "rescale": 1, "merged": 2}


def listed():
    return [
        # the smallest ring: what a unit of work costs when launches and latency are all there is
        {"name": "hmult_toy", "kind": "hmult", "set": "toy4", "level": 3, "flags": "rescale"},
        # the last levels before bootstrapping: few limbs, the whole auxiliary basis
        {"name": "hrot_l1", "kind": "hrot", "set": "d3", "level": 1, "r": 5},
        # an ordinary multiplication in the middle of a circuit
        {"name": "hmult_l20", "kind": "hmult", "set": "d3", "level": 20, "flags": "rescale"},
        # the headline parameter set at its top level: multiply and rotate
        {"name": "hmult_l39", "kind": "hmult", "set": "d3", "level": 39, "flags": "rescale"},
        {"name": "hrot_l39", "kind": "hrot", "set": "d3", "level": 39, "r": 1},
        # more digits, the last one partial, and no rescaling (sums of products rescale once)
        {"name": "hmult_d5_l27", "kind": "hmult", "set": "d5", "level": 27, "flags": "none"},
        # the 25-30 prime system: ModDown merged into the rational rescaling
        {"name": "hmult_2530_l6", "kind": "hmult", "set": "2530", "level": 6, "flags": "merged"},
        # weighted sums: plaintext product, sum and rescale, no key switch
        {"name": "weighted_l30", "kind": "weighted", "set": "d3", "level": 30},
        # rotations of one ciphertext (inner sums, baby steps)
        {"name": "hoisted_l24", "kind": "hoisted", "set": "d3", "level": 24, "count": 8},
        # matrix times vector: one linear transform
        {"name": "transform_l33", "kind": "transform", "set": "d3", "level": 33, "count": 16},
        # the client's side: message to plaintext and back
        {"name": "encode_decode_l5", "kind": "encode_decode", "set": "d3", "level": 5, "scale_bits": 40},
        # throughput: independent operations of many users at mixed levels, replayed as one graph on four lanes
        {"name": "batch_48", "kind": "batch", "set": "d3", "count": 48, "low": 1, "high": 39, "mix": 7},
    ]


def draw(rng):
    def level(name):
        if name == "2530":
            return rng.randint(1, 8)
        if name.startswith("toy"):
            return rng.randint(1, 3)
        return max(1, min(39, round(2 ** rng.uniform(0, 5.33))))

    kind = rng.choice(("hmult", "hmult", "hmult", "hrot", "hrot", "weighted", "hoisted", "transform", "encode_decode",
                       "batch"))
    if kind == "hmult":
        name = rng.choice(("d3", "d3", "d5", "d1", "2530", "toy4", "toy1"))
        flags = rng.choice(("none", "rescale", "rescale", "merged"))
        return {"kind": kind, "set": name, "level": level(name), "flags": flags}
    if kind == "hrot":
        name = rng.choice(("d3", "d3", "d5", "d1", "2530", "toy4"))
        return {"kind": kind, "set": name, "level": level(name), "r": rng.choice((1, 2, 5, 64, 1001))}
    if kind == "weighted":
        return {"kind": kind, "set": "d3", "level": level("d3")}
    if kind == "hoisted":
        name = rng.choice(("d3", "d5"))
        return {"kind": kind, "set": name, "level": level(name), "count": rng.randint(2, 8)}
    if kind == "transform":
        return {"kind": kind, "set": "d3", "level": level("d3"), "count": rng.randint(3, 16)}
    if kind == "encode_decode":
        return {"kind": kind, "set": "d3", "level": rng.randint(1, 8), "scale_bits": rng.randint(25, 45)}
    low = rng.randint(1, 12)
    return {"kind": "batch", "set": "d3", "count": rng.randint(5, 40), "low": low, "high": rng.randint(low + 2, 39),
            "mix": rng.randint(0, 1000)}


class Params:
    """A parameter set's context, primes and evaluation keys."""

    def __init__(self, name):
        self.log_n, n_q, n_p, self.dnum = SETS[name]
        self.N, self.alpha = 1 << self.log_n, n_p
        self.levels = None
        if name == "2530":
            self.q, self.p, self.levels = K.ckks_gen_prime_system_2530(self.log_n, n_p)
        else:
            self.q, self.p = K.ckks_gen_primes(self.log_n, n_q, n_p)
        self.scale = 2.0**40 if self.log_n == 16 else 2.0**28
        self.ctx = K.ckks_ctx_create(self.log_n, self.q, self.p, self.dnum, scale=self.scale,
                                     stream=torch.cuda.current_stream().cuda_stream, levels=self.levels)
        self._keys = {}

    def primes(self, level):
        if self.levels is None:
            return self.q[: level + 1]
        first, count = self.levels[level]
        return self.q[first:first + count]

    def key(self, galois):
        """Evaluation key for a Galois element (0: relinearization)."""
        if galois not in self._keys:
            g = torch.Generator(device="cuda").manual_seed(1000 + galois)
            every = np.concatenate([self.q, self.p])
            host = uniform((self.dnum, 2), every, self.N, g).cpu().numpy().view(np.uint32)
            self._keys[galois] = K.ckks_evk_import(self.ctx, host, galois)
        return self._keys[galois]

    def rotation_key(self, r):
        return self.key(pow(5, r % (self.N // 2), 2 * self.N))


@functools.lru_cache(maxsize=None)
def params(name):
    return Params(name)


def uniform(lead, primes, n, g):
    """int32 residues [*lead][len(primes)][n], limb i uniform in [0, primes[i])."""
    out = torch.empty((*lead, len(primes), n), dtype=torch.int32, device="cuda")
    for i, q in enumerate(primes):
        out[..., i, :] = torch.randint(0, int(q), (*lead, n), generator=g, device="cuda").to(torch.int32)
    return out


class State:
    """Handles of one state; they are freed with it."""

    def __init__(self, p, seed):
        self.p, self.ctx = p, p.ctx
        self.g = torch.Generator(device="cuda").manual_seed(seed)
        self.tensors, self._free, self.go = [], [], None
        weakref.finalize(self, _release, self._free)

    def owned(self, free, handle):
        self._free.append((free, handle))
        return handle

    def wrap(self, t, level, scale):
        self.tensors.append(t)
        return self.owned(K.ckks_free, K.ckks_ct_wrap_device(self.ctx, t.data_ptr(), level, scale))

    def ciphertext(self, level, scale=None):
        t = uniform((2,), self.p.primes(level), self.p.N, self.g)
        return self.wrap(t, level, self.p.scale if scale is None else scale)

    def output(self, level):
        t = torch.zeros((2, len(self.p.primes(level)), self.p.N), dtype=torch.int32, device="cuda")
        return t, self.wrap(t, level, self.p.scale)

    def plaintext(self, level, scale, extended=False):
        every = self.p.primes(level)
        if extended:
            every = np.concatenate([every, self.p.p])
        host = uniform((), every, self.p.N, self.g).cpu().numpy().view(np.uint32)
        make = K.ckks_pt_import_ext if extended else K.ckks_pt_import
        return self.owned(K.ckks_free, make(self.ctx, host, level, scale))


def _release(handles):
    torch.cuda.synchronize()
    for free, h in reversed(handles):
        free(h)


def prepare(case, seed):
    p = params(case["set"])
    s = State(p, seed)
    globals()["_prepare_" + case["kind"]](s, case, seed)
    torch.cuda.synchronize()
    return s


def run(state):
    return state.go()


def _prepare_hmult(s, case, seed):
    level, flags = case["level"], FLAGS[case["flags"]]
    a, b, key = s.ciphertext(level), s.ciphertext(level), s.p.key(0)
    out, h = s.output(level - 1 if flags else level)
    ctx = s.ctx

    def go():
        K.ckks_hmult(ctx, a, b, key, flags, h)
        return out
    s.go = go


def _prepare_hrot(s, case, seed):
    level, r = case["level"], case["r"]
    a, key = s.ciphertext(level), s.p.rotation_key(r)
    out, h = s.output(level)
    ctx = s.ctx

    def go():
        K.ckks_hrot(ctx, a, r, key, h)
        return out
    s.go = go


def _prepare_weighted(s, case, seed):
    """rescale(a * w + b): a sum of one product and a ciphertext of the product's scale."""
    level = case["level"]
    a, b = s.ciphertext(level), s.ciphertext(level, s.p.scale * s.p.scale)
    w = s.plaintext(level, s.p.scale)
    prod, hp = s.output(level)
    out, h = s.output(level - 1)
    ctx = s.ctx

    def go():
        K.ckks_pmult(ctx, a, w, hp)
        K.ckks_hadd(ctx, hp, b, hp)
        K.ckks_rescale(ctx, hp, h)
        return prod, out
    s.go = go


def _prepare_hoisted(s, case, seed):
    level, rs = case["level"], list(range(1, case["count"] + 1))
    a, keys = s.ciphertext(level), [s.p.rotation_key(r) for r in rs]
    outs = [s.output(level) for _ in rs]
    hs, ts, ctx = [h for _, h in outs], [t for t, _ in outs], s.ctx

    def go():
        K.ckks_hrot_hoisted(ctx, a, rs, keys, hs)
        return ts
    s.go = go


def _prepare_transform(s, case, seed):
    level, rs = case["level"], list(range(case["count"]))
    a, keys = s.ciphertext(level), [s.p.rotation_key(r) if r else None for r in rs]
    pts = [s.plaintext(level, s.p.scale, extended=True) for _ in rs]
    out, h = s.output(level)
    ctx = s.ctx

    def go():
        K.ckks_linear_transform(ctx, a, rs, keys, pts, h)
        return out
    s.go = go


def _message(case, seed):
    rng = np.random.default_rng(seed)
    slots = 1 << (SETS[case["set"]][0] - 1)
    return rng.uniform(-1, 1, slots) + 1j * rng.uniform(-1, 1, slots)


def _prepare_encode_decode(s, case, seed):
    level, scale, u, ctx = case["level"], 2.0 ** case["scale_bits"], _message(case, seed), s.ctx

    def go():
        pt = K.ckks_encode(ctx, u, level, scale)
        back = K.ckks_decode(ctx, pt, len(u))
        K.ckks_free(pt)
        return back
    s.go = go


def _batch_ops(case):
    """(operation, level) of each entry: which operations a batch has is the case's, its data the seed's."""
    rng = np.random.default_rng(case["mix"])
    kinds = ("hmult", "hrot", "hmult", "hrot", "pmult", "rescale")
    return [(kinds[i % len(kinds)], int(rng.integers(case["low"], case["high"] + 1))) for i in range(case["count"])]


def _prepare_batch(s, case, seed):
    ops, outs = [], []
    for i, (kind, level) in enumerate(_batch_ops(case)):
        a = s.ciphertext(level)
        if kind == "hmult":
            t, h = s.output(level - 1)
            ops.append({"op": K.CKKS_OP_HMULT, "flags": K.CKKS_RESCALE, "a": a, "b": s.ciphertext(level),
                        "evk": s.p.key(0), "out": h})
        elif kind == "hrot":
            r = 1 + i % 8
            t, h = s.output(level)
            ops.append({"op": K.CKKS_OP_HROT, "r": r, "a": a, "evk": s.p.rotation_key(r), "out": h})
        elif kind == "pmult":
            t, h = s.output(level)
            ops.append({"op": K.CKKS_OP_PMULT, "a": a, "pt": s.plaintext(level, s.p.scale), "out": h})
        else:
            t, h = s.output(level - 1)
            ops.append({"op": K.CKKS_OP_RESCALE, "a": a, "out": h})
        outs.append(t)
    ctx = s.ctx
    batch = s.owned(K.ckks_batch_destroy, K.ckks_batch_create(ctx, ops, 4, K.CKKS_BATCH_GRAPH))

    def go():
        K.ckks_batch_run(ctx, batch)
        return outs
    s.go = go


def exact(case, seed):
    """Residues are whole numbers and have no rounding; a decoded message is rounded once, at the encoding."""
    if case["kind"] != "encode_decode":
        return None
    # m(X) interpolates slot j at zeta^(5^j), zeta = exp(i pi / N), and its conjugate at the inverse
    u, n = _message(case, seed), 1 << SETS[case["set"]][0]
    at = np.empty(n // 2, dtype=np.int64)
    e = 1
    for j in range(n // 2):
        at[j] = e
        e = e * 5 % (2 * n)
    values = np.empty(n, dtype=np.complex128)  # m(zeta^(2k + 1))
    values[(at - 1) // 2] = u
    values[(2 * n - at - 1) // 2] = u.conj()
    twist = np.exp(1j * np.pi * np.arange(n) / n)
    scale = 2.0 ** case["scale_bits"]
    coeffs = (np.fft.fft(values) / n * twist.conj()).real * scale
    coeffs = np.copysign(np.floor(np.abs(coeffs) + 0.5), coeffs)
    back = np.fft.ifft(coeffs * twist) * n / scale
    return back[(at - 1) // 2]


def _key_switch_work(p, n, digits, moddown_targets):
    """Modular products of one key switch of n limbs: (ModUp part, KeyMult and ModDown part)."""
    rows = p.N // 2 * p.log_n
    ext = n + p.alpha
    up = n * rows
    for j in range(digits):
        k = min(n, (j + 1) * p.alpha) - j * p.alpha
        up += (ext - k) * (rows + k * p.N)
    down = 2 * digits * ext * p.N + 2 * (p.alpha * rows + moddown_targets * (rows + p.alpha * p.N))
    return up, down


def _op_work(p, kind, level, rescale=True, count=1):
    """(bytes, modular products) of one operation: inputs and keys read once, outputs written once."""
    n = len(p.primes(level))
    limb = 4 * p.N
    digits = -(-n // p.alpha)
    key = 2 * digits * (n + p.alpha)
    up, down = _key_switch_work(p, n, digits, n)
    n1 = len(p.primes(level - 1)) if level else n
    if kind == "hmult":
        return (4 * n + key + 2 * (n1 if rescale else n)) * limb, up + down + 4 * n * p.N
    if kind == "hrot":
        return (2 * n + key + 2 * n) * limb, up + down
    if kind == "hoisted":
        return (2 * n + count * (key + 2 * n)) * limb, up + count * down
    if kind == "transform":
        muls = up + down + (count - 1) * 2 * (digits + 1) * (n + p.alpha) * p.N
        return (2 * n + (count - 1) * key + count * (n + p.alpha) + 2 * n) * limb, muls
    rows = p.N // 2 * p.log_n
    if kind == "pmult":
        return (2 * n + n + 2 * n) * limb, 2 * n * p.N
    return (2 * n + 2 * n1) * limb, 2 * (1 + n1) * rows + 2 * n1 * p.N  # rescale


def work(case):
    p = params(case["set"])
    kind = case["kind"]
    if kind == "batch":
        parts = [_op_work(p, k, level) for k, level in _batch_ops(case)]
    elif kind == "weighted":
        # read: both ciphertexts and the plaintext; written: the sum and its rescaled form
        n = len(p.primes(case["level"]))
        parts = [((2 * n + n + 2 * n + 2 * n + 2 * (n - 1)) * 4 * p.N,
                  _op_work(p, "pmult", case["level"])[1] + _op_work(p, "rescale", case["level"])[1])]
    elif kind == "encode_decode":
        parts = [(2 * 16 * (p.N // 2), 2 * 5 * p.N * p.log_n + 2 * (case["level"] + 1) * (p.N // 2) * p.log_n)]
    else:
        parts = [_op_work(p, kind, case["level"], case.get("flags") != "none", case.get("count", 1))]
    # a modular product counts as one multiplication and one addition
    return {"bytes": float(sum(b for b, _ in parts)), "flops": 2.0 * sum(m for _, m in parts)}
