"""Encoding and decoding on the device against the definition: every ring size,
one limb up to all of them, plain and extended plaintexts, positive and negative
values, values of one limb's size and of hundreds of bits, and numbers that are
not finite."""
import numpy as np
import pytest

from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu
EPS = 2.0**-53


@pytest.fixture(scope="module")
def K():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks
    return ckks


RINGS = [(8, 4, 2, 2), (12, 4, 1, 4), (16, 6, 2, 3), (8, 30, 3, 10)]


@pytest.mark.parametrize("log_n,L,dnum,alpha", RINGS)
@pytest.mark.parametrize("bits", [12, 30, 45])
def test_encode_matches_definition(K, O, log_n, L, dnum, alpha, bits):
    P = O.make_params(log_n, L, dnum, alpha)
    ctx = K.ckks_ctx_create(log_n, P.q, P.p, dnum, scale=2.0**30)
    scale, u = 2.0**bits, inputs.messages(171 + bits, P.n // 2)
    want = np.array([int(c) for c in O.encode_coeffs(u, scale, log_n)], dtype=object)
    # two FFTs of binary64, each off by at most 4 log2(N) roundings of a mean of values below sqrt(2)
    # (butterfly products and sums, twiddles, twist), and one rounding to a whole number on either side
    bound = 1 + int(2 * 4 * (log_n + 1) * EPS * 1.5 * scale)
    for level in sorted({0, 1, L - 1}):
        for ext in (False, True):
            pt = (K.ckks_encode_ext if ext else K.ckks_encode)(ctx, u, level, scale)
            res = K.ckks_pt_export(ctx, pt, level, P.n)[0]
            K.ckks_free(pt)
            primes = P.q[:level + 1]
            coeffs = O.intt(res, primes).astype(np.int64)
            for c, q in zip(coeffs, primes):
                diff = (c - np.array([w % int(q) for w in want], dtype=np.int64)) % int(q)
                diff = np.minimum(diff, int(q) - diff)
                assert diff.max() <= bound, (level, ext, int(q))
    K.ckks_ctx_destroy(ctx)


@pytest.mark.parametrize("log_n,L,dnum,alpha", RINGS)
def test_decode_matches_definition(K, O, log_n, L, dnum, alpha):
    P = O.make_params(log_n, L, dnum, alpha)
    ctx = K.ckks_ctx_create(log_n, P.q, P.p, dnum, scale=2.0**30)
    rng = np.random.default_rng(173)
    for level in sorted({0, 1, L // 2, L - 1}):
        primes = P.q[:level + 1]
        Q = 1
        for q in primes:
            Q *= int(q)
        half, scale = (Q - 1) // 2, 2.0**25
        for size in (1, 1 << 20, half):
            # whole numbers in [-size, size], both ends and zero among them
            size = min(size, half)
            words = rng.integers(0, 2**32, (P.n, (size.bit_length() + 95) // 32), dtype=np.uint64)
            m = [sum(int(w) << (32 * i) for i, w in enumerate(row)) % (2 * size + 1) - size for row in words]
            m[0], m[1], m[2] = size, -size, 0
            res = np.stack([np.array([x % int(q) for x in m], dtype=np.uint32) for q in primes])
            pt = K.ckks_pt_import(ctx, O.ntt(res, primes), level, scale)
            got = K.ckks_decode(ctx, pt, P.n // 2)
            K.ckks_free(pt)
            want = O.decode_coeffs(np.array([float(x) for x in m]), scale, log_n)
            # Horner: one rounding per limb and coefficient; FFTs on both sides: 4 log2(N) roundings; the sum
            # of N values of at most `size`
            bound = (level + 1 + 2 * 4 * (log_n + 1)) * EPS * float(size) * P.n / scale
            assert np.max(np.abs(got - want)) <= bound, (level, size)
    K.ckks_ctx_destroy(ctx)


@pytest.mark.parametrize("log_n", [8, 12, 16])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 1e308])
def test_not_finite(K, O, log_n, bad):
    """Slots that are not finite, or overflow, are taken, and the context goes on as before."""
    P = O.make_params(log_n, 4, 2, 2)
    ctx = K.ckks_ctx_create(log_n, P.q, P.p, 2, scale=2.0**30)
    u = inputs.messages(175, P.n // 2)
    v = u.copy()
    v[5] = bad
    pt = K.ckks_encode(ctx, v, 3, 2.0**40)
    K.ckks_decode(ctx, pt, P.n // 2)
    K.ckks_free(pt)
    pt = K.ckks_encode(ctx, u, 3, 2.0**40)
    # half a unit of rounding per coefficient
    assert np.max(np.abs(K.ckks_decode(ctx, pt, P.n // 2) - u)) <= P.n / 2.0**40
    K.ckks_free(pt)
    K.ckks_ctx_destroy(ctx)
