"""The automorphism's gather: HRot and HConj (word by word) of a borrowed
ciphertext that starts at any 4-byte address equal those of an aligned copy, and
a hoisted rotation (whole quads in another order) equals the single one, for
Galois elements of both residues modulo 4 and every ring size (whole numbers:
equality); and a linear transform with several unrotated terms, whose products
with a and b ride on the key switch, equals the sum of its parts made one by one."""
import numpy as np
import pytest

from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks
    return ckks


def context(K, O, log_n, L, dnum, alpha):
    P = O.make_params(log_n, L, dnum, alpha)
    return P, K.ckks_ctx_create(log_n, P.q, P.p, dnum, scale=2.0**30)


def key(P, seed):
    allp = P.all_primes()
    return np.stack([np.stack([inputs.uniform_residues(seed, allp, P.n, 10 * j + t) for t in range(2)])
                     for j in range(P.dnum)])


@pytest.mark.parametrize("log_n,L,dnum,alpha", [(8, 4, 2, 2), (12, 4, 4, 1), (16, 4, 2, 2)])
def test_unaligned_borrowed_ciphertext(K, O, log_n, L, dnum, alpha):
    import torch
    P, ctx = context(K, O, log_n, L, dnum, alpha)
    ct = np.stack([inputs.uniform_residues(951, P.q, P.n, t) for t in (0, 1)])
    dev = torch.empty(ct.size + 4, dtype=torch.int32, device="cuda")
    handles = []
    try:
        a = K.ckks_ct_import(ctx, ct, L - 1, 2.0**30)
        out = K.ckks_ct_create(ctx, L - 1)
        handles += [a, out]
        # device words of the imported ciphertext, by way of an addition of zero into the buffer
        zero = K.ckks_ct_import(ctx, np.zeros_like(ct), L - 1, 2.0**30)
        base = K.ckks_ct_wrap_device(ctx, dev.data_ptr(), L - 1, 2.0**30)
        handles += [zero, base]
        K.ckks_hadd(ctx, a, zero, base)
        K.ckks_sync(ctx)
        words = dev[:ct.size].clone()
        for r, conj in ((1, False), (2, False), (0, True)):
            k = O.conj_k(log_n) if conj else O.rot_k(r, log_n)
            ek = K.ckks_evk_import(ctx, key(P, 953 + r), k)
            handles.append(ek)
            run = (lambda c: K.ckks_hconj(ctx, c, ek, out)) if conj else (lambda c: K.ckks_hrot(ctx, c, r, ek, out))
            run(a)
            want = K.ckks_ct_export(ctx, out, P.n)[0]
            if not conj:
                K.ckks_hrot_hoisted(ctx, a, [r], [ek], [out])
                assert np.array_equal(K.ckks_ct_export(ctx, out, P.n)[0], want), k
            for offset in (1, 2, 3):
                dev[offset:offset + ct.size] = words
                torch.cuda.synchronize()
                b = K.ckks_ct_wrap_device(ctx, dev.data_ptr() + 4 * offset, L - 1, 2.0**30)
                handles.append(b)
                run(b)
                assert np.array_equal(K.ckks_ct_export(ctx, out, P.n)[0], want), (k, offset)
    finally:
        for h in handles:
            K.ckks_free(h)
        K.ckks_ctx_destroy(ctx)


@pytest.mark.parametrize("log_n,L,dnum,alpha,level", [(8, 6, 3, 2, 4), (12, 4, 1, 4, 3), (16, 6, 2, 3, 5)])
def test_unrotated_terms_ride_on_the_key_switch(K, O, log_n, L, dnum, alpha, level):
    P, ctx = context(K, O, log_n, L, dnum, alpha)
    n, handles = level + 1, []
    q = P.q[:n]
    try:
        c = K.ckks_ct_import(ctx, np.stack([inputs.uniform_residues(961, q, P.n, t) for t in (0, 1)]), level, 2.0**30)
        handles.append(c)
        every = np.concatenate([q, P.p])
        pts = [K.ckks_pt_import_ext(ctx, inputs.uniform_residues(963, every, P.n, i), level, 2.0**20) for i in range(4)]
        ek = K.ckks_evk_import(ctx, key(P, 965), O.rot_k(3, log_n))
        outs = [K.ckks_ct_create(ctx, level) for _ in range(3)]
        handles += pts + [ek] + outs
        get = lambda h: K.ckks_ct_export(ctx, h, P.n)[0].astype(np.uint64)
        K.ckks_linear_transform(ctx, c, [0, 3, 0, 0], [None, ek, None, None], pts, outs[0])
        got = get(outs[0])
        K.ckks_linear_transform(ctx, c, [3], [ek], [pts[1]], outs[0])
        want = get(outs[0])
        K.ckks_linear_transform(ctx, c, [0, 0, 0], [None] * 3, [pts[0], pts[2], pts[3]], outs[1])
        want = want + get(outs[1])
        assert np.array_equal(got, want % q.astype(np.uint64)[None, :, None])
        for i, o in ((0, outs[1]), (2, outs[2])):  # and the plain form against PMult
            K.ckks_pmult(ctx, c, pts[i], o)
        K.ckks_linear_transform(ctx, c, [0, 0], [None] * 2, [pts[0], pts[2]], outs[0])
        assert np.array_equal(get(outs[0]), (get(outs[1]) + get(outs[2])) % q.astype(np.uint64)[None, :, None])
    finally:
        for h in handles:
            K.ckks_free(h)
        K.ckks_ctx_destroy(ctx)
