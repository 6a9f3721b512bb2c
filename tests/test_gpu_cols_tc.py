"""The tensor-core column kernel against the CUDA-core ones and the oracle at
the sizes where it can go wrong: target counts around the groups of four that
a product converts and around the split of an item between blocks, one to
sixteen sources, primes on both sides of 2^29 and 2^30 (the 25-30 system's
2^25 and 2^30 windows, the 31-bit auxiliary primes), one-source rescaling on
both sides of its dispatch line, every residue at its extreme. Whole numbers:
equality, no tolerance."""
import numpy as np
import pytest

from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu

TENSOR, CORES = (8, 4, 1, 16), (8, 4, 1, 1)
_ctx = {}


@pytest.fixture(scope="module")
def K():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks
    yield ckks
    for ctx, _, _ in _ctx.values():
        ckks.ckks_ctx_destroy(ctx)
    _ctx.clear()


def get(K, O, name):
    """(context, oracle parameters, windows per level)"""
    if name not in _ctx:
        if name == "2530":
            P, levels = O.prime_system_2530(16, 5)
            ctx = K.ckks_ctx_create(16, P.q, P.p, P.dnum, scale=2.0**30, levels=levels)
        else:
            log_n, L, dnum, alpha = name
            P = O.make_params(log_n, L, dnum, alpha)
            levels = [(0, n + 1) for n in range(L)]
            ctx = K.ckks_ctx_create(log_n, P.q, P.p, dnum, scale=2.0**30)
        _ctx[name] = (ctx, P, levels)
    return _ctx[name]


def residues(P, window, seed, extreme):
    q = P.q[window[0]:window[0] + window[1]]
    if extreme:
        return np.stack([np.broadcast_to((q.astype(np.uint64) - 1)[:, None], (len(q), P.n))] * 2).astype(np.uint32)
    return np.stack([inputs.uniform_residues(seed, q, P.n, t) for t in (0, 1)])


def results(K, ctx, P, level, c1, c2, evk, k):
    a, b = K.ckks_ct_import(ctx, c1, level, 2.0**30), K.ckks_ct_import(ctx, c2, level, 2.0**30)
    rk, gk = K.ckks_evk_import(ctx, evk, 0), K.ckks_evk_import(ctx, evk, k)
    out = K.ckks_ct_create(ctx, level)
    got = {}
    try:
        K.ckks_hrot(ctx, a, 1, gk, out)
        got["hrot"] = K.ckks_ct_export(ctx, out, P.n)[0]
        for name, flag in (("rescale", K.CKKS_RESCALE), ("merged", K.CKKS_RESCALE_MERGED)) if level else ():
            K.ckks_hmult(ctx, a, b, rk, flag, out)
            got[name] = K.ckks_ct_export(ctx, out, P.n)[0]
    finally:
        for h in (a, b, rk, gk, out):
            K.ckks_free(h)
    return got


CASES = [(n, lv) for n, lvs in (((16, 40, 3, 14), (0, 1, 4, 5, 12, 13, 14, 27, 28, 39)),
                                ((16, 17, 2, 16), (0, 15, 16)),      # 16 sources, and 17 in the fused rescale
                                ((16, 16, 8, 2), (3, 15)),           # eight digits, two sources
                                ((12, 4, 4, 1), (1, 3)), ("2530", (0, 1, 2, 4, 8))) for lv in lvs]


@pytest.mark.parametrize("extreme", [False, True])
@pytest.mark.parametrize("name,level", CASES)
def test_tensor_columns_equal_cuda_core_columns(K, O, name, level, extreme):
    ctx, P, levels = get(K, O, name)
    c1, c2 = (residues(P, levels[level], s, extreme) for s in (901, 903))
    allp = P.all_primes()
    evk = np.stack([np.stack([inputs.uniform_residues(905, allp, P.n, 10 * j + t) for t in range(2)])
                    for j in range(P.dnum)])
    k = O.rot_k(1, P.log_n)
    kernels = (K.CKKS_COL_MODUP, K.CKKS_COL_MODDOWN, K.CKKS_COL_RS_FUSED)
    got = {}
    try:
        for shape in (TENSOR, CORES):
            for kern in kernels:
                K.ckks_tune_set(ctx, kern, level, *shape)
            got[shape] = results(K, ctx, P, level, c1, c2, evk, k)
    finally:
        for kern in kernels:
            K.ckks_tune_set(ctx, kern, level, 0, 4, 1, 1)
    for op, want in got[CORES].items():
        assert np.array_equal(got[TENSOR][op], want), op


@pytest.mark.parametrize("n_q", [2, 12, 13, 14, 40])
def test_rescale_on_both_sides_of_its_line(K, O, n_q):
    ctx, P, levels = get(K, O, (16, 40, 3, 14))
    for extreme in (False, True):
        c = residues(P, levels[n_q - 1], 911, extreme)
        a, out = K.ckks_ct_import(ctx, c, n_q - 1, 2.0**30), K.ckks_ct_create(ctx, n_q - 1)
        try:
            K.ckks_rescale(ctx, a, out)
            assert np.array_equal(K.ckks_ct_export(ctx, out, P.n)[0], O.rescale(c, P.q[:n_q]))
        finally:
            K.ckks_free(a)
            K.ckks_free(out)
