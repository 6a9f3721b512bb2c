"""The ModDown step on a context with level windows converts to the first n_q
primes, whether or not a level has that window, equal to the oracle: at every
count, with the default column shapes and with a tensor-core shape set for the
level whose number the count happens to have."""
import numpy as np
import pytest

from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def system(O):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks as K
    P, levels = O.prime_system_2530(16, 5)
    ctx = K.ckks_ctx_create(16, P.q, P.p, P.dnum, scale=2.0**30, levels=levels)
    yield K, ctx, P, levels
    K.ckks_ctx_destroy(ctx)


@pytest.mark.parametrize("n_q", range(1, 16))
def test_moddown_step_of_the_first_primes(system, O, n_q):
    K, ctx, P, levels = system
    assert n_q <= len(P.q)
    primes = np.concatenate([P.q[:n_q], P.p])
    acc = np.stack([inputs.uniform_residues(701 + n_q, primes, P.n, t) for t in (0, 1)])
    want = O.moddown(P, acc, n_q)
    assert np.array_equal(K.ckks_step_moddown(ctx, acc, n_q), want)
    if n_q <= len(levels):
        K.ckks_tune_set(ctx, K.CKKS_COL_MODDOWN, n_q - 1, 8, 4, 1, 16)
        try:
            assert np.array_equal(K.ckks_step_moddown(ctx, acc, n_q), want)
        finally:
            K.ckks_tune_set(ctx, K.CKKS_COL_MODDOWN, n_q - 1, 0, 4, 1, 1)
