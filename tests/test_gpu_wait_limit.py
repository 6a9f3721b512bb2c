"""The tensor-core column kernels' waits run out when their limit says so: with
a shape set by hand and a limit of one cycle, an operation ends, the next
synchronizing call reports CKKS_ETIMEOUT, and the same operations are right
again under the default limit. A level whose blocks hold several segments and
one whose blocks hold one; by rule (no shape set) the limit has a floor."""
import numpy as np
import pytest

import test_gpu_cols_tc as T
from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def system(O):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks as K
    P = O.make_params(16, 24, 6, 4)
    ctx = K.ckks_ctx_create(16, P.q, P.p, 6, scale=2.0**30)
    allp = P.all_primes()
    key = np.stack([np.stack([inputs.uniform_residues(935, allp, P.n, 10 * j + t) for t in range(2)])
                    for j in range(P.dnum)])
    yield K, ctx, P, K.ckks_evk_import(ctx, key, 0), K.ckks_evk_import(ctx, key, O.rot_k(1, 16))
    K.ckks_ctx_destroy(ctx)


@pytest.mark.parametrize("level", [23, 3])
def test_waits_run_out_and_the_context_goes_on(system, level):
    K, ctx, P, relin, rot = system
    a, b = (K.ckks_ct_import(ctx, T.residues(P, (0, level + 1), s, False), level, 2.0**30) for s in (931, 933))
    out = K.ckks_ct_create(ctx, level)
    ops = (lambda: K.ckks_hrot(ctx, a, 1, rot, out),                      # ModUp and ModDown columns
           lambda: K.ckks_hmult(ctx, a, b, relin, K.CKKS_RESCALE, out))   # and the fused rescale's
    get = lambda: K.ckks_ct_export(ctx, out, P.n)[0]
    want = []
    kernels = (K.CKKS_COL_MODUP, K.CKKS_COL_MODDOWN, K.CKKS_COL_RS_FUSED)
    try:
        for op in ops:
            op()
            want.append(get())
        K.ckks_set_wait_limit(ctx, 1)
        for op, w in zip(ops, want):  # by rule: the floor
            op()
            assert np.array_equal(get(), w)
        for kern in kernels:
            K.ckks_tune_set(ctx, kern, level, *T.TENSOR)
            for op in ops[1:] if kern == K.CKKS_COL_RS_FUSED else ops[:1]:
                op()
                with pytest.raises(K.CkksError) as e:
                    K.ckks_sync(ctx)
                assert e.value.code == K.CKKS_ETIMEOUT
            K.ckks_tune_set(ctx, kern, level, 0, 4, 1, 1)
        K.ckks_set_wait_limit(ctx, 1 << 32)
        for kern in kernels:
            K.ckks_tune_set(ctx, kern, level, *T.TENSOR)
        for op, w in zip(ops, want):
            op()
            assert np.array_equal(get(), w)
    finally:
        K.ckks_set_wait_limit(ctx, 1 << 32)
        for kern in kernels:
            K.ckks_tune_set(ctx, kern, level, 0, 4, 1, 1)
        for h in (a, b, out):
            K.ckks_free(h)
