"""A batch whose operations may use different numbers of lanes (many limbs share
two of them, few use all) gives what the operations give one by one, for one
lane up to more lanes than operations, issued directly and as a graph."""
import numpy as np
import pytest

from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case(O):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks as K
    P = O.make_params(16, 16, 2, 8)
    ctx = K.ckks_ctx_create(16, P.q, P.p, 2, scale=2.0**30)
    allp = P.all_primes()
    key = np.stack([np.stack([inputs.uniform_residues(981, allp, P.n, 10 * j + t) for t in range(2)])
                    for j in range(P.dnum)])
    relin, rot = K.ckks_evk_import(ctx, key, 0), K.ckks_evk_import(ctx, key, O.rot_k(1, 16))
    ops, want = [], []
    for i, level in enumerate((15, 1, 14, 13, 2, 12, 15)):
        a = K.ckks_ct_import(ctx, np.stack([inputs.uniform_residues(983 + i, P.q[:level + 1], P.n, t) for t in (0, 1)]),
                             level, 2.0**30)
        out = K.ckks_ct_create(ctx, level)
        if i % 3 == 0:
            ops.append(dict(op=K.CKKS_OP_HMULT, flags=K.CKKS_RESCALE, a=a, b=a, evk=relin, out=out))
            K.ckks_hmult(ctx, a, a, relin, K.CKKS_RESCALE, out)
        elif i % 3 == 1:
            ops.append(dict(op=K.CKKS_OP_HROT, r=1, a=a, evk=rot, out=out))
            K.ckks_hrot(ctx, a, 1, rot, out)
        else:
            ops.append(dict(op=K.CKKS_OP_RESCALE, a=a, out=out))
            K.ckks_rescale(ctx, a, out)
        want.append(K.ckks_ct_export(ctx, out, P.n)[0])
    yield K, P, ctx, ops, want
    K.ckks_ctx_destroy(ctx)


@pytest.mark.parametrize("lanes", [1, 2, 3, 9])
@pytest.mark.parametrize("graph", [False, True])
def test_lanes_by_size(case, lanes, graph):
    K, P, ctx, ops, want = case
    batch = K.ckks_batch_create(ctx, ops, lanes, graph)
    for o in ops:  # what the batch's own first run left there
        K.ckks_hadd(ctx, o["out"], o["out"], o["out"])
    for _ in range(2):
        K.ckks_batch_run(ctx, batch)
    for o, w in zip(ops, want):
        assert np.array_equal(K.ckks_ct_export(ctx, o["out"], P.n)[0], w), o["op"]
    K.ckks_batch_destroy(batch)
