"""Batches without a key switch use every lane they are given: rescalings of
one level, each of which leaves most of the chip idle, take clearly less time
on eight lanes than on two (measured at level 10 of this ring: 156 us and 239;
on two lanes whatever is given: the same), and the results are those of the
operations one by one."""
import time

import numpy as np
import pytest

from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level", [10])
def test_rescalings_use_every_lane(O, level):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks as K
    P = O.make_params(16, 40, 3, 14)
    ctx = K.ckks_ctx_create(16, P.q, P.p, 3, scale=2.0**30)
    ops, want = [], []
    for i in range(24):
        c = np.stack([inputs.uniform_residues(941 + i, P.q[:level + 1], P.n, t) for t in (0, 1)])
        a, out = K.ckks_ct_import(ctx, c, level, 2.0**30), K.ckks_ct_create(ctx, level - 1)
        K.ckks_rescale(ctx, a, out)
        want.append(K.ckks_ct_export(ctx, out, P.n)[0])
        ops.append(dict(op=K.CKKS_OP_RESCALE, a=a, out=out))
    us = {}
    try:
        for lanes in (2, 8):
            batch = K.ckks_batch_create(ctx, ops, lanes, True)
            runs = []
            for _ in range(9):
                K.ckks_sync(ctx)
                t = time.perf_counter()
                for _ in range(10):
                    K.ckks_batch_run(ctx, batch)
                K.ckks_sync(ctx)
                runs.append((time.perf_counter() - t) / 10 * 1e6)
            us[lanes] = min(runs)
            K.ckks_batch_destroy(batch)
            for o, w in zip(ops, want):
                assert np.array_equal(K.ckks_ct_export(ctx, o["out"], P.n)[0], w)
    finally:
        K.ckks_ctx_destroy(ctx)
    assert us[8] < 0.85 * us[2], us
