"""Batches without a key switch use every lane they are given: rescalings of
one level, each of which leaves most of the chip idle, take clearly less time
on eight lanes than on two (measured: level 10 156 us and 239, on two lanes
whatever is given the same; level 30 408 and 552, in the tensor-core form on
eight lanes 522; the 25-30 system's level 7 221 and 301, 284), and the results
are those of the operations one by one."""
import time

import numpy as np
import pytest

from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,level", [("single", 10), ("single", 30), ("2530", 7)])
def test_rescalings_use_every_lane(O, name, level):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks as K
    if name == "2530":
        P, levels = O.prime_system_2530(16, 5)
        ctx = K.ckks_ctx_create(16, P.q, P.p, P.dnum, scale=2.0**30, levels=levels)
    else:
        P, levels = O.make_params(16, 40, 3, 14), [(0, n + 1) for n in range(40)]
        ctx = K.ckks_ctx_create(16, P.q, P.p, 3, scale=2.0**30)
    first, count = levels[level]
    primes = P.q[first:first + count]
    ops, want = [], []
    for i in range(24):
        c = np.stack([inputs.uniform_residues(941 + i, primes, P.n, t) for t in (0, 1)])
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
