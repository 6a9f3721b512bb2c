"""Conversions to more targets than a segment of the tensor-core column kernel
holds: an item is cut inside one block, which converts its sources once more
and stores the digits over those that the products before it have read. Equal
to the CUDA-core columns (whole numbers: equality), run after run."""
import numpy as np
import pytest

import test_gpu_cols_tc as T
from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks
    return ckks


# ModUp to 64 targets; the fused rescale (15 + 1 sources) to 59, a partial group of four
@pytest.mark.parametrize("L,dnum,alpha,level", [(64, 4, 16, 63), (64, 4, 16, 56), (60, 4, 15, 59)])
def test_items_cut_inside_a_block(K, O, L, dnum, alpha, level):
    P = O.make_params(16, L, dnum, alpha)
    ctx = K.ckks_ctx_create(16, P.q, P.p, dnum, scale=2.0**30)
    c1, c2 = (T.residues(P, (0, level + 1), s, False) for s in (921, 923))
    allp = P.all_primes()
    evk = np.stack([np.stack([inputs.uniform_residues(925, allp, P.n, 10 * j + t) for t in range(2)])
                    for j in range(dnum)])
    kernels = (K.CKKS_COL_MODUP, K.CKKS_COL_MODDOWN, K.CKKS_COL_RS_FUSED)
    try:
        for kern in kernels:
            K.ckks_tune_set(ctx, kern, level, *T.CORES)
        want = T.results(K, ctx, P, level, c1, c2, evk, O.rot_k(1, 16))
        for kern in kernels:
            K.ckks_tune_set(ctx, kern, level, *T.TENSOR)
        for _ in range(3):
            got = T.results(K, ctx, P, level, c1, c2, evk, O.rot_k(1, 16))
            for op in want:
                assert np.array_equal(got[op], want[op]), op
    finally:
        K.ckks_ctx_destroy(ctx)
