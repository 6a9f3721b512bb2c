"""The bytes a context reports contain the workspaces that it keeps: encoding
adds N complex values and N / 2 slots, decoding the limbs of the largest level
decoded so far, repeated calls nothing, and a clone counts its own."""
import pytest

from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n", [8, 16])
def test_encoding_workspaces_are_counted(O, log_n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks as K
    P = O.make_params(log_n, 6, 2, 3)
    ctx = K.ckks_ctx_create(log_n, P.q, P.p, 2, scale=2.0**30)
    lane = K.ckks_ctx_clone(ctx, torch.cuda.Stream().cuda_stream)
    held = lambda c: K.lib.ckks_ctx_device_bytes(c)
    start, lane_start = held(ctx), held(lane)
    u, limb, workspace = inputs.messages(177, P.n // 2), 4 * P.n, 24 * P.n
    pts = {level: K.ckks_encode(ctx, u, level, 2.0**30) for level in (1, 4, 2)}
    assert held(ctx) == start + workspace
    for level, limbs in ((1, 2), (4, 5), (2, 5), (4, 5)):
        K.ckks_decode(ctx, pts[level], P.n // 2)
        assert held(ctx) == start + workspace + limbs * limb
    assert held(lane) == lane_start
    K.ckks_decode(lane, pts[2], P.n // 2)
    assert held(lane) == lane_start + workspace + 3 * limb
    for pt in pts.values():
        K.ckks_free(pt)
    K.ckks_ctx_destroy(lane)
    K.ckks_ctx_destroy(ctx)
