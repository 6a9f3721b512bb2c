"""A linear transform of one unrotated term gives PMult's limbs and takes about
its time (the same bytes; measured at level 39 of this ring: 7.5 us and 6.2,
with blocks too small to start fast enough 11.4; fifty calls as one graph each,
so that the host's time does not count)."""
import numpy as np
import pytest

from paper_2407_13055_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_one_unrotated_term(O):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2407_13055_gb300 import ckks as K
    P, level = O.make_params(16, 40, 3, 14), 39
    stream = torch.cuda.Stream()
    ctx = K.ckks_ctx_create(16, P.q, P.p, 3, scale=2.0**30, stream=stream.cuda_stream)
    c = K.ckks_ct_import(ctx, np.stack([inputs.uniform_residues(971, P.q, P.n, t) for t in (0, 1)]), level, 2.0**30)
    w = K.ckks_pt_import_ext(ctx, inputs.uniform_residues(973, np.concatenate([P.q, P.p]), P.n, 0), level, 2.0**20)
    out = K.ckks_ct_create(ctx, level)
    runs = {"term": lambda: K.ckks_linear_transform(ctx, c, [0], [None], [w], out),
            "pmult": lambda: K.ckks_pmult(ctx, c, w, out)}
    got, us = {}, {}
    try:
        for name, run in runs.items():
            run()
            got[name] = K.ckks_ct_export(ctx, out, P.n)[0]
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                for _ in range(50):
                    run()
            best = []
            for _ in range(20):
                begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                with torch.cuda.stream(stream):
                    begin.record()
                    graph.replay()
                    end.record()
                torch.cuda.synchronize()
                best.append(begin.elapsed_time(end) / 50 * 1e3)
            us[name] = min(best)
            del graph
    finally:
        K.ckks_ctx_destroy(ctx)
    assert np.array_equal(got["term"], got["pmult"])
    assert us["term"] < 1.5 * us["pmult"], us
