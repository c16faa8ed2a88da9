"""A registration captured into the caller's graph allocates nothing: a context whose workspace an earlier call
of the same size has made large enough takes the call, also where that earlier call ran without a stop rule (the
strip-and-band sweep keeps d for the stop rule's SSD) or on fewer levels of this form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_capture_after_a_call_without_stop_rule():
    import torch
    import paper_1907_05993_gb300 as P
    B, H, W, R = 152, 300, 311, 3
    rng = np.random.default_rng(5)
    y, x = np.mgrid[0:H, 0:W]
    refs = np.stack([np.cos(0.2 * x + 0.1 * k * y) + np.cos(0.13 * y + k) for k in range(R)]).astype(np.float32)
    idx = (np.arange(B) % R).astype(np.int32)
    tests = np.stack([np.roll(refs[i], (int(rng.integers(-2, 3)), int(rng.integers(-2, 3))), (0, 1)) for i in idx])
    tests = tests + 0.05 * rng.standard_normal(tests.shape, dtype=np.float32)
    refs, tests, idx = (torch.from_numpy(a).cuda() for a in (refs, tests, idx))
    plain = P.demons_params(1, [25])
    stop = P.demons_params(1, [25], 1.0, 1.0, 1.0, 1e-3, 5)

    def run(ctx, prm, out):
        P.hrebsd_demons_register_batch(ctx, refs, tests, idx, R, B, H, W, prm, None, *out)

    outs = lambda: (torch.empty((B, 2, H, W), device="cuda"), torch.empty((B, 1), dtype=torch.int32, device="cuda"),
                    torch.empty((B,), dtype=torch.int32, device="cuda"))
    own = P.hrebsd_create(0)
    expect = outs()
    run(own, stop, expect)
    P.hrebsd_device_error(own)
    P.hrebsd_destroy(own)
    assert expect[1].min() < 25   # the stop rule acts

    ctx = P.hrebsd_create(0)
    run(ctx, plain, outs())
    for _ in range(2):   # the second time after a call with the rule has made room for d
        out = outs()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run(ctx, stop, out)
        graph.replay()
        torch.cuda.synchronize()
        P.hrebsd_device_error(ctx)
        for a, b in zip(out, expect):
            assert torch.equal(a, b)
        del graph
        run(ctx, stop, outs())
    P.hrebsd_destroy(ctx)
