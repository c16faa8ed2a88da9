"""The preprocessing's chunks of 8 pixels per thread at sizes that do not fill them (fewer pixels than threads,
one pixel past a chunk, odd widths), in place, several sizes through one context's plans, and repeated calls."""
import numpy as np
import pytest

from synth import kikuchi as K

pytestmark = pytest.mark.gpu


def test_preprocess_chunks():
    import torch
    import oracle
    import paper_1907_05993_gb300 as P
    ctx = P.hrebsd_create(0)
    sizes = [(8, 8), (9, 57), (17, 31), (64, 64), (1, 513)[::-1], (65, 63), (4096 // 16 + 1, 16), (100, 92), (23, 1500)]
    for rep in range(2):   # more sizes than the context keeps plans for, twice
        for H, W in sizes:
            if min(H, W) < 3:
                continue
            spec = K.ScanSpec(n_pairs=3, H=H, W=W, seed=11)
            x = np.stack([K.render_test(spec, p) for p in range(3)]).astype(np.float32)
            for flat in (0, 1):
                d = torch.from_numpy(x).cuda()
                out = torch.empty_like(d)
                P.hrebsd_preprocess_batch(ctx, d, 3, H, W, flat, out)
                P.hrebsd_preprocess_batch(ctx, d, 3, H, W, flat, d)   # in place
                got = out.cpu().numpy()
                assert np.array_equal(got, d.cpu().numpy())
                for b in range(3):
                    exp = oracle.preprocess(x[b].astype(np.float64), flat=bool(flat))
                    ulps = np.abs(got[b] - exp) / np.spacing(np.maximum(np.abs(exp), 1.0).astype(np.float32))
                    assert ulps.max() <= 32   # the bar of the parity test at the usual sizes
    P.hrebsd_destroy(ctx)
