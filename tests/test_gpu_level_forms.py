"""Which form a level runs in (hrebsd_level_form), and that the forms chosen by estimate give what the shape they
stand in for gives: the strip-and-band sweep without a stop rule, and both forms on autotuned contexts, where
the stop rule's SSD is regrouped as the tuned shape sums it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _batch(B, H, W):
    rng = np.random.default_rng(B + H * W)
    y, x = np.mgrid[0:H, 0:W]
    refs = np.zeros((2, H, W))
    for r in refs:
        for _ in range(6):
            a, p = rng.uniform(0, np.pi), rng.uniform(0, 6)
            r += np.cos(rng.uniform(8, 30) / 100 * (np.cos(a) * x + np.sin(a) * y) + p)
    refs = (refs / refs.std(axis=(1, 2), keepdims=True)).astype(np.float32)
    idx = (np.arange(B) % 2).astype(np.int32)
    tests = np.stack([np.roll(refs[i], (int(rng.integers(-2, 3)), int(rng.integers(-2, 3))), (0, 1)) for i in idx])
    return refs, tests + 0.05 * rng.standard_normal(tests.shape, dtype=np.float32), idx


def _run(ctx, data, prm):
    import torch
    import paper_1907_05993_gb300 as P
    refs, tests, idx = (torch.from_numpy(a).cuda() for a in data)
    B, H, W = tests.shape
    out = (torch.empty((B, 2, H, W), device="cuda"), torch.empty((B, prm.levels), dtype=torch.int32, device="cuda"),
           torch.empty((B,), dtype=torch.int32, device="cuda"))
    P.hrebsd_demons_register_batch(ctx, refs, tests, idx, len(refs), B, H, W, prm, None, *out)
    P.hrebsd_device_error(ctx)
    return [t.cpu().numpy() for t in out], [P.hrebsd_level_form(ctx, l) for l in range(prm.levels)]


def _pinned(data, prm, shapes):
    import paper_1907_05993_gb300 as P
    ctx = P.hrebsd_create(0)
    for l, v in enumerate(shapes):
        P.hrebsd_set_tile_variant(ctx, data[1].shape[1] >> l, data[1].shape[2] >> l, v)
    out = _run(ctx, data, prm)
    P.hrebsd_destroy(ctx)
    return out


def test_form_of_each_level():
    import paper_1907_05993_gb300 as P
    ctx = P.hrebsd_create(0)
    with pytest.raises(P.HrebsdError):
        P.hrebsd_level_form(ctx, 0)                      # no registration yet
    data = _batch(1, 128, 128)
    assert _run(ctx, data, P.demons_params(2, [5, 5]))[1] == [P.FORM_CLUSTER] * 2
    for l in (-1, 2, 8):
        with pytest.raises(P.HrebsdError):
            P.hrebsd_level_form(ctx, l)                  # a level that the registration did not have
    P.hrebsd_destroy(ctx)
    for shape, ran in ((0, 0), (4, 4), (5, 6), (6, 6)):  # one pair: shape 5 in its one-launch form
        assert _pinned(data, P.demons_params(1, [5]), [shape])[1] == [ran]
    assert _pinned(data, P.demons_params(1, [1]), [5])[1] == [5]
    assert _pinned(_batch(1, 64, 64), P.demons_params(1, [5]), [7])[1] == [7]
    assert _pinned(_batch(1, 64, 61), P.demons_params(1, [5]), [0])[1] == [P.FORM_PLAIN]


@pytest.mark.parametrize("B,H,W,levels,cap", [(16, 1024, 1244, 2, 6), (600, 92, 100, 1, 1), (400, 77, 270, 1, 7),
                                              (60, 61, 1021, 1, 12)])
def test_strip_band_sweep_runs_without_stop_rule(B, H, W, levels, cap):
    import paper_1907_05993_gb300 as P
    data, prm = _batch(B, H, W), P.demons_params(levels, [cap] * levels)
    ctx = P.hrebsd_create(0)
    out, forms = _run(ctx, data, prm)
    P.hrebsd_destroy(ctx)
    assert forms[0] == P.FORM_STRIPS
    for a, b in zip(out, _pinned(data, prm, [0] * levels)[0]):
        assert np.array_equal(a, b)


# form: the one that the finest level has to run in (None: as the estimate for the tuned shape says)
@pytest.mark.parametrize("B,H,W,levels,form", [(1, 128, 128, 3, 8), (3, 64, 64, 2, None), (40, 64, 64, 2, None),
                                               (5, 100, 92, 3, 8), (150, 100, 92, 3, 8), (152, 300, 312, 1, None),
                                               (16, 512, 624, 3, None), (600, 92, 100, 1, None)])
def test_autotuned_levels_count_as_the_tuned_shape(B, H, W, levels, form):
    import paper_1907_05993_gb300 as P
    data, prm = _batch(B, H, W), P.demons_params(levels, [40] * levels, 1.0, 1.0, 1.0, 1e-3, 5)
    ctx = P.hrebsd_create(0)
    P.hrebsd_autotune(ctx, B, H, W, prm)
    shapes = [P.hrebsd_get_tile_variant(ctx, H >> l, W >> l) for l in range(levels)]
    out, forms = _run(ctx, data, prm)
    P.hrebsd_destroy(ctx)
    assert form is None or forms[0] == form
    pinned, ran = _pinned(data, prm, shapes)
    assert all(f not in (P.FORM_CLUSTER, P.FORM_STRIPS) for f in ran)
    for a, b in zip(out, pinned):
        assert np.array_equal(a, b)
    assert out[1].min() < 40   # the stop rule acts
