"""ROIs with non-finite pixels: a NaN or an infinity makes the whole correlation NaN (through the mean), so there
is no peak.  Such a ROI reports what a ROI outside the image does (q NaN, no peak, height 0, no tie) and the
other ROIs are those of the finite image, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [16, 32, 64, 128, 256])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("where", ["test", "reference"])
def test_nonfinite_roi_has_no_peak(S, bad, where):
    import torch
    import paper_1907_05993_gb300 as P
    rng = np.random.default_rng(S)
    H, W, B = S, 2 * S, 2
    ref = rng.standard_normal((B, H, W)).astype(np.float32)
    test = np.roll(ref, (1, -2), (1, 2)) + 0.1 * rng.standard_normal(ref.shape).astype(np.float32)
    roi = torch.from_numpy(np.array([[S // 2, S // 2], [S + S // 2, S // 2]], np.int32)).cuda()   # side by side
    ctx = P.hrebsd_create(0)

    def run(r, t):
        q, peak = torch.empty((B, 2, 2), device="cuda"), torch.full((B, 2, 2), -7, dtype=torch.int32, device="cuda")
        ph, tie = torch.empty((B, 2), device="cuda"), torch.full((B, 2), -7, dtype=torch.int32, device="cuda")
        P.hrebsd_xcf_roi_batch(ctx, torch.from_numpy(r).cuda(), torch.from_numpy(t).cuda(), B, H, W, roi, 2, S, 1, q,
                               peak, ph, tie)
        P.hrebsd_device_error(ctx)
        return [x.cpu().numpy() for x in (q, peak, ph, tie)]

    good = run(ref, test)
    assert np.isfinite(good[0]).all()
    r, t = ref.copy(), test.copy()
    (t if where == "test" else r)[1, S // 3, S + S // 5] = bad   # pair 1, ROI 1
    out = run(r, t)
    q, peak, ph, tie = (x[1, 1] for x in out)
    assert np.isnan(q).all() and (peak == 0).all() and ph == 0 and tie == 0
    for a, b in zip(out, good):
        a[1, 1] = b[1, 1] = 0
        assert np.array_equal(a, b)
    P.hrebsd_destroy(ctx)
