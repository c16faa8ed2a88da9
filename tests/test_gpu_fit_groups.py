"""The lane-group forms of the Eq. 3 fits (4 lanes or a warp per pair) at the edges of their ranges:
few and many pairs, ROI counts below, at and above the lane and shared-memory limits."""
import math

import numpy as np
import pytest

from synth import kikuchi as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 7, 700])      # a warp per pair; 700: 4 lanes per pair while N <= 64
@pytest.mark.parametrize("N", [4, 5, 25, 64, 65, 512])
def test_fit_groups_parity(B, N):
    import torch
    import oracle
    import paper_1907_05993_gb300 as P
    H, W, geom = 96, 128, K.Geometry()
    rng = np.random.default_rng(N + B)
    cells = rng.choice(27 * 20, N, replace=False)
    roi = np.stack([10 + 4 * (cells % 27), 10 + 4 * (cells // 27)], 1).astype(np.int32)
    if N < 25:   # random placements of so few points can be degenerate
        roi = np.array([[20, 20], [100, 24], [30, 80], [90, 70], [60, 50]], np.int32)[:N]
    x, y = np.meshgrid(np.arange(W) + 0.5 - 0.5 * W, np.arange(H) + 0.5 - 0.5 * H)
    zs = 0.6 * W
    fields, Rs = [], []
    for b in range(min(B, 7)):
        R = K.axis_angle(rng.normal(size=3), math.radians(rng.uniform(0.1, 8)))
        v = np.einsum("ba,bhw->ahw", R, np.stack([x, y, np.full_like(x, zs)]))   # R^T r'
        fields.append(np.stack([x - zs * v[0] / v[2], y - zs * v[1] / v[2]]) + rng.normal(0, 0.05, (2, H, W)))
        Rs.append(R)
    fields = np.stack(fields).astype(np.float32)
    q = rng.normal(0, 0.3, (len(Rs), N, 2)).astype(np.float32)
    pick = np.arange(B) % len(Rs)
    ctx = P.hrebsd_create(0)
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)
    F1, Rf, F = (torch.empty((B, 9), dtype=torch.float64, device="cuda") for _ in range(3))
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    g, d_roi = P.hrebsd_geometry(geom.xstar, geom.ystar, geom.zstar), dev(roi, torch.int32)
    P.hrebsd_fit_rotation(ctx, dev(fields[pick], torch.float32), B, H, W, d_roi, N, g, F1, Rf, st)
    P.hrebsd_solve_F(ctx, dev(q[pick], torch.float32), d_roi, N, B, H, W, g,
                     dev(np.stack(Rs)[pick].reshape(B, 9), torch.float64), F, st)
    assert not st.cpu().numpy().any()
    F1, Rf, F = (t.cpu().numpy().reshape(B, 3, 3) for t in (F1, Rf, F))
    P.hrebsd_destroy(ctx)
    for b in range(len(Rs)):
        eF, eR = oracle.fit_rotation(fields[b].astype(np.float64), roi, geom)
        # the field is sampled in FP32 on the GPU: 1e-6 px of sampling error moves F by at most ~1e-6 / Z*, more
        # where 4 or 5 points determine it; the second pass has no sampling and agrees to FP64 rounding
        assert np.abs(F1[b] - eF).max() < 1e-6 and np.abs(Rf[b] - eR).max() < 1e-6
        assert np.abs(F[b] - oracle.solve_F(q[b].astype(np.float64), roi, H, W, geom, Rs[b])).max() < 1e-10
    for b in range(len(Rs), B):   # the same pair at another place of the batch
        k = pick[b]
        assert np.array_equal(F1[b], F1[k]) and np.array_equal(Rf[b], Rf[k]) and np.array_equal(F[b], F[k])
