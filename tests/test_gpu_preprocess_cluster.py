"""A pattern preprocessed by a cluster of CTAs (few patterns) and by one CTA (many) gives the same bits: the
threads' partial sums are added exactly.  Sizes at the edge of the rule, of 2, 4 and 8 CTAs, whose last chunk is
partial or belongs to any rank, with a fit that is not positive everywhere and with non-finite pixels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W", [(128, 256), (181, 181), (182, 181), (256, 256), (300, 219), (480, 640), (1024, 131)])
@pytest.mark.parametrize("flat", [True, False])
def test_preprocess_cluster_matches_one_cta(H, W, flat):
    import torch
    import paper_1907_05993_gb300 as P
    rng = np.random.default_rng(H * W)
    y, x = np.meshgrid(np.linspace(-1, 1, H), np.linspace(-1, 1, W), indexing="ij")
    pat = np.stack([100.0 * (b + 0.2 * x - 0.3 * y - 0.4 * x * x + 0.1 * x * y - 0.3 * y * y
                             + 0.1 * rng.standard_normal((H, W))) for b in (1.1, 1.3, 0.2)]).astype(np.float32)
    pat = np.concatenate([pat, pat[:1]])
    pat[3, H // 2, W // 3] = np.inf
    ctx = P.hrebsd_create(0)
    many = torch.from_numpy(np.repeat(pat, 100, 0)).cuda()   # 400 patterns: one CTA each
    out = torch.empty_like(many)
    P.hrebsd_preprocess_batch(ctx, many, 400, H, W, flat, out)
    exp = out.cpu().numpy()[::100]
    for n in (1, 2, 4):
        d = torch.from_numpy(pat).cuda()
        for k in range(0, 4, n):   # in place
            P.hrebsd_preprocess_batch(ctx, d[k:k + n], n, H, W, flat, d[k:k + n])
        assert np.array_equal(d.cpu().numpy(), exp, equal_nan=True)
    P.hrebsd_destroy(ctx)
