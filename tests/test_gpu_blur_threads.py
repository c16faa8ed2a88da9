"""The blur's shared-memory limit belongs to the kernel, not to a handle: calls of different radii from two host
threads, each with a handle and a stream of its own, may not lower each other's."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_blurs_of_different_radii_from_two_threads():
    import torch
    import paper_1907_05993_gb300 as P
    x = torch.from_numpy(np.random.default_rng(0).uniform(1, 2, (1, 256, 256)).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    failed, results = [], {}

    def work(sigma):   # radii 66 and 96: both need more than the 48 KB that every launch may use
        ctx, out, stream = P.hrebsd_create(0), torch.empty_like(x), torch.cuda.Stream()
        try:
            for _ in range(4000):
                P.hrebsd_bandpass_batch(ctx, x, 1, 256, 256, sigma, 0.0, out, stream=stream)
            stream.synchronize()
            results[sigma] = out.cpu().numpy()
        except P.HrebsdError as e:
            failed.append((sigma, str(e)))
        stream.synchronize()
        P.hrebsd_destroy(ctx)

    threads = [threading.Thread(target=work, args=(s,)) for s in (22.0, 32.0)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    ctx, out = P.hrebsd_create(0), torch.empty_like(x)
    for sigma, r in results.items():
        P.hrebsd_bandpass_batch(ctx, x, 1, 256, 256, sigma, 0.0, out)
        assert np.array_equal(out.cpu().numpy(), r)
    P.hrebsd_destroy(ctx)
