"""The reference arrays behind the texture gathers are bounded in number; the sizes that the strip-and-band sweep
meets first may not use up those of the row sweep (levels 64, 128 and 256 pixels wide)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_other_widths_leave_the_row_sweep_its_arrays():
    import torch
    import paper_1907_05993_gb300 as P
    ctx = P.hrebsd_create(0)
    P.hrebsd_set_option(ctx, P.OPT_GRAPHS, 0)
    rng = np.random.default_rng(0)

    def register(R, B, H, W):
        ref = torch.from_numpy(rng.standard_normal((R, H, W)).astype(np.float32)).cuda()
        idx = torch.zeros(B, dtype=torch.int32, device="cuda")
        out = (torch.empty((B, 2, H, W), device="cuda"), torch.empty((B, 1), dtype=torch.int32, device="cuda"),
               torch.empty((B,), dtype=torch.int32, device="cuda"))
        tests = ref[:1].expand(B, H, W).contiguous()
        free = []
        for tex in (0, 1):   # without the gathers first: it grows everything else
            P.hrebsd_set_option(ctx, P.OPT_TEX_GATHER, tex)
            P.hrebsd_demons_register_batch(ctx, ref, tests, idx, R, B, H, W, P.demons_params(1, [2]), None, *out)
            torch.cuda.synchronize()
            free.append(torch.cuda.mem_get_info()[0])
        P.hrebsd_device_error(ctx)
        return free[0] - free[1]

    for w in range(195, 211):   # sizes of the strip-and-band sweep
        register(1, 300, 150, w)
    P.hrebsd_set_tile_variant(ctx, 256, 256, 5)
    assert register(120, 4, 256, 256) >= 28 << 20   # 120 references of 256 x 256: an array of 30 MiB
    P.hrebsd_destroy(ctx)
