"""The independent-warp bispectrum kernel at the edges of its work split: fewer groups
than an item has warps, groups that end inside a stage, items of one group and of the
longest, sub-tiles below bin 0 (several channels) and the sub-tiles of isolated
points.  Against the 64 x 64 tiles of k2=84s2: both within 1e-5 of the definition.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,T,m,G", [(1, 8, 4, 2), (1, 64, 5, 3), (1, 256, 11, 7),
                                     (1, 32, 3, 5000), (1, 1024, 10, 700), (2, 8, 3, 5),
                                     (2, 16, 4, 2), (3, 64, 5, 9), (2, 256, 6, 300),
                                     (4, 32, 7, 1000)])
def test_warp_items_match_the_tiles(C, T, m, G):
    import paper_2505_01231_gb300 as mod
    n = T * m * G + 5
    z = synth.ar1_quadratic(n, seed=T + G) if C == 1 else synth.multichannel_shared(C, n, seed=G)
    z = torch.from_numpy(np.ascontiguousarray(z)).cuda()
    outs = []
    for form in ("k2=84s2", "k2=84w"):
        plan = mod.Plan(channels=C, T=T, dt=0.5, m=m, orders=(3,))
        mod.ss_set_tuning(plan.handle, form)
        plan.accumulate(z)
        outs.append(plan.finalize())
        plan.close()
    a, b = outs
    assert np.max(np.abs(a["S3"] - b["S3"])) <= 2e-5 * np.max(np.abs(a["S3"]))
    assert np.max(np.abs(a["S3_err"] - b["S3_err"])) <= 2e-4 * np.max(a["S3_err"])
