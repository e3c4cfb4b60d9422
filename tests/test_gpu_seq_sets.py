"""Several blocks of sequential spectra in one batch: the sums of each block kept apart by
every kernel (S2 in the resident, the two-kernel and the register forms of K1, K2, the S4
contraction, the tensor-core S4 and its column kernel), calls that start inside a block,
fewer blocks kept than completed, more blocks than one set holds.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL, TOL_ERR = 1e-5, 1e-4


@pytest.mark.parametrize("T,m,B,G,orders,precision,keep,cuts", [
    (64, 6, 5, 43, (2, 3, 4), "fp32", 6, (0.13, 0.31)),
    (128, 5, 3, 40, (2, 3, 4), "fp16x3", 99, ()),
    (128, 10, 7, 61, (2, 3, 4), "tf32x3", 8, (0.5,)),
    (256, 4, 2, 31, (2, 4), "fp32", 99, (0.2,)),
    (1024, 3, 4, 21, (2,), "fp32", 99, (0.4,)),
    (2048, 4, 2, 6, (2, 3), "fp32", 99, ()),
    (16, 3, 9, 5200, (2, 3), "fp32", 560, ()),
])
def test_block_sets_match_the_oracle(T, m, B, G, orders, precision, keep, cuts):
    import paper_2505_01231_gb300 as mod
    z = synth.ar1_quadratic(T * m * G + 11, seed=T + B)
    ref = oracle.sequential_spectra(z, T, 0.5, m, B, orders=orders)
    full = oracle.polyspectra(z, T, 0.5, m, orders=orders, group_chunk=32)
    plan = mod.Plan(T=T, dt=0.5, m=m, orders=orders, precision=precision)
    plan.sequential(B, keep)
    zd = torch.from_numpy(z).cuda()
    at = [0] + [int(c * z.size) for c in cuts] + [z.size]
    for _ in range(2):                                    # and again after a reset
        plan.reset()
        for a, b in zip(at, at[1:]):
            plan.accumulate(zd[a:b])
        out = plan.finalize()
    assert mod.ss_sequential_info(plan.handle)[1] == G // B == ref["blocks"]
    got = plan.blocks()
    plan.close()
    assert len(got) == min(keep, G // B)
    for o in orders:
        key = f"S{o}"
        r = full[key]
        assert np.max(np.abs(out[key][0].reshape(r.shape) - r)) <= TOL * np.max(np.abs(r))
        for b, blk in enumerate(got):
            r, re = ref[key][b], ref[key + "_err"][b]
            assert np.max(np.abs(blk[key][0].reshape(r.shape) - r)) <= TOL * np.max(np.abs(r)), (key, b)
            e = blk[key + "_err"][0].reshape(re.shape)
            assert np.max(np.abs(e - re)) <= TOL_ERR * np.max(re), (key, b)
