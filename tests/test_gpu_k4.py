"""K4's outputs wherever the caller keeps them: device memory at 16-byte and at odd 8-byte
addresses, page-locked and pageable host memory, some outputs left out; grids of one tile,
ragged tiles and many tiles, mirrored from [k][l] and from [l][k]; the values are the same
bits whatever the destination.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KEYS = ("S2", "S3", "S4", "S2_err", "S3_err", "S4_err")


@pytest.mark.parametrize("C,T,precision", [(1, 8, "fp32"), (1, 64, "fp32"), (1, 256, "tf32x3"),
                                           (1, 1024, "fp32"), (2, 32, "fp32")])
def test_destinations_agree(C, T, precision):
    import paper_2505_01231_gb300 as mod
    m, G = 6, 9
    n = T * m * G
    z = synth.ar1_quadratic(n, seed=T) if C == 1 else synth.multichannel_shared(C, n, seed=T)
    plan = mod.Plan(channels=C, T=T, dt=0.5, m=m, precision=precision)
    plan.accumulate(torch.from_numpy(np.ascontiguousarray(z)).cuda())
    sh = plan.shapes()
    size = {k: 2 * int(np.prod(sh[k[:2]])) for k in KEYS}
    ref = plan.finalize()                                    # pageable host memory
    want = {}
    for k in KEYS:
        v = ref[k]
        want[k] = (v if k.endswith("err") else np.stack([v.real, v.imag], -1)).reshape(-1)
    M = T // 2 + 1
    if C == 1:
        for key in ("S3", "S4"):
            assert np.array_equal(ref[key][0], ref[key][0].T)
        k, l = np.indices((M, M))
        assert np.all(ref["S3"][0][k + l > M - 1] == 0)

    def run(bufs):
        mod.ss_finalize(plan.handle, *[bufs.get(k) for k in KEYS])
        torch.cuda.synchronize()
        for k, b in bufs.items():
            got = b.cpu().numpy() if hasattr(b, "cpu") else b
            assert np.array_equal(got.reshape(-1), want[k]), k

    run({k: torch.empty(size[k], dtype=torch.float64, device="cuda") for k in KEYS})
    run({k: torch.empty(size[k] + 1, dtype=torch.float64, device="cuda")[1:] for k in KEYS})
    run({k: torch.empty(size[k], dtype=torch.float64).pin_memory() for k in KEYS})
    run({"S3": torch.empty(size["S3"], dtype=torch.float64, device="cuda"),
         "S4_err": np.empty(size["S4_err"])})
    plan.close()
