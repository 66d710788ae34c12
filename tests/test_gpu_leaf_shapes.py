"""P2M and L2P at the block shapes that the mean leaf picks (a few elements to several tiles a
leaf): FP32 against the FP64 context of the same tree and p, far field only, for vortex elements,
filaments and the scalar case."""
import numpy as np
import pytest

import workloads
from tests.gpu_util import dev, host3, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [3, 8, 13, 24])
@pytest.mark.parametrize("n,level", [(3000, 4), (1500, 2), (2500, 2), (3500, 2), (6000, 2), (30000, 2)])
def test_fp32_far_field_equals_fp64(p, n, level):
    """Mean leaves from about 1 to 470 elements.  Every coefficient and every field value sums at
    most 2 p^2 rounded terms: sqrt(2 24^2) 2^-24 = 2e-6."""
    import torch
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.cube(n, level)
    q = workloads.charges(n, 2)
    got = {}
    for prec in ("fp32", "fp64"):
        c = LHV(p=p, leaf_max=1, core_a=0.0, precision=prec, terms="far", max_level=level)
        t = torch.float64 if prec == "fp64" else torch.float32
        v4, s4 = c.evaluate_velocity_stretching(dev(x, prec), dev(w, prec))
        pg = c.evaluate_potential_gradient(dev(x, prec), torch.from_numpy(q).to("cuda", t))
        assert c.stats()["leaf_level"] == level
        got[prec] = (host3(v4), host3(s4), pg.double().cpu().numpy())
        c.close()
    for a, b in zip(got["fp32"], got["fp64"]):
        assert rel(a, b) < 2e-6, rel(a, b)


@pytest.mark.parametrize("n", [900, 4000, 20000])
def test_filaments_need_only_the_velocity(n):
    import torch
    from paper_1201_5430_gb300 import LHV
    th = 2 * np.pi * np.arange(n) / n
    x = np.stack([np.cos(th), np.sin(th), 0.05 * np.sin(3 * th)], axis=1).astype(np.float32)
    got = []
    for prec in ("fp32", "fp64"):
        c = LHV(p=12, leaf_max=1, core_a=0.0, precision=prec, terms="far", max_level=5)
        t = torch.float64 if prec == "fp64" else torch.float32
        got.append(host3(c.evaluate_filaments([0, n], [True], dev(x, prec), torch.ones(n, device="cuda", dtype=t))))
        c.close()
    assert rel(got[0], got[1]) < 2e-6, rel(got[0], got[1])
