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


@pytest.mark.parametrize("prec", ["fp32", "fp64", "tf32x3"])
@pytest.mark.parametrize("n,leaf", [(600, 8), (4000, 300)])
def test_one_term_expansions(prec, n, leaf):
    """p = 1, the smallest truncation number: a far field of constants per leaf, so v, s and grad phi are zero
    and phi is the oracle's, for vortex elements, filaments, the scalar case and a leaf level of p = 1 below
    longer expansions.  Positive charges: phi adds positive terms, at most the elements of a leaf, 8 L children and
    189 L pairs in a chain, each one rounding, 20 more for the tables' own."""
    import torch
    from oracle import scalar
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.cube(n, 5)
    q = np.abs(workloads.charges(n, 6))
    e = "fp64" if prec == "fp64" else "fp32"
    t = torch.float64 if prec == "fp64" else torch.float32
    ref = scalar.fmm_scalar(x, q, 1, leaf_max=leaf, near=False)
    assert ref.tree.L >= 2
    c = LHV(p=1, leaf_max=leaf, core_a=0.0, precision=prec, terms="far")
    v4, s4 = c.evaluate_velocity_stretching(dev(x, e), dev(w, e))
    assert c.stats()["leaf_level"] == ref.tree.L
    assert not v4.any() and not s4.any()
    pg = c.evaluate_potential_gradient(dev(x, e), torch.from_numpy(q.astype(np.float64)).to("cuda", t))
    assert not pg[:, :3].any()
    eps = 2.0 ** (-53 if prec == "fp64" else -24)
    bound = (leaf + 197 * ref.tree.L + 20) * eps
    assert np.max(np.abs(pg[:, 3].double().cpu().numpy() - ref.phi) / ref.phi) < bound
    assert not c.evaluate_filaments([0, n], [True], dev(x, e), torch.ones(n, device="cuda", dtype=t)).any()
    c.close()
    c = LHV(p=6, leaf_max=leaf, core_a=0.0, precision=prec, terms="far")
    c.set_level_p([0] * ref.tree.L + [1])
    v4, s4 = c.evaluate_velocity_stretching(dev(x, e), dev(w, e))
    assert not v4.any() and not s4.any()
    c.close()


@pytest.mark.parametrize("n,leaf", [(600, 8), (4000, 300)])
def test_two_term_expansions(n, leaf):
    """p = 2: v and s of the FP64 context are the oracle's (1e-10, as at every other p), the FP32 one's
    to 2e-6 as above."""
    from oracle import fmm
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.cube(n, 5)
    ref = fmm.fmm(x, w, 2, leaf_max=leaf, near=False)
    assert ref.tree.L >= 2
    for prec, tol in (("fp64", 1e-10), ("fp32", 2e-6)):
        c = LHV(p=2, leaf_max=leaf, core_a=0.0, precision=prec, terms="far")
        v4, s4 = c.evaluate_velocity_stretching(dev(x, prec), dev(w, prec))
        assert rel(host3(v4), ref.v) < tol and rel(host3(s4), ref.s) < tol, (rel(host3(v4), ref.v), rel(host3(s4), ref.s))
        c.close()
