"""The Gaussian core of the near field (Eq. vem1), pair by pair: two elements at distances from far
inside the core to beyond its cut, each pair a system of its own, against the closed form in FP64."""
import numpy as np
import pytest

from oracle.direct import core_dK, core_K
from tests.gpu_util import dev, host3

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a", [1e-4, 0.006283, 0.37, 12.0])
@pytest.mark.parametrize("tpt", [1, 2, 4])
def test_pairs_across_the_core(a, tpt):
    """Each term of v and s carries 1/r^3 or 1/r^5 from rsqrt.approx (2^-22.9, five times), the fit
    (2.3e-7) and about ten roundings: 5 2^-22.9 + 2.3e-7 + 10 2^-24 = 1.5e-6 of its size."""
    from paper_1201_5430_gb300 import LHV
    rng = np.random.default_rng(5)
    x = np.concatenate([np.geomspace(0.02, 9.0, 300), [1.4999, 1.5, 1.5001, 6.4999, 6.5, 6.5001]])
    n = x.size
    u = rng.standard_normal((n, 3))
    d = (u / np.linalg.norm(u, axis=1)[:, None] * (x * a)[:, None]).astype(np.float32)
    w = rng.standard_normal((2 * n, 3)).astype(np.float32)
    pos = np.zeros((2 * n, 3), dtype=np.float32)
    pos[1::2] = d  # the first of each pair at the origin: the FP32 difference is exact
    c = LHV(p=4, leaf_max=64, core_a=a, precision="fp32", terms="near")
    c.set_launch_shape(p2p_targets_per_thread=tpt)
    v4, s4 = c.evaluate_batched(list(range(0, 2 * n + 1, 2)), dev(pos, "fp32"), dev(w, "fp32"))
    v, s = host3(v4), host3(s4)
    r = np.linalg.norm(d.astype(np.float64), axis=1)
    K, dK = core_K(r, a), core_dK(r, a)
    small = r < 0.1 * a  # the series of K where its closed form cancels
    y = (r / a) ** 2
    ser = np.sqrt(2 / np.pi) * (1 / 3 - y / 10 + y ** 2 / 56 - y ** 3 / 432)
    f = np.where(small, ser / a ** 3, K / r ** 3)
    g = np.where(small, np.sqrt(2 / np.pi) * (-1 / 5 + y / 14 - y ** 2 / 72) / a ** 5, (dK / r ** 3 - 3 * K / r ** 4) / r)
    for i in (0, 1):  # target i of each pair, source 1 - i
        dd = (d if i == 1 else -d).astype(np.float64)
        wj, wi = w[1 - i::2].astype(np.float64), w[i::2].astype(np.float64)
        cr = np.cross(wj, dd)
        ve = f[:, None] * cr
        se = f[:, None] * np.cross(wj, wi) + (g * np.sum(wi * dd, axis=1))[:, None] * cr
        nj, ni = np.linalg.norm(wj, axis=1), np.linalg.norm(wi, axis=1)
        sv, ss = f * nj * r, (f + np.abs(g) * r * r) * nj * ni
        assert np.max(np.linalg.norm(v[i::2] - ve, axis=1) / sv) < 1.5e-6
        assert np.max(np.linalg.norm(s[i::2] - se, axis=1) / ss) < 1.5e-6


@pytest.mark.parametrize("n,leaf", [(300, 4), (2000, 12), (4000, 24), (4000, 48), (3001, 150)])
@pytest.mark.parametrize("a", [0.0, 0.03])
def test_fp64_source_strands_equal_one_strand(n, leaf, a):
    """FP64 near field with 1 to 8 source strands (mean leaves from a few elements to more than a
    tile) against the unsplit kernel (two targets per thread): the same terms in another order,
    n 2^-53 of the sum of their sizes at most; s cancels to about 1e-3 of it."""
    import workloads
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.cube(n, 3)
    got = []
    for tpt in (1, 2):
        c = LHV(p=4, leaf_max=leaf, core_a=a, precision="fp64", terms="near")
        c.set_launch_shape(p2p_targets_per_thread=tpt)
        v4, s4 = c.evaluate_velocity_stretching(dev(x, "fp64"), dev(w, "fp64"))
        got.append((host3(v4), host3(s4), c.stats()["p2p_pairs"]))
        c.close()
    assert got[0][2] == got[1][2]
    for p, q in zip(got[0][:2], got[1][:2]):
        assert np.linalg.norm(p - q) < n * 2.0 ** -53 * 1e3 * np.linalg.norm(q)
