"""M2L by rotation - coaxial translation - back rotation (Sec. 4.4, Eq. rcr1) on the GPU,
against the oracle's FMM with every translation by RCR (same p and tree): FP32 within
1e-6 relative L2 of v and s; the form against the fused-table form on the same inputs at
p = 12, 16, 20 (multi-level trees with full interaction lists); an RK4 step and a CUDA
graph replay of it equal to the uncaptured step; the unsupported configurations."""
import numpy as np
import pytest

import workloads
from oracle import rcr
from tests.gpu_util import dev, host3, rel

pytestmark = pytest.mark.gpu


def _ctx(p, leaf, a, prec="fp32", form="rcr", terms="all"):
    from paper_1201_5430_gb300 import LHV
    c = LHV(p=p, leaf_max=leaf, core_a=a, eps=1e-6, precision=prec, terms=terms)
    c.set_form(form)
    return c


@pytest.mark.parametrize("case", ["cube", "ring"])
def test_parity_with_oracle_rcr(case):
    if case == "cube":
        x, w = workloads.cube(2500, 41)
        a, p, leaf = 0.01, 8, 24
    else:
        x, w = workloads.ring(8000, 1)
        a, p, leaf = workloads.RING_CORE_A, 12, 64
    ref = rcr.fmm_rcr(x, w, p, leaf_max=leaf, a=a)
    c = _ctx(p, leaf, a)
    v4, s4 = c.evaluate_velocity_stretching(dev(x, "fp32"), dev(w, "fp32"))
    assert c.stats()["leaf_level"] == ref.tree.L >= 3
    ev, es = rel(host3(v4), ref.v), rel(host3(s4), ref.s)
    print(f"rcr {case} p={p}: rel L2 v {ev:.2e} s {es:.2e}")
    assert ev < 1e-6 and es < 1e-6, (ev, es)


@pytest.mark.parametrize("p", [12, 16, 20])
def test_equals_fused_form(p):
    x, w = workloads.cube(60000, 7)
    out = {}
    for form in ("phi_chi", "rcr"):
        c = _ctx(p, 32, 0.002, "fp32", form, terms="far")
        v4, s4 = c.evaluate_velocity_stretching(dev(x, "fp32"), dev(w, "fp32"))
        out[form] = (host3(v4), host3(s4))
        assert c.stats()["leaf_level"] >= 4
    ev = rel(out["rcr"][0], out["phi_chi"][0])
    es = rel(out["rcr"][1], out["phi_chi"][1])
    print(f"rcr vs fused p={p}: far field rel L2 v {ev:.2e} s {es:.2e}")
    assert ev < 2e-6 and es < 2e-6, (ev, es)


def test_step_and_graph_replay():
    import torch
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.ring(6000, 3)
    a = workloads.RING_CORE_A
    res = []
    for form, graph in (("phi_chi", False), ("rcr", False), ("rcr", True)):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            c = LHV(p=12, leaf_max=64, core_a=a, eps=1e-6, precision="fp32")
            c.set_form(form)
            if graph:
                c.set_graph(True)
            x4, w4 = dev(x, "fp32"), dev(w, "fp32")
            for _ in range(3):
                c.step(x4, w4, 1e-3)
        s.synchronize()
        res.append((host3(x4), host3(w4)))
        if graph:
            assert c.stats()["graph"]["replays"] >= 1
    x0 = x.astype(np.float64)
    assert rel(res[1][0] - x0, res[0][0] - x0) < 1e-5
    assert rel(res[1][1], res[0][1]) < 1e-6
    assert rel(res[2][0] - x0, res[1][0] - x0) < 1e-5
    assert rel(res[2][1], res[1][1]) < 1e-6


def test_unsupported():
    from paper_1201_5430_gb300 import LHVError
    x, w = workloads.cube(3000, 2)
    for kw, lp in ((dict(p=8, prec="fp64"), None), (dict(p=22, prec="fp32"), None), (dict(p=8, prec="fp32"), [0, 0, 6, 8])):
        c = _ctx(kw["p"], 16, 0.01, kw["prec"])
        if lp:
            c.set_level_p(lp)
        with pytest.raises(LHVError) as e:
            c.evaluate_velocity_stretching(dev(x, kw["prec"]), dev(w, kw["prec"]))
        assert e.value.status == -6


def _default_and_fused(run, **kw):
    """run(context) with the default M2L of the two-potential form and with the fused tables
    (chosen by a CUDA-core chunk)."""
    from paper_1201_5430_gb300 import LHV
    out = []
    for nc in (0, 64):
        c = LHV(**kw)
        c.set_launch_shape(m2l_pairs_per_chunk=nc)
        out.append(run(c))
        assert c.stats()["m2l_pairs"] > 0
        c.close()
    return out


@pytest.mark.parametrize("prec,p", [("fp32", p) for p in (3, 4, 5, 7, 8, 10, 13, 17, 20, 21)]
                         + [("fp64", p) for p in (4, 7, 12, 16, 17)] + [("tf32x3", 10)])
@pytest.mark.parametrize("n,leaf", [(700, 8), (6000, 16)])
def test_default_translations_equal_the_fused_tables(prec, p, n, leaf):
    """The default M2L of the two-potential form (RCR where its tables fit) against the fused
    tables, far field only, few and many pairs a chunk, p outside RCR's range included.  Both
    sides round about 2 p^2 terms: sqrt(2 21^2) 2^-24 = 2e-6 in FP32; in FP64 the quadrature of the
    rotation blocks adds 2 p^2 terms of its own, 1e-12."""
    x, w = workloads.cube(n, 11)
    e = "fp64" if prec == "fp64" else "fp32"

    def run(c):
        v4, s4 = c.evaluate_velocity_stretching(dev(x, e), dev(w, e))
        return host3(v4), host3(s4)

    a, b = _default_and_fused(run, p=p, leaf_max=leaf, core_a=0.0, precision=prec, terms="far")
    tol = 1e-12 if prec == "fp64" else 2e-6
    assert rel(a[0], b[0]) < tol and rel(a[1], b[1]) < tol, (rel(a[0], b[0]), rel(a[1], b[1]))


def test_default_translations_of_filaments_and_batches():
    import torch
    th = 2 * np.pi * np.arange(3000) / 3000
    x = np.stack([np.cos(th), np.sin(th), np.zeros(3000)], axis=1).astype(np.float32)
    g = torch.ones(3000, device="cuda")
    a, b = _default_and_fused(lambda c: host3(c.evaluate_filaments([0, 3000], [True], dev(x, "fp32"), g)),
                              p=12, leaf_max=16, core_a=0.0, precision="fp32", terms="far")
    assert rel(a, b) < 2e-6, rel(a, b)
    systems = workloads.blob_systems(nsys=3, seed=9, n_lo=1e3, n_hi=4e3)
    xs, ws = (np.concatenate([q[k] for q in systems]) for k in (0, 1))
    off = np.cumsum([0] + [q[0].shape[0] for q in systems]).tolist()
    a, b = _default_and_fused(lambda c: host3(c.evaluate_batched(off, dev(xs, "fp32"), dev(ws, "fp32"))[0]),
                              p=8, leaf_max=16, core_a=0.0, precision="fp32", terms="far")
    assert rel(a, b) < 2e-6, rel(a, b)


@pytest.mark.parametrize("n,leaf,nsys", [(65, 1, 1), (700, 1, 1), (3000, 8, 1), (20000, 4, 1), (900, 4, 7)])
def test_pair_list_against_the_definition(n, leaf, nsys):
    """The M2L pair list (blocks of target boxes, pairs ranked per offset slot): as many pairs as the
    interaction lists of the exported boxes hold, and as the list of the route with a truncation number
    per level (the interaction table); few and many boxes a block, several systems.  What the pairs
    carry is compared with the oracle elsewhere."""
    from paper_1201_5430_gb300 import LHV
    rng = np.random.default_rng(n)
    x = rng.random((n * nsys, 3)).astype(np.float32)
    w = rng.standard_normal((n * nsys, 3)).astype(np.float32)
    off = [n * k for k in range(nsys + 1)]
    got = []
    for mixed in (False, True):
        c = LHV(p=6, leaf_max=leaf, core_a=0.0, precision="fp32", terms="far")
        c.set_launch_shape(m2l_pairs_per_chunk=64)
        if mixed:
            c.set_level_p([0, 0, 5])
        c.evaluate_batched(off, dev(x, "fp32"), dev(w, "fp32"))
        st = c.stats()
        if not mixed:
            L = st["leaf_level"]
            want = 0
            for l in range(2, L + 1):
                keys = c.export("box_keys", l).cpu().numpy().astype(np.uint64)
                sysid = keys >> np.uint64(3 * l)
                q = np.zeros((keys.size, 3), dtype=np.int64)
                for b in range(l):
                    for d in range(3):
                        q[:, d] |= ((keys >> np.uint64(3 * b + d)) & np.uint64(1)).astype(np.int64) << b
                for i in range(keys.size):
                    same = sysid == sysid[i]
                    far = np.abs(q - q[i]).max(axis=1) > 1
                    near_parent = np.abs((q >> 1) - (q[i] >> 1)).max(axis=1) <= 1
                    want += int(np.sum(same & far & near_parent))
            assert st["m2l_pairs"] == want
        got.append(st["m2l_pairs"])
        c.close()
    assert got[0] == got[1]


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("n,leaf", [(700, 8), (40000, 8)])
def test_form_of_few_terms_equals_the_fused_tables(p, n, leaf):
    """LHV_FORM_RCR at the smallest p, one and many chunks a block: rows of 8 to 128 bytes, of which those of
    p = 2 are whole 16-byte pieces but too short for the 16-byte route.  The locals of every level and the far
    field against the fused tables', to the rounding of the sums as above (2e-6)."""
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.cube(n, 12)
    got = []
    for form in ("rcr", "phi_chi"):
        c = LHV(p=p, leaf_max=leaf, core_a=0.0, precision="fp32", terms="far")
        c.set_form(form)
        if form == "phi_chi":
            c.set_launch_shape(m2l_pairs_per_chunk=64)
        v4, s4 = c.evaluate_velocity_stretching(dev(x, "fp32"), dev(w, "fp32"))
        L = c.stats()["leaf_level"]
        assert L >= 2
        got.append([host3(v4), host3(s4)] + [c.export("local", l).double().cpu().numpy() for l in range(2, L + 1)])
        c.close()
    for a, b in zip(*got):
        assert np.linalg.norm(a - b) <= 2e-6 * np.linalg.norm(b), (np.linalg.norm(a - b), np.linalg.norm(b))
