"""Tensor-core (tcgen05, TF32) path: descriptor self-test and split-precision parity."""
import ctypes

import numpy as np
import pytest

import workloads
from oracle import fmm as ofmm
from tests.gpu_util import dev, host3, rel

pytestmark = pytest.mark.gpu


def _tf32(a):
    """Round FP32 to TF32 (10 mantissa bits), to nearest, ties away from zero."""
    b = np.asarray(a, dtype=np.float32).view(np.uint32).astype(np.uint64)
    b = (b + 0x1000) & 0xFFFFE000
    return b.astype(np.uint32).view(np.float32)


@pytest.mark.parametrize("N,K", [(16, 32), (144, 64), (256, 96)])
def test_tc_selftest_matches_reference(N, K):
    import torch
    from paper_1201_5430_gb300 import _lib
    lib = _lib.load()
    rng = np.random.default_rng(N + K)
    X = rng.normal(size=(128, K)).astype(np.float32)
    B = rng.normal(size=(N, K)).astype(np.float32)
    Xd, Bd = torch.from_numpy(X).cuda(), torch.from_numpy(B).cuda()
    Dd = torch.zeros(128, N, device="cuda")
    torch.cuda.synchronize()
    st = lib.lhv_tc_selftest(ctypes.c_void_p(Xd.data_ptr()), ctypes.c_void_p(Bd.data_ptr()),
                             ctypes.c_void_p(Dd.data_ptr()), N, K)
    assert st == 0
    want = _tf32(X).astype(np.float64) @ _tf32(B).astype(np.float64).T
    got = Dd.cpu().numpy()
    scale = np.abs(_tf32(X)).astype(np.float64) @ np.abs(_tf32(B)).astype(np.float64).T
    assert np.max(np.abs(got - want) / scale) < 1e-6


@pytest.mark.parametrize("case", ["cube", "ring"])
def test_tf32x3_parity(case):
    from paper_1201_5430_gb300 import LHV
    if case == "cube":
        x, w = workloads.cube(6000, 5)
        a, leaf = 0.01, 32
    else:
        x, w = workloads.ring(12000, 1)
        a, leaf = workloads.RING_CORE_A, 64
    p = 12
    ref = ofmm.fmm(x, w, p, leaf_max=leaf, a=a)
    ctx = LHV(p=p, leaf_max=leaf, core_a=a, precision="tf32x3")
    v4, s4 = ctx.evaluate_velocity_stretching(dev(x, "fp32"), dev(w, "fp32"))
    ctx.stats()  # raises if a tensor-core wait timed out
    ev, es = rel(host3(v4), ref.v), rel(host3(s4), ref.s)
    print(f"tf32x3 {case} p=12: rel L2 v {ev:.2e} s {es:.2e}")
    assert ev < 1e-6 and es < 1e-6, (ev, es)


@pytest.mark.parametrize("p", [4, 8, 12, 16, 20, 24])
@pytest.mark.parametrize("n,leaf", [(700, 8), (5000, 16)])
def test_m2l_converts_like_the_fused_table(p, n, leaf):
    """One translation block with the conversion in the epilogue against the fused tables on the
    CUDA cores, far field only: v and s, and the scalar case.  Covers one and several column
    ranges (p = 20, 24), one and two accumulator buffers, full and partly filled chunks.  Both
    sides round 2 p^2 FP32 terms a coefficient: sqrt(2 24^2) 2^-24 = 2e-6."""
    import torch
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.cube(n, 9)
    q = torch.from_numpy(workloads.charges(n, 3)).cuda()
    got = {}
    for tc in (1, 0):
        ctx = LHV(p=p, leaf_max=leaf, core_a=0.0, precision="tf32x3", terms="far")
        ctx.set_launch_shape(m2l_pairs_per_chunk=64, m2l_tensor_cores=tc)
        v4, s4 = ctx.evaluate_velocity_stretching(dev(x, "fp32"), dev(w, "fp32"))
        pg = ctx.evaluate_potential_gradient(dev(x, "fp32"), q)
        st = ctx.stats()  # raises if a tensor-core wait timed out
        assert st["leaf_level"] >= 2 and st["m2l_pairs"] > 0
        got[tc] = (host3(v4), host3(s4), pg.cpu().numpy())
        ctx.close()
    for a, b in zip(got[1], got[0]):
        assert rel(a, b) < 2e-6, rel(a, b)


@pytest.mark.parametrize("p", [4, 8, 12, 16, 20])
@pytest.mark.parametrize("n,leaf,nsys", [(3000, 4, 1), (60, 1, 5)])
def test_levels_translate_like_the_fused_tables(p, n, leaf, nsys):
    """M2M and L2L on the tensor cores (several levels, few and many boxes an octant) against the
    fused tables on the CUDA cores: the exported multipoles of every level, the locals of the leaves
    and the field.  A coefficient passes up to seven levels of 2 p^2 rounded terms:
    7 sqrt(2 20^2) 2^-24 = 1.2e-5 at most, 2e-6 a level."""
    import torch
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.cube(n * nsys, 21)
    off = [n * k for k in range(nsys + 1)]
    q = torch.from_numpy(workloads.charges(n * nsys, 4)).cuda()
    got = {}
    for tc in (1, 0):
        ctx = LHV(p=p, leaf_max=leaf, core_a=0.0, precision="tf32x3", terms="far")
        ctx.set_launch_shape(m2l_pairs_per_chunk=64, m2l_tensor_cores=tc)
        v4, s4 = ctx.evaluate_batched(off, dev(x, "fp32"), dev(w, "fp32"))
        L = ctx.stats()["leaf_level"]
        assert L >= 4
        out = [ctx.export("multipole", l).double().cpu().numpy() for l in range(2, L + 1)]
        out += [ctx.export("local", l).double().cpu().numpy() for l in range(2, L + 1)]
        out += [host3(v4), host3(s4)]
        out.append(ctx.evaluate_potential_gradient(dev(x, "fp32"), q).double().cpu().numpy())
        got[tc] = out
        ctx.close()
    for a, b in zip(got[1], got[0]):
        assert np.linalg.norm(a - b) < 1.2e-5 * np.linalg.norm(b), np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("p,n,leaf", [(4, 100000, 2), (8, 20000, 4)])
def test_levels_of_many_boxes_take_the_tensor_cores(p, n, leaf):
    """Low p: a level needs p^4 boxes > 1.6e7 for the tensor cores; the levels above stay with the
    grouped GEMM, which splits the same list's chunks of 128.  Bound as above."""
    test_levels_translate_like_the_fused_tables(p, n, leaf, 1)


@pytest.mark.parametrize("p", [8, 16, 20])
def test_a_schedule_of_one_p_equals_the_context_of_that_p(p):
    """set_level_p with one p at every level (M2L, M2M and L2L tiles of a p that is not the context's) against
    a context of that p: the same products, bound as for the levels above, 1.2e-5; far field."""
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.cube(20000, 8)
    got = []
    for schedule in (True, False):
        ctx = LHV(p=12 if schedule else p, leaf_max=8, core_a=0.0, precision="tf32x3", terms="far")
        if schedule:
            ctx.set_level_p([p] * 12)
        v4, s4 = ctx.evaluate_velocity_stretching(dev(x, "fp32"), dev(w, "fp32"))
        assert ctx.stats()["leaf_level"] >= 4
        got.append((host3(v4), host3(s4)))
        ctx.close()
    for a, b in zip(*got):
        assert rel(a, b) < 1.2e-5, rel(a, b)


@pytest.mark.parametrize("scalar", [False, True])
def test_waits_that_give_up_end_the_translations(scalar):
    """Short limits let the waits of a launch's roles run out at any of its items: every call ends, the
    status says so once, and with the default limit the same context gives its first results again."""
    import torch
    from paper_1201_5430_gb300 import LHV, LHVError
    from paper_1201_5430_gb300 import _lib
    x, w = workloads.cube(20000, 8)
    x4, w4 = dev(x, "fp32"), dev(w, "fp32")
    q = torch.from_numpy(workloads.charges(20000, 3)).cuda()
    ctx = LHV(p=12, leaf_max=16, core_a=0.0, precision="tf32x3", terms="far")
    call = (lambda: ctx.evaluate_potential_gradient(x4, q)) if scalar else \
        (lambda: ctx.evaluate_velocity_stretching(x4, w4)[0])
    want = call().double().cpu().numpy()
    ctx.stats()
    gave_up = 0
    for limit in [1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 64, 128, 256, 1024] * 3:
        ctx.set_wait_limit(limit)
        call()
        torch.cuda.synchronize()
        try:
            ctx.stats()
        except LHVError as e:
            assert e.status == _lib.LHV_ETIMEOUT
            gave_up += 1
    assert gave_up > 0
    ctx.set_wait_limit()
    got = call().double().cpu().numpy()
    ctx.stats()
    assert rel(got, want) < 2e-6
    for bad in (-1, (1 << 24) + 1):
        assert ctx.lib.lhv_set_wait_limit(ctx.h, bad) == _lib.LHV_EINVAL
    ctx.close()


@pytest.mark.parametrize("p", [8, 12, 16])
def test_multipoles_are_as_exact_as_in_fp32(p):
    """M2M of a TF32x3 context runs in FP32: the multipoles of every level with a thousand boxes below it are no
    further from the FP64 context's than the FP32 context's.  Both add the same products in another order; the
    norm of 1000 x 2 p^2 rounding errors scatters by about a percent, and ten are allowed."""
    from paper_1201_5430_gb300 import LHV
    x = np.random.default_rng(6).standard_normal((100003, 3))
    x = (x / np.linalg.norm(x, axis=1)[:, None]).astype(np.float32)
    w = np.random.default_rng(7).standard_normal((100003, 3)).astype(np.float32)
    got = {}
    for prec in ("tf32x3", "fp32", "fp64"):
        ctx = LHV(p=p, leaf_max=32, core_a=0.0, precision=prec, terms="far")
        e = "fp64" if prec == "fp64" else "fp32"
        ctx.evaluate_velocity_stretching(dev(x, e), dev(w, e))
        st = ctx.stats()
        L = st["leaf_level"]
        levels = [l for l in range(2, L) if st["nbox"][l + 1] >= 1000]
        got[prec] = [ctx.export("multipole", l).double().cpu().numpy() for l in levels]
        ctx.close()
    assert len(levels) >= 2
    for a, b, c in zip(got["tf32x3"], got["fp32"], got["fp64"]):
        assert np.linalg.norm(a - c) <= 1.1 * np.linalg.norm(b - c), (rel(a, c), rel(b, c))
