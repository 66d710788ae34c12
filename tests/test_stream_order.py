"""Tables reach the GPU on the stream whose kernels read them."""
import glob
import os
import re

import pytest

import workloads
from tests.gpu_util import dev, host3, rel

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1201_5430_gb300", "csrc")


def test_no_upload_on_the_default_stream():
    """A plain cudaMemcpy from pageable memory may return before its transfer is done, and a non-blocking
    stream does not wait for the default one: every upload names its stream."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for call in re.findall(r"\bcudaMemcpy\s*\((?:[^()]|\([^()]*\))*\)", text):
            if "HostToDevice" in call:
                found.append((os.path.basename(path), call))
    assert not found, found


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_first_evaluations_on_a_stream_of_their_own(prec):
    """Fresh contexts on a non-blocking stream, each with tables of its own p, against contexts on the default
    stream: the same kernels, to the rounding of differently ordered sums (2e-6, FP64 1e-13)."""
    import torch
    from paper_1201_5430_gb300 import LHV
    x, w = workloads.cube(3000, 4)
    s = torch.cuda.Stream()
    for p in (3, 5, 9, 12):
        got = []
        for stream in (s, None):
            x4, w4 = dev(x, prec), dev(w, prec)
            torch.cuda.synchronize()
            c = LHV(p=p, leaf_max=16, core_a=0.0, precision=prec, terms="far", stream=stream)
            with torch.cuda.stream(stream or torch.cuda.current_stream()):
                v4, s4 = c.evaluate_velocity_stretching(x4, w4)
            torch.cuda.synchronize()
            got.append((host3(v4), host3(s4)))
            c.close()
        for a, b in zip(*got):
            assert rel(a, b) < (2e-6 if prec == "fp32" else 1e-13), (p, rel(a, b))
