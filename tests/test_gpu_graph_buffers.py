"""A captured graph keeps replaying correctly when calls in between need larger buffers of its
handle: the replays agree bit for bit with those of a handle that was left alone."""
import numpy as np
import pytest

from helpers import DT, population32
from paper_1903_06479_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def N():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_06479_gb300 import npfem
    npfem.lib()
    return npfem


# FP32 cells above one per SM keep vectors in the handle's scratch; BF16 cells and their carried
# pairs in its trajectory buffers
@pytest.mark.parametrize("precision,n,cells,more,warm", [("fp32", 642, 160, 330, 2), ("fp32", 642, 160, 330, 0),
                                                         ("fp32", 258, 310, 700, 2), ("bf16", 642, 40, 200, 1),
                                                         ("bf16", 642, 40, 200, 2), ("fp64", 162, 160, 620, 2)])
def test_replays_after_larger_calls(N, precision, n, cells, more, warm):
    import torch
    td = torch.float64 if precision == "fp64" else torch.float32
    rest, tris = W.discocyte(n)
    p = population32(n, more, seed=950, forces="shear", noise_pN=0.5, box=60.0)
    big = [torch.tensor(W.to_soa(p[k]), dtype=td, device="cuda") for k in "xvf"]
    out = []
    for disturbed in (False, True):
        h = N.Handle(rest, tris, N.material(), N.default_opts(precision=precision, tol=1e-6, warm_history=warm), dt=DT)
        x, v, f = (b[:cells].clone() for b in big)
        loop = N.StepGraph([h], [cells], x, v, f, DT, steps=2)
        loop.launch()
        if disturbed:
            torch.cuda.synchronize()
            bx, bv, bf = (b.clone() for b in big)
            grad, parts = torch.zeros_like(bx), torch.zeros(more * 8, dtype=torch.float64, device="cuda")
            h.eval(more, bx, bx, grad, parts)
            N.step([h], [more], bx, bv, bf, DT)
            second = N.StepGraph([h], [more], bx, bv, bf, DT, steps=1)
            second.launch()
            torch.cuda.synchronize()
            # memory the library gave back, if any, is taken and written by others
            junk = [torch.full((1 << 22,), float("nan"), device="cuda") for _ in range(16)]
        for _ in range(3):
            loop.launch()
        torch.cuda.synchronize()
        out.append((x.clone(), v.clone()))
        loop.close()
        if disturbed:
            second.close()
            N.step([h], [more], bx, bv, bf, DT)
            torch.cuda.synchronize()
            assert bool(torch.isfinite(bx).all()) and len(junk) == 16
        h.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
