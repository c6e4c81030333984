"""The immersed-boundary gathers cell by cell (a box of lattice nodes in shared memory) against
vertex by vertex, at the edges of the rule that chooses between them: the number of cells, the
vertices per cell, the lattice spacing, and boxes that do not fit."""
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


# 250 cells of 642: both gathers cell by cell at 1 um, vertex by vertex at 0.5 um; 258: Step 4 only;
# stretched: a third of the cells 1.8 times as long, whose boxes do not fit; two groups
@pytest.mark.parametrize("sizes,cells,dx,stretch", [((642,), (250,), 1.0, 1.0), ((642,), (250,), 0.5, 1.0),
                                                    ((642,), (249,), 1.0, 1.0), ((642,), (260,), 1.0, 1.8),
                                                    ((258,), (250,), 1.0, 1.0), ((1026, 258), (240, 20), 1.3, 1.0)])
def test_gathers_cell_by_cell(N, sizes, cells, dx, stretch):
    """Interpolation and one cycle of the forcing over all cells, against interpolations of
    batches of 100 cells (vertex by vertex): the same sums in another order, 1e-5 of the largest
    value (FP32 sums of 64 products; the slip divides by the time step on both sides)."""
    import torch
    hs, xs = [], []
    for n, c in zip(sizes, cells):
        rest, tris = W.discocyte(n)
        hs.append(N.Handle(rest, tris, N.material(), N.default_opts(), dt=DT))
        x = population32(n, c, seed=1000 + n, forces="noise", box=30.0)["x"]
        centre = x.mean(1, keepdims=True)
        x[::3] = (centre + stretch * (x - centre))[::3]
        xs.append(torch.tensor(W.to_soa(x), dtype=torch.float32, device="cuda"))
    x = torch.cat([t.reshape(-1) for t in xs])
    v = torch.randn_like(x)
    side = int(30.0 / dx)
    dims = (side, side + 1, side + 2)
    lat = N.lattice((0.0, 0.0, 0.0), dx, dims)  # some cells lie partly outside
    nodes = int(np.prod(dims))
    u = torch.randn(nodes * 4, device="cuda")

    def in_batches(field):
        out, at = torch.zeros_like(x), 0
        for h, t in zip(hs, xs):
            for a in range(0, t.shape[0], 100):
                part = t[a:a + 100].contiguous()
                o = torch.zeros_like(part)
                N.ibm_interpolate([h], [part.shape[0]], part, lat, field, o)
                out[at:at + o.numel()] = o.reshape(-1)
                at += o.numel()
        return out

    close = lambda a, b: float((a.double() - b.double()).abs().max()) <= 1e-5 * float(b.double().abs().max())
    whole = torch.zeros_like(x)
    N.ibm_interpolate(hs, cells, x, lat, u, whole)
    parts = in_batches(u)
    assert float(parts.abs().max()) > 0 and close(whole, parts)
    f0, f1, spread = torch.zeros_like(x), torch.zeros_like(x), torch.zeros(nodes * 4, device="cuda")
    N.ibm_forcing(hs, cells, x, v, lat, u, DT, 0, f0, spread)
    assert close(f0, (v - parts) / DT)
    # one cycle: f_1 = f_0 + (U - u_l) / dt with u_l = u* + dt (the spread of f_0)
    N.ibm_forcing(hs, cells, x, v, lat, u, DT, 1, f1, torch.zeros_like(spread))
    ul = u + DT * spread
    assert close(f1, f0 + (v - in_batches(ul)) / DT)
