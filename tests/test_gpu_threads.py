"""Host threads that step handles of their own on streams of their own, each needing another
amount of shared memory of the same kernel."""
import threading

import numpy as np
import pytest

from helpers import DT, population32
from paper_1903_06479_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,sizes", [("fp32", (66, 258, 642)), ("bf16", (66, 162, 258)), ("fp64", (66, 162, 258))])
def test_threads_with_handles_of_their_own(precision, sizes):
    """Each thread's cells come out bit for bit as when stepped alone."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_06479_gb300 import npfem as N
    N.lib()
    td = torch.float64 if precision == "fp64" else torch.float32
    cells, steps = 2, 60

    def make(n):
        rest, tris = W.discocyte(n)
        h = N.Handle(rest, tris, N.material(), N.default_opts(precision=precision, tol=1e-6), dt=DT)
        p = population32(n, cells, seed=1100 + n, forces="shear", noise_pN=0.5, box=20.0)
        return h, [torch.tensor(W.to_soa(p[k]), dtype=td, device="cuda") for k in "xvf"]

    def run(job, stream, fails):
        h, (x, v, f) = job
        try:
            for _ in range(steps):
                N.step([h], [cells], x, v, f, DT, stream=stream.cuda_stream)
                # a smaller or larger launch of the same kernel now and then
                N.step([h], [1], x, v, f, DT, stream=stream.cuda_stream)
        except N.NpfemError as e:
            fails.append(str(e))

    out = []
    for together in (False, True):
        jobs = [make(n) for n in sizes]
        streams = [torch.cuda.Stream() for _ in sizes]
        torch.cuda.synchronize()
        fails = []
        workers = [threading.Thread(target=run, args=(j, s, fails)) for j, s in zip(jobs, streams)]
        for w in workers:
            w.start()
            if not together:
                w.join()
        for w in workers:
            w.join()
        torch.cuda.synchronize()
        assert not fails, fails[0]
        out.append([j[1][0].clone() for j in jobs])
    for a, b in zip(*out):
        assert torch.equal(a, b) and bool(np.isfinite(a.double().cpu().numpy()).all())
