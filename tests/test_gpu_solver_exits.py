"""What a solve leaves behind when it returns, and how it ends when a vector
vanishes or is not finite."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import make_lattice, wc

pytestmark = pytest.mark.gpu

DIMS, KAPPA, CSW, TBC = (6, 4, 4, 8), 0.12, 1.0, -1
KINDS = [dict(), dict(even_odd=True), dict(solver=1), dict(solver=1, krylov_prec=2), dict(solver=1, even_odd=True),
         dict(solver=2), dict(solver=2, even_odd=True, krylov_prec=2)]


@pytest.mark.parametrize("kw", KINDS)
def test_a_returned_solve_has_left_its_stream(kw):
    """The step queued ahead of the last one is off the stream when a solve
    returns, converged, stopped by max_iter or by a NaN in the links: the
    stream is idle, and the next solve, on another stream, takes the steps to
    the bits of a solve on a lattice of its own."""
    import torch
    U = synth.exp_links(DIMS, 0.3, 301)
    src = synth.gaussian_source(DIMS, 302)
    alone = make_lattice(DIMS, U, CSW, KAPPA, TBC)
    x = alone.field(0)
    alone.solve(x, alone.field(0).load(src), tol=1e-10, **kw)
    ref = x.store(np.zeros_like(src))
    streams = [torch.cuda.Stream() for _ in range(3)]
    lat = wc().Lattice(DIMS, TBC, stream=streams[0]).load_gauge(U).load_clover(CSW, KAPPA)
    b = lat.field(0).load(src)
    lat.sync()
    for k in range(6):
        s = streams[k % 3]
        lat.set_stream(s)
        x = lat.field(0)
        if k == 3:
            lat.solve(x, b, tol=1e-10, max_iter=2, max_restarts=0, check=False, **kw)
            assert s.query()
            continue
        lat.solve(x, b, tol=1e-10, **kw)
        assert s.query()
        assert np.array_equal(x.store(np.zeros_like(src)), ref)
    bad = U.copy()
    bad.reshape(-1)[5] = np.nan
    lat.load_gauge(bad).load_clover(0.0, KAPPA)
    if not kw.get("even_odd"):
        info = lat.solve(lat.field(0), b, tol=1e-10, max_restarts=1, check=False, **kw)
        assert info.status != 0 and s.query()
