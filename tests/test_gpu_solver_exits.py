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


NESTED = [dict(precond=p, krylov_prec=k, even_odd=e) for p in (0, 1) for k in (1, 2) for e in (False, True)]


@pytest.mark.parametrize("kw", NESTED)
def test_nested_solve_whose_half_step_is_exact(kw):
    """M = 1 (kappa = 0, csw = 0) and a point source: the first half step is
    exact, so the second inner solve starts from a zero vector and has to
    return a zero correction."""
    dims = (4, 4, 4, 6)
    U = synth.exp_links(dims, 0.3, 311)
    lat = make_lattice(dims, U, 0.0, 0.0, TBC)
    src = np.zeros((int(np.prod(dims)), 4, 3), complex)
    src[0, 1, 2] = 1.0
    x = lat.field(0)
    info = lat.solve(x, lat.field(0).load(src), tol=1e-10, solver=2, block=(2, 2, 2, 2), overlap=0, mr_iters=2,
                     **kw)
    assert info.status == 0
    assert np.abs(x.store(np.zeros_like(src)) - src).max() <= 1e-10


@pytest.mark.parametrize("kw", NESTED[::2])
def test_nested_solve_on_links_with_a_nan(kw):
    """The inner solves meet a NaN, their second one in its source: the solve
    ends as WC_ERR_NAN (6)."""
    dims = (4, 4, 4, 6)
    U = synth.exp_links(dims, 0.3, 312)
    U[0, 0, 1, 1] = np.nan      # (the third row is rebuilt from the other two)
    lat = make_lattice(dims, U, 0.0, KAPPA, TBC)
    src = synth.gaussian_source(dims, 313)
    info = lat.solve(lat.field(0), lat.field(0).load(src), tol=1e-10, solver=2, check=False,
                     block=(2, 2, 2, 2), overlap=0, mr_iters=2, **kw)
    assert info.status == 6
