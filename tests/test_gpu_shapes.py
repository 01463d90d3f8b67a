"""Pinned launch shapes and the rules that choose without one."""
import numpy as np
import pytest

import synth
from gpu_common import make_lattice, wc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arith", [0, 1])
def test_a_pinned_shape_is_used_in_solves_and_can_be_taken_back(arith):
    """Three steps of a whole-lattice solve: every pinned shape (a site per
    thread) gives the same bits, the kernels on four warps others, and these
    are back once the pin is taken back."""
    dims, kappa, csw, tbc = (4, 6, 8, 6), 0.12, 1.0, -1
    U = synth.exp_links(dims, 0.3, 401)
    src = synth.gaussian_source(dims, 402)
    lat = make_lattice(dims, U, csw, kappa, tbc).set_fp64_arith(arith)
    b = lat.field(0).load(src)

    def steps():
        x, y = lat.field(0), lat.field(0)
        lat.solve(x, b, tol=1e-13, max_iter=3, max_restarts=0, check=False)
        lat.apply_M(y, b)
        return np.stack([f.store(np.zeros_like(src)) for f in (x, y)])

    free = steps()
    assert lat.apply_shape(0, 0)[2] == 64
    pinned = []
    for shape in (0, 22):
        assert lat.apply_shape(0, 0, force=shape)[2] != 64
        pinned.append(steps())
    assert np.array_equal(pinned[0], pinned[1])
    assert not np.array_equal(pinned[0][0], free[0]) and not np.array_equal(pinned[0][1], free[1])
    assert lat.apply_shape(0, 0, force=-2) == (-1, (-1,) * 4, -1)
    assert np.array_equal(steps(), free)
    with pytest.raises(wc().WCError):
        lat.apply_shape(0, 0, force=-3)


@pytest.mark.parametrize("dims,split", [((32, 16, 16, 32), True), ((34, 16, 16, 32), False)])
def test_double_fp32_form_depends_on_the_size_only(dims, split):
    """On both sides of the line at 2^18 sites."""
    lat = make_lattice(dims, synth.unit_links(dims), 1.0, 0.12, -1).set_fp64_arith(1)
    f, g = lat.field(0), lat.field(0)
    lat.apply_M(g, f)
    assert (lat.apply_shape(0, 0)[2] == 64) == split
