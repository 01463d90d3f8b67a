"""Rounding errors of the FP64 and double-FP32 operators against extended
precision.

The bounds are the errors that operators taking one site per thread, one hop
after the other, had on the same inputs (their clover inverse by pivoted
elimination, the leaves of its plaquettes one by one): a faster form may not
be less accurate."""
import numpy as np
import pytest

import synth
from extended import Extended, rel_err
from gpu_common import make_lattice

pytestmark = pytest.mark.gpu

DIMS = (4, 6, 4, 8)
CASES = {   # links, csw, kappa: errors of M, M^+, H, M^, M^^+ in units of 1e-16
    "smooth": (lambda: synth.exp_links(DIMS, 0.3, 71), 1.0, 0.12, (3.601, 3.619, 6.785, 2.940, 2.947)),
    "smooth csw 1.9": (lambda: synth.exp_links(DIMS, 0.3, 71), 1.9, 0.137, (4.234, 4.263, 6.785, 4.094, 4.103)),
    "random": (lambda: synth.haar_links(DIMS, 72), 1.4, 0.115, (3.387, 3.478, 5.782, 2.953, 3.002)),
    "random csw 3": (lambda: synth.haar_links(DIMS, 72), 3.0, 0.13, (4.531, 4.570, 5.782, 4.899, 5.064)),
    "rounded to FP32": (lambda: synth.haar_links(DIMS, 72).astype(np.complex64).astype(complex), 1.2, 0.12,
                        (2.031, 2.012, 1.472, 1.814, 1.813)),
}


@pytest.mark.parametrize("name", CASES)
def test_fp64_operators_are_no_less_accurate(name):
    links, csw, kappa, bounds = CASES[name]
    U = links()
    psi = synth.gaussian_source(DIMS, 73)
    lat = make_lattice(DIMS, U, csw, kappa, -1)
    ext = Extended(DIMS, U, csw, kappa, -1)
    refs = [ext.M(psi), ext.M(psi, -1), ext.H(psi), ext.schur(psi), ext.schur(psi, -1)]
    f, g = lat.field(0).load(psi), lat.field(0)
    ops = [lambda: lat.apply_M(g, f), lambda: lat.apply_Mdag(g, f), lambda: lat.apply_hop(g, f),
           lambda: lat.apply_schur(g, f), lambda: lat.apply_schur(g, f, True)]
    for op, ref, bound in zip(ops, refs, bounds):
        op()
        assert rel_err(g.store(np.zeros_like(psi)), ref) <= bound * 1e-16


DF_CASES = {   # links, csw, kappa: errors of M, H, M^ in units of 1e-15
    "smooth": (lambda: synth.exp_links(DIMS, 0.3, 71), 1.0, 0.12, (6.089, 9.035, 15.08)),
    "smooth csw 1.9": (lambda: synth.exp_links(DIMS, 0.3, 71), 1.9, 0.137, (8.005, 9.035, 17.17)),
    "random": (lambda: synth.haar_links(DIMS, 72), 1.0, 0.125, (4.577, 10.16, 15.52)),
}


@pytest.mark.parametrize("name", DF_CASES)
def test_double_fp32_operators_are_no_less_accurate(name):
    """By the kernels an application takes and, for M, by every other launch
    shape too."""
    links, csw, kappa, bounds = DF_CASES[name]
    U = links()
    psi = synth.gaussian_source(DIMS, 73)
    lat = make_lattice(DIMS, U, csw, kappa, -1).set_fp64_arith(1)
    ext = Extended(DIMS, U, csw, kappa, -1)
    refs = [ext.M(psi), ext.H(psi), ext.schur(psi)]
    f, g = lat.field(0).load(psi), lat.field(0)
    for op, ref, bound in zip((lat.apply_M, lat.apply_hop, lat.apply_schur), refs, bounds):
        op(g, f)
        assert rel_err(g.store(np.zeros_like(psi)), ref) <= bound * 1e-15
    for shape in (0, 3, 22):
        lat.apply_shape(0, 0, force=shape)
        lat.apply_M(g, f)
        assert rel_err(g.store(np.zeros_like(psi)), refs[0]) <= bounds[0] * 1e-15
