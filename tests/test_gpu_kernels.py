"""Edges of the kernels' tiles and of the rules that choose between kernels.

Each test compares one path with the oracle, or with the general path, at
the sizes where it can go wrong: remainders of tiles, the smallest extents,
a workspace that grows and is reused.  Tolerances as in the parity tests:
1e-12 (FP64), 1e-5 (FP32), 5e-3 (binary16 storage) relative.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import assert_elementwise, make_lattice, wc
from oracle.evenodd import EvenOdd

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 1e-5, 2: 5e-3}


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 10)])
def test_schur_workspaces_are_reused_and_grow(dims):
    """Single and multi-field Schur applications in turn on one lattice,
    with the count and the precision changing between calls."""
    csw, kappa, tbc = 1.3, 0.12, -1
    U = synth.exp_links(dims, 0.4, 31)
    lat = make_lattice(dims, U, csw, kappa, tbc)
    op = oracle.Operator(dims, U, csw, kappa, tbc)
    eo = EvenOdd(dims, tbc, kappa, U, op.T)
    for call, (n, prec, dagger) in enumerate([(3, 1, False), (12, 2, True), (16, 1, True), (1, 2, False), (5, 1, False)]):
        srcs = [synth.gaussian_source(dims, 40 + 20 * call + r) for r in range(n)]
        ins = [lat.field(prec).load(s) for s in srcs]
        outs = [lat.field(prec).load(s) for s in srcs]      # old contents, odd sites included, must go
        lat.apply_schur_multi(outs, ins, dagger)
        one = lat.field(prec)
        for s, f, g in zip(srcs, outs, ins):
            ref = eo.schur(s, dagger)
            out = f.store(np.zeros_like(s))
            assert np.abs(out[eo.odd]).max() == 0.0
            assert_elementwise(out, ref, TOL[prec])
            lat.apply_schur(one, g, dagger)
            assert_elementwise(one.store(np.zeros_like(s)), ref, TOL[prec])
