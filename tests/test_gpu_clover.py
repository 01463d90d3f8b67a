"""The clover term and its inverse at fields made for their weak points."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import assert_elementwise, make_lattice, wc
from oracle.evenodd import EvenOdd

pytestmark = pytest.mark.gpu

DIMS = (4, 4, 4, 4)


def three_zero_modes():
    """Links, csw and kappa for which both blocks of A at site 0 are
    [[1, Q^+], [Q, 1]] with Q unitary up to rounding: three zero modes each.
    All links are 1 but U_z(0 + y) and U_z(0 + x), which are the yz and the xz
    leaf of site 0: their anti-Hermitian parts are made such that Q = X, 0.3
    radians off the cyclic permutation of the three colours (so that no other
    block, which has one of the two leaves, is singular)."""
    X = np.exp(0.3j) * np.roll(np.eye(3), 1, axis=0)
    s = 0.7

    def link(H):
        """SU(3) matrix whose anti-Hermitian traceless part is i s H."""
        w, v = np.linalg.eigh(H)
        lo, hi = -1 - s * w.min(), 1 - s * w.max()
        for _ in range(200):
            m = (lo + hi) / 2
            lo, hi = (lo, m) if np.arcsin(s * w + m).sum() > 0 else (m, hi)
        return (v * np.exp(1j * np.arcsin(s * w + m))) @ v.conj().T

    U = synth.unit_links(DIMS)
    U[DIMS[0], 2] = link((X + X.conj().T) / 2)
    U[1, 2] = link(1j * (X - X.conj().T) / 2)
    return U, 4.0 / s / 0.13, 0.13


def blocks(U, csw, kappa):
    A = oracle.Operator(DIMS, U, csw, kappa, -1).T + np.eye(12)
    return [A[:, b:b + 6, b:b + 6] for b in (0, 6)]


def test_clover_block_with_three_zero_modes_is_singular():
    """Nothing of the block's lower half is left after the elimination of its
    upper one but rounding, which is as regular as any matrix: the call has to
    see that it is small against the block."""
    U, csw, kappa = three_zero_modes()
    for B in blocks(U, csw, kappa):
        assert np.sort(np.abs(np.linalg.eigvalsh(B[0])))[2] < 1e-14
    lat = make_lattice(DIMS, U, csw, kappa, -1)
    for prec in (0, 1, 2):
        with pytest.raises(wc().WCError) as e:
            lat.apply_schur(lat.field(prec), lat.field(prec))
        assert e.value.status == 5


def test_clover_block_beside_three_zero_modes_is_inverted():
    """The same field at 0.999 of that csw: condition 2e3, which the FP64
    tolerance scales with."""
    U, csw, kappa = three_zero_modes()
    csw *= 0.999
    cond = max(np.linalg.cond(B).max() for B in blocks(U, csw, kappa))
    assert 1e3 < cond < 1e4
    lat = make_lattice(DIMS, U, csw, kappa, -1)
    op = oracle.Operator(DIMS, U, csw, kappa, -1)
    psi = synth.gaussian_source(DIMS, 331)
    fi, fo = lat.field(0).load(psi), lat.field(0)
    lat.apply_schur(fo, fi)
    assert_elementwise(fo.store(np.zeros_like(psi)), EvenOdd(DIMS, -1, kappa, U, op.T).schur(psi), 1e-12 * cond)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 4, 5, 2), (4, 4, 4, 6)])
def test_clover_term_of_links_rounded_to_fp32(dims):
    """Links kept in FP32, as configurations often are: unitary to 1e-7 only.
    The clover term is the one of these links (two rows as given, the third
    their cross product, as the library and here the oracle have it), not
    one that assumes U^+ U = 1: FP64 tolerance."""
    csw, kappa, tbc = 1.3, 0.12, -1
    U = synth.haar_links(dims, 341).astype(np.complex64).astype(complex)
    U[..., 2, :] = np.conj(np.cross(U[..., 0, :], U[..., 1, :]))
    lat = make_lattice(dims, U, csw, kappa, tbc)
    psi = synth.gaussian_source(dims, 342)
    fi, fo = lat.field(0).load(psi), lat.field(0)
    lat.apply_M(fo, fi)
    assert_elementwise(fo.store(np.zeros_like(psi)), oracle.apply_M(dims, tbc, kappa, csw, U, psi), 1e-12)
