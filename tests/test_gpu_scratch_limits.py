"""Calls that run out of device memory: the error, and the call after it."""
import gc

import numpy as np
import pytest

import synth
from gpu_common import make_lattice, wc

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _leave(mbytes):
    """A tensor that leaves about so much device memory free."""
    import torch
    gc.collect()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(free - mbytes * MB, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("left", [100, 300])
def test_even_odd_call_after_one_that_ran_out_of_memory(left):
    """At 16^3x32 the inverse clover term takes 208 MB and the parity-ordered
    one 192 MB, 75 MB of each in its first array: with 100 MB left the second
    array of the first store does not fit, with 300 MB that of the second.
    The call reports it, and with memory free again the next one is right."""
    import torch
    dims, kappa, csw, tbc = (16, 16, 16, 32), 0.12, 1.0, -1
    U = synth.pool_links(dims, 321)
    src = synth.gaussian_source(dims, 322)
    ref_lat = make_lattice(dims, U, csw, kappa, tbc)
    f, g = ref_lat.field(0).load(src), ref_lat.field(0)
    ref_lat.apply_schur(g, f)
    ref = g.store(np.zeros_like(src))
    ref_lat.close()
    lat = make_lattice(dims, U, csw, kappa, tbc)
    f, g = lat.field(0).load(src), lat.field(0)
    lat.sync()
    hog = _leave(left)
    with pytest.raises(wc().WCError) as e:
        lat.apply_schur(g, f)
    assert e.value.status == 2
    del hog
    torch.cuda.empty_cache()
    lat.apply_schur(g, f)
    assert np.array_equal(g.store(np.zeros_like(src)), ref)


def test_schur_workspaces_above_their_bound_are_given_back():
    """16 half-lattice FP32 fields of 32^4 are 805 MB and freed with the call, 8
    are 403 MB and kept for the next one."""
    import torch

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    dims = (32, 32, 32, 32)
    lat = make_lattice(dims, synth.unit_links(dims), 1.0, 0.12, -1)
    fields = [lat.field(1) for _ in range(32)]
    lat.apply_schur_multi(fields[:1], fields[16:17])
    before = free()
    lat.apply_schur_multi(fields[:16], fields[16:])
    assert free() >= before
    lat.apply_schur_multi(fields[:8], fields[16:24])
    kept = free()
    assert before - kept >= 7 * 48 * 32 ** 4      # the first call had kept one field
    lat.apply_schur_multi(fields[:8], fields[16:24])
    assert free() == kept


@pytest.mark.parametrize("kw", [dict(solver=1, even_odd=True), dict(), dict(solver=1, even_odd=True, krylov_prec=2)])
def test_force_in_the_memory_of_its_fields_and_xi(kw):
    """At 16^3x32 a force needs two fields (50 MB) and Xh (57 MB) once its
    solver's vectors exist: it runs with 140 MB left, and gives the same bits."""
    import torch
    dims, kappa, csw, tbc = (16, 16, 16, 32), 0.11, 1.0, -1
    U = synth.pool_links(dims, 351)
    phi = synth.gaussian_source(dims, 352)
    lat = make_lattice(dims, U, csw, kappa, tbc)
    b = lat.field(0).load(phi)
    F = [torch.zeros(int(np.prod(dims)), 4, 3, 3, dtype=torch.complex128, device="cuda") for _ in range(2)]
    S0 = lat.action_force(b, F[0], tol=1e-10, **kw)
    hog = _leave(140)
    S1 = lat.action_force(b, F[1], tol=1e-10, **kw)
    del hog
    torch.cuda.empty_cache()
    assert S0 == S1 and torch.equal(F[0], F[1])
