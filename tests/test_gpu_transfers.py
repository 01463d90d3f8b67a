"""Imports on both sides of the rule that chooses between their kernels."""
import numpy as np
import pytest

import synth
from gpu_common import wc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(8, 8, 8, 37), (8, 8, 8, 38), (9, 13, 17, 11)])
@pytest.mark.parametrize("offset", [0, 1])
def test_imports_of_a_thread_per_site_and_turned_round(dims, offset):
    """A CTA of 128 sites less than one per SM (152) takes the turned-round
    form, from one on a thread per site does, but for complex64 -> binary16;
    ragged volumes, and complex64 rows 8 bytes off a 16-byte boundary.  FP64
    holds the values, FP32 their roundings, binary16 components lie within
    2^-11 of the site's largest."""
    import torch
    V = int(np.prod(dims))
    ref = torch.from_numpy(synth.gaussian_source(dims, 371))
    lat = wc().Lattice(dims)
    for dtype in (torch.complex64, torch.complex128):
        store = torch.zeros(V * 12 + 1, dtype=dtype, device="cuda")
        src = store[offset:offset + V * 12].view(V, 4, 3)
        src.copy_(ref)
        want = ref.to(dtype).to(torch.complex128)
        for prec in (0, 1, 2):
            got = torch.zeros(V, 4, 3, dtype=torch.complex128)
            lat.field(prec).load(src).store(got.numpy())
            if prec == 2:
                r, w = torch.view_as_real(got), torch.view_as_real(want)
                big = w.abs().amax(dim=(1, 2, 3), keepdim=True)
                assert ((r - w).abs() <= 2.0 ** -11 * big * (1 + 1e-5)).all()
            else:
                assert torch.equal(got, want if prec == 0 else ref.to(torch.complex64).to(torch.complex128))
