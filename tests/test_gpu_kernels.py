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


@pytest.mark.parametrize("csw", [1.0, 5.0])
def test_clover_inverse_by_blocks_and_by_elimination(csw):
    """csw = 1: every 6x6 block of A is inverted by 3x3 blocks.  csw = 5 on
    Haar links: 31 of the 768 blocks have a 3x3 determinant so small that
    they take the pivoted elimination, and the blocks' condition numbers
    reach 1.4e3 (1.7 at csw = 1), which the FP64 tolerance scales with."""
    dims, kappa, tbc = (4, 4, 4, 6), 0.13, -1
    U = synth.haar_links(dims, 5)
    lat = make_lattice(dims, U, csw, kappa, tbc)
    op = oracle.Operator(dims, U, csw, kappa, tbc)
    A = op.T + np.eye(12)
    cond = max(np.linalg.cond(A[:, b:b + 6, b:b + 6]).max() for b in (0, 6))
    psi = synth.gaussian_source(dims, 6)
    fi, fo = lat.field(wc().F64).load(psi), lat.field(wc().F64)
    lat.apply_schur(fo, fi)
    assert_elementwise(fo.store(np.zeros_like(psi)), EvenOdd(dims, tbc, kappa, U, op.T).schur(psi), 1e-12 * cond)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 2, 5, 4), (7, 3, 2, 11)])
def test_clover_from_shared_plaquettes(dims):
    """The clover term through M on extents where the corners of a
    plaquette wrap onto themselves, odd ones and ragged CTAs; links and
    term loaded twice, so that the second build starts from used stores."""
    csw, kappa, tbc = 1.5, 0.13, -1
    lat = make_lattice(dims, synth.haar_links(dims, 7), 0.7, 0.11, tbc)
    U = synth.haar_links(dims, 8)
    lat.load_gauge(U).load_clover(csw, kappa)
    psi = synth.gaussian_source(dims, 9)
    ref = oracle.apply_M(dims, tbc, kappa, csw, U, psi)
    for prec in (0, 1, 2):
        fi, fo = lat.field(prec).load(psi), lat.field(prec)
        lat.apply_M(fo, fi)
        assert_elementwise(fo.store(np.zeros_like(psi)), ref, TOL[prec])


@pytest.mark.parametrize("dims,tbc", [((2, 2, 2, 2), -1), ((3, 5, 2, 7), 1), ((5, 3, 7, 4), -1), ((8, 4, 4, 4), -1)])
def test_fp64_operator_with_directions_on_four_warps(dims, tbc):
    """M, M^+ and H in FP64 with no shape pinned: volumes of half a CTA of 32
    sites, ragged ones and a whole number of CTAs, both time boundaries; and
    the same as the shapes that take a site per thread."""
    csw, kappa = 1.2, 0.13
    U = synth.haar_links(dims, 60 + sum(dims))
    lat = make_lattice(dims, U, csw, kappa, tbc)
    op = oracle.Operator(dims, U, csw, kappa, tbc)
    psi = synth.gaussian_source(dims, 61)
    F64 = wc().F64
    fi, fo = lat.field(F64).load(psi), lat.field(F64)
    ref = {"M": op.M(psi), "Mdag": op.Mdag(psi), "hop": oracle.apply_hop(dims, tbc, U, psi)}
    outs = {}
    for kind, name in enumerate(ref):
        getattr(lat, "apply_" + name)(fo, fi)
        assert lat.apply_shape(F64, kind)[2] == 64
        outs[name] = fo.store(np.zeros_like(psi))
        assert_elementwise(outs[name], ref[name], 1e-12)
    for kind, name in enumerate(ref):
        lat.apply_shape(F64, kind, force=22)
        getattr(lat, "apply_" + name)(fo, fi)
        assert_elementwise(fo.store(np.zeros_like(psi)), outs[name], 1e-14)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 3, 5, 2), (4, 4, 4, 2), (5, 3, 3, 3), (6, 7, 5, 9)])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("offset", [0, 1])
def test_transfers_turn_rows_round_at_ragged_sizes(dims, prec, offset):
    """Import and export of complex64 and complex128 tensors at volumes below,
    at and above the 128 sites of a CTA; offset 1 starts the complex64 rows
    8 bytes off a 16-byte boundary.  FP64 round trips are exact, FP32 ones
    round once, binary16 components lie within 2^-11 of the site's largest."""
    import torch
    V = int(np.prod(dims))
    lat = wc().Lattice(dims)
    ref = torch.from_numpy(synth.gaussian_source(dims, 77))
    for dtype in (torch.complex64, torch.complex128):
        store = torch.zeros(V * 12 + 1 + 8, dtype=dtype, device="cuda")
        src = store[offset:offset + V * 12].view(V, 4, 3)
        src.copy_(ref)
        f = lat.field(prec).load(src)
        store2 = torch.full((V * 12 + 1 + 8,), 7.0, dtype=dtype, device="cuda")
        f.store(store2[offset:offset + V * 12].view(V, 4, 3))
        out = store2.cpu()
        assert (out[:offset] == 7).all() and (out[offset + V * 12:] == 7).all()
        got = out[offset:offset + V * 12].view(V, 4, 3)
        want = ref.to(dtype)
        if prec == 0 or (prec == 1 and dtype == torch.complex64):
            assert torch.equal(got, want)
        elif prec == 1:
            assert torch.equal(got, ref.to(torch.complex64).to(dtype))
        else:
            r, w = torch.view_as_real(got.to(torch.complex128)), torch.view_as_real(want.to(torch.complex128))
            big = w.abs().amax(dim=(1, 2, 3), keepdim=True)
            assert ((r - w).abs() <= 2.0 ** -11 * big * (1 + 1e-5)).all()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (5, 3, 17, 2), (16, 8, 8, 8), (24, 24, 24, 24)])
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_reductions_of_one_two_and_three_sums(dims, prec):
    """Inner product, norm and axpy with norm from one block (16 sites) to
    more partials than threads, against numpy on the stored values.  Sums
    of n = 24 V products in FP64, in trees with at most 12 V / (256 grid) +
    60 sequential additions: relative error of the sum of magnitudes below
    1e-13 at these sizes; twice the same bits."""
    V = int(np.prod(dims))
    lat = wc().Lattice(dims)
    a, b = lat.field(prec).load(synth.gaussian_source(dims, 5)), lat.field(prec).load(synth.gaussian_source(dims, 6))
    na, nb = (f.store(np.zeros((V, 4, 3), complex)) for f in (a, b))
    mag = np.sum(np.abs(na) * np.abs(nb))
    assert abs(lat.dot(a, b) - np.vdot(na, nb)) <= 1e-13 * mag
    assert abs(lat.norm2(a) - np.sum(np.abs(na) ** 2)) <= 1e-13 * np.sum(np.abs(na) ** 2)
    assert lat.dot(a, b) == lat.dot(a, b) and lat.norm2(b) == lat.norm2(b)
    got = lat.axpy_norm(0.5 - 0.25j, a, b)
    tol = {0: 1e-13, 1: 2e-7, 2: 2e-3}[prec]     # the norm is of the values before they are stored
    assert abs(got - np.sum(np.abs(b.store(np.zeros((V, 4, 3), complex))) ** 2)) <= tol * got


SOLVERS = [dict(), dict(even_odd=True), dict(solver=1), dict(solver=1, even_odd=True), dict(solver=1, even_odd=True, krylov_prec=2),
           dict(solver=2, even_odd=True), dict(solver=2)]


@pytest.mark.parametrize("kw", SOLVERS)
def test_steps_queued_ahead_do_not_run(kw):
    """A host-driven solve queues a step before it has seen the last one's
    outcome: it stops after exactly max_iter steps, goes on from there, and
    two solves of one source take the same steps to the same bits."""
    dims, kappa, csw, tbc = (6, 4, 4, 8), 0.12, 1.0, -1
    U = synth.exp_links(dims, 0.3, 91)
    lat = make_lattice(dims, U, csw, kappa, tbc)
    src = synth.gaussian_source(dims, 92)
    b = lat.field(0).load(src)
    xs, infos = [], []
    for _ in range(2):
        x = lat.field(0)
        infos.append(lat.solve(x, b, tol=1e-10, **kw))
        xs.append(x.store(np.zeros_like(src)))
    assert infos[0].iters == infos[1].iters and np.array_equal(xs[0], xs[1])
    r = src - oracle.apply_M(dims, tbc, kappa, csw, U, xs[0])
    assert np.linalg.norm(r) <= 1.5e-10 * np.linalg.norm(src)
    for n in (1, 2, 3):
        if n >= infos[0].iters:
            continue
        x = lat.field(0)
        info = lat.solve(x, b, tol=1e-10, max_iter=n, check=False, **kw)
        assert info.iters == n and info.status != 0
        assert lat.solve(x, b, tol=1e-10, **kw).status == 0


def test_solves_of_two_threads_on_their_own_streams():
    """Each thread solves on its own lattice and stream; the solutions have
    the bits of the same solves one after the other."""
    import threading

    import torch
    dims, kappa, csw, tbc = (4, 6, 4, 8), 0.12, 1.0, -1
    kinds = [dict(), dict(solver=1, even_odd=True), dict(solver=2, even_odd=True)]
    lats, srcs, streams = [], [], []
    for k in range(3):
        streams.append(torch.cuda.Stream())
        U = synth.exp_links(dims, 0.3, 95 + k)
        lats.append(wc().Lattice(dims, tbc, stream=streams[k]).load_gauge(U).load_clover(csw, kappa))
        srcs.append(synth.gaussian_source(dims, 97 + k))

    def solve(k, out):
        for _ in range(4):
            x, b = lats[k].field(0), lats[k].field(0).load(srcs[k])
            lats[k].solve(x, b, tol=1e-10, **kinds[k])
            out.append(x.store(np.zeros_like(srcs[k])))

    alone = [[] for _ in kinds]
    for k in range(3):
        solve(k, alone[k])
    together = [[] for _ in kinds]
    threads = [threading.Thread(target=solve, args=(k, together[k])) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(3):
        assert len(together[k]) == 4
        for a in together[k]:
            assert np.array_equal(a, alone[k][0])


@pytest.mark.parametrize("dims,tbc", [((2, 2, 2, 2), -1), ((3, 5, 2, 7), 1), ((5, 3, 7, 4), -1), ((8, 4, 4, 4), -1)])
def test_double_fp32_operator_with_directions_on_four_warps(dims, tbc):
    """M, M^+ and H in double-FP32 arithmetic on ragged volumes, by the kernel
    that splits its input per hop (whatever shape is chosen), and by the
    solves, which split a vector once: one step from x = 0 gives the same
    x as the FP64 arithmetic's to 1e-11 (the step's scalars amplify the
    2^-45 of the operator)."""
    csw, kappa = 1.2, 0.12
    U = synth.haar_links(dims, 160 + sum(dims))
    lat = make_lattice(dims, U, csw, kappa, tbc)
    op = oracle.Operator(dims, U, csw, kappa, tbc)
    psi = synth.gaussian_source(dims, 161)
    F64 = wc().F64
    fi, fo, fx = lat.field(F64).load(psi), lat.field(F64), lat.field(F64)
    lat.solve(fx, fi, tol=1e-13, max_iter=2, max_restarts=0, check=False)
    x64 = fx.store(np.zeros_like(psi))
    lat.set_fp64_arith(wc().ARITH_DF32)
    ref = {"M": op.M(psi), "Mdag": op.Mdag(psi), "hop": oracle.apply_hop(dims, tbc, U, psi)}
    for name in ref:
        getattr(lat, "apply_" + name)(fo, fi)
        assert_elementwise(fo.store(np.zeros_like(psi)), ref[name], 1e-12)
    fx = lat.field(F64)
    lat.solve(fx, fi, tol=1e-13, max_iter=2, max_restarts=0, check=False)
    assert_elementwise(fx.store(np.zeros_like(psi)), x64, 1e-11)


@pytest.mark.parametrize("dims,tbc", [((2, 2, 2, 2), -1), ((6, 2, 10, 4), 1), ((4, 4, 4, 4), -1)])
@pytest.mark.parametrize("arith", [0, 1])
def test_even_odd_passes_of_a_solve(dims, tbc, arith):
    """The source preparation, reconstruction and both residual halves of an
    even-odd solve (modes 4, 2, 5, 1) in FP64 and double-FP32: stopped after
    one step, the reported residual is the oracle's of the returned x; M and
    M^+ (the force's two solves) to 1e-12."""
    csw, kappa = 1.1, 0.11
    U = synth.exp_links(dims, 0.4, 171)
    lat = make_lattice(dims, U, csw, kappa, tbc).set_fp64_arith(arith)
    src = synth.gaussian_source(dims, 172)
    b, x = lat.field(0).load(src), lat.field(0)
    info = lat.solve(x, b, tol=1e-30, max_iter=1, max_restarts=0, even_odd=True, check=False)
    r = src - oracle.apply_M(dims, tbc, kappa, csw, U, x.store(np.zeros_like(src)))
    rel = np.linalg.norm(r) / np.linalg.norm(src)
    assert abs(info.true_rel_resid - rel) <= 1e-11 * max(1.0, rel) + 1e-13
    F = np.zeros((int(np.prod(dims)), 4, 3, 3), complex)
    S = lat.action_force(b, F, tol=1e-13, even_odd=True)
    S0, F0, _, _ = oracle.action_and_force(oracle.Operator(dims, U, csw, kappa, tbc), src, tol=1e-14)
    assert abs(S - S0) <= 1e-11 * S0
    assert_elementwise(F, F0, 1e-9)


@pytest.mark.parametrize("n", [4, 5, 6, 7, 16])
@pytest.mark.parametrize("dims,tbc", [((3, 5, 2, 3), -1), ((4, 4, 4, 4), 1), ((6, 2, 2, 6), -1)])
def test_multi_field_operators_on_16_and_32_sites(n, dims, tbc):
    """M and M^+ of n fields on both sides of the rule for a CTA's sites (4
    and 6 fields), on ragged volumes and odd n (a warp of one and a half
    fields); the Schur form where all extents are even."""
    csw, kappa = 1.2, 0.12
    U = synth.haar_links(dims, 190 + n)
    lat = make_lattice(dims, U, csw, kappa, tbc)
    op = oracle.Operator(dims, U, csw, kappa, tbc)
    srcs = [synth.gaussian_source(dims, 200 + r) for r in range(n)]
    ins, outs = [lat.field(1).load(s) for s in srcs], [lat.field(1) for _ in srcs]
    for dagger in (False, True):
        lat.apply_multi(outs, ins, dagger)
        for s, f in zip(srcs, outs):
            assert_elementwise(f.store(np.zeros_like(s)), op.Mdag(s) if dagger else op.M(s), 1e-5)
    if any(d % 2 for d in dims):
        return
    eo = EvenOdd(dims, tbc, kappa, U, op.T)
    for prec in (1, 2):
        ins, outs = [lat.field(prec).load(s) for s in srcs], [lat.field(prec) for _ in srcs]
        lat.apply_schur_multi(outs, ins, True)
        for s, f in zip(srcs, outs):
            assert_elementwise(f.store(np.zeros_like(s)), eo.schur(s, True), TOL[prec])


@pytest.mark.parametrize("n", [5, 7, 12])
def test_lockstep_group_whose_members_stop_apart(n):
    """The fused inner products of a lockstep group with n members, one of
    which has a zero source: its lanes leave while the other field of the
    warp goes on."""
    dims, kappa, csw, tbc = (4, 4, 4, 6), 0.12, 1.0, -1
    U = synth.exp_links(dims, 0.3, 210)
    lat = make_lattice(dims, U, csw, kappa, tbc)
    srcs = [synth.gaussian_source(dims, 211 + r) if r != 2 else np.zeros((int(np.prod(dims)), 4, 3), complex) for r in range(n)]
    xs = [lat.field(0) for _ in srcs]
    infos = wc().solve_batch([lat] * n, xs, [lat.field(0).load(s) for s in srcs], tol=1e-10, solver=wc().SOLVER_RELIABLE,
                             even_odd=True)
    for s, x, info in zip(srcs, xs, infos):
        sol = x.store(np.zeros_like(s))
        r = s - oracle.apply_M(dims, tbc, kappa, csw, U, sol)
        assert info.status == 0 and np.linalg.norm(r) <= 1.5e-10 * np.linalg.norm(s)


@pytest.mark.parametrize("dims,tbc", [((2, 2, 2, 2), -1), ((2, 4, 6, 2), 1), ((3, 2, 5, 3), -1), ((4, 4, 4, 6), -1)])
@pytest.mark.parametrize("csw", [0.0, 1.3])
def test_force_from_shared_plaquettes(dims, tbc, csw):
    """The force where a plaquette's corners wrap onto each other (extent 2),
    on odd and ragged volumes, with and without the clover part: every link
    against the oracle (its F of the same solutions; solves to 1e-13), and
    traceless and anti-Hermitian to rounding."""
    kappa = 0.11
    U = synth.haar_links(dims, 230 + sum(dims))
    lat = make_lattice(dims, U, csw, kappa, tbc)
    phi = synth.gaussian_source(dims, 231)
    F = np.full((int(np.prod(dims)), 4, 3, 3), 9.0, complex)      # old contents must not matter
    S = lat.action_force(lat.field(0).load(phi), F, tol=1e-13)
    S0, F0, _, _ = oracle.action_and_force(oracle.Operator(dims, U, csw, kappa, tbc), phi, tol=1e-14)
    assert abs(S - S0) <= 1e-11 * S0
    assert_elementwise(F, F0, 1e-9)
    scale = np.abs(F).max()
    assert np.abs(F + F.conj().swapaxes(-1, -2)).max() == 0.0
    assert np.abs(np.trace(F, axis1=-2, axis2=-1)).max() <= 1e-14 * scale


@pytest.mark.parametrize("kw,dims", [
    # FP64, whole lattice: CTAs of 32 sites, the last grid that forms its sums
    # in the operator pass (152 SMs) and the first that does not
    (dict(), (2, 2, 2, 2)), (dict(), (5, 3, 7, 9)), (dict(), (8, 8, 8, 76)), (dict(), (8, 8, 8, 78)),
    (dict(even_odd=True), (2, 2, 2, 2)), (dict(even_odd=True), (6, 2, 10, 4)),
    # low precisions: CTAs of one warp up to 9728 even sites, of four from 38912 on
    (dict(even_odd=True, solver=1, krylov_prec=1), (2, 2, 2, 2)),
    (dict(even_odd=True, solver=1, krylov_prec=1), (6, 2, 10, 4)),
    (dict(even_odd=True, solver=1, krylov_prec=1), (8, 8, 8, 38)),
    (dict(even_odd=True, solver=1, krylov_prec=1), (8, 8, 8, 40)),
    (dict(even_odd=True, solver=1, krylov_prec=1), (10, 14, 18, 34)),
    (dict(even_odd=True, solver=1, krylov_prec=2), (6, 2, 10, 4)),
    (dict(even_odd=True, solver=1, krylov_prec=2), (10, 14, 18, 34))])
def test_sums_formed_by_the_operator_pass(kw, dims):
    """x after one step from x = 0 is alpha b + omega s: the scalars of a step
    whether its operator passes form the sums or separate passes do.  The
    source lives on even sites, so that M^ is all that an even-odd step
    applies to it.  x is first order in both scalars and in the vectors as
    stored: the tolerance of the Krylov vectors."""
    U = synth.exp_links(dims, 0.3, 121)
    lat = make_lattice(dims, U, 1.0, 0.12, -1)
    eo = bool(kw)
    c = np.indices(dims[::-1]).sum(axis=0).reshape(-1) % 2 == 0
    src = synth.gaussian_source(dims, 122)
    if eo:
        src = src * c.reshape(-1, *[1] * (src.ndim - 1))
    f, g = lat.field(0), lat.field(0)

    def op(a):
        (lat.apply_schur if eo else lat.apply_M)(g, f.load(a))
        return g.store(np.zeros_like(a))

    v = op(src)
    alpha = np.vdot(src, src) / np.vdot(src, v)
    s = src - alpha * v
    t = op(s)
    assert abs(np.vdot(t, s)) > 0.75 * np.linalg.norm(t) * np.linalg.norm(s)     # omega as it is
    ref = alpha * src + np.vdot(t, s) / np.vdot(t, t) * s
    x = lat.field(0)
    info = lat.solve(x, lat.field(0).load(src), tol=1e-14, max_iter=1, check=False, **kw)
    assert info.iters == 1
    out = x.store(np.zeros_like(src))
    if eo:
        out = out * c.reshape(-1, *[1] * (src.ndim - 1))
    assert np.linalg.norm(out - ref) <= TOL[kw.get("krylov_prec", 0)] * np.linalg.norm(ref)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 3, 7), (4, 4, 4, 6)])
@pytest.mark.parametrize("krylov", [1, 2])
def test_refresh_on_half_warps_of_ragged_lattices(dims, krylov):
    """A refresh replaces the recurrence's residual 16 sites to a warp.  Lost
    sites or a wrong rho would leave the recurrence with another residual than
    the true one: the solve would need further refreshes and steps, and it
    would not take the steps of the FP64 solve within a factor of two."""
    kappa, csw, tbc = 0.12, 1.0, -1
    U = synth.exp_links(dims, 0.3, 131)
    lat = make_lattice(dims, U, csw, kappa, tbc)
    src = synth.gaussian_source(dims, 132)
    b = lat.field(0).load(src)
    plain = lat.solve(lat.field(0), b, tol=1e-11)
    x = lat.field(0)
    info = lat.solve(x, b, tol=1e-11, solver=1, krylov_prec=krylov)
    r = src - oracle.apply_M(dims, tbc, kappa, csw, U, x.store(np.zeros_like(src)))
    assert np.linalg.norm(r) <= 1.5e-11 * np.linalg.norm(src)
    assert info.iters <= 2 * plain.iters + 4


@pytest.mark.parametrize("dims", [(4, 4, 4, 6), (8, 8, 8, 8)])
@pytest.mark.parametrize("kappa,csw", [(0.12, 1.0), (0.137, 1.9)])
def test_double_fp32_operators_keep_their_accuracy(dims, kappa, csw):
    """Relative L2 distance of the double-FP32 operators from the FP64 ones.
    A pair of floats rounds at 2^-49 = 1.8e-15.  With a chain of double-word
    multiply-adds per row, M stood at 6.6e-15 (kappa 0.12) and 8.5e-15 and M^,
    two dot products longer, at 1.53e-14 and 1.74e-14: the dot products may not
    be worse."""
    U = synth.exp_links(dims, 0.3, 141)
    lat = make_lattice(dims, U, csw, kappa, -1)
    src = synth.gaussian_source(dims, 142)
    f, g = lat.field(0).load(src), lat.field(0)
    out = {}
    for arith in (0, 1):
        lat.set_fp64_arith(arith)
        for name, op in (("M", lat.apply_M), ("S", lat.apply_schur)):
            op(g, f)
            out[name, arith] = g.store(np.zeros_like(src))
    bound = {"M": 6.6e-15 if kappa == 0.12 else 8.5e-15, "S": 1.53e-14 if kappa == 0.12 else 1.74e-14}
    for name in ("M", "S"):
        a, b = out[name, 0], out[name, 1]
        assert np.linalg.norm(a - b) <= bound[name] * np.linalg.norm(a), name
