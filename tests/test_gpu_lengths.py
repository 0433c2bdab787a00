"""GPU parity of the two-factor FFT stages at the edges of their dispatch: one
shape per register class (larger factor up to 16, 24 and 32) along every axis,
column counts that leave part of the last 8-column group, coil counts that
leave part of a coil group, against the oracle (relative L2 <= 1e-5)."""
import numpy as np
import pytest

import synth
from oracle import pp_oracle as O

pytestmark = pytest.mark.gpu

TOL_APPLY = 1e-5


@pytest.fixture(scope="module")
def pp():
    from paper_2204_10252_gb300.build import build_library
    build_library()
    import paper_2204_10252_gb300 as m
    m.lib()
    return m


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def err(t, ref):
    got = t.cpu().numpy().astype(np.complex128)
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


# nz, ny, nx: 16-point and smaller factors; 18 x 18 and 18 x 24; 20 x 25 and 16 x 32
@pytest.mark.parametrize("shape,coils", [((20, 36, 100), 1), ((36, 108, 20), 5), ((324, 16, 12), 3), ((16, 432, 12), 4),
                                         ((500, 16, 8), 2), ((16, 512, 20), 3), ((16, 20, 480), 5), ((12, 16, 324), 9)])
def test_cartesian_3d_lengths(pp, shape, coils):
    import torch
    sens = synth.coil_maps(shape, coils, 11)
    mask = synth.line_mask(shape, 2, 8, 12)
    x = synth.crandn(shape, 13)
    y = synth.crandn((coils,) + shape, 14)
    with pp.pp_plan_create(shape, coils, dev(sens), mask=mask, power_iters=0) as plan:
        gy = torch.empty((coils,) + shape, dtype=torch.complex64, device="cuda")
        gx = torch.empty(shape, dtype=torch.complex64, device="cuda")
        gn = torch.empty(shape, dtype=torch.complex64, device="cuda")
        pp.pp_forward_apply(plan, dev(x), gy)
        pp.pp_adjoint_apply(plan, dev(y), gx)
        pp.pp_normal_apply(plan, dev(x), gn)
        assert err(gy, O.cart_forward(x, sens, mask)) <= TOL_APPLY
        assert err(gx, O.cart_adjoint(y, sens, mask)) <= TOL_APPLY
        assert err(gn, O.cart_normal(x, sens, mask)) <= TOL_APPLY


LENGTHS = [32, 36, 40, 48, 60, 64, 72, 80, 96, 100, 108, 120, 128, 144, 160, 180, 192, 200, 216, 240, 256, 288, 300, 320,
           324, 360, 384, 400, 432, 480, 500, 512]


@pytest.mark.parametrize("ny", LENGTHS)
def test_column_resident_chain(pp, ny):
    """Every compiled length of the column-resident operator, one application
    and a Horner chain, with every width (a ragged last group), one to four coil
    groups (maps resident and streamed)."""
    import torch
    nx, c = 12, [1.5, -2.0, 1.25]
    for coils in (1 + ny % 8, 8, 27):
        shape = (ny, nx)
        sens = synth.coil_maps(shape, coils, 21)
        mask = synth.line_mask(shape, 3, 6, 22)
        x = synth.crandn(shape, 23)
        nrm = lambda v: O.cart_normal(v, sens, mask) / 1.25  # noqa: E731
        ref1, ref2 = nrm(x), O.horner_apply(c, nrm, x)
        with pp.pp_plan_create(shape, coils, dev(sens), mask=mask, power_iters=0) as plan:
            pp.pp_plan_set_scale(plan, 1.25)
            out = torch.empty(shape, dtype=torch.complex64, device="cuda")
            for w in (1, 2, 4, 8):
                pp.pp_plan_set_tuning(plan, w, 0, 8)
                pp.pp_normal_apply(plan, dev(x), out)
                assert err(out, ref1) <= TOL_APPLY, (coils, w)
                pp.pp_poly_apply(plan, c, 2, dev(x), out)
                assert err(out, ref2) <= TOL_APPLY, (coils, w)


@pytest.mark.parametrize("tile", [-8, -16, -32])
def test_column_resident_batch_of_mixed_lengths(pp, tile):
    """Slices of several lengths (one launch each, every launch after the first
    beside its predecessor), one long enough for no 4-column form."""
    import torch
    shapes, coils = [(180, 20), (128, 12), (500, 8), (128, 36), (36, 16)], [5, 9, 3, 17, 8]
    sens = [synth.coil_maps(s, c, 31 + i) for i, (s, c) in enumerate(zip(shapes, coils))]
    masks = [synth.line_mask(s, 3, 6, 41 + i) for i, s in enumerate(shapes)]
    b = pp.pp_batch_create(shapes, coils, [dev(s) for s in sens], masks, power_iters=0)
    try:
        pp.pp_batch_set_tile(b, tile)
        assert pp.pp_batch_tile(b)[0] == tile
        L = np.linspace(0.8, 1.4, len(shapes))
        pp.pp_batch_set_scales(b, L)
        xs = [synth.crandn(s, 51 + i) for i, s in enumerate(shapes)]
        x = dev(np.concatenate([v.ravel() for v in xs]))
        y = torch.empty_like(x)
        for _ in range(3):
            pp.pp_batch_normal_apply(b, x, y)
        got = y.cpu().numpy().astype(np.complex128)
        for i, s in enumerate(shapes):
            ref = O.cart_normal(xs[i], sens[i], masks[i]) / L[i]
            g = got[b.image_off[i]:b.image_off[i + 1]].reshape(s)
            assert np.linalg.norm(g - ref) <= TOL_APPLY * np.linalg.norm(ref)
    finally:
        b.destroy()


# image axes (multiples of 4 up to 512), and the other compiled lengths as grids of an
# image axis n oversampled by s: (length, n, s, n and length of the other axis)
AXES = [16, 20, 24, 32, 36, 40, 48, 60, 64, 72, 80, 96, 100, 108, 120, 128, 144, 160, 180, 192, 200, 216, 240, 256, 288,
        300, 320, 324, 360, 384, 400, 432, 480, 500, 512]
GRIDS = [(50, 40, 1.25), (54, 48, 1.125), (90, 72, 1.25), (150, 120, 1.25), (162, 144, 1.125), (250, 200, 1.25),
         (270, 240, 1.125), (450, 360, 1.25), (486, 432, 1.125), (540, 480, 1.125), (576, 512, 1.125), (600, 480, 1.25),
         (640, 512, 1.25), (648, 324, 2.0), (720, 360, 2.0), (750, 500, 1.5), (768, 384, 2.0), (800, 400, 2.0),
         (810, 432, 1.875), (864, 432, 2.0), (900, 480, 1.875), (960, 480, 2.0), (1024, 512, 2.0)]


@pytest.mark.parametrize("n", AXES)
def test_row_and_column_stages_at_every_image_length(pp, n):
    """Forward and adjoint with rows and with columns of every compiled image length,
    beside 20 points (three rows or columns past a group of eight), three coils."""
    import torch
    for shape in ((n, 20), (20, n)):
        sens = synth.coil_maps(shape, 3, 31)
        mask = synth.line_mask(shape, 2, 4, 32)
        x, y = synth.crandn(shape, 33), synth.crandn((3,) + shape, 34)
        with pp.pp_plan_create(shape, 3, dev(sens), mask=mask, power_iters=0) as plan:
            gy = torch.empty((3,) + shape, dtype=torch.complex64, device="cuda")
            gx = torch.empty(shape, dtype=torch.complex64, device="cuda")
            pp.pp_forward_apply(plan, dev(x), gy)
            pp.pp_adjoint_apply(plan, dev(y), gx)
            assert err(gy, O.cart_forward(x, sens, mask)) <= TOL_APPLY, shape
            assert err(gx, O.cart_adjoint(y, sens, mask)) <= TOL_APPLY, shape


@pytest.mark.parametrize("length,n,s", GRIDS)
def test_row_and_column_stages_at_every_grid_length(pp, length, n, s):
    """The same for the lengths that only oversampled grids have."""
    import torch
    assert int(n * s) == length
    for shape in ((n, 64), (64, n)):
        sens = synth.coil_maps(shape, 2, 41)
        traj = (np.random.default_rng(42).uniform(-0.499, 0.499, (301, 2)) * [shape[1], shape[0]]).astype(np.float32)
        x, y = synth.crandn(shape, 43), synth.crandn((2, len(traj)), 44)
        with pp.pp_plan_create(shape, 2, dev(sens), traj=traj, oversamp=s, power_iters=0) as plan:
            gy = torch.empty((2, len(traj)), dtype=torch.complex64, device="cuda")
            gx = torch.empty(shape, dtype=torch.complex64, device="cuda")
            pp.pp_forward_apply(plan, dev(x), gy)
            pp.pp_adjoint_apply(plan, dev(y), gx)
            assert err(gy, O.nc_forward(x, sens, traj, 4, s)) <= TOL_APPLY, shape
            assert err(gx, O.nc_adjoint(y, sens, traj, 4, s)) <= TOL_APPLY, shape


@pytest.mark.parametrize("coils", [3, 5, 9, 27])
@pytest.mark.parametrize("ny", [64, 128, 300, 500])
def test_gradient_and_horner_chain_in_every_form(pp, ny, coils):
    """A preconditioned solve (gradient and Horner recursion in one launch, the
    gradient re-read by the streamed form) with every width, as a plan and as a batch
    of two lengths; 3, 5 and 9 coils give the streamed form 1, 2 and 4 slots where they
    fit.  Tolerance of the repository's solves, 1e-4."""
    import torch
    iters, lam, c = 4, 1e-3, [float(v) for v in O.poly_coeffs_l2(2)]
    shapes = [(ny, 20), (96, 12)]
    sens = [synth.coil_maps(s, coils, 51 + i) for i, s in enumerate(shapes)]
    masks = [synth.line_mask(s, 2, 6, 53 + i) for i, s in enumerate(shapes)]
    ys = [(synth.crandn((coils,) + s, 55 + i) * m[None]).astype(np.complex64) for i, (s, m) in enumerate(zip(shapes, masks))]
    refs = [O.pfista(lambda v: O.cart_normal(v, s, m), lambda y: O.cart_adjoint(y, s, m), y.astype(np.complex128), lam, c,
                     iters, 1.1) for s, m, y in zip(sens, masks, ys)]
    with pp.pp_plan_create(shapes[0], coils, dev(sens[0]), mask=masks[0], power_iters=0) as plan:
        pp.pp_plan_set_scale(plan, 1.1)
        out = torch.empty(shapes[0], dtype=torch.complex64, device="cuda")
        for w in (1, 2, 4, 8):
            pp.pp_plan_set_tuning(plan, w, 0, 8)
            pp.pp_fista_solve(plan, dev(ys[0]), lam, iters, c, 2, out)
            assert err(out, refs[0]) <= 1e-4, w
    b = pp.pp_batch_create(shapes, [coils] * 2, [dev(s) for s in sens], masks, power_iters=0)
    try:
        pp.pp_batch_set_scales(b, np.full(2, 1.1))
        y = dev(np.concatenate([v.ravel() for v in ys]))
        for tile in (-8, -16, -32):
            pp.pp_batch_set_tile(b, tile)
            out = torch.empty(int(b.image_off[-1]), dtype=torch.complex64, device="cuda")
            pp.pp_batch_fista_solve(b, y, lam, iters, c, 2, out)
            for i, s in enumerate(shapes):
                assert err(out[b.image_off[i]:b.image_off[i + 1]].view(s), refs[i]) <= 1e-4, (tile, i)
    finally:
        b.destroy()


def test_coils_split_over_more_ctas_than_a_slice_has(pp):
    """Slices of one length with 1, 27 and 2 coils: the streamed form splits the coils of
    all of them over four CTAs, some of which then have none."""
    import torch
    shapes, coils, c = [(96, 20), (96, 12), (96, 8)], [1, 27, 2], [1.5, -2.0, 1.25]
    sens = [synth.coil_maps(s, n, 61 + i) for i, (s, n) in enumerate(zip(shapes, coils))]
    masks = [synth.line_mask(s, 2, 6, 64 + i) for i, s in enumerate(shapes)]
    xs = [synth.crandn(s, 67 + i) for i, s in enumerate(shapes)]
    b = pp.pp_batch_create(shapes, coils, [dev(s) for s in sens], masks, power_iters=0)
    try:
        pp.pp_batch_set_tile(b, -8)
        pp.pp_batch_set_scales(b, np.full(3, 1.25))
        x = dev(np.concatenate([v.ravel() for v in xs]))
        out = torch.empty_like(x)
        for _ in range(3):
            pp.pp_batch_normal_apply(b, x, out)
        # the chain of the unrolled solve's reverse pass (every result kept) and of its steps
        y = torch.empty(int(b.kspace_off[-1]), dtype=torch.complex64, device="cuda")
        pp.pp_batch_forward_apply(b, x, y)
        sol = torch.empty_like(x)
        pp.pp_batch_fista_solve(b, y, 1e-3, 3, c, 2, sol)
        for i, s in enumerate(shapes):
            lo, hi = b.image_off[i], b.image_off[i + 1]
            nrm = lambda v: O.cart_normal(v, sens[i], masks[i])  # noqa: E731
            assert err(out[lo:hi].view(s), nrm(xs[i]) / 1.25) <= TOL_APPLY
            ref = O.pfista(nrm, lambda v: O.cart_adjoint(v, sens[i], masks[i]), O.cart_forward(xs[i], sens[i], masks[i]),
                           1e-3, c, 3, 1.25)
            assert err(sol[lo:hi].view(s), ref) <= 1e-4
    finally:
        b.destroy()


@pytest.mark.parametrize("coils", [4, 12, 33])
def test_adjoint_rows_of_the_register_lengths(pp, coils):
    """The adjoint's row stage at 16 x {8, 12, 16, 20, 24} points and four coils or more:
    rows as long as the image, and padded ones of a grid (one coil group and several)."""
    import torch
    for nx in (128, 192, 256, 320, 384):
        sens, mask, y = synth.coil_maps((20, nx), coils, 71), synth.line_mask((20, nx), 2, 4, 72), synth.crandn((coils, 20, nx), 73)
        with pp.pp_plan_create((20, nx), coils, dev(sens), mask=mask, power_iters=0) as plan:
            out = torch.empty((20, nx), dtype=torch.complex64, device="cuda")
            pp.pp_adjoint_apply(plan, dev(y), out)
            assert err(out, O.cart_adjoint(y, sens, mask)) <= TOL_APPLY, nx
    for nx, s in ((128, 1.5), (160, 2.0), (256, 1.25)):
        sens = synth.coil_maps((64, nx), coils, 74)
        traj = (np.random.default_rng(75).uniform(-0.499, 0.499, (301, 2)) * [nx, 64]).astype(np.float32)
        y = synth.crandn((coils, len(traj)), 76)
        with pp.pp_plan_create((64, nx), coils, dev(sens), traj=traj, oversamp=s, power_iters=0) as plan:
            out = torch.empty((64, nx), dtype=torch.complex64, device="cuda")
            ref = O.nc_adjoint(y, sens, traj, 4, s)
            pp.pp_plan_set_tuning(plan, 1, 0, 8)
            pp.pp_adjoint_apply(plan, dev(y), out)
            assert err(out, ref) <= TOL_APPLY, nx


def test_batch_forms_of_applications_and_chains(pp):
    """A batch keeps one form for a single application and one for chains; whichever the
    timing takes, both agree with the oracle, also after another form was forced."""
    import torch
    for shapes, coils in (([(256, 24)], [9]), ([(128, 40)] * 3, [5, 17, 3]), ([(512, 12), (64, 60)], [6, 20])):
        sens = [synth.coil_maps(s, n, 81 + i) for i, (s, n) in enumerate(zip(shapes, coils))]
        masks = [synth.line_mask(s, 2, 6, 84 + i) for i, s in enumerate(shapes)]
        xs = [synth.crandn(s, 87 + i) for i, s in enumerate(shapes)]
        ys = [O.cart_forward(v, s, m).astype(np.complex64) for v, s, m in zip(xs, sens, masks)]
        c = [1.5, -2.0, 1.25]
        refs = [O.pfista(lambda v: O.cart_normal(v, s, m), lambda k: O.cart_adjoint(k, s, m),
                         y.astype(np.complex128), 1e-3, c, 3, 1.25)
                for s, m, y in zip(sens, masks, ys)]
        b = pp.pp_batch_create(shapes, coils, [dev(s) for s in sens], masks, power_iters=0)
        try:
            pp.pp_batch_set_scales(b, np.full(b.n, 1.25))
            x, y = (dev(np.concatenate([v.ravel() for v in vs])) for vs in (xs, ys))
            for tile in (None, -16, -32, -8):
                if tile:
                    pp.pp_batch_set_tile(b, tile)
                out, sol = torch.empty_like(x), torch.empty_like(x)
                pp.pp_batch_normal_apply(b, x, out)
                pp.pp_batch_fista_solve(b, y, 1e-3, 3, c, 2, sol)
                for i, s in enumerate(shapes):
                    lo, hi = b.image_off[i], b.image_off[i + 1]
                    assert err(out[lo:hi].view(s), O.cart_normal(xs[i], sens[i], masks[i]) / 1.25) <= TOL_APPLY, (tile, i)
                    assert err(sol[lo:hi].view(s), refs[i]) <= 1e-4, (tile, i)
        finally:
            b.destroy()


@pytest.mark.parametrize("ny", [36, 60, 100, 180, 256, 480])
def test_split_coils_of_one_application(pp, ny):
    """One application whose coils are split over two and four CTAs: every rank adds and
    writes its share of the rows, with and without an operand (a polynomial of degree 0
    and 1 in the streamed form)."""
    import torch
    for coils in (6, 16, 40):
        shape = (ny, 20)
        sens, mask, x = synth.coil_maps(shape, coils, 91), synth.line_mask(shape, 2, 4, 92), synth.crandn(shape, 93)
        with pp.pp_plan_create(shape, coils, dev(sens), mask=mask, power_iters=0) as plan:
            pp.pp_plan_set_scale(plan, 1.25)
            pp.pp_plan_set_tuning(plan, 8, 0, 8)
            ref = O.cart_normal(x, sens, mask) / 1.25
            out = torch.empty(shape, dtype=torch.complex64, device="cuda")
            pp.pp_normal_apply(plan, dev(x), out)
            assert err(out, ref) <= TOL_APPLY, coils
            pp.pp_poly_apply(plan, [0.5, -2.0], 1, dev(x), out)
            assert err(out, 0.5 * x.astype(np.complex128) - 2.0 * ref) <= TOL_APPLY, coils
            y = (synth.crandn((coils,) + shape, 94) * mask[None]).astype(np.complex64)
            pp.pp_fista_solve(plan, dev(y), 1e-3, 4, None, 0, out)
            sol = O.pfista(lambda v: O.cart_normal(v, sens, mask), lambda k: O.cart_adjoint(k, sens, mask),
                           y.astype(np.complex128), 1e-3, None, 4, 1.25)
            assert err(out, sol) <= 1e-4, coils
