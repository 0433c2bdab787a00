"""GPU parity of the gridding applies (forward: interpolation, adjoint: the
gathered spread) at the edges of their dispatch: every lanes-per-point form (8,
16, 32 coils and one past each), more than one chunk of coils, the
coil-innermost and the coil-major grid, samples on the periodic edge and many
samples in one cell."""
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


def trajectory(shape, seed):
    """Uniform samples, samples at -n/2 and just below n/2 on either axis (taps
    that wrap), 300 samples within one cell, and an odd total."""
    ny, nx = shape
    g = np.random.default_rng(seed)
    half = np.array([nx / 2.0, ny / 2.0])
    u = g.uniform(-1.0, 1.0, (400, 2)) * half * 0.999
    e = g.uniform(-1.0, 1.0, (40, 2)) * half * 0.999
    e[:10, 0], e[10:20, 0] = -half[0], np.nextafter(np.float32(half[0]), np.float32(0))
    e[20:30, 1], e[30:, 1] = -half[1], np.nextafter(np.float32(half[1]), np.float32(0))
    c = g.uniform(0.0, 0.4, (301, 2))
    return np.concatenate([u, e, c]).astype(np.float32)


@pytest.mark.parametrize("coils", [1, 8, 9, 16, 17, 32, 33])
@pytest.mark.parametrize("shape,oversamp", [((64, 96), 2.0), ((64, 80), 1.25)], ids=["register_grid", "other_grid"])
def test_gridding_applies_match_oracle(pp, shape, oversamp, coils):
    import torch
    sens = synth.coil_maps(shape, coils, 3)
    traj = trajectory(shape, 5)
    x = synth.crandn(shape, 7)
    y = synth.crandn((coils, len(traj)), 8)
    fwd = O.nc_forward(x, sens, traj, 4, oversamp)
    adj = O.nc_adjoint(y, sens, traj, 4, oversamp)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    with pp.pp_plan_create(shape, coils, dev(sens), traj=traj, oversamp=oversamp, power_iters=0) as plan:
        variants = [pp.pp_plan_tuning(plan)]
        if oversamp == 2.0 and coils <= 32:   # both grid layouts of a plan that has both
            variants = [(1, 1, 8), (1, 9, 8), (4, 9, 8)]
        for v in variants:
            pp.pp_plan_set_tuning(plan, *v)
            gy = torch.empty((coils, len(traj)), dtype=torch.complex64, device="cuda")
            gx = torch.empty(shape, dtype=torch.complex64, device="cuda")
            gs = torch.empty(shape, dtype=torch.complex64, device="cuda")
            pp.pp_forward_apply(plan, dev(x), gy)
            pp.pp_adjoint_apply(plan, dev(y), gx)
            pp.pp_adjoint_apply_static(plan, dev(y), gs)
            for got, ref in ((gy, fwd), (gx, adj), (gs, adj)):
                got = got.cpu().numpy().astype(np.complex128)
                assert np.linalg.norm(got - ref) <= TOL_APPLY * np.linalg.norm(ref)


@pytest.mark.parametrize("coils", [3, 12, 32])
@pytest.mark.parametrize("shape", [(72, 40), (40, 120)], ids=str)
def test_gridding_applies_on_partial_tiles(pp, shape, coils):
    """Grids that the spread's 4 x 4 tiles do not divide (90 x 50, 50 x 150),
    with 300 samples in the corner cells, whose taps wrap on both axes.  FP32 sums of at most 1000 terms: 1e-5 holds."""
    import torch
    sens = synth.coil_maps(shape, coils, 3)
    corner = -np.array([shape[1], shape[0]]) / 2.0 * np.random.default_rng(1).uniform(0.98, 1.0, (300, 2))
    traj = np.concatenate([trajectory(shape, 5), corner.astype(np.float32)])
    x = synth.crandn(shape, 7)
    y = synth.crandn((coils, len(traj)), 8)
    fwd = O.nc_forward(x, sens, traj, 4, 1.25)
    adj = O.nc_adjoint(y, sens, traj, 4, 1.25)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    with pp.pp_plan_create(shape, coils, dev(sens), traj=traj, oversamp=1.25, power_iters=0) as plan:
        gy = torch.empty((coils, len(traj)), dtype=torch.complex64, device="cuda")
        gx = torch.empty(shape, dtype=torch.complex64, device="cuda")
        gs = torch.empty(shape, dtype=torch.complex64, device="cuda")
        pp.pp_forward_apply(plan, dev(x), gy)
        pp.pp_adjoint_apply(plan, dev(y), gx)
        pp.pp_adjoint_apply_static(plan, dev(y), gs)
        for got, ref in ((gy, fwd), (gx, adj), (gs, adj)):
            got = got.cpu().numpy().astype(np.complex128)
            assert np.linalg.norm(got - ref) <= TOL_APPLY * np.linalg.norm(ref)
