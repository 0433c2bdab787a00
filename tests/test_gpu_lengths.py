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
