"""Plans on a nearly full GPU: workspaces that only make things faster shrink, and the
operators give what they give with all of them.  This also holds the loops over chunks
of coils (3-D) and of slices (batched adjoint) to the results of a single chunk.

Tolerance: the same FP32 sums over coils in another grouping, 2e-6."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

TOL = 2e-6
MB = 1 << 20


@pytest.fixture(scope="module")
def pp():
    from paper_2204_10252_gb300.build import build_library
    build_library()
    import paper_2204_10252_gb300 as m
    m.lib()
    return m


def noise(shape, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=g, device="cuda"))


def fill(leave):
    """Takes the device's memory but for `leave` bytes, until the result is dropped."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room, _ = torch.cuda.mem_get_info()
    assert room > leave
    return torch.empty(room - leave, dtype=torch.uint8, device="cuda")


def compare(make, apply, leave):
    """apply(plan) with all the memory, and with `leave` bytes when the plan is made."""
    import torch
    want = []
    with make() as plan:
        apply(plan, want)
        torch.cuda.synchronize()
    got = [torch.empty_like(w) for w in want]
    held = fill(leave)
    try:
        with make() as plan:
            del held
            apply(plan, got)
            torch.cuda.synchronize()
    finally:
        held = None
        torch.cuda.empty_cache()
    for w, g in zip(want, got):
        assert float(torch.linalg.vector_norm(g - w)) <= TOL * float(torch.linalg.vector_norm(w))


def put(outs, i, like):
    """Output i: made on the first pass."""
    import torch
    if len(outs) <= i:
        outs.append(torch.empty(like, dtype=torch.complex64, device="cuda"))
    return outs[i]


def test_3d_plan_with_a_chunk_of_coils(pp):
    """11 coils of 44 MB: one chunk of 487 MB with all the memory; with 760 MB, of which
    the images and one volume take 400, three coils at a time (3 + 3 + 3 + 2)."""
    shape, coils = (96, 240, 240), 11
    sens = noise((coils,) + shape, 1) / coils
    mask = synth.line_mask(shape, 3, 8, 2)
    x, y = noise(shape, 3), noise((coils,) + shape, 4)

    def apply(plan, outs):
        pp.pp_plan_set_scale(plan, 0.3)
        pp.pp_forward_apply(plan, x, put(outs, 0, y.shape))
        pp.pp_adjoint_apply(plan, y, put(outs, 1, shape))
        pp.pp_normal_apply(plan, x, put(outs, 2, shape))
        pp.pp_poly_apply(plan, [1.5, -2.0, 1.25], 2, x, put(outs, 3, shape))

    compare(lambda: pp.pp_plan_create(shape, coils, sens, mask=mask, power_iters=0), apply, 760 * MB)


def test_spread_without_its_transposed_kspace(pp):
    """2^20 samples of 32 coils: 268 MB of transposed k-space, with 300 MB left."""
    shape, coils, K = (128, 128), 32, 1 << 20
    sens = noise((coils,) + shape, 1) / coils
    traj = np.random.default_rng(2).uniform(-63.9, 63.9, (K, 2)).astype(np.float32)
    x, y = noise(shape, 3), noise((coils, K), 4)

    def apply(plan, outs):
        pp.pp_adjoint_apply(plan, y, put(outs, 0, shape))
        pp.pp_normal_apply(plan, x, put(outs, 1, shape))

    compare(lambda: pp.pp_plan_create(shape, coils, sens, traj=traj, power_iters=0), apply, 300 * MB)


def test_batch_with_one_slice_of_adjoint_workspace(pp):
    """12 slices with 63 MB of k-space: one adjoint chunk with all the memory; with
    100 MB, of which the images take 50, one slice at a time."""
    shapes, coils = [(256, 240), (240, 256), (256, 256)] * 4, [10] * 12
    sens = [noise((c,) + s, 10 + i) / c for i, (s, c) in enumerate(zip(shapes, coils))]
    masks = [synth.line_mask(s, 3, 8, i) for i, s in enumerate(shapes)]
    n = sum(a * b for a, b in shapes)
    x, y = noise((n,), 3), noise((10 * n,), 4)

    class Made:
        def __enter__(self):
            self.b = pp.pp_batch_create(shapes, coils, sens, masks, power_iters=0)
            return self.b

        def __exit__(self, *a):
            self.b.destroy()

    def apply(batch, outs):
        pp.pp_batch_forward_apply(batch, x, put(outs, 0, (10 * n,)))
        pp.pp_batch_adjoint_apply(batch, y, put(outs, 1, (n,)))
        pp.pp_batch_normal_apply(batch, x, put(outs, 2, (n,)))

    compare(Made, apply, 100 * MB)
