"""Performance cases of the library: what a reconstruction program has it do.

Every case calls the package's public entry points on data that is already on
the GPU.  A case names an operation ("op"), the sampling it works on ("kind")
and its sizes.  The inputs are drawn on the GPU from the seed alone: smooth
coil maps with sum_c |S_c|^2 = 1, an ellipse phantom with a smooth phase and
white noise, variable-density line or (ky, kz) masks, Archimedean spirals.

exact() evaluates the same definitions in 64 bits with plain torch calls (FFT,
index_add, eigh, autograd).
"""
import math
from fractions import Fraction

import numpy as np
import torch

import paper_2204_10252_gb300 as pp

C64, C128, F64 = torch.complex64, torch.complex128, torch.float64

# even lengths with prime factors 2, 3 and 5 that are multiples of 4 (the
# two-level wavelet tile): the matrix sizes that scanners and their zero-filled
# reconstructions use
SMOOTH = [n for n in range(16, 513, 4) if not [p for p in (7, 11, 13, 17, 19, 23, 29, 31, 37, 41, 43, 47, 53, 59, 61,
                                                           67, 71, 73, 79, 83, 89, 97, 101, 103, 107, 109, 113, 127)
                                               if n % p == 0]]
SPIRAL_N = [64, 80, 96, 128, 144, 160, 192, 200, 240, 256, 288, 320, 384]
TOEPLITZ_N = [64, 96, 128, 160, 192, 256]


def listed():
    return [
        # One application of the normal operator inside a user's own solver on a
        # small slice: the smallest call, one launch.
        dict(name="normal_cart2d_small", op="normal", kind="cart2d", ny=128, nx=128, coils=8, R=4.0),
        # The same for a brain slice of an ordinary scanner matrix that is not a
        # power of two, with a 13-channel head coil.
        dict(name="normal_cart2d_odd", op="normal", kind="cart2d", ny=180, nx=240, coils=13, R=3.0),
        # The spiral workload's operator (256 x 256, 32 coils, 16 x 4096 samples),
        # gridding form: it is nearly all of a spiral reconstruction.
        dict(name="normal_spiral", op="normal", kind="spiral", ny=256, nx=256, coils=32, interleaves=16, samples=4096,
             turns=4.0),
        # The same through the exact Toeplitz form.
        dict(name="normal_toeplitz", op="normal", kind="toeplitz", ny=256, nx=256, coils=32, interleaves=16,
             samples=4096, turns=4.0),
        # The largest operator: a 256 x 256 x 128 volume, 32 coils.
        dict(name="normal_cart3d", op="normal", kind="cart3d", nz=128, ny=256, nx=256, coils=32, R=8.0),
        # A stack of 64 slices of different protocols, one call for all of them.
        dict(name="normal_batch", op="normal", kind="batch", slices=64, lo=128, hi=384, coils_lo=8, coils_hi=32),
        # A whole small reconstruction with the Daubechies wavelet, as on a
        # scanner's console: 160 operator applications at launch latency.
        dict(name="solve_cart2d_db4", op="solve", kind="cart2d", ny=128, nx=128, coils=8, R=4.0, d=3, iters=40,
             lam=1e-3, wavelet="db4"),
        # The headline reconstruction: spiral, d = 5, Haar prox, to the number of
        # iterations at which it reaches its target accuracy.
        dict(name="solve_spiral", op="solve", kind="spiral", ny=256, nx=256, coils=32, interleaves=16, samples=4096,
             turns=4.0, d=5, iters=20, lam=5e-4, wavelet="haar"),
        # Simulated acquisition and its adjoint for a volume of uneven size, the
        # two halves of a user's own data-consistency step.
        dict(name="fwdadj_cart3d", op="fwdadj", kind="cart3d", nz=80, ny=180, nx=200, coils=12, R=6.0),
        # The same for the spiral: gather and spread gridding.
        dict(name="fwdadj_spiral", op="fwdadj", kind="spiral", ny=256, nx=256, coils=32, interleaves=16, samples=4096,
             turns=4.0),
        # One training step of an unrolled reconstruction network: forward and
        # backward on eight 256 x 256 slices, gradients for data, lambda and p.
        dict(name="train_unrolled", op="train", kind="batch", slices=8, lo=256, hi=256, coils_lo=16, coils_hi=16, d=1,
             iters=3, every=2, lam=3e-5),
        # Locally-low-rank prox of five coefficient images of a volume, as each
        # outer iteration of a fingerprinting reconstruction calls it.
        dict(name="prox_llr", op="llr", kind="image", nz=128, ny=256, nx=256, T=5, block=8, lam=1.5),
    ]


def _log_pick(rng, values, lo, hi):
    """One of the sorted values in [lo, hi], even over their logarithm."""
    v = [x for x in values if lo <= x <= hi]
    t = math.exp(rng.uniform(math.log(v[0]), math.log(v[-1])))
    return min(v, key=lambda x: abs(math.log(x / t)))


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["normal/cart2d", "normal/cart2d", "normal/spiral", "normal/toeplitz", "normal/cart3d",
                       "normal/batch", "solve/cart2d", "solve/spiral", "fwdadj/cart2d", "fwdadj/cart3d",
                       "fwdadj/spiral", "train/batch", "llr/image"])
    op, kind = what.split("/")
    c = dict(op=op, kind=kind)
    if kind == "cart2d":
        c.update(ny=_log_pick(rng, SMOOTH, 64, 512), nx=_log_pick(rng, SMOOTH, 64, 512), coils=_log_int(rng, 4, 32),
                 R=round(rng.uniform(2.0, 6.0), 2))
    elif kind == "cart3d":
        c.update(nz=_log_pick(rng, SMOOTH, 32, 128), ny=_log_pick(rng, SMOOTH, 64, 256),
                 nx=_log_pick(rng, SMOOTH, 64, 256), coils=_log_int(rng, 4, 24), R=round(rng.uniform(4.0, 10.0), 2))
        while c["nz"] * c["ny"] * c["nx"] * c["coils"] > 48000000:
            c["coils"] = max(4, c["coils"] // 2)
            c["ny"] = max(64, SMOOTH[SMOOTH.index(c["ny"]) - 1])
    elif kind in ("spiral", "toeplitz"):
        n = TOEPLITZ_N if kind == "toeplitz" else SPIRAL_N
        ny = _log_pick(rng, n, 64, 384)
        c.update(ny=ny, nx=_log_pick(rng, n, 64, 384) if rng.random() < 0.3 else ny, coils=_log_int(rng, 4, 32),
                 interleaves=rng.randint(6, 32), samples=_log_int(rng, 512, 4096), turns=round(rng.uniform(2.0, 8.0), 2))
    elif kind == "batch" and op == "normal":
        c.update(slices=_log_int(rng, 2, 64), lo=rng.choice([64, 128]), hi=rng.choice([256, 320, 384]), coils_lo=4,
                 coils_hi=rng.randint(8, 32))
    elif kind == "batch":
        c.update(slices=rng.randint(1, 8), lo=rng.choice([96, 128, 192]), hi=256, coils_lo=4, coils_hi=rng.randint(6, 16),
                 d=rng.randint(0, 1), iters=3, every=rng.randint(1, 3), lam=3e-5)
    else:
        three = rng.random() < 0.6
        b = rng.choice([4, 8]) if three else rng.choice([4, 8, 16])
        n = [x for x in SMOOTH if x % b == 0]
        c.update(nz=_log_pick(rng, n, 32, 128) if three else 1, ny=_log_pick(rng, n, 64, 256),
                 nx=_log_pick(rng, n, 64, 256), T=rng.randint(2, 8), block=b, lam=round(rng.uniform(0.5, 2.0), 2))
        while c["nz"] * c["ny"] * c["nx"] * c["T"] > 30000000:
            c["T"] = max(2, c["T"] - 1)
            c["nz"] = max(32, c["nz"] // 2 // b * b)
    if op == "solve":
        c.update(d=rng.randint(0, 5), iters=rng.randint(8, 40), lam=round(rng.uniform(3e-4, 2e-3), 5),
                 wavelet=rng.choice(["haar", "haar", "db4"]))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _cnoise(shape, g, scale):
    s = scale / math.sqrt(2.0)
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=g, device="cuda") * s)


def _axis(n):
    return (torch.arange(n, device="cuda", dtype=torch.float32) - n // 2) / n


def _maps(shape, coils, rng):
    """Gaussian-bump maps on a ring (2-D) or sphere (3-D) around the object."""
    nd = len(shape)
    k = np.arange(coils) + 0.5
    if nd == 2:
        th = 2 * math.pi * k / coils
        ctr = np.stack([np.sin(th), np.cos(th)], 1)
    else:
        phi, th = np.arccos(1 - 2 * k / coils), math.pi * (1 + math.sqrt(5.0)) * k
        ctr = np.stack([np.cos(phi), np.sin(th) * np.sin(phi), np.cos(th) * np.sin(phi)], 1)
    ctr = 0.7 * ctr + rng.uniform(-0.05, 0.05, ctr.shape)
    slope = rng.uniform(-1.0, 1.0, ctr.shape)
    f, sq = [], []
    for a, n in enumerate(shape):
        r = _axis(n)[None]
        c = torch.tensor(ctr[:, a], device="cuda", dtype=torch.float32)[:, None]
        p = torch.tensor(slope[:, a], device="cuda", dtype=torch.float32)[:, None]
        mag = torch.exp(-2.0 * (r - c) ** 2)
        f.append(torch.polar(mag, 2 * math.pi * p * r))
        sq.append(mag * mag)
    out = torch.empty((coils,) + tuple(shape), dtype=C64, device="cuda")
    letters = "zyx"[3 - nd:]
    rss = torch.einsum(",".join("c" + a for a in letters) + "->" + letters, *sq).rsqrt()
    for c in range(coils):
        m = f[0][c].view((-1,) + (1,) * (nd - 1))
        for a in range(1, nd):
            m = m * f[a][c].view((1,) * a + (-1,) + (1,) * (nd - 1 - a))
        out[c] = m * rss
    return out


def _phantom(shape, rng, g, noise=0.03):
    """Ellipses with a smooth phase, plus white noise."""
    nd = len(shape)
    ax = [_axis(n).view((1,) * a + (-1,) + (1,) * (nd - 1 - a)) for a, n in enumerate(shape)]
    img = torch.zeros(tuple(shape), device="cuda")
    for _ in range(12):
        q = 0.0
        for a in range(nd):
            q = q + ((ax[a] - float(rng.uniform(-0.4, 0.4))) / float(rng.uniform(0.05, 0.4))) ** 2
        img += float(rng.uniform(0.1, 1.0)) * (q <= 1.0)
    phase = math.pi * (0.6 * ax[-1] + 0.4 * ax[-2])
    return torch.polar(img, phase.expand(tuple(shape)).contiguous()) + _cnoise(shape, g, noise)


def _mask(shape, R, rng):
    """Variable-density sampling, constant along the readout, centre fully sampled."""
    ph = shape[:-1]
    q = [np.abs(np.arange(n) - n // 2) / (n / 2.0) for n in ph]
    rho = q[0] if len(ph) == 1 else np.sqrt((q[0][:, None] ** 2 + q[1][None, :] ** 2) / 2)
    p = (1.0 - np.minimum(rho, 1.0)) ** 2 + 1e-3
    keep = np.zeros(rho.size, dtype=bool)
    centre = q[0] <= 24.0 / ph[0] if len(ph) == 1 else (q[0] <= 24.0 / ph[0])[:, None] & (q[1] <= 24.0 / ph[1])[None, :]
    want = max(8, int(round(rho.size / R)))
    keep[rng.choice(rho.size, size=want, replace=False, p=(p / p.sum()).ravel())] = True
    keep = keep.reshape(rho.shape) | centre
    return np.ascontiguousarray(np.broadcast_to(keep[..., None], shape)).astype(np.uint8)


def _spiral(case, rng):
    t = np.arange(case["samples"]) / case["samples"]
    turn = 2 * math.pi * (case["turns"] * t[None] + np.arange(case["interleaves"])[:, None] / case["interleaves"]
                          + rng.uniform(0.0, 1.0))
    k = (t[None] * np.exp(1j * turn)).ravel()
    return np.stack([k.real * case["nx"] / 2, k.imag * case["ny"] / 2], 1).astype(np.float32)


def _waves(traj, axis, r, n, dtype):
    """exp(+2 pi i kappa r / n), [K, len(r)]."""
    k = torch.tensor(traj[:, axis], device="cuda", dtype=F64)
    u = k[:, None] * (r.to(F64) / n)[None]
    u = u - torch.round(u)
    f = F64 if dtype == C128 else torch.float32
    a = (2 * math.pi * u).to(f)
    return torch.polar(torch.ones_like(a), a)


def _kernel(traj, ny, nx, dtype):
    """FFT on the 2ny x 2nx circulant of h(d) = 1/n sum_k exp(2 pi i kappa_k d / n)."""
    dy, dx = torch.arange(-ny + 1, ny, device="cuda"), torch.arange(-nx + 1, nx, device="cuda")
    h = torch.zeros((2 * ny - 1, 2 * nx - 1), dtype=dtype, device="cuda")
    for k in range(0, len(traj), 16384):
        t = traj[k:k + 16384]
        h += _waves(t, 1, dy, ny, dtype).T @ _waves(t, 0, dx, nx, dtype)
    full = torch.zeros((2 * ny, 2 * nx), dtype=dtype, device="cuda")
    full[(dy % (2 * ny))[:, None], (dx % (2 * nx))[None]] = h / (ny * nx)
    return torch.fft.fft2(full)


def _scale(traj, ny, nx):
    """A bound on lambda_max(A^H A) from F^H F (the maps have unit sum of squares)."""
    T = _kernel(traj, ny, nx, C64)
    x = torch.ones((ny, nx), dtype=C64, device="cuda")
    top = 1.0
    for _ in range(30):
        x = torch.fft.ifft2(T * torch.fft.fft2(x, s=(2 * ny, 2 * nx)))[:ny, :nx]
        top = float(torch.linalg.vector_norm(x))
        x = x / top
    return 1.05 * top


def _ndft(img, traj):
    """[C, ny, nx] -> [C, K], the exact non-uniform DFT in 32 bits."""
    C, ny, nx = img.shape
    ry, rx = torch.arange(ny, device="cuda") - ny // 2, torch.arange(nx, device="cuda") - nx // 2
    flat = img.reshape(C * ny, nx).T.contiguous()
    out = []
    for k in range(0, len(traj), 8192):
        t = traj[k:k + 8192]
        u = (_waves(t, 0, rx, nx, C64).conj() @ flat).view(len(t), C, ny)
        out.append(torch.bmm(u, _waves(t, 1, ry, ny, C64).conj().unsqueeze(2)).squeeze(2))
    return (torch.cat(out).T / math.sqrt(ny * nx)).contiguous()


def _fft(x, axes, inverse=False):
    f = torch.fft.ifftn if inverse else torch.fft.fftn
    return torch.fft.fftshift(f(torch.fft.ifftshift(x, axes), dim=axes, norm="ortho"), axes)


def _shape(case):
    return (case["nz"], case["ny"], case["nx"]) if case["kind"] == "cart3d" else (case["ny"], case["nx"])


def _slices(case, rng):
    """(ny, nx, coils, R) of a batch's slices."""
    sizes = [n for n in (64, 96, 128, 160, 192, 256, 320, 384) if case["lo"] <= n <= case["hi"]]
    return [(int(rng.choice(sizes)), int(rng.choice(sizes)), int(rng.integers(case["coils_lo"], case["coils_hi"] + 1)),
             int(rng.integers(3, 7))) for _ in range(case["slices"])]


def _inputs(case, seed):
    """Everything that is drawn: the same for prepare() and exact()."""
    rng, g = np.random.default_rng(int(seed)), _gen(seed)
    op, kind = case["op"], case["kind"]
    if kind == "image":
        shape = ((case["nz"],) if case["nz"] > 1 else ()) + (case["ny"], case["nx"])
        base = [_phantom(shape, rng, g) for _ in range(2)]
        w = rng.standard_normal((case["T"], 2)) * 0.7 ** np.arange(case["T"])[:, None]
        x = torch.stack([float(a) * base[0] + float(b) * base[1] for a, b in w]) + _cnoise((case["T"],) + shape, g, 0.05)
        return dict(shape=shape, x=x, shift=[int(v) for v in rng.integers(0, case["block"], len(shape))])
    if kind == "batch":
        # the slices of a protocol do not change with the data in them
        dims = _slices(case, np.random.default_rng(case["slices"] * 1000 + case["hi"] + case["coils_hi"]))
        s = dict(dims=dims, maps=[_maps((a, b), c, rng) for a, b, c, _ in dims],
                 masks=[_mask((a, b), r, rng) for a, b, _, r in dims])
        # training on noisy, weakly regularised data: its images have detail everywhere
        img = [_phantom((a, b), rng, g, 0.03 if op == "normal" else 0.3) for a, b, _, _ in dims]
        if op == "normal":
            s["x"] = torch.cat([v.reshape(-1) for v in img])
        else:
            m = [torch.tensor(k, device="cuda", dtype=torch.float32) for k in s["masks"]]
            s["b"] = torch.cat([((_fft(v * t, (-2, -1)) + _cnoise(t.shape, g, 0.1)) * k).reshape(-1)
                                for v, t, k in zip(img, s["maps"], m)])
            s["target"] = torch.cat([v.reshape(-1) for v in img])
        return s
    shape = _shape(case)
    s = dict(shape=shape, maps=_maps(shape, case["coils"], rng), x=_phantom(shape, rng, g))
    if kind in ("cart2d", "cart3d"):
        s["mask"], s["L"] = _mask(shape, case["R"], rng), 1.0
        if op == "solve":
            m = torch.tensor(s["mask"], device="cuda", dtype=torch.float32)
            s["b"] = (_fft(s["x"] * s["maps"], (-2, -1)) + _cnoise(s["maps"].shape, g, 1e-2)) * m
    else:
        s["traj"] = _spiral(case, rng)
        s["L"] = _scale(s["traj"], *shape)
        if op == "solve":
            b = _ndft(s["x"] * s["maps"], s["traj"])
            s["b"] = b + _cnoise(b.shape, g, 1e-2)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    op, kind = case["op"], case["kind"]
    s["case"] = case
    empty = lambda n: torch.empty(n, dtype=C64, device="cuda")  # noqa: E731
    if kind == "image":
        s["out"] = torch.empty_like(s["x"])
        return s
    if kind == "batch":
        dims = s["dims"]
        s["plan"] = pp.pp_batch_create([d[:2] for d in dims], [d[2] for d in dims], s["maps"], s["masks"], power_iters=0)
        pp.pp_batch_set_scales(s["plan"], np.ones(len(dims)))
        if op == "normal":
            s["out"] = torch.empty_like(s["x"])
        else:
            s["b"].requires_grad_(True)
            s["lam"] = torch.tensor(case["lam"], dtype=torch.float32, requires_grad=True)
            s["c"] = torch.tensor(pp.pp_poly_coeffs_l2(case["d"]), dtype=torch.float32, requires_grad=True)
        return s
    kw = dict(mask=s["mask"]) if "mask" in s else dict(traj=s["traj"], toeplitz=kind == "toeplitz")
    s["plan"] = pp.pp_plan_create(s["shape"], case["coils"], s["maps"], power_iters=0, **kw)
    pp.pp_plan_set_scale(s["plan"], s["L"])
    s["out"] = torch.empty_like(s["x"])
    if op == "solve":
        s["c"] = pp.pp_poly_coeffs_l2(case["d"])
    elif op == "fwdadj":
        s["y"] = empty(s["plan"].kspace_shape)
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "normal":
        (pp.pp_batch_normal_apply if case["kind"] == "batch" else pp.pp_normal_apply)(s["plan"], s["x"], s["out"])
        return s["out"]
    if op == "solve":
        pp.pp_fista_solve(s["plan"], s["b"], case["lam"], case["iters"], s["c"], case["d"], s["out"],
                          wavelet=case["wavelet"])
        return s["out"]
    if op == "fwdadj":
        pp.pp_forward_apply(s["plan"], s["x"], s["y"])
        pp.pp_adjoint_apply(s["plan"], s["y"], s["out"])
        return s["y"], s["out"]
    if op == "llr":
        pp.pp_prox_llr(s["shape"], case["T"], case["block"], case["lam"], s["x"], s["out"], shift=s["shift"])
        return s["out"]
    y = pp.unrolled_pfista(s["plan"], s["b"], s["lam"], s["c"], case["iters"], checkpoint_every=case["every"])
    gb, gl, gc = torch.autograd.grad(y, (s["b"], s["lam"], s["c"]), grad_outputs=y.detach() - s["target"])
    return y.detach(), gb, gl, gc


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _lines(n, count):
    """5 n log2 n flops for each of `count` complex FFTs of length n."""
    return 5.0 * n * math.log2(n) * count


def _normal_work(kind, ny, nx, nz, C, K, table):
    """(bytes, flops) of one A^H A: maps and image in, image out; the readout is not transformed under a line mask."""
    n = ny * nx * nz
    if kind == "cart":
        f = 2 * _lines(ny, C * nx * nz) + (2 * _lines(nz, C * nx * ny) if nz > 1 else 0.0)
        return 8.0 * (C * n + 2 * n) + ny * nz, f + 16.0 * C * n
    gy, gx = (2 * ny, 2 * nx) if kind == "toeplitz" else (math.ceil(1.25 * ny), math.ceil(1.25 * nx))
    f = 2 * _lines(gx, C * ny) + 2 * _lines(gy, C * gx)
    if kind == "toeplitz":
        return 8.0 * (C * n + 2 * n) + 4.0 * gx * gy, f + C * (16.0 * n + 2.0 * gx * gy)
    # gridding: 16 taps a sample out and in
    return 8.0 * (C * n + 2 * n) + 8.0 * K, f + C * (16.0 * n + 4.0 * 16 * 2 * K)


def work(case):
    op, kind = case["op"], case["kind"]
    if op == "llr":
        n = case["nz"] * case["ny"] * case["nx"]
        T = case["T"]
        # the Gram matrix of every block and the product with its T x T factor
        return {"bytes": 16.0 * n * T, "flops": n * (8.0 * T * (T + 1) / 2 + 8.0 * T * T)}
    if kind == "batch":
        dims = _slices(case, np.random.default_rng(case["slices"] * 1000 + case["hi"] + case["coils_hi"]))
        w = [_normal_work("cart", a, b, 1, c, 0, 0) for a, b, c, _ in dims]
        one = {"bytes": sum(v[0] for v in w), "flops": sum(v[1] for v in w)}
        if op == "normal":
            return one
        n, y = sum(a * b for a, b, _, _ in dims), sum(a * b * c for a, b, c, _ in dims)
        # adjoint of b, iters (d + 1) applications forward, as many again in
        # reverse, the forward operator for b's gradient
        full = sum(2 * (_lines(a, b * c) + _lines(b, a * c)) + 16.0 * a * b * c for a, b, c, _ in dims)
        return {"bytes": 8.0 * (y + 2 * y + 3 * n), "flops": 2 * case["iters"] * (case["d"] + 1) * one["flops"] + full}
    C = case["coils"]
    ny, nx, nz = case["ny"], case["nx"], case.get("nz", 1)
    n, K = ny * nx * nz, case.get("interleaves", 0) * case.get("samples", 0)
    cart = kind in ("cart2d", "cart3d")
    by, fl = _normal_work("cart" if cart else kind, ny, nx, nz, C, K, None)
    if op == "normal":
        return {"bytes": by, "flops": fl}
    ksp = C * (n if cart else K)
    if cart:
        half = sum(_lines(m, C * n // m) for m in (ny, nx, nz) if m > 1) + 8.0 * C * n
    else:
        half = fl / 2
    if op == "fwdadj":
        return {"bytes": 8.0 * (2 * ksp + C * n + 2 * n), "flops": 2 * half}
    its = case["iters"]
    prox = (32.0 if case["wavelet"] == "haar" else 64.0) * n
    return {"bytes": by + 8.0 * ksp, "flops": half + its * ((case["d"] + 1) * fl + prox)}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _cart_ops(maps, mask):
    S = maps.to(C128)
    m = torch.tensor(mask, device="cuda", dtype=F64)
    ax = tuple(range(-mask.ndim, 0))
    fwd = lambda x: torch.stack([m * _fft(x * s, ax) for s in S])  # noqa: E731
    adj = lambda y: sum(s.conj() * _fft(m * v, ax, True) for s, v in zip(S, y))  # noqa: E731
    ph = ax[:-1]
    nrm = lambda x: sum(s.conj() * _fft(m * _fft(x * s, ph), ph, True) for s in S)  # noqa: E731
    return fwd, adj, nrm


def _grid_ops(maps, traj, ny, nx):
    """Kaiser-Bessel gridding of width 4, oversampling 1.25 (Beatty et al. 2005)."""
    W, sig = 4, 1.25
    gy, gx = math.ceil(sig * ny), math.ceil(sig * nx)
    beta = math.pi * math.sqrt((W / sig) ** 2 * (sig - 0.5) ** 2 - 0.8)

    def taps(axis, n, G):
        s = torch.tensor(traj[:, axis], device="cuda", dtype=F64) * (G / n)
        m = (torch.floor(s - W / 2.0) + 1)[:, None] + torch.arange(W, device="cuda", dtype=F64)[None]
        t = 1 - (2 * (s[:, None] - m) / W) ** 2
        w = torch.where(t >= 0, torch.special.i0(beta * torch.sqrt(t.clamp(min=0))), torch.zeros_like(t))
        return m.long() % G, w

    def apod(n, G):
        a = beta ** 2 - (math.pi * W * (torch.arange(n, device="cuda", dtype=F64) - n // 2) / G) ** 2
        r = torch.sqrt(a.abs())
        return torch.where(a > 0, torch.sinh(r), torch.sin(r)) * W / r

    (iy, wy), (ix, wx) = taps(1, ny, gy), taps(0, nx, gx)
    idx = (iy[:, :, None] * gx + ix[:, None, :]).reshape(-1)
    w = (wy[:, :, None] * wx[:, None, :]).reshape(-1, 1, 1)
    d = (apod(ny, gy)[:, None] * apod(nx, gx)[None]).reciprocal() / math.sqrt(ny * nx)
    S = maps.to(C128) * d
    C, K = S.shape[0], len(traj)
    py = (torch.arange(ny, device="cuda") - ny // 2) % gy
    px = (torch.arange(nx, device="cuda") - nx // 2) % gx

    def fwd(x):
        g = torch.zeros((C, gy, gx), dtype=C128, device="cuda")
        g[:, py[:, None], px[None]] = x * S
        g = torch.view_as_real(torch.fft.fft2(g).permute(1, 2, 0).reshape(gy * gx, C).contiguous())
        return torch.view_as_complex((g[idx] * w).view(K, 16, C, 2).sum(1).contiguous()).T

    def adj(y):
        v = torch.view_as_real(y.T.contiguous()).repeat_interleave(16, 0) * w
        g = torch.zeros((gy * gx, C, 2), dtype=F64, device="cuda").index_add_(0, idx, v)
        g = torch.view_as_complex(g).view(gy, gx, C).permute(2, 0, 1)
        return (S.conj() * (torch.fft.ifft2(g, norm="forward")[:, py[:, None], px[None]])).sum(0)
    return fwd, adj, lambda x: adj(fwd(x))


def _toeplitz_op(maps, traj, ny, nx):
    T, S = _kernel(traj, ny, nx, C128), maps.to(C128)
    return lambda x: (S.conj() * torch.fft.ifft2(T * torch.fft.fft2(x * S, s=(2 * ny, 2 * nx)))[:, :ny, :nx]).sum(0)


def _soft(v, lam):
    a = v.abs()
    on = a > lam
    safe = torch.where(on, a, torch.ones_like(a))
    return torch.where(on, v * (1 - lam / safe), torch.zeros_like(v))


def _haar(v, lam, levels=2):
    """Two-level orthonormal Haar prox of a 2-D image."""
    if levels == 0:
        return _soft(v, lam)
    a, b, c, d = v[0::2, 0::2], v[0::2, 1::2], v[1::2, 0::2], v[1::2, 1::2]
    s = _haar((a + b + c + d) / 2, lam, levels - 1)
    x, y, z = (_soft(t / 2, lam) for t in (a - b + c - d, a + b - c - d, a - b - c + d))
    rows = [torch.stack([s + x + y + z, s - x + y - z], -1), torch.stack([s + x - y - z, s - x - y + z], -1)]
    return torch.stack([r.flatten(-2) for r in rows], 1).reshape(v.shape) / 2


def _db4(v, lam, levels=2):
    """Prox of the periodic four-coefficient Daubechies transform."""
    if levels == 0:
        return _soft(v, lam)
    r = math.sqrt(3.0)
    h = [c / (4 * math.sqrt(2.0)) for c in (1 + r, 3 + r, 3 - r, 1 - r)]
    g = [h[3], -h[2], h[1], -h[0]]

    def split(x, ax):
        t = [torch.roll(x, -k, ax).index_select(ax, torch.arange(0, x.shape[ax], 2, device="cuda")) for k in range(4)]
        return sum(h[k] * t[k] for k in range(4)), sum(g[k] * t[k] for k in range(4))

    def join(a, d, ax):
        shape = list(a.shape)
        shape[ax] *= 2
        out = torch.zeros(shape, dtype=a.dtype, device="cuda")
        even = torch.arange(0, shape[ax], 2, device="cuda")
        for k in range(4):
            out.index_add_(ax, (even + k) % shape[ax], h[k] * a + g[k] * d)
        return out
    lo, hi = split(v, 1)
    (ll, lh), (hl, hh) = split(lo, 0), split(hi, 0)
    ll = _db4(ll, lam, levels - 1)
    return join(join(ll, _soft(lh, lam), 0), join(_soft(hl, lam), _soft(hh, lam), 0), 1)


def _l2(d):
    """Minimiser of int_0^1 (1 - z p(z))^2 dz: the normal equations in exact rationals."""
    m = [[Fraction(1, i + j + 3) for j in range(d + 1)] + [Fraction(1, i + 2)] for i in range(d + 1)]
    for i in range(d + 1):
        m[i] = [v / m[i][i] for v in m[i]]
        for k in range(d + 1):
            if k != i:
                m[k] = [a - m[k][i] * b for a, b in zip(m[k], m[i])]
    return [float(r[-1]) for r in m]


def _pfista(nrm, ahb, prox, lam, c, iters):
    y = z = torch.zeros_like(ahb)
    for k in range(iters):
        g = nrm(z) - ahb
        u = c[-1] * g
        for i in range(len(c) - 2, -1, -1):
            u = c[i] * g + nrm(u)
        new = prox(z - u, lam)
        z = new + k / (k + 3.0) * (new - y)
        y = new
    return y


def exact(case, seed):
    s = _inputs(case, seed)
    op, kind = case["op"], case["kind"]
    if kind == "image":
        b, shape, T = case["block"], s["shape"], case["T"]
        nd = len(shape)
        ax, sh = tuple(range(1, nd + 1)), list(reversed(s["shift"]))
        x = torch.roll(s["x"].to(C128), [-v for v in sh], ax)
        x = x.reshape([T] + [k for n in shape for k in (n // b, b)])
        perm = [1 + 2 * i for i in range(nd)] + [2 + 2 * i for i in range(nd)] + [0]
        x = x.permute(perm)
        M = x.reshape(-1, b ** nd, T)
        out = torch.empty_like(M)
        for i in range(0, len(M), 4096):
            m = M[i:i + 4096]
            e, V = torch.linalg.eigh(m.mH @ m)
            e = torch.sqrt(e.clamp(min=0))
            f = torch.where(e > case["lam"], 1 - case["lam"] / e.clamp(min=1e-300), torch.zeros_like(e))
            out[i:i + 4096] = m @ ((V * f[:, None]) @ V.mH)
        out = out.reshape(x.shape).permute([int(v) for v in np.argsort(perm)]).reshape((T,) + tuple(shape))
        return torch.roll(out, sh, ax)
    if kind == "batch":
        ops = [_cart_ops(m, k) for m, k in zip(s["maps"], s["masks"])]
        dims = [d[:2] for d in s["dims"]]
        if op == "normal":
            xs = torch.split(s["x"].to(C128), [a * b for a, b in dims])
            return torch.cat([o[2](v.view(d)).reshape(-1) for o, v, d in zip(ops, xs, dims)])
        b = s["b"].to(C128).requires_grad_(True)
        lam = torch.tensor(float(np.float32(case["lam"])), dtype=F64, device="cuda", requires_grad=True)
        c = torch.tensor(np.float32(_l2(case["d"])), dtype=F64, device="cuda", requires_grad=True)
        bs = torch.split(b, [d[0] * d[1] * d[2] for d in s["dims"]])
        y = torch.cat([_pfista(o[2], o[1](v.view(d[2], d[0], d[1])), _haar, lam, c, case["iters"]).reshape(-1)
                       for o, v, d in zip(ops, bs, s["dims"])])
        y32 = y.detach().to(C64)
        grads = torch.autograd.grad(y, (b, lam, c), grad_outputs=(y32 - s["target"]).to(C128))
        return (y.detach(),) + tuple(grads)
    shape = s["shape"]
    if "mask" in s:
        fwd, adj, nrm = _cart_ops(s["maps"], s["mask"])
    elif kind == "toeplitz":
        fwd, adj, nrm = None, None, _toeplitz_op(s["maps"], s["traj"], *shape)
    else:
        fwd, adj, nrm = _grid_ops(s["maps"], s["traj"], *shape)
    if op == "normal":
        return nrm(s["x"].to(C128)) / s["L"]
    if op == "fwdadj":
        y = fwd(s["x"].to(C128))
        return y, adj(y)
    b = s["b"].to(C128)
    ahb = adj(b / torch.linalg.vector_norm(b)) / math.sqrt(s["L"])
    return _pfista(lambda v: nrm(v) / s["L"], ahb, _db4 if case["wavelet"] == "db4" else _haar, case["lam"], _l2(case["d"]),
                   case["iters"])
