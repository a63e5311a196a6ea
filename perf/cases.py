"""Performance cases of the reconstruction library: what its users run, through the public API.

Kinds of work (a case is one of these at one size):

* ``forward`` / ``adjoint``: one application of A or A^H of a plan whose geometry and coil maps are
  set.  The operator on its own is what simulation, data-consistency layers and any outer
  solver written by the user call.
* ``recon``: one whole reconstruction of a new scan with an existing plan: new trajectory and
  maps into the plan, then the PDHG solve with the multi-channel preconditioner and lambda_max
  computed inside (the scanner's work for each scan).
* ``frame``: one frame of a series with fixed geometry: the PDHG solve alone, the preconditioner
  and lambda_max computed once beforehand.
* ``batch``: a mix of independent 2D cases solved together, as a serving process does.
* ``unrolled``: one training step through the unrolled solver: forward, then the gradients with
  respect to the measurements, lambda and the trajectory.
* ``precond``: the multi-channel preconditioner of a new set of maps.

Inputs are drawn on the GPU from the seed: random ellipses, Gaussian-bump coil maps normalised to
unit sum of squares, golden-angle radial, variable-density spiral and 3D centre-out radial
trajectories turned by a random angle, and measurements of the drawn image with 1 % noise.  The
64-bit expressions of the method further down serve ``exact`` and the measurements.
"""
import functools
import math

import numpy as np
import torch

from paper_1902_09657_gb300 import autograd
from paper_1902_09657_gb300.api import Batch, Plan, to_storage

DEV = "cuda"
W = 4                      # Kaiser-Bessel width
POWER_ITERS = 30


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one frame's forward operator of a small real-time 2D radial scan: the smallest call
        dict(name="forward_2d_small", kind="forward", n0=128, n1=128, n2=0, coils=4, traj="radial", shots=64, read=256,
             alpha=2.0, maps="c64", y="c64"),
        # an odd-sized 2D radial forward operator (ragged field of view, odd coil and sample counts)
        dict(name="forward_2d_ragged", kind="forward", n0=217, n1=186, n2=0, coils=7, traj="radial", shots=151, read=433,
             alpha=1.25, maps="c64", y="c64"),
        # adjoint (gridding reconstruction) of a 2D spiral scan kept in 16-bit storage
        dict(name="adjoint_2d_half", kind="adjoint", n0=256, n1=256, n2=0, coils=12, traj="spiral", shots=24, read=4096,
             alpha=1.25, maps="fp16", y="bf16"),
        # 3D forward operator at the full size of the UTE scan, half-precision maps
        dict(name="forward_3d", kind="forward", n0=192, n1=192, n2=192, coils=8, traj="radial3d", shots=24000, read=256,
             alpha=1.25, maps="fp16", y="c64"),
        # 3D adjoint on an uneven volume with odd coil, spoke and sample counts
        dict(name="adjoint_3d_ragged", kind="adjoint", n0=150, n1=132, n2=116, coils=5, traj="radial3d", shots=9001,
             read=187, alpha=1.25, maps="c64", y="c64"),
        # whole small 2D radial reconstruction, l2
        dict(name="recon_2d_l2", kind="recon", n0=128, n1=128, n2=0, coils=4, traj="radial", shots=64, read=256,
             alpha=2.0, maps="c64", y="c64", reg="l2", lam=1e-3, levels=0, iters=30),
        # whole 2D spiral compressed-sensing reconstruction, l1-wavelet, 16-bit storage
        dict(name="recon_2d_l1", kind="recon", n0=256, n1=256, n2=0, coils=12, traj="spiral", shots=24, read=4096,
             alpha=1.25, maps="fp16", y="bf16", reg="l1_wavelet", lam=1e-3, levels=4, iters=100),
        # one frame of a 2D radial series with total variation, geometry fixed
        dict(name="frame_2d_tv", kind="frame", n0=192, n1=192, n2=0, coils=16, traj="radial", shots=120, read=384,
             alpha=1.25, maps="c64", y="c64", reg="tv", lam=1e-3, levels=0, iters=50),
        # a serving batch of uneven 2D cases, radial and spiral, l2 and l1 mixed, bf16 k-space
        dict(name="batch_2d", kind="batch", cases=12, iters=20, nmin=96, nmax=320, cmin=4, cmax=32, mix=1000),
        # training step of the unrolled solver
        dict(name="unrolled_2d", kind="unrolled", n0=256, n1=256, n2=0, coils=16, traj="spiral", shots=16, read=4096,
             alpha=1.25, maps="c64", y="c64", lam=1e-2, iters=10),
        # preconditioner of a many-coil 2D scan (the set-up of every reconstruction)
        dict(name="precond_2d", kind="precond", n0=320, n1=320, n2=0, coils=32, traj="radial", shots=400, read=640,
             alpha=1.25, maps="c64", y="c64"),
        # whole 3D UTE compressed-sensing reconstruction: the largest and the headline
        dict(name="recon_3d_l1", kind="recon", n0=192, n1=192, n2=192, coils=8, traj="radial3d", shots=24000, read=256,
             alpha=1.25, maps="fp16", y="c64", reg="l1_wavelet", lam=1e-3, levels=3, iters=30),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi, mult):
    """An image side: mostly a scanner matrix size (a multiple of 8), at times any size; a multiple
    of `mult` where the wavelet levels ask for it."""
    n = _log(rng, lo, hi)
    if mult > 1:
        return max(mult, n // mult * mult)
    return max(8, n // 8 * 8) if rng.random() < 0.7 else n


def draw(rng):
    kind = rng.choice(["forward", "adjoint", "forward", "adjoint", "recon", "recon", "recon", "frame", "batch",
                       "unrolled", "precond"])
    if kind == "batch":
        nmin = 16 * rng.randint(6, 12)
        return dict(kind="batch", cases=rng.randint(3, 12), iters=rng.randint(10, 20), nmin=nmin,
                    nmax=min(320, nmin + 16 * rng.randint(1, 10)), cmin=4, cmax=rng.randint(8, 32), mix=rng.randint(1, 10 ** 6))
    three = kind in ("forward", "adjoint", "recon") and rng.random() < 0.4
    reg, levels = "l2", 0
    if kind in ("recon", "frame"):
        reg = rng.choice(["l2", "l1_wavelet", "l1_wavelet", "tv"])
        levels = rng.randint(2, 3 if three else 4) if reg == "l1_wavelet" else 0
    mult = 1 << levels
    if three:
        big = 160 if kind == "recon" else 192
        ns = [_side(rng, 40, big, mult) for _ in range(3)]
        if rng.random() < 0.6:
            ns = [ns[0]] * 3
        coils = rng.randint(1, 8)
        read = rng.randint(int(1.0 * max(ns)), int(1.35 * max(ns)))
        shots = _log(rng, 10 * max(ns), 125 * max(ns))
        traj, alpha = "radial3d", rng.choice([1.25, 1.25, 1.25, 1.5])
        iters = rng.randint(10, 30)
    else:
        lo, hi = (64, 320) if kind != "unrolled" else (64, 256)
        ns = [_side(rng, lo, hi, mult) for _ in range(2)] + [0]
        if rng.random() < 0.6:
            ns[1] = ns[0]
        coils = _log(rng, 1, 16 if kind == "unrolled" else 32)
        traj = rng.choice(["radial", "spiral"])
        read = rng.randint(int(1.9 * max(ns)), int(2.4 * max(ns))) if traj == "radial" else _log(rng, 800, 4096)
        shots = _log(rng, 16, 400) if traj == "radial" else _log(rng, 6, 32)
        alpha = rng.choice([1.25, 1.25, 1.5, 2.0])
        iters = rng.randint(4, 10) if kind == "unrolled" else rng.randint(20, 100)
    c = dict(kind=kind, n0=ns[0], n1=ns[1], n2=ns[2], coils=coils, traj=traj, shots=shots, read=read, alpha=alpha,
             maps="c64" if kind == "unrolled" else rng.choice(["c64", "c64", "fp16"]),
             y="c64" if kind in ("unrolled", "precond", "forward") else rng.choice(["c64", "c64", "bf16"]))
    if kind in ("recon", "frame"):
        c.update(reg=reg, lam=1e-3, levels=levels, iters=iters)
    if kind == "unrolled":
        c.update(lam=1e-2, iters=iters)
    return c


def _shape(case):
    return tuple(case[k] for k in ("n0", "n1", "n2") if case[k])


def _batch_cases(case):
    """The uneven cases of a batch: side, coils, shots, trajectory and regulariser from the mix's number."""
    out = []
    for i in range(case["cases"]):
        r = np.random.default_rng(case["mix"] + i)
        n = int(r.integers(case["nmin"] // 16, case["nmax"] // 16 + 1)) * 16
        coils = int(r.integers(case["cmin"], case["cmax"] + 1))
        shots = int(r.integers(32, 401))
        traj = "radial" if r.uniform() < 0.5 else "spiral"
        l1 = r.uniform() < 0.5
        out.append(dict(kind="recon", n0=n, n1=n, n2=0, coils=coils, traj=traj, shots=shots, read=2 * n, alpha=1.25,
                        maps="c64", y="bf16", reg="l1_wavelet" if l1 else "l2", lam=1e-3, levels=4 if l1 else 0,
                        iters=case["iters"]))
    return out


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _coords(shape):
    return torch.meshgrid(*[(torch.arange(n, device=DEV, dtype=torch.float64) - n // 2) / n for n in shape], indexing="ij")


def _phantom(shape, g):
    """Twelve random ellipses (ellipsoids) with a smooth phase, complex64."""
    pos, d = _coords(shape), len(shape)
    img = torch.zeros(shape, device=DEV, dtype=torch.float64)
    r = _rand(g, 12, 3 * d + 1).cpu()
    for row in r.tolist():
        q = torch.linalg.qr(torch.tensor(row[2 * d:3 * d], dtype=torch.float64).outer(torch.ones(d)) + torch.eye(d))[0]
        rel = [p - 0.7 * (row[k] - 0.5) for k, p in enumerate(pos)]
        rad = torch.zeros_like(img)
        for k in range(d):
            axis = sum(float(q[j, k]) * rel[j] for j in range(d))
            rad += (axis / (0.05 + 0.3 * row[d + k])) ** 2
        img += (0.1 + 0.9 * row[3 * d]) * (rad <= 1)
    return (img * torch.exp(0.2j * math.pi * sum(pos))).to(torch.complex64)


def _maps(shape, coils, g):
    """Gaussian-bump coil maps on a circle (sphere) around the field of view, sum |s_c|^2 = 1, complex64."""
    pos, d = _coords(shape), len(shape)
    out = torch.empty((coils,) + shape, device=DEV, dtype=torch.complex64)
    jit = _rand(g, coils).tolist()
    sos = torch.zeros(shape, device=DEV, dtype=torch.float64)
    for c in range(coils):
        if d == 2:
            centre = [0.6 * math.cos(2 * math.pi * c / coils), 0.6 * math.sin(2 * math.pi * c / coils)]
        else:
            z = 1 - (2 * c + 1) / coils
            rho, phi = math.sqrt(max(0.0, 1 - z * z)), c * math.pi * (3 - math.sqrt(5))
            centre = [0.6 * z, 0.6 * rho * math.sin(phi), 0.6 * rho * math.cos(phi)]
        w = 0.4 * (1 + 0.1 * (jit[c] - 0.5))
        b = torch.exp(-sum((p - q) ** 2 for p, q in zip(pos, centre)) / (2 * w * w))
        out[c] = (b * complex(math.cos(math.pi * c / coils), math.sin(math.pi * c / coils))).to(torch.complex64)
        sos += b * b
    return (out / torch.sqrt(sos).to(torch.float32)).contiguous()


def _traj(case, g):
    """Trajectory [M, D] in cycles per field of view, turned by a random angle, float32."""
    shape, S, R = _shape(case), case["shots"], case["read"]
    turn = 2 * math.pi * float(_rand(g, 1))
    s = torch.arange(S, device=DEV, dtype=torch.float64)
    j = torch.arange(R, device=DEV, dtype=torch.float64)
    if case["traj"] == "radial":
        ang = s * (math.pi * (math.sqrt(5) - 1) / 2) + turn
        r = -1 + 2 * j / R
        k = torch.stack([torch.sin(ang)[:, None] * r, torch.cos(ang)[:, None] * r], -1)
    elif case["traj"] == "spiral":
        turns = max(shape) / 2 / (3 * S)
        ph = 2 * math.pi * (turns * (j / R)[None, :] + s[:, None] / S) + turn
        k = torch.stack([(j / R) * torch.sin(ph), (j / R) * torch.cos(ph)], -1)
    else:
        z = 1 - (2 * s + 1) / S
        rho, phi = torch.sqrt(torch.clamp(1 - z * z, min=0)), s * (math.pi * (3 - math.sqrt(5))) + turn
        dirs = torch.stack([z, rho * torch.sin(phi), rho * torch.cos(phi)], -1)
        k = dirs[:, None, :] * (j / R)[None, :, None]
    half = torch.tensor([n / 2 for n in shape], device=DEV, dtype=torch.float64)
    k = (k.reshape(-1, len(shape)) * half).to(torch.float32)
    return torch.minimum(torch.maximum(k, -half.float()), half.float()).contiguous()


def _store(t, kind):
    return t.contiguous() if kind == "c64" else to_storage(t, kind)


def _stored64(t):
    """The values of a storage tensor in complex128."""
    return t.to(torch.complex128) if t.is_complex() else torch.view_as_complex(t.double().contiguous())


def _inputs(case, seed):
    """Trajectory, image, maps and measurements of one case."""
    g = _gen(seed)
    shape = _shape(case)
    d = dict(traj=_traj(case, g), x=_phantom(shape, g), maps=_store(_maps(shape, case["coils"], g), case["maps"]))
    M = d["traj"].shape[0]
    if case["kind"] in ("forward", "precond"):
        return d
    noise = torch.randn((case["coils"], M), generator=g, device=DEV, dtype=torch.complex64)
    y = Nufft(d["traj"], shape, case["alpha"]).forward(d["x"].to(torch.complex128), _stored64(d["maps"]))
    d["y"] = _store((y + 0.01 * float(y.abs().max()) * noise).to(torch.complex64), case["y"])
    if case["kind"] == "unrolled":
        d["gx"] = torch.randn(shape, generator=g, device=DEV, dtype=torch.complex64)
    return d


def _lambda(case, peak):
    """The regularisation weight: itself for l2 and unrolled, else relative to max |A^H y| (three digits)."""
    if case.get("reg", "l2") == "l2":
        return case["lam"]
    return float("%.2e" % (case["lam"] * peak))


def _plan(case, d):
    p = Plan(_shape(case), case["coils"], d["traj"].shape[0], oversamp=case["alpha"],
             wavelet_levels=case.get("levels", 0), device=DEV)
    return p.set_trajectory(d["traj"]).set_maps(d["maps"])


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        cs = _batch_cases(case)
        ds = [_inputs(c, 1009 * seed + i) for i, c in enumerate(cs)]
        plans = [_plan(c, d) for c, d in zip(cs, ds)]
        lams = [_lambda(c, float(p.sense_adjoint(d["y"]).abs().max())) for c, d, p in zip(cs, ds, plans)]
        return dict(kind=kind, plans=plans, batch=Batch(plans), ys=[d["y"] for d in ds], regs=[c["reg"] for c in cs],
                    lams=lams, iters=case["iters"])
    d = _inputs(case, seed)
    s = dict(d, kind=kind, case=case, plan=_plan(case, d))
    if kind in ("recon", "frame"):
        s["lam"] = _lambda(case, float(s["plan"].sense_adjoint(d["y"]).abs().max()))
    if kind in ("frame", "unrolled"):
        s["p"] = s["plan"].make_preconditioner()
        s["lmax"] = s["plan"].max_eig(s["p"])
    if kind == "unrolled":
        s["lam"] = torch.tensor(case["lam"], device=DEV, requires_grad=True)
        s["y"].requires_grad_(True)
        s["traj"].requires_grad_(True)
    return s


def run(s):
    kind = s["kind"]
    if kind == "forward":
        return s["plan"].sense_forward(s["x"])
    if kind == "adjoint":
        return s["plan"].sense_adjoint(s["y"])
    if kind == "precond":
        return s["plan"].make_preconditioner()
    if kind == "recon":
        s["plan"].set_trajectory(s["traj"]).set_maps(s["maps"])
        return s["plan"].pdhg_solve(s["y"], None, s["case"]["reg"], s["lam"], s["case"]["iters"])[0]
    if kind == "frame":
        return s["plan"].pdhg_solve(s["y"], s["p"], s["case"]["reg"], s["lam"], s["case"]["iters"], lmax=s["lmax"])[0]
    if kind == "batch":
        return s["batch"].solve(s["ys"], None, s["regs"], s["lams"], s["iters"])
    x = autograd.unrolled_pdhg(s["y"], s["lam"], s["traj"], s["plan"], s["p"], s["case"]["iters"], s["lmax"])
    gy, gl, gt = torch.autograd.grad(x, [s["y"], s["lam"], s["traj"]], grad_outputs=s["gx"])
    return dict(x=x.detach(), gy=gy, glam=gl, gtraj=gt)


# ------------------------------------------------------------------ work
def _grid(shape, alpha):
    out = []
    for n in shape:
        g = int(math.ceil(alpha * n - 1e-9))
        out.append(g + g % 2)
    return tuple(out)


def work(case):
    """Bytes and operations: every input read once and every output written once; an iterative
    solve does so in each iteration with the operands of A and A^H and of the two updates (maps,
    coordinates, measurements, p, and the iterates)."""
    if case["kind"] == "batch":
        ws = [work(c) for c in _batch_cases(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    shape, C = _shape(case), case["coils"]
    D, N, M = len(shape), math.prod(shape), case["shots"] * case["read"]
    g = _grid(shape, case["alpha"])
    G = math.prod(g)
    mb, yb = (8 if case[k] == "c64" else 4 for k in ("maps", "y"))
    op_b = 8 * N + mb * C * N + 4 * D * M + yb * C * M
    op_f = 8 * C * N + 5 * C * G * math.log2(G) + 4 * C * M * W ** D
    kind, it = case["kind"], case.get("iters", 0)
    nb = 2 ** D * N
    pre_b = mb * C * N + 4 * D * M + 4 * C * M
    pre_f = C * (C + 1) // 2 * (5 * nb * math.log2(nb) + 6 * N + 3 * nb) + 2 * C * M * W ** D
    if kind in ("forward", "adjoint"):
        return {"bytes": op_b, "flops": op_f}
    if kind == "precond":
        return {"bytes": pre_b, "flops": pre_f}
    it_b = 2 * mb * C * N + 8 * D * M + (yb + 4 + 16) * C * M + 32 * N
    it_f = 2 * op_f + 12 * C * M + 20 * N
    if kind == "unrolled":       # the reverse sweep: A, A^H, two trajectory gradients per iteration
        return {"bytes": it * (3 * it_b + 16 * D * M), "flops": it * (4 * it_f + 16 * D * C * M * W ** D)}
    b, f = it * it_b, it * it_f
    if kind == "recon":
        b += pre_b + POWER_ITERS * 2 * op_b
        f += pre_f + POWER_ITERS * 2 * op_f
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the method in 64 bits
class Nufft:
    """A and A^H as the method defines them (Kaiser-Bessel, width 4), complex128; scale = 2 gives the
    preconditioner's operator on the 2N image."""

    def __init__(self, traj, shape, alpha, scale=1):
        self.shape, self.g = shape, _grid(shape, alpha)
        self.N, self.G = math.prod(shape), math.prod(self.g)
        self.k0, self.w, ap = [], [], []
        for d, (n, g) in enumerate(zip(shape, self.g)):
            a = g / n
            beta = math.pi * math.sqrt((W / a) ** 2 * (a - 0.5) ** 2 - 0.8)
            t = traj[:, d].double() * scale * g / n
            k0 = torch.ceil(t.detach()) - W // 2
            self.k0.append(k0.long())
            u = [t - (k0 + j) for j in range(W)]
            self.w.append([torch.special.i0(beta * torch.sqrt(1 - (v / 2) ** 2 + 1e-30)) for v in u])
            z = beta * beta - (math.pi * W * (torch.arange(n, device=DEV, dtype=torch.float64) - n // 2) / g) ** 2
            r = torch.sqrt(z.abs())
            ap.append(W * torch.where(z > 0, torch.sinh(r) / r, torch.sin(r) / r))
        self.apod = functools.reduce(lambda x, y: x[..., None] * y, ap)
        self.pad = [(torch.arange(n, device=DEV) - n // 2) % g for n, g in zip(shape, self.g)]

    def _taps(self):
        for q in range(W ** len(self.g)):
            j = [q // W ** d % W for d in range(len(self.g))]
            f, w = 0, 1.0
            for d, g in enumerate(self.g):
                f = f * g + (self.k0[d] + j[d]) % g
                w = w * self.w[d][j[d]]
            yield f, w

    def _crop(self, grid):
        for d, p in enumerate(self.pad):
            grid = grid.index_select(d + 1, p)
        return grid

    def forward(self, x, maps):
        v = maps * (x / self.apod)
        for d, (p, g) in enumerate(zip(self.pad, self.g)):   # zero padding, axis by axis
            shp = list(v.shape)
            shp[d + 1] = g
            v = torch.zeros(shp, device=DEV, dtype=torch.complex128).index_copy(d + 1, p, v)
        # grid points outermost: one row of coils per tap
        v = torch.fft.fftn(v, dim=tuple(range(1, len(self.g) + 1))).reshape(maps.shape[0], -1).T.contiguous()
        y = 0
        for f, w in self._taps():
            y = y + w[:, None] * v[f]
        return (y / math.sqrt(self.N)).T.contiguous()

    def adjoint(self, y, maps):
        grid = torch.zeros((self.G, maps.shape[0], 2), device=DEV, dtype=torch.float64)
        yr = torch.view_as_real(y.T.contiguous())
        for f, w in self._taps():
            grid = grid.index_add(0, f, w[:, None, None] * yr)
        grid = torch.view_as_complex(grid).T.reshape((maps.shape[0],) + self.g)
        img = self._crop(torch.fft.ifftn(grid, dim=tuple(range(1, len(self.g) + 1))) * self.G)
        return (maps.conj() * img).sum(0) / self.apod / math.sqrt(self.N)


def _precond64(traj, maps, alpha):
    """Multi-channel preconditioner by the fast route (pair products on the 2N grid)."""
    shape = tuple(maps.shape[1:])
    C, N, big = maps.shape[0], math.prod(shape), tuple(2 * n for n in shape)
    dims = tuple(range(len(shape)))
    idx = torch.meshgrid(*[(torch.arange(n, device=DEV) - n // 2) % (2 * n) for n in shape], indexing="ij")
    op = Nufft(traj, big, alpha, scale=2)
    one = torch.ones((1,) + big, device=DEV, dtype=torch.complex128)
    h = op.adjoint(torch.ones((1, traj.shape[0]), device=DEV, dtype=torch.complex128), one) * math.sqrt(2 ** len(shape))
    R = [torch.zeros(big, device=DEV, dtype=torch.float64) for _ in range(C)]
    for c in range(C):
        for e in range(c, C):
            q = torch.zeros(big, device=DEV, dtype=torch.complex128)
            q[idx] = maps[c] * maps[e].conj()
            a = torch.view_as_real(torch.fft.fftn(q)).square().sum(-1)
            R[c] += a
            if e != c:
                R[e] += torch.roll(torch.flip(a, dims), [1] * len(dims), dims)
    p = []
    for c in range(C):
        r = torch.fft.fftshift(torch.fft.ifftn(R[c].to(torch.complex128)))
        s = op.forward(r * h, one)[0] * math.sqrt(math.prod(big))
        p.append(maps[c].abs().square().sum() * math.sqrt(N) / s.real)
    return torch.stack(p)


def _lmax64(A, AH, p, shape):
    v = torch.ones(shape, device=DEV, dtype=torch.complex128)
    v = v / v.norm()
    for _ in range(POWER_ITERS):
        w = AH(p * A(v))
        L = float(w.norm())
        v = w / L
    return L


@functools.lru_cache(None)
def _db4():
    """The 8-tap extremal-phase Daubechies filter by spectral factorisation."""
    poly = np.ones(1)
    for y in np.roots([20.0, 10.0, 4.0, 1.0]):
        b = 2 - 4 * y
        z = (b + np.sqrt(b * b - 4 + 0j)) / 2
        poly = np.convolve(poly, [1, -(z if abs(z) < 1 else 1 / z)])
    for _ in range(4):
        poly = np.convolve(poly, [1, 1])
    h = np.real(poly) * math.sqrt(2) / np.real(poly).sum()
    return h.tolist(), [(-1) ** n * h[7 - n] for n in range(8)]


def _dwt_axis(x, d):
    h, g = _db4()
    even = lambda v: v.unflatten(d, (v.shape[d] // 2, 2)).select(d + 1, 0)  # noqa: E731
    sh = [even(torch.roll(x, -n, d)) for n in range(8)]
    return torch.cat([sum(a * v for a, v in zip(f, sh)) for f in (h, g)], d)


def _idwt_axis(c, d):
    h, g = _db4()
    a, b = c.chunk(2, d)
    up = lambda v: torch.stack([v, torch.zeros_like(v)], d + 1).flatten(d, d + 1)  # noqa: E731
    a, b = up(a), up(b)
    return sum(torch.roll(h[n] * a + g[n] * b, n, d) for n in range(8))


def _wprox(z, t, levels):
    c = z.clone()
    blocks = [tuple(slice(0, n >> lev) for n in z.shape) for lev in range(levels)]
    for b in blocks:
        v = c[b]
        for d in range(z.dim()):
            v = _dwt_axis(v, d)
        c[b] = v
    m = c.abs()
    c = torch.where(m > t, c * (1 - t / torch.clamp(m, min=1e-300)), torch.zeros_like(c))
    for b in reversed(blocks):
        v = c[b]
        for d in reversed(range(z.dim())):
            v = _idwt_axis(v, d)
        c[b] = v
    return c


def _pdhg64(A, AH, y, p, L, shape, reg, lam, iters, levels=0):
    x = torch.zeros(shape, device=DEV, dtype=torch.complex128)
    xbar, u = x, torch.zeros_like(y)
    pmin = float(p.min())
    if reg == "tv":
        D = len(shape)
        tau, v = 1.0 / (L + 4 * D), [torch.zeros_like(x) for _ in range(D)]
        for _ in range(iters):
            u = (u + p * (A(xbar) - y)) / (1 + p)
            v = [a + torch.roll(xbar, -1, d) - xbar for d, a in enumerate(v)]
            v = [a * torch.clamp(lam / torch.clamp(a.abs(), min=1e-300), max=1) for a in v]
            new = x - tau * (AH(u) + sum(torch.roll(a, 1, d) - a for d, a in enumerate(v)))
            x, xbar = new, 2 * new - x
        return x
    sig, tau = 1.0, 1.0 / L
    for _ in range(iters):
        theta = 1 / (1 + 2 * sig * pmin)
        u = (u + sig * p * (A(xbar) - y)) / (1 + sig * p)
        z = x - tau * AH(u)
        new = z / (1 + tau * lam) if reg == "l2" else _wprox(z, tau * lam, levels)
        x, xbar = new, new + theta * (new - x)
        sig, tau = theta * sig, tau / theta
    return x


def _recon64(case, d):
    traj, maps, y, shape = d["traj"], _stored64(d["maps"]), _stored64(d["y"].detach()), _shape(case)
    op = Nufft(traj, shape, case["alpha"])
    A, AH = (lambda v: op.forward(v, maps)), (lambda v: op.adjoint(v, maps))
    lam = _lambda(case, float(AH(y).abs().max()))
    p = _precond64(traj, maps, case["alpha"])
    return _pdhg64(A, AH, y, p, _lmax64(A, AH, p, shape), shape, case["reg"], lam, case["iters"], case["levels"])


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_recon64(c, _inputs(c, 1009 * seed + i)) for i, c in enumerate(_batch_cases(case))]
    M = case["shots"] * case["read"]
    if len(_shape(case)) == 3 and kind == "recon" and (POWER_ITERS + case["iters"]) * M * case["coils"] > 2e8:
        return None          # minutes in 64 bits
    d = _inputs(case, seed)
    if kind in ("recon", "frame"):
        return _recon64(case, d)
    maps = _stored64(d["maps"])
    if kind == "precond":
        return _precond64(d["traj"], maps, case["alpha"])
    if kind in ("forward", "adjoint"):
        op = Nufft(d["traj"], _shape(case), case["alpha"])
        return op.forward(d["x"].to(torch.complex128), maps) if kind == "forward" else op.adjoint(_stored64(d["y"]), maps)
    # unrolled: p, lambda_max and the step sizes are constants
    shape, y = _shape(case), d["y"].to(torch.complex128).requires_grad_(True)
    op = Nufft(d["traj"], shape, case["alpha"])
    A, AH = (lambda v: op.forward(v, maps)), (lambda v: op.adjoint(v, maps))
    p = _precond64(d["traj"], maps, case["alpha"])
    L = _lmax64(A, AH, p, shape)
    traj = d["traj"].double().requires_grad_(True)
    lam = torch.tensor(case["lam"], device=DEV, dtype=torch.float64, requires_grad=True)
    op = Nufft(traj, shape, case["alpha"])
    x = _pdhg64(lambda v: op.forward(v, maps), lambda v: op.adjoint(v, maps), y, p, L, shape, "l2", lam, case["iters"])
    gy, gl, gt = torch.autograd.grad(x, [y, lam, traj], grad_outputs=d["gx"].to(torch.complex128))
    return dict(x=x.detach(), gy=gy, glam=gl, gtraj=gt)
