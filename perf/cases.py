"""Performance cases of the solver and of the learned start, through the Python binding.

A case is a dict of plain values; ``kind`` selects the calls it makes:

``solve``      a solver whose phases and reference medium are set; a pass is one ``Solver.solve`` of
               unit strains from E = 0 and the read-out of the strain fields.  ``iters`` > 0 runs that
               many iterations (tol = 0), ``iters`` = 0 solves to ``tol``.  ``reference`` includes the
               table build (``set_reference``) in the pass, as a parameter sweep over materials does.
``batch``      ``solve_batch`` over seeded 2-D microstructures of uneven sizes, strain fields read out.
``infer``      the learned start's network on one or more microstructures: input channels, forward.
``train``      a training step of that network: gradients of ``acc`` accumulated batches, read out as
               a checkpoint does, and the Adam update.

Single-precision solves hand back single-precision numbers (fields and averages); double-precision
solves double-precision ones.  ``exact`` evaluates the same equations in 64 bits with torch.fft on the
natural grid of M; it shares nothing with the package.  Where the package stores the points in an order
of its own (a sheared M) only the averages have a value there.
"""
import math

import numpy as np
import torch

import paper_1701_04685_gb300 as fh

NU = 0.3
PREC = {"fp64": fh.FH_PREC_FP64, "fp32": fh.FH_PREC_FP32, "mixed": fh.FH_PREC_MIXED}


def listed():
    return [
        # a small 2-D unit cell in double precision: the smallest call a user makes, bound by latency
        dict(name="disk32_fp64", kind="solve", d=2, n=32, shear=0, nz=0, gen="dirichlet", field="balls", contrast=10.0,
             count=1, prec="fp64", loads=3, iters=40, tol=0.0, method=0, form=0, reference=False),
        # the anisotropic 2-D pattern of the benchmark in single precision
        dict(name="sheared128_fp32", kind="solve", d=2, n=128, shear=32, nz=0, gen="dlvp", field="balls", contrast=100.0,
             count=20, prec="fp32", loads=3, iters=100, tol=0.0, method=0, form=0, reference=False),
        # a graded 2-D material, every point its own stiffness (whole-GPU passes)
        dict(name="graded512_fp32", kind="solve", d=2, n=512, shear=0, nz=0, gen="dlvp", field="graded", contrast=20.0,
             count=0, prec="fp32", loads=3, iters=40, tol=0.0, method=0, form=0, reference=False),
        # a parameter study: many 2-D microstructures of uneven sizes, all loads, to the tolerance
        dict(name="batch64_mixed", kind="batch", items=64, tol=1e-6),
        # the learned start's volume in single precision, where the fields stay in the L2 cache
        dict(name="volume64_fp32", kind="solve", d=3, n=64, shear=0, nz=0, gen="dirichlet", field="balls", contrast=40.0,
             count=40, prec="fp32", loads=6, iters=40, tol=0.0, method=0, form=0, reference=False),
        # a volume from a voxel image of a hundred points a side: no power of two
        dict(name="volume100_fp32", kind="solve", d=3, n=100, shear=0, nz=0, gen="dirichlet", field="balls", contrast=30.0,
             count=40, prec="fp32", loads=6, iters=20, tol=0.0, method=0, form=0, reference=False),
        # the whole call of the benchmark: table, solve of all six loads to 1e-6, effective stiffness, fields
        dict(name="volume128_mixed", kind="solve", d=3, n=128, shear=0, nz=0, gen="box4", field="balls", contrast=50.0,
             count=50, prec="mixed", loads=6, iters=0, tol=1e-6, method=0, form=0, reference=True),
        # the same volume in double precision throughout
        dict(name="volume128_fp64", kind="solve", d=3, n=128, shear=0, nz=0, gen="box4", field="balls", contrast=50.0,
             count=50, prec="fp64", loads=6, iters=8, tol=0.0, method=0, form=0, reference=False),
        # BiCGStab in mixed precision, which produces the network's training fields
        dict(name="krylov64_mixed", kind="solve", d=3, n=64, shear=0, nz=0, gen="dirichlet", field="balls", contrast=20.0,
             count=40, prec="mixed", loads=6, iters=36, tol=0.0, method=1, form=0, reference=False),
        # anisotropic phases with an anisotropic reference medium: the general table and the full stress product
        dict(name="ortho64_reference", kind="solve", d=3, n=64, shear=0, nz=0, gen="box4", field="ortho", contrast=8.0,
             count=20, prec="fp64", loads=6, iters=4, tol=0.0, method=0, form=0, reference=True),
        # the learned start of one microstructure (36 output channels: six unit loads at once)
        dict(name="infer64", kind="infer", n=64, width=32, modes=12, layers=4, batch=1),
        # a training step of the same network
        dict(name="train64", kind="train", n=64, width=32, modes=12, layers=4, batch=4, acc=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plane", "plane", "graded", "volume", "volume", "volume", "krylov", "ortho", "batch", "infer", "train"])
    if kind == "batch":
        return dict(kind="batch", items=rng.randint(3, 63), tol=1e-6)
    if kind in ("infer", "train"):
        n = rng.choice([16, 20, 24, 30, 32, 40, 48, 50, 60, 64])
        c = dict(kind=kind, n=n, width=rng.choice([8, 12, 16, 24, 32, 48 if n <= 48 else 32]), modes=rng.randint(2, min(12, n // 2)),
                 layers=rng.randint(2, 4), batch=rng.randint(1, 3 if kind == "infer" else 4))
        if kind == "train":
            c["acc"] = rng.randint(1, 3)
        return c
    c = dict(kind="solve", d=3, n=0, shear=0, nz=0, gen=rng.choice(["dirichlet", "dlvp", "box2"]), field="balls",
             contrast=round(math.exp(rng.uniform(math.log(5.0), math.log(60.0))), 2), count=rng.randint(5, 40),
             prec=rng.choice(["fp32", "fp32", "fp64", "mixed"]), loads=rng.randint(1, 6), iters=rng.randint(5, 40), tol=0.0, method=0,
             form=0, reference=False)
    if kind == "plane":
        n = _log_int(rng, 24, 400)
        c.update(d=2, n=n, shear=rng.choice([0, 1, n // 8, n // 4, n // 3]), loads=rng.randint(1, 3), iters=rng.randint(20, 45))
        if c["gen"] == "dirichlet" and rng.random() < 0.2:
            c["form"] = 1
    elif kind == "graded":
        c.update(d=2, n=_log_int(rng, 40, 600), field="graded", loads=rng.randint(1, 3), prec=rng.choice(["fp32", "fp64"]))
    elif kind == "volume":
        n = _log_int(rng, 12, 128)
        c.update(n=n, nz=2 * n if n <= 64 and rng.random() < 0.3 else 0, reference=rng.random() < 0.3)
        most = (2e7 if c["prec"] == "fp32" else 5e6) / (n * n * (c["nz"] or n))
        c["iters"] = max(3, min(c["iters"], int(most)))
    elif kind == "krylov":
        c.update(n=_log_int(rng, 20, 72), prec="mixed", contrast=round(rng.uniform(5.0, 30.0), 2), iters=36, method=1)
    else:
        c.update(n=_log_int(rng, 16, 64), field="ortho", contrast=round(rng.uniform(2.0, 12.0), 2), gen=rng.choice(["dlvp", "box2", "box4"]),
                 prec="fp64", iters=rng.randint(2, 6), reference=True)
    return c


# ---------------------------------------------------------------- inputs
def _matrix(c):
    if c["d"] == 2:
        return [[c["n"], c["shear"]], [0, c["n"]]]
    return [[c["n"], 0, 0], [0, c["n"], 0], [0, 0, c["nz"] or c["n"]]]


def _generator(c):
    """(kind, half ramp widths, box-spline order, alias radius)"""
    return {"dirichlet": ("dirichlet", 0.0, 0, 1), "dlvp": ("dlvp", 0.25, 0, 1), "box2": ("box", 0.0, 2, 2), "box4": ("box", 0.0, 2, 4)}[c["gen"]]


def _fh_generator(c):
    kind, alpha, order, radius = _generator(c)
    if kind == "box":
        return fh.tensor_boxspline(c["d"], order, radius)
    return fh.generator(kind, alpha=[alpha] * c["d"])


def _balls(rng, d, count):
    """Non-overlapping periodic balls, as many of `count` as find a place."""
    lo, hi = (0.03, 0.08) if d == 2 else (0.05, 0.1)
    if count == 1:
        return np.array([rng.uniform(-0.5, 0.5, d)]), np.array([0.25])
    cs, rs = [], []
    for _ in range(2000):
        if len(cs) == count:
            break
        x, r = rng.uniform(-0.5, 0.5, d), rng.uniform(lo, hi)
        if all(np.linalg.norm((x - y + 0.5) % 1.0 - 0.5) > r + q for y, q in zip(cs, rs)):
            cs.append(x)
            rs.append(r)
    return np.array(cs), np.array(rs)


def _phase(y, centres, radii):
    """uint8 phase of the points y (m, d), a CUDA float64 tensor."""
    ph = torch.zeros(y.shape[0], dtype=torch.uint8, device=y.device)
    for x, r in zip(centres, radii):
        t = y - torch.tensor(x, device=y.device)
        t -= torch.round(t)
        ph[(t * t).sum(1) < r * r] = 1
    return ph


def _axis_points(n):
    t = np.arange(n, dtype=np.float64) / n
    return np.where(t >= 0.5, t - 1.0, t)


def _natural_points(c):
    """Points M^-1 n of the natural grid (row-major n), in [-1/2, 1/2)."""
    if c["d"] == 2:
        n, s = c["n"], c["shear"]
        n1, n2 = np.meshgrid(np.arange(n, dtype=np.int64), np.arange(n, dtype=np.int64), indexing="ij")
        num = np.stack([n1 * n - s * n2, n2 * n], -1).reshape(-1, 2)
        num = num % (n * n)
        num = np.where(2 * num >= n * n, num - n * n, num)
        return torch.from_numpy(num / float(n * n)).cuda()
    ax = [torch.from_numpy(_axis_points(k)).cuda() for k in (c["n"], c["n"], c["nz"] or c["n"])]
    return torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)


def _identity_order(c):
    return c["d"] == 3 or c["shear"] == 0


def _material(c, rng):
    """Phase matrices (nphase, nv, nv) and C0 (None: the solver's rule), or for a graded field None."""
    d = c["d"]
    if c["field"] == "balls":
        return np.stack([_iso(1.0, NU, d), _iso(c["contrast"], NU, d)]), None
    soft, hard = _iso(1.0, NU, 3), np.zeros((6, 6))
    a = rng.uniform(0.6, 1.0, 3) * c["contrast"]
    hard[:3, :3] = 0.3 * c["contrast"] + np.diag(a)
    hard[3:, 3:] = np.diag(rng.uniform(0.4, 0.9, 3) * c["contrast"])
    return np.stack([soft, hard]), 0.5 * (soft + hard)


def _iso(E, nu, d):
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    nv = 3 if d == 2 else 6
    m = np.zeros((nv, nv))
    m[:d, :d] = lam
    m[np.arange(nv), np.arange(nv)] = 2 * mu
    m[np.arange(d), np.arange(d)] = lam + 2 * mu
    return m


def _graded(y, contrast, rng):
    """(m, 3, 3) stiffness of a continuously varying isotropic plane material."""
    k = rng.integers(1, 4, 2)
    t = 0.5 * (1 + torch.sin(2 * math.pi * (k[0] * y[:, 0] + k[1] * y[:, 1] + rng.uniform())))
    E = 1.0 + (contrast - 1.0) * t
    nu = 0.2 + 0.15 * (0.5 + 0.5 * torch.cos(2 * math.pi * (y[:, 0] - y[:, 1]) + rng.uniform()))
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    C = torch.zeros(y.shape[0], 3, 3, dtype=torch.float64, device=y.device)
    C[:, :2, :2] = lam[:, None, None]
    C[:, 0, 0] += 2 * mu
    C[:, 1, 1] += 2 * mu
    C[:, 2, 2] = 2 * mu
    return C


def _batch_item(rng, sizes):
    """One microstructure; its pattern comes from `sizes` (the same for every seed), the rest from `rng`."""
    N = int(sizes.choice([64, 96, 128, 192, 256]))
    s = 0 if sizes.random() < 0.5 else N // int(sizes.choice([8, 4, 2]))
    return dict(d=2, n=N, shear=s, nz=0, gen="dirichlet", field="balls", count=int(rng.integers(5, 31)),
                contrast=float(math.exp(rng.uniform(math.log(5.0), math.log(200.0)))))


def _solver(c, rng, loads, patterns=None):
    key = str(_matrix(c))
    p = patterns.get(key) if patterns is not None else None
    if p is None:
        p = fh.Pattern(_matrix(c))
        if patterns is not None:
            patterns[key] = p
    y = _natural_points(c) if _identity_order(c) else torch.from_numpy(p.points()).cuda()
    s = fh.Solver(p, _fh_generator(c), loads)
    if c["field"] == "graded":
        s.set_stiffness_field(_graded(y, c["contrast"], rng).contiguous())
        C0 = None
    else:
        ph = _phase(y, *_balls(rng, c["d"], c["count"]))
        Cp, C0 = _material(c, rng)
        s.set_stiffness_phases(ph, Cp)
    s.set_reference(C0)
    return s, C0


def _net_params(c, seed):
    """Weights of a network that starts its training, and the seeded source of its inputs."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    W, L, nm = c["width"], c["layers"], 4 * c["modes"] ** 3

    def n(k, s):
        return torch.randn(k, generator=gen, device="cuda") * s
    parts = [n(W, 1.0), n(W, 0.1), n(L * W * W, W ** -0.5), n(L * W, 0.1), n(L * nm * W * W, 1.0 / W), n(L * nm * W * W, 1.0 / W),
             n(36 * W, 0.1 * W ** -0.5), n(36, 0.01)]
    return torch.cat(parts), gen


def _two_phase(gen, n, vf):
    """A two-phase n^3 map of blobs with volume fraction about vf (uint8)."""
    z = torch.randn(n, n, n, generator=gen, device="cuda")
    k = torch.fft.fftfreq(n, device="cuda") * n
    w = torch.exp(-(k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2) / 18.0)
    z = torch.fft.ifftn(torch.fft.fftn(z) * w).real
    z = z / z.std()
    t = torch.tensor(vf, device="cuda")
    return (z > math.sqrt(2) * torch.erfinv(1 - 2 * t)).to(torch.uint8).reshape(-1)


def _net_inputs(c, gen, rng, count):
    """`count` phase maps with their contrasts."""
    return ([_two_phase(gen, c["n"], float(rng.uniform(0.1, 0.35))) for _ in range(count)],
            [float(rng.uniform(10.0, 100.0)) for _ in range(count)])


def _targets(maps, gen):
    """Strain-like fields: each channel follows the map, with a rough part."""
    B, m = len(maps), maps[0].numel()
    a = torch.randn(B, 36, 1, generator=gen, device="cuda")
    f = torch.stack(maps).float()[:, None, :]
    return (a * (f - f.mean(2, keepdim=True)) + 0.2 * torch.randn(B, 36, m, generator=gen, device="cuda")).contiguous()


def prepare(case, seed):
    c, rng = case, np.random.default_rng(seed)
    if c["kind"] == "solve":
        s, C0 = _solver(c, rng, c["loads"])
        dt = torch.float64 if c["prec"] == "fp64" else torch.float32
        return dict(c=c, s=s, C0=C0, eps0=np.eye(s.nv)[: c["loads"]], E=torch.empty(c["loads"], s.nv, s.m, dtype=dt, device="cuda"))
    if c["kind"] == "batch":
        pats, sizes = {}, np.random.default_rng(c["items"])
        ss = [_solver(_batch_item(rng, sizes), rng, 3, pats)[0] for _ in range(c["items"])]
        return dict(c=c, ss=ss, eps0=[np.eye(3)] * len(ss), E=torch.empty(9 * sum(s.m for s in ss), dtype=torch.float32, device="cuda"))
    flat, gen = _net_params(c, seed)
    net = fh.FNO(c["n"], 1, 36, c["width"], c["modes"], c["layers"], max_batch=c["batch"])
    net.set_params(flat.cpu().numpy())
    m = c["n"] ** 3
    if c["kind"] == "infer":
        maps, E = _net_inputs(c, gen, rng, c["batch"])
        return dict(c=c, net=net, maps=maps, logE=[[0.0, math.log10(e)] for e in E], e0=np.zeros(6),
                    x=torch.empty(c["batch"], 1, m, device="cuda"), y=torch.empty(c["batch"], 36, m, device="cuda"))
    sets = []
    for _ in range(c["acc"]):
        maps, E = _net_inputs(c, gen, rng, c["batch"])
        x = torch.empty(c["batch"], 1, m, device="cuda")
        for b in range(c["batch"]):
            net.make_input(maps[b], [0.0, math.log10(E[b])], np.zeros(6), x[b])
        sets.append((x, _targets(maps, gen)))
    return dict(c=c, net=net, sets=sets, step=0)


# ---------------------------------------------------------------- one pass
def run(state):
    c = state["c"]
    if c["kind"] == "solve":
        s, E = state["s"], state["E"]
        if c["reference"]:
            s.set_reference(state["C0"])
        r = s.solve(state["eps0"], tol=c["tol"], max_iter=c["iters"] or 20000, precision=PREC[c["prec"]], form=c["form"], method=c["method"])
        for k in range(c["loads"]):
            if c["prec"] == "fp64":
                s.get_strain(k, E[k])
            else:
                fh.get_strain_f32(s, k, E[k])
        out = {"strain": E, "mean_stress": r["mean_stress"]}
        if c["loads"] == s.nv:
            out["ceff"] = s.get_ceff()
        if c["prec"] != "fp64":
            return {k: v if k == "strain" else v.astype(np.float32) for k, v in out.items()}
        return out
    if c["kind"] == "batch":
        _, rs = fh.solve_batch(state["ss"], state["eps0"], tol=c["tol"])
        o = 0
        for s in state["ss"]:
            for k in range(3):
                fh.get_strain_f32(s, k, state["E"][o:o + 3 * s.m])
                o += 3 * s.m
        return {"strain": state["E"], "mean_stress": np.stack([r["mean_stress"] for r in rs]).astype(np.float32),
                "ceff": np.stack([s.get_ceff() for s in state["ss"]]).astype(np.float32)}
    net = state["net"]
    if c["kind"] == "infer":
        for b in range(c["batch"]):
            net.make_input(state["maps"][b], state["logE"][b], state["e0"], state["x"][b])
        return {"y": net.forward(state["x"], state["y"])}
    state["step"] += 1
    net.zero_grad()
    loss = [net.loss_grad(x, t) for x, t in state["sets"]]
    g = net.get_grads()
    net.adam_step(2e-3, state["step"])
    return {"loss": np.array(loss, dtype=np.float32), "grads": g}


# ---------------------------------------------------------------- work
def _points(c):
    return c["n"] ** 2 if c["d"] == 2 else c["n"] ** 2 * (c["nz"] or c["n"])


def _solve_flops(nv, m, loads, iters):
    # per point, load and iteration: FFTs of n_v real fields both ways, the stress and Green products, update and residual
    return float(iters) * loads * m * (5 * nv * math.log2(max(2, m)) + 4 * nv * nv + 6 * nv)


def _net_flops(c):
    # lift and projection, and per layer the 1 x 1 layer, FFTs of every channel both ways and the mode mixing
    N3, W = c["n"] ** 3, c["width"]
    layer = 2.0 * W * W * N3 + 5.0 * W * N3 * math.log2(N3) + 8.0 * W * W * 4 * c["modes"] ** 3
    return 2.0 * 37 * W * N3 + c["layers"] * layer


def work(case):
    c = case
    if c["kind"] == "solve":
        m, nv = _points(c), 3 if c["d"] == 2 else 6
        b = 8 if c["prec"] == "fp64" else 4
        mat = nv * (nv + 1) // 2 * b * m if c["field"] == "graded" else m
        its = c["iters"] or 168
        f = _solve_flops(nv, m, c["loads"], its * (2 if c["method"] else 1))
        return {"bytes": mat + nv * (nv + 1) // 2 * b * m / 2.0 + c["loads"] * nv * m * b, "flops": f}
    if c["kind"] == "batch":
        m = c["items"] * 27400.0   # the mean of the sizes
        return {"bytes": m + 6 * 4 * m / 2 + 9 * 4 * m, "flops": _solve_flops(3, 27400, 3, 220) * c["items"]}
    N3, W = c["n"] ** 3, c["width"]
    prm = c["layers"] * 8 * c["modes"] ** 3 * W * W
    if c["kind"] == "infer":
        return {"bytes": c["batch"] * 37 * 4 * N3 + 2 * prm, "flops": c["batch"] * _net_flops(c)}
    n = c["batch"] * c["acc"]
    # forward with its 16-bit weights, gradients written, and the update's weights and two moments read and written
    return {"bytes": n * 37 * 4 * N3 + (2 + 4 + 4 + 24) * prm, "flops": 3.0 * n * _net_flops(c)}


# ---------------------------------------------------------------- the same in 64 bits
PAIRS = {2: ([0, 1, 0], [0, 1, 1]), 3: ([0, 1, 2, 1, 0, 0], [0, 1, 2, 2, 2, 1])}


class _Grid:
    """DFT over P(M) on the natural grid n = (n1, n2[, n3]): for M = [[a, s], [0, a]] an FFT along n1, a
    phase factor exp(2 pi i h1 s n2 / a^2), an FFT along n2; for a diagonal M an ordinary real FFT."""

    def __init__(self, c):
        self.c, self.d = c, c["d"]
        self.nv = 3 if self.d == 2 else 6
        n = c["n"]
        self.shape = (n, n) if self.d == 2 else (n, n, c["nz"] or n)
        self.m = int(np.prod(self.shape))
        self.real = self.d == 3
        ar = [torch.arange(k, device="cuda", dtype=torch.int64) for k in self.shape]
        if self.real:
            ar[-1] = ar[-1][: self.shape[-1] // 2 + 1]
        self.h = list(torch.meshgrid(*ar, indexing="ij"))
        if self.d == 2:
            h1, n2 = torch.meshgrid(ar[0], ar[1], indexing="ij")
            ang = 2 * math.pi * ((h1 * c["shear"] * n2) % (n * n)).double() / (n * n)
            self.tw = torch.complex(torch.cos(ang), torch.sin(ang))

    def fwd(self, x):
        if self.real:
            return torch.fft.rfftn(x, dim=(-3, -2, -1))
        return torch.fft.fft(torch.fft.fft(x + 0j, dim=-2) * self.tw, dim=-1)

    def inv(self, X):
        if self.real:
            return torch.fft.irfftn(X, s=self.shape, dim=(-3, -2, -1))
        return torch.fft.ifft(torch.fft.ifft(X, dim=-1) * self.tw.conj(), dim=-2).real

    def frequencies(self):
        """h reduced to G(M^T) and the numerators of u = M^-T h over the common denominator D."""
        if self.d == 2:
            n, s = self.c["n"], self.c["shear"]
            D, Mt = n * n, [[n, 0], [s, n]]
            u = [self.h[0] * n, self.h[1] * n - s * self.h[0]]
        else:
            D = self.shape[2]
            Mt = [[self.shape[i] if i == j else 0 for j in range(3)] for i in range(3)]
            u = [h * (D // k) for h, k in zip(self.h, self.shape)]
        z = [torch.div(2 * v + D, 2 * D, rounding_mode="floor") for v in u]
        h = [self.h[i] - sum(Mt[i][j] * z[j] for j in range(self.d)) for i in range(self.d)]
        return h, [v - D * w for v, w in zip(u, z)], D, Mt

    def table(self, C0):
        """Gamma^p, (nv, nv, *frequencies): the alias sum of Gamma^0 with the orthonormalised weights."""
        kind, alpha, order, R = _generator(self.c)
        d, nv = self.d, self.nv
        h, un, D, Mt = self.frequencies()
        zs = list(range(-R, R + 2))

        def symbol(v):
            two = 2 * v.abs()
            if kind == "dirichlet":
                g = (two < D).double() + 0.5 * (two == D).double()
            elif kind == "dlvp":
                g = ((0.5 + alpha - v.abs().double() / D) / (2 * alpha)).clamp(0.0, 1.0)
            else:
                g = torch.special.sinc(v.double() / D) ** order
                g = torch.where((v != 0) & (v % D == 0), torch.zeros_like(g), g)
            return torch.where(two > (2 * R + 1) * D, torch.zeros_like(g), g * g)

        w = [[symbol(un[i] + D * z) for z in zs] for i in range(d)]
        total = [sum(x) for x in w]
        I, J = PAIRS[d]
        C0 = np.asarray(C0, dtype=np.float64)
        sc = [1.0 if I[a] == J[a] else math.sqrt(2.0) for a in range(nv)]
        C4 = np.zeros((d,) * 4)
        for a in range(nv):
            for b in range(nv):
                for i, j in ((I[a], J[a]), (J[a], I[a])):
                    for p, q in ((I[b], J[b]), (J[b], I[b])):
                        C4[i, j, p, q] = C0[a, b] / (sc[a] * sc[b])
        G = torch.zeros((nv, nv) + self.h[0].shape, dtype=torch.float64, device="cuda")
        for z in np.ndindex(*(len(zs),) * d):
            if any(float(w[i][z[i]].max()) == 0.0 for i in range(d)):
                continue
            wt = w[0][z[0]] / total[0]
            for i in range(1, d):
                wt = wt * (w[i][z[i]] / total[i])
            k = [(h[i] + sum(Mt[i][j] * zs[z[j]] for j in range(d))).double() for i in range(d)]
            r2 = sum(x * x for x in k)
            zero = r2 == 0
            k = [x / torch.sqrt(torch.where(zero, torch.ones_like(r2), r2)) for x in k]
            wt = torch.where(zero, torch.zeros_like(wt), wt)
            K = [[sum(C4[i, j, p, q] * k[j] * k[q] for j in range(d) for q in range(d) if C4[i, j, p, q] != 0.0) + torch.zeros_like(r2)
                  for p in range(d)] for i in range(d)]
            if d == 2:
                det = K[0][0] * K[1][1] - K[0][1] * K[1][0]
                N = [[K[1][1], -K[0][1]], [-K[1][0], K[0][0]]]
            else:
                def cof(a, b):
                    r, s = [x for x in range(3) if x != a], [x for x in range(3) if x != b]
                    return (-1) ** (a + b) * (K[r[0]][s[0]] * K[r[1]][s[1]] - K[r[0]][s[1]] * K[r[1]][s[0]])
                N = [[cof(b, a) for b in range(3)] for a in range(3)]
                det = sum(K[0][b] * N[b][0] for b in range(3))
            wt = wt / torch.where(zero, torch.ones_like(det), det)
            for a in range(nv):
                for b in range(a, nv):
                    i, j, p, q = I[a], J[a], I[b], J[b]
                    G[a, b] += (0.25 * sc[a] * sc[b]) * wt * (k[i] * (N[j][p] * k[q] + N[j][q] * k[p]) + k[j] * (N[i][p] * k[q] + N[i][q] * k[p]))
        for a in range(nv):
            for b in range(a):
                G[a, b] = G[b, a]
        return G


class _Medium:
    """Stiffness on the natural grid and the operator of the discrete equation."""

    def __init__(self, c, seed):
        rng = np.random.default_rng(seed)
        self.g = g = _Grid(c)
        y = _natural_points(c)
        if c["field"] == "graded":
            C = _graded(y, c["contrast"], rng)
            lam, mu = C[:, 0, 1], 0.5 * C[:, -1, -1]
            C0 = None
        else:
            ph = _phase(y, *_balls(rng, c["d"], c["count"]))
            Cp, C0 = _material(c, rng)
            C = torch.from_numpy(Cp).cuda()[ph.long()]
            lam, mu = torch.from_numpy(Cp[:, 0, 1]), torch.from_numpy(0.5 * Cp[:, -1, -1])
        if C0 is None:
            l0, m0 = 0.5 * float(lam.min() + lam.max()), 0.5 * float(mu.min() + mu.max())
            C0 = np.zeros((g.nv, g.nv))
            C0[: g.d, : g.d] = l0
            C0 += 2 * m0 * np.eye(g.nv)
        self.C = C.permute(1, 2, 0).reshape((g.nv, g.nv) + g.shape).contiguous()
        self.form = c["form"]
        self.dC = self.C if self.form else self.C - torch.from_numpy(C0).cuda()[(...,) + (None,) * g.d]
        self.G = g.table(C0)
        self.G[(slice(None), slice(None)) + (0,) * g.d] = 0.0

    @staticmethod
    def dot(A, x):
        return torch.stack([sum(A[a, b] * x[b] for b in range(x.shape[0])) for a in range(x.shape[0])])

    def green(self, x):
        """Gamma^p applied to the stress dC : x"""
        g = self.g
        return g.inv(self.dot(self.G, g.fwd(self.dot(self.dC, x))))

    def step(self, E, e0):
        y = self.green(E + e0)
        return E - y if self.form else -y

    def solution(self, e0, tol=1e-11):
        """E + Gamma^p dC E = -Gamma^p dC e0 by BiCGStab."""
        x = torch.zeros_like(self.C[0])
        b = -self.green(x + e0)
        r = b.clone()
        x = torch.zeros_like(b)
        rh, p = r.clone(), r.clone()
        rho = (rh * r).sum()
        for _ in range(200):
            v = p + self.green(p)
            al = rho / (rh * v).sum()
            s = r - al * v
            t = s + self.green(s)
            om = (t * s).sum() / (t * t).sum()
            x = x + al * p + om * s
            r = s - om * t
            if float(r.norm()) <= tol * float((x + e0).norm()):
                break
            new = (rh * r).sum()
            p = r + (new / rho) * (al / om) * (p - om * v)
            rho = new
        return x


def _exact_solve(c, seed):
    M = _Medium(c, seed)
    g = M.g
    Es, ms = [], []
    for k in range(c["loads"]):
        e0 = torch.zeros((g.nv,) + (1,) * g.d, dtype=torch.float64, device="cuda")
        e0[k] = 1.0
        if c["iters"] and not c["method"]:
            E = torch.zeros((g.nv,) + g.shape, dtype=torch.float64, device="cuda")
            # a mixed solve adds one iteration in double precision to the ones in single precision
            for _ in range(c["iters"] + (c["prec"] == "mixed")):
                E = M.step(E, e0)
        else:
            E = M.solution(e0)
        Es.append(E.reshape(g.nv, g.m))
        ms.append(M.dot(M.C, E + e0).reshape(g.nv, -1).mean(1).cpu().numpy())
    out = {"strain": torch.stack(Es) if _identity_order(c) else None, "mean_stress": np.stack(ms)}
    if c["loads"] == g.nv:
        out["ceff"] = out["mean_stress"].T.copy()
    return out


def _unflatten(flat, c):
    """Views of the parameter vector (P, p, W, w, Re R, Im R, Q, q)."""
    W, L, m = c["width"], c["layers"], c["modes"]
    sizes = [(W, 1), (W,), (L, W, W), (L, W), (L, 2 * m, 2 * m, m, W, W), (L, 2 * m, 2 * m, m, W, W), (36, W), (36,)]
    out, o = [], 0
    for s in sizes:
        k = int(np.prod(s))
        out.append(flat[o:o + k].view(s))
        o += k
    return out


def _net64(P, x, c):
    """The network in 64 bits for one sample x (1, n, n, n)."""
    n, m, W = c["n"], c["modes"], c["width"]
    ix = torch.cat([torch.arange(m), torch.arange(n - m, n)]).cuda()
    lift, bl, w1, b1, rr, ri, proj, bp = P
    v = torch.einsum("oc,cxyz->oxyz", lift, x) + bl[:, None, None, None]
    for q in range(c["layers"]):
        vh = torch.fft.rfftn(v, dim=(1, 2, 3))[:, ix][:, :, ix][..., :m]
        k = torch.einsum("abkoi,iabk->oabk", torch.complex(rr[q], ri[q]), vh)
        full = torch.zeros(W, n, n, n // 2 + 1, dtype=torch.complex128, device="cuda")
        full = full.index_put((torch.arange(W, device="cuda")[:, None, None, None], ix[None, :, None, None], ix[None, None, :, None],
                               torch.arange(m, device="cuda")[None, None, None, :]), k)
        u = torch.einsum("oi,ixyz->oxyz", w1[q], v) + b1[q][:, None, None, None] + torch.fft.irfftn(full, s=(n, n, n), dim=(1, 2, 3))
        v = torch.nn.functional.gelu(u)
    return torch.einsum("oc,cxyz->oxyz", proj, v) + bp[:, None, None, None]


def _exact_net(c, seed):
    flat, gen = _net_params(c, seed)
    rng = np.random.default_rng(seed)
    P32 = _unflatten(flat, c)
    # the hidden and the spectral weights are applied in bfloat16
    P = [(t.bfloat16() if k in (2, 4, 5) else t).double() for k, t in enumerate(P32)]
    n = c["n"]

    def channel(mp, e):
        return (mp.double() * float(np.float32(0.5 * math.log10(e)))).reshape(1, n, n, n)
    if c["kind"] == "infer":
        maps, E = _net_inputs(c, gen, rng, c["batch"])
        return {"y": torch.stack([_net64(P, channel(mp, e), c).reshape(36, -1) for mp, e in zip(maps, E)])}
    P = [t.requires_grad_(True) for t in P]
    losses = []
    for _ in range(c["acc"]):
        maps, E = _net_inputs(c, gen, rng, c["batch"])
        T = _targets(maps, gen).double()
        tot = 0.0
        for b in range(c["batch"]):
            part = ((_net64(P, channel(maps[b], E[b]), c).reshape(36, -1) - T[b]) ** 2).sum() / T.numel()
            part.backward()
            tot += float(part.detach())
        losses.append(tot)
    return {"loss": np.array(losses), "grads": torch.cat([t.grad.reshape(-1) for t in P])}


def exact(case, seed):
    if case["kind"] == "solve":
        return _exact_solve(case, seed)
    if case["kind"] == "batch":
        return None   # hundreds of converged solutions at high contrast: minutes
    return _exact_net(case, seed)
