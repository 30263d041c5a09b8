"""The calls by which this library's speed is judged: what they are, how their inputs are
made, how one pass of them is run, and what they compute in plain 64-bit torch and numpy.

Every case is a whole unwrap of wrapped-phase maps (the method's outer reweighting loop
around an inner preconditioned CG solve) through ``native.Plan``, or one gradient of the
learned preconditioner's training loss through ``native.Unet``.  A case is a dict:

  kind      "unwrap" (one map), "batch" (n uneven maps on one plan) or "train"
  precond   preconditioner; precision "f64" or "mixed"
  H, W      rows and columns (batch: lo, hi the range of the maps' sides)
  p, tau    the L^p exponent and the weights' regularisation
  stop      "rel": inner ||r|| <= tol ||b||; "paper": the paper's criteria (inner test
            delta_new <= tol^2 delta_0, outer tolerance 1e-6)
  noise     standard deviation of the phase noise in rad; mask: masked share of the pixels
"""
import math

import numpy as np
import torch

from paper_2203_13675_gb300 import native

F64 = torch.float64


# ------------------------------------------------------------------ the cases
def _unwrap(name, precond, precision, H, W, p=1.0, stop="rel", tol=1e-6, passes=5, noise=0.5, mask=0.05, bumps=12,
            ramp=0.02, wide=1.0):
    c = dict(kind="unwrap", precond=precond, precision=precision, H=H, W=W, p=p, tau=1e-2, stop=stop, tol=tol,
             passes=passes, noise=noise, mask=mask, bumps=bumps, ramp=ramp, wide=wide)
    return dict(c, name=name) if name else c


def _paper(name, precond, precision, H, W, p=1.0):
    """The paper's study: no mask, 6 bumps whose widths grow with the map, its stopping criteria."""
    return _unwrap(name, precond, precision, H, W, p=p, stop="paper", tol=0.005, passes=20, noise=0.3, mask=0.0,
                   bumps=6, ramp=0.05, wide=max(H, W) / 256.0)


def _batch(name, precond, n, lo, hi):
    c = dict(kind="batch", precond=precond, precision="mixed", n=n, lo=lo, hi=hi, tau=1e-2, stop="rel", tol=1e-6,
             passes=5)
    return dict(c, name=name) if name else c


def _train(name, B, H, W):
    c = dict(kind="train", B=B, H=H, W=W, p=0.5, tau=1e-2, noise=0.3)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small interferogram, as in an interactive tool or a tile of a larger scene:
        # latency and launches are what it waits for
        _unwrap("mg_mixed_256", "mg", "mixed", 256, 256, noise=0.3, mask=0.0, bumps=6, ramp=0.05),
        # the benchmark's map: the fastest form on a noisy scene with an excluded region
        _unwrap("mg_mixed_2048", "mg", "mixed", 2048, 2048),
        # the largest scene of the repository's workloads, p < 1
        _unwrap("mg_mixed_4096", "mg", "mixed", 4096, 4096, p=0.5, noise=0.7, mask=0.0),
        # a scene of odd, ragged size in full FP64 with the fastest FP64 form
        _unwrap("mg_f64_1251x937", "mg", "f64", 937, 1251, p=0.0),
        # the paper's own study, its map size and criteria: Jacobi in FP64
        _paper("jacobi_f64_640x480", "jacobi", "f64", 480, 640),
        # the paper's triangular preconditioners in its natural order, at sizes of its Table 1
        _paper("ilu_f64_480x360", "ilu0", "f64", 360, 480),
        _paper("ssor_f64_320x240", "ssor", "f64", 240, 320),
        # the paper's method in mixed precision on a megapixel scene
        _unwrap("jacobi_mixed_1024", "jacobi", "mixed", 1024, 1024),
        # the Fourier-basis preconditioner on the same scene
        _unwrap("dct_f64_1024", "dct", "f64", 1024, 1024),
        # a stack of uneven scenes unwrapped together
        _batch("batch_mg_mixed_12", "mg", 12, 256, 1024),
        # the same with the persistent Krylov solver: one launch per pass for all maps
        _batch("batch_jacobi_mixed_8", "jacobi", 8, 160, 400),
        # training the learned preconditioner: the batch of its own training run
        _train("train_8x512x512", 8, 512, 512),
    ]


def _side(rng, lo, hi):
    """Log-uniform; every other size is a multiple of 8, the others fall where they fall."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, v // 8 * 8) if rng.random() < 0.5 else v


def draw(rng):
    what = rng.choice(["mg_mixed", "mg_mixed", "mg_f64", "jacobi_f64", "sweep", "jacobi_mixed", "dct", "batch_mg",
                       "batch_jacobi", "train"])
    p = rng.choice([0.0, 0.5, 1.0, 1.0, 1.5])
    noise = round(rng.uniform(0.2, 0.7), 2)
    mask = rng.choice([0.0, 0.05])
    if what == "mg_mixed":
        return _unwrap(None, "mg", "mixed", _side(rng, 96, 3072), _side(rng, 96, 3072), p=p, noise=noise, mask=mask)
    if what == "mg_f64":
        return _unwrap(None, "mg", "f64", _side(rng, 96, 1536), _side(rng, 96, 1536), p=p, noise=noise, mask=mask)
    if what == "jacobi_f64":
        return _paper(None, "jacobi", "f64", _side(rng, 240, 640), _side(rng, 240, 640))
    if what == "sweep":
        return _paper(None, rng.choice(["ilu0", "ic0", "ssor"]), "f64", _side(rng, 200, 360), _side(rng, 200, 420))
    if what == "jacobi_mixed":
        return _unwrap(None, "jacobi", "mixed", _side(rng, 200, 1024), _side(rng, 200, 1024), p=p, noise=noise,
                       mask=mask)
    if what == "dct":
        return _unwrap(None, "dct", "f64", _side(rng, 128, 1024), _side(rng, 128, 1024), p=p, noise=noise, mask=mask)
    if what == "batch_mg":
        lo = _side(rng, 128, 256)
        return _batch(None, "mg", rng.randint(4, 12), lo, lo * rng.randint(2, 4))
    if what == "batch_jacobi":
        lo = _side(rng, 96, 200)
        return _batch(None, "jacobi", rng.randint(4, 8), lo, 2 * lo)
    return _train(None, rng.randint(1, 8), 128 * rng.randint(1, 4), 128 * rng.randint(1, 4))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _scene(H, W, seed, bumps, ramp, noise, mask, wide):
    """Wrapped phase in (-pi, pi] of a ramp, Gaussian bumps and noise; with mask, a disk of
    zero amplitude (uniform phase) covering that share of the pixels, and its mask."""
    g = _gen(seed)
    u = torch.rand(bumps + 1, 4, generator=g, device="cuda", dtype=F64).cpu()
    i = torch.arange(H, device="cuda", dtype=F64)[:, None]
    j = torch.arange(W, device="cuda", dtype=F64)[None, :]
    phi = ramp * j + torch.zeros(H, 1, device="cuda", dtype=F64)
    for k in range(bumps):
        ci, cj, sb, amp = (float(v) for v in u[k])
        sb, amp = wide * (10.0 + 30.0 * sb), 60.0 * amp - 30.0
        phi = phi + amp * torch.exp(-(i - ci * H) ** 2 / (2 * sb * sb)) * torch.exp(-(j - cj * W) ** 2 / (2 * sb * sb))
    phi = phi + noise * torch.randn(H, W, generator=g, device="cuda", dtype=F64)
    m = None
    if mask > 0:
        rad = math.sqrt(mask * H * W / math.pi)
        rad = min(rad, 0.45 * min(H, W))
        ci, cj = rad + float(u[bumps, 0]) * (H - 2 * rad), rad + float(u[bumps, 1]) * (W - 2 * rad)
        inside = (i - ci) ** 2 + (j - cj) ** 2 <= rad * rad
        free = (2 * torch.rand(H, W, generator=g, device="cuda", dtype=F64) - 1) * math.pi
        phi = torch.where(inside, free, phi)
        m = inside.to(torch.uint8).contiguous()
    psi = torch.atan2(torch.sin(phi), torch.cos(phi))
    psi = torch.where(psi <= -math.pi, psi + 2 * math.pi, psi)
    return psi.contiguous(), m


def _batch_specs(case, seed):
    """The sizes belong to the case (a plan is made for them); p, noise and phase to the seed."""
    shape = np.random.Generator(np.random.PCG64([case["n"], case["lo"], case["hi"]]))
    rng = np.random.Generator(np.random.PCG64(seed))
    specs = []
    for t in range(case["n"]):
        h, w = (int(round(math.exp(shape.uniform(math.log(case["lo"]), math.log(case["hi"]))))) for _ in range(2))
        specs.append(dict(H=h, W=w, p=float(rng.integers(0, 2)), noise=float(rng.uniform(0.1, 0.8)),
                          seed=seed * 1000 + t))
    return specs


def _weights(phi, dx, dy, mask, p, tau):
    """Edge weights tau / (|e|^(2-p) + tau), 0 on edges that leave the grid or touch a masked pixel."""
    def w(e):
        a = e.abs()
        t = torch.ones_like(a) if p == 2 else a if p == 1 else a * a if p == 0 else a ** (2 - p)
        return tau / (t + tau)
    U, V = torch.zeros_like(phi), torch.zeros_like(phi)
    U[:, :-1] = w(phi[:, 1:] - phi[:, :-1] - dx[:, :-1])
    V[:-1] = w(phi[1:] - phi[:-1] - dy[:-1])
    if mask is not None:
        keep = (mask == 0).to(phi.dtype)
        U[:, :-1] *= keep[:, 1:] * keep[:, :-1]
        V[:-1] *= keep[1:] * keep[:-1]
    return U, V


def _diffs(psi):
    def wrap(x):
        return x - 2 * math.pi * torch.ceil((x - math.pi) / (2 * math.pi))
    dx, dy = torch.zeros_like(psi), torch.zeros_like(psi)
    dx[:, :-1] = wrap(psi[:, 1:] - psi[:, :-1])
    dy[:-1] = wrap(psi[1:] - psi[:-1])
    return dx, dy


def _diag(U, V):
    D = U + V
    D[:, 1:] += U[:, :-1]
    D[1:] += V[:-1]
    return D


def _mul(U, V, D, x):
    y = D * x
    y[:, :-1] -= U[:, :-1] * x[:, 1:]
    y[:, 1:] -= U[:, :-1] * x[:, :-1]
    y[:-1] -= V[:-1] * x[1:]
    y[1:] -= V[:-1] * x[:-1]
    return y


_LAYERS = [(3, 16), (16, 32), (32, 64), (64, 128), (192, 64), (96, 32), (48, 16)]


def _train_inputs(case, seed):
    """Network parameters (He-uniform) and B pairs r = A e of residual and error with the weights of A."""
    B, H, W = case["B"], case["H"], case["W"]
    g = _gen(seed)
    parts = []
    for cin, cout in _LAYERS:
        lim = math.sqrt(6.0 / (9 * cin))
        parts.append((2 * torch.rand(cout * cin * 9, generator=g, device="cuda") - 1) * lim)
        parts.append(0.05 * torch.randn(cout, generator=g, device="cuda"))
    parts.append((2 * torch.rand(16, generator=g, device="cuda") - 1) * math.sqrt(6.0 / 16))
    parts.append(0.05 * torch.randn(1, generator=g, device="cuda"))
    planes = {k: torch.empty(B, H, W, device="cuda", dtype=F64) for k in ("r", "U", "V", "e")}
    for k in range(B):
        psi, _ = _scene(H, W, seed * 100 + k, 6, 0.05, case["noise"], 0.0, max(H, W) / 256.0)
        dx, dy = _diffs(psi)
        near = 0.3 * torch.randn(H, W, generator=g, device="cuda", dtype=F64)
        U, V = _weights(torch.cumsum(dx, 1) + near, dx, dy, None, case["p"], case["tau"])
        # an error as an iterate leaves it: smooth, with a rough part
        e = torch.randn(1, 1, H // 16, W // 16, generator=g, device="cuda", dtype=F64)
        e = torch.nn.functional.interpolate(e, size=(H, W), mode="bilinear", align_corners=False)[0, 0]
        e = e + 0.05 * torch.randn(H, W, generator=g, device="cuda", dtype=F64)
        e = e - e.mean()
        planes["r"][k], planes["U"][k], planes["V"][k], planes["e"][k] = _mul(U, V, _diag(U, V), e), U, V, e
    return torch.cat(parts), planes


# ------------------------------------------------------------------ a pass
def _options(case):
    mixed = native.ULP_PRECISION_MIXED if case["precision"] == "mixed" else native.ULP_PRECISION_FP64
    if case["stop"] == "paper":
        return dict(precision=mixed, stop_mode=native.ULP_STOP_PAPER, outer_tol=1e-6)
    return dict(precision=mixed, outer_tol=0.0)


def prepare(case, seed):
    if case["kind"] == "train":
        params, planes = _train_inputs(case, seed)
        net = native.Unet(seed=1)
        net.set_params(params.cpu())
        return dict(case=case, net=net, **planes)
    if case["kind"] == "batch":
        specs = _batch_specs(case, seed)
        maps = []
        for s in specs:
            psi, _ = _scene(s["H"], s["W"], s["seed"], 12, 0.02, s["noise"], 0.0, 1.0)
            maps.append(dict(psi=psi, mask=None, phi=torch.empty_like(psi), p=s["p"], eps=case["tau"]))
        plan = native.Plan(0, sizes=[(s["H"], s["W"]) for s in specs], **_options(case))
        return dict(case=case, plan=plan, maps=maps)
    psi, mask = _scene(case["H"], case["W"], seed, case["bumps"], case["ramp"], case["noise"], case["mask"],
                       case["wide"])
    plan = native.Plan(case["H"], case["W"], **_options(case))
    return dict(case=case, plan=plan, psi=psi, mask=mask)


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        loss, grad = state["net"].loss_grad(state["r"], state["U"], state["V"], state["e"])
        return {"loss": loss, "grad": grad}
    call = dict(precond=case["precond"], tol=case["tol"], max_outer=case["passes"], stats=False)
    if case["kind"] == "batch":
        state["plan"].unwrap_batched(state["maps"], **call)
        return [m["phi"] for m in state["maps"]]
    phi, _ = state["plan"].unwrap(state["psi"], state["mask"], p=case["p"], eps=case["tau"], **call)
    return phi


# ------------------------------------------------------------------ work
# Inner iterations of a whole call that the method needs (all passes): a multigrid or Fourier
# preconditioner's do not grow with the map; the others' grow with its side.
def _iterations(precond, px):
    side = math.sqrt(px)
    return {"mg": 45.0, "dct": 120.0, "jacobi": 10.0 * side, "ilu0": 3.0 * side, "ic0": 3.0 * side,
            "ssor": 3.0 * side}[precond]


# Operations per pixel and iteration: 19 of CG (stencil, updates, dots) and the preconditioner's.
_OPS = {"mg": 19 + 110, "jacobi": 20, "ilu0": 19 + 9, "ic0": 19 + 9, "ssor": 19 + 9}


def work(case):
    if case["kind"] == "train":
        px = case["B"] * case["H"] * case["W"]
        area = [1, 1 / 4, 1 / 16, 1 / 64, 1 / 16, 1 / 4, 1]
        fwd = sum(2 * 9 * ci * co * a for (ci, co), a in zip(_LAYERS, area)) + 32
        return {"bytes": px * 4 * 8 + 2 * 4 * 242721, "flops": 3.0 * fwd * px}
    if case["kind"] == "batch":
        sizes = [(s["H"], s["W"]) for s in _batch_specs(case, 0)]
    else:
        sizes = [(case["H"], case["W"])]
    nbytes = flops = 0.0
    for h, w in sizes:
        px = float(h * w)
        it = _iterations(case["precond"], px)
        # the Fourier preconditioner: a fast transform each way
        ops = _OPS.get(case["precond"]) or 19 + 2 * 2.5 * math.log2(px)
        nbytes += px * (16 + (1 if case.get("mask") else 0))
        flops += px * ops * it
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ the same in plain 64 bits
def _coarsen(U, V):
    """Weights of the grid whose cells are 2x2 cells of this one: sums of the edges between them."""
    H, W = U.shape
    Hc, Wc = (H + 1) // 2, (W + 1) // 2
    u = torch.zeros(2 * Hc, 2 * Wc, device=U.device, dtype=F64)
    v = torch.zeros_like(u)
    u[:H, :W], v[:H, :W] = U, V
    return u[0::2, 1::2] + u[1::2, 1::2], v[1::2, 0::2] + v[1::2, 1::2]


class _Multigrid:
    """One V-cycle: 2 + 2 damped-Jacobi sweeps (2/3), 2x2 aggregates, correction x 1.5, thirty
    sweeps on the coarsest grid (at most 16 cells)."""

    def __init__(self, U, V):
        self.g = []
        while True:
            D = _diag(U, V)
            self.g.append((U, V, D, torch.where(D > 0, 1 / D, torch.zeros_like(D))))
            if U.numel() <= 16:
                break
            U, V = _coarsen(U, V)

    def cycle(self, b, k=0):
        U, V, D, Di = self.g[k]
        om = 2.0 / 3.0
        x = torch.zeros_like(b)
        if k + 1 == len(self.g):
            for _ in range(30):
                x = x + om * Di * (b - _mul(U, V, D, x))
            return x
        x = om * Di * b
        x = x + om * Di * (b - _mul(U, V, D, x))
        H, W = b.shape
        Hc, Wc = (H + 1) // 2, (W + 1) // 2
        r = torch.zeros(2 * Hc, 2 * Wc, device=b.device, dtype=F64)
        r[:H, :W] = b - _mul(U, V, D, x)
        xc = self.cycle(r.view(Hc, 2, Wc, 2).sum((1, 3)), k + 1)
        x = x + 1.5 * xc.repeat_interleave(2, 0).repeat_interleave(2, 1)[:H, :W]
        for _ in range(2):
            x = x + om * Di * (b - _mul(U, V, D, x))
        return x


def _cosines(n):
    k = torch.arange(n, device="cuda", dtype=F64)[:, None]
    i = torch.arange(n, device="cuda", dtype=F64)[None, :]
    C = torch.cos(math.pi * k * (2 * i + 1) / (2 * n)) * math.sqrt(2.0 / n)
    C[0] /= math.sqrt(2.0)
    return C, 2 - 2 * torch.cos(math.pi * k[:, 0] / n)


class _Skewed:
    """A grid laid out by anti-diagonals: row d holds the cells with i + j = d, at place i."""

    def __init__(self, H, W):
        i, j = np.meshgrid(np.arange(H), np.arange(W), indexing="ij")
        self.at, self.shape = (i + j, i), (H + W - 1, H)

    def put(self, x):
        s = np.zeros(self.shape)
        s[self.at] = x
        return s

    def get(self, s):
        return s[self.at]


def _triangular(kind, U, V, D):
    """s = M^-1 r of the no-fill factorisations in row-major order, cell by cell along anti-diagonals."""
    H, W = U.shape
    sk = _Skewed(H, W)
    Uw, Vn = np.zeros_like(U), np.zeros_like(V)
    Uw[:, 1:], Vn[1:] = U[:, :-1], V[:-1]
    if kind == "ssor":
        P = np.where(D > 0, D, 1.0)
    else:
        a, uw, vn = sk.put(D), sk.put(Uw), sk.put(Vn)
        p = np.ones(sk.shape)
        for d in range(sk.shape[0]):
            v = a[d].copy()
            if d:
                v -= uw[d] ** 2 / p[d - 1]
                v[1:] -= vn[d][1:] ** 2 / p[d - 1][:-1]
            p[d] = np.where((v > 1e-12 * a[d]) & (v > 0), v, np.where(a[d] > 0, a[d], 1.0))
        P = sk.get(p)
    cw, cn, ce, cs = (sk.put(x / P) for x in (Uw, Vn, U, V))
    cn1, cs1 = cn[:, 1:].copy(), cs[:, :-1].copy()
    n, t = sk.shape[0], np.empty(H)

    def apply(r):
        z = sk.put(r / P)
        for d in range(1, n):
            np.multiply(cw[d], z[d - 1], out=t)
            z[d] += t
            np.multiply(cn1[d], z[d - 1, :-1], out=t[1:])
            z[d, 1:] += t[1:]
        for d in range(n - 2, -1, -1):
            np.multiply(ce[d], z[d + 1], out=t)
            z[d] += t
            np.multiply(cs1[d], z[d + 1, 1:], out=t[:-1])
            z[d, :-1] += t[:-1]
        return sk.get(z)

    return apply


def _solver_step(precond, U, V, D, mask, dct):
    """r -> M^-1 r"""
    if precond == "jacobi":
        Di = torch.where(D > 0, 1 / D, torch.zeros_like(D))
        return lambda r: Di * r
    keep = None if mask is None else (mask == 0).to(F64)
    if precond == "mg":
        mg = _Multigrid(U, V)
        return lambda r: mg.cycle(r) if keep is None else mg.cycle(r) * keep
    if precond == "dct":
        Ch, Cw, lam = dct
        def apply(r):
            s = Ch.T @ ((Ch @ r @ Cw.T) * lam) @ Cw
            return s if keep is None else s * keep
        return apply
    tri = _triangular(precond, U.numpy(), V.numpy(), D.numpy())
    return lambda r: torch.from_numpy(tri(r.numpy()))


def _exact_unwrap(psi, mask, p, case):
    precond, tol2 = case["precond"], case["tol"] ** 2
    if precond in ("ilu0", "ic0", "ssor"):  # a wavefront: on the host
        psi, mask = psi.cpu(), None if mask is None else mask.cpu()
    H, W = psi.shape
    dct = None
    if precond == "dct":
        (Ch, lh), (Cw, lw) = _cosines(H), _cosines(W)
        lam = lh[:, None] + lw[None, :]
        lam[0, 0] = 1.0
        lam = 1 / lam
        lam[0, 0] = 0.0
        dct = (Ch, Cw, lam)
    dx, dy = _diffs(psi)
    phi = torch.zeros_like(psi)
    for _ in range(case["passes"]):
        U, V = _weights(phi, dx, dy, mask, p, case["tau"])
        D = _diag(U, V)
        b = -U * dx - V * dy
        b[:, 1:] += U[:, :-1] * dx[:, :-1]
        b[1:] += V[:-1] * dy[:-1]
        M = _solver_step(precond, U, V, D, mask, dct)
        before = phi
        r = b - _mul(U, V, D, phi)
        s = M(r)
        delta = delta0 = float((r * s).sum())
        bb, d = float((b * b).sum()), s
        for _ in range(2 * H * W):
            stop = delta <= tol2 * delta0 if case["stop"] == "paper" else float((r * r).sum()) <= tol2 * bb
            if stop or bb == 0:
                break
            q = _mul(U, V, D, d)
            alpha = delta / float((d * q).sum())
            phi = phi + alpha * d
            r = r - alpha * q
            s = M(r)
            new = float((r * s).sum())
            d = s + (new / delta) * d
            delta = new
        base = float(before.norm())
        err = float((phi - before).norm()) / base if base > 0 else math.inf
        if not err > (1e-6 if case["stop"] == "paper" else 0.0):
            break
    return phi


def _exact_train(case, seed):
    params, planes = _train_inputs(case, seed)
    params = params.double().requires_grad_(True)
    conv = torch.nn.functional.conv2d
    with torch.backends.cudnn.flags(enabled=False):
        total = torch.zeros((), device="cuda", dtype=F64)
        for k in range(case["B"]):
            at, ws = 0, []
            for cin, cout in _LAYERS:
                ws.append((params[at: at + cout * cin * 9].view(cout, cin, 3, 3), params[at + cout * cin * 9:][:cout]))
                at += cout * cin * 9 + cout
            r, U, V, e = (planes[n][k] for n in ("r", "U", "V", "e"))
            rho = (r * r).mean().sqrt()
            relu = lambda x, i: conv(x, ws[i][0], ws[i][1], padding=1).relu()  # noqa: E731
            pool = lambda x: torch.nn.functional.avg_pool2d(x, 2)  # noqa: E731
            up = lambda x: x.repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
            e0 = relu(torch.stack([r / rho, U, V])[None], 0)
            e1 = relu(pool(e0), 1)
            e2 = relu(pool(e1), 2)
            b3 = relu(pool(e2), 3)
            d2 = relu(torch.cat([e2, up(b3)], 1), 4)
            d1 = relu(torch.cat([e1, up(d2)], 1), 5)
            d0 = relu(torch.cat([e0, up(d1)], 1), 6)
            y = (d0[0] * params[at: at + 16, None, None]).sum(0) + params[at + 16]
            D = _diag(U, V)
            x = r / rho
            s = torch.where(D > 0, x / D, torch.zeros_like(x)) + y
            loss = 1 - (s * x).sum() ** 2 / ((s * _mul(U, V, D, s)).sum() * ((e / rho) * x).sum())
            (loss / case["B"]).backward()
            total += loss.detach() / case["B"]
    return {"loss": float(total), "grad": params.grad}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "batch":
        out = []
        for s in _batch_specs(case, seed):
            psi, _ = _scene(s["H"], s["W"], s["seed"], 12, 0.02, s["noise"], 0.0, 1.0)
            out.append(_exact_unwrap(psi, None, s["p"], case))
        return out
    psi, mask = _scene(case["H"], case["W"], seed, case["bumps"], case["ramp"], case["noise"], case["mask"],
                       case["wide"])
    return _exact_unwrap(psi, mask, case["p"], case)
