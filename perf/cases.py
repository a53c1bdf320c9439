"""Measured work of the library: what a user has it do, through its public entry points.

Whole calls (a plan is made once per image shape, as a user's program keeps one):

* ``unwrap``  one image through ``Plan.unwrap``;
* ``batch``   many images of uneven sizes through ``Batch.unwrap``;
* ``train``   forward and backward through ``unwrap_differentiable``.

Single operators:

* ``precond`` one application of the Laplacian preconditioner (``precond_laplacian``);
* ``matvec``  one product with the system's matrix (``apply_A``);
* ``post``    the 2 pi congruent rounding and the best-shift error of an unwrapped image.

Images are synthetic interferograms drawn on the GPU from the seed alone, after the laws of the
package's test workloads: a phase ramp and Gaussian bumps, noise, a smoothed coherence map, and
for the "mixed" law low-coherence patches and 3 pi steps.  Whole solves take fewer outer steps
than a full unwrap where a full one would take seconds: every outer step is the same work.

``exact`` restates each operation in 64 bits with plain torch: the IRLS iteration and its
preconditioned conjugate gradients, the adjoint sweep, and the single operators.
"""
import math

import torch

import paper_2401_09961_gb300 as irls

TAU, DELTA = 1e-2, 1e-3
TWO_PI = 2.0 * math.pi


# ---- cases -------------------------------------------------------------------------------------
def listed():
    return [
        # a small crop with uniform weights and the library's default (float32) options: many
        # short dependent launches, latency decides
        {"name": "unwrap 256 fp32", "kind": "unwrap", "H": 256, "W": 256, "law": "uniform",
         "precision": "fp32", "form": "auto", "system": "full", "outer": 10, "tol": 1e-5},
        # a ragged mid-size crop in the default options
        {"name": "unwrap 701x1003 fp32", "kind": "unwrap", "H": 701, "W": 1003,
         "law": "coherence", "precision": "fp32", "form": "auto", "system": "full", "outer": 20,
         "tol": 1e-6},
        # a full burst crop in the default options
        {"name": "unwrap 2048 fp32", "kind": "unwrap", "H": 2048, "W": 2048, "law": "coherence",
         "precision": "fp32", "form": "auto", "system": "full", "outer": 3, "tol": 1e-6},
        # the large scene on the tensor-core preconditioner (split bfloat16)
        {"name": "unwrap 4096 bf16x3", "kind": "unwrap", "H": 4096, "W": 4096, "law": "mixed",
         "precision": "bf16x3", "form": "auto", "system": "full", "outer": 3, "tol": 1e-6},
        # a wide scene on the fast-transform preconditioner and the U-only system: the
        # quickest form for the lengths that it takes
        {"name": "unwrap 4000x8000 fft", "kind": "unwrap", "H": 4000, "W": 8000, "law": "mixed",
         "precision": "fp32", "form": "fft", "system": "schur", "outer": 3, "tol": 1e-6},
        # an uneven set of tiles in one call
        {"name": "batch 64 tiles", "kind": "batch", "tiles": 64, "lo": 256, "hi": 1536,
         "step": 128, "precision": "bf16x3", "outer": 3, "tol": 1e-6, "layout": 1000},
        # one training step: forward with checkpoints, gradients of the phase and the coherence
        {"name": "train 1024 bf16x3", "kind": "train", "H": 1024, "W": 1024, "law": "coherence",
         "precision": "bf16x3", "form": "auto", "outer": 15, "tol": 1e-8},
        # the preconditioner by itself, in each of its forms
        {"name": "precond 300x451 fp32", "kind": "precond", "H": 300, "W": 451,
         "precision": "fp32", "form": "auto"},
        {"name": "precond 2047x1999 bf16x3", "kind": "precond", "H": 2047, "W": 1999,
         "precision": "bf16x3", "form": "auto"},
        {"name": "precond 4096 fft", "kind": "precond", "H": 4096, "W": 4096,
         "precision": "fp32", "form": "fft"},
        # one product with the matrix, for a caller's own Krylov method
        {"name": "matvec 2047x1999", "kind": "matvec", "H": 2047, "W": 1999},
        # the outputs a user keeps: integer map, congruent phase, error against a reference
        {"name": "post 4096", "kind": "post", "H": 4096, "W": 4096},
    ]


def draw(rng):
    """One more case of the ranges above: sides spread over their logarithm, odd ones among them."""
    def side(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    def pow2(lo, hi):
        return 2 ** rng.randint(lo, hi)

    kind = rng.choice(["unwrap"] * 4 + ["precond"] * 3 + ["batch", "train", "matvec", "post"])
    c = {"kind": kind}
    if kind in ("unwrap", "precond"):
        form = rng.choice(["fp32", "bf16x3", "fft"])
        if form == "fp32":       # the default: any sides
            c |= {"H": side(64, 1500), "W": side(64, 1500), "precision": "fp32", "form": "auto"}
        elif form == "bf16x3":   # tensor-core products
            c |= {"H": side(256, 3000), "W": side(256, 3000), "precision": "bf16x3",
                  "form": "auto"}
        else:                    # fast transforms: the lengths they take
            c |= {"H": rng.choice([2000, 4000, pow2(7, 12), pow2(7, 12)]),
                  "W": rng.choice([2000, 4000, pow2(7, 12), pow2(7, 12)]),
                  "precision": "fp32", "form": "fft"}
        if kind == "unwrap":
            small = c["H"] * c["W"] <= 512 * 512
            c |= {"law": "coherence" if form == "fp32" else rng.choice(["coherence", "mixed"]),
                  "system": "full" if form != "fft" else rng.choice(["full", "schur"]),
                  "outer": rng.randint(2, 4) if small else 1, "tol": 1e-6}
    elif kind == "batch":
        c |= {"tiles": rng.randint(8, 48), "lo": 256, "hi": rng.choice([768, 1024, 1536]),
              "step": rng.choice([64, 101, 128]), "precision": "bf16x3", "outer": 1, "tol": 1e-6,
              "layout": rng.randrange(1 << 20)}
    elif kind == "train":
        c |= {"H": side(256, 1024), "W": side(256, 1024), "law": "coherence",
              "precision": rng.choice(["fp32", "bf16x3"]), "form": "auto", "outer": rng.randint(2, 5),
              "tol": 1e-8}
    else:
        c |= {"H": side(100, 4096), "W": side(100, 4096)}
    return c


# ---- synthetic interferograms ------------------------------------------------------------------
def scene(H, W, seed, law):
    """(X, coherence or None, noise-free phase less its mean): the package's test laws, drawn on
    the GPU.  The ramp is 0.195 rad per pixel of the longer side (800 rad over 4096)."""
    dev = "cuda"
    few = torch.Generator().manual_seed(seed * 7919 + 17)
    many = torch.Generator(device=dev).manual_seed(seed * 104729 + 29)
    u = lambda *n: torch.rand(*n, generator=few, dtype=torch.float64)  # noqa: E731
    y = torch.arange(H, device=dev, dtype=torch.float64)
    x = torch.arange(W, device=dev, dtype=torch.float64)
    side = max(H, W)
    th = float(u(1)) * TWO_PI
    proj = y[:, None] * math.sin(th) + x[None, :] * math.cos(th)
    proj -= proj.min()
    phi = proj * ((40.0 / 256 if law == "uniform" else 800.0 / 4096) * side / max(float(proj.max()), 1.0))
    n = 5 if law == "uniform" else max(1, round(80 * side / 4096))
    amp, sig = (5 + 25 * u(n)).to(dev), (10 + 50 * u(n)).to(dev)
    cy, cx = (u(n) * H).to(dev), (u(n) * W).to(dev)
    by = torch.exp(-0.5 * ((y[:, None] - cy) / sig) ** 2) * amp
    bx = torch.exp(-0.5 * ((x[:, None] - cx) / sig) ** 2)
    phi += by @ bx.T
    sigma = 0.3 if law == "uniform" else 0.5
    coh = None
    if law != "uniform":
        f = torch.fft.rfft2(torch.rand(H, W, generator=many, device=dev))
        fy, fx = torch.fft.fftfreq(H, device=dev)[:, None], torch.fft.rfftfreq(W, device=dev)
        c = torch.fft.irfft2(f * torch.exp(-2 * (math.pi * 16.0) ** 2 * (fy * fy + fx * fx)), s=(H, W))
        coh = 0.05 + 0.95 * (c - c.min()) / (c.max() - c.min()).clamp_min(1e-20)
    if law == "mixed":
        low = torch.zeros(H, W, dtype=torch.bool, device=dev)
        for e in u(28, 5).tolist():   # ellipses over about a fifth of the pixels
            a, b = ((0.02 + 0.06 * t) * min(H, W) for t in e[:2])
            co, si = math.cos(e[2] * TWO_PI), math.sin(e[2] * TWO_PI)
            dy, dx = y[:, None] - e[3] * H, x[None, :] - e[4] * W
            low |= ((dx * co + dy * si) / a) ** 2 + ((dy * co - dx * si) / b) ** 2 <= 1
        for e in u(2, 3).tolist():    # two half-planes 3 pi higher
            t = e[0] * math.pi
            phi += 3 * math.pi * ((x - e[1] * W) * math.cos(t) + (y[:, None] - e[2] * H) * math.sin(t) > 0)
        coh = torch.where(low, 0.05 + 0.15 * torch.rand(H, W, generator=many, device=dev), coh)
        sigma = torch.where(low, 1.2, 0.5)
    obs = phi + sigma * torch.randn(H, W, generator=many, device=dev, dtype=torch.float64)
    X = (obs - TWO_PI * torch.round(obs / TWO_PI)).float()
    return X, None if coh is None else coh.float().contiguous(), phi - phi.mean()


def noise(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed * 15485863 + 5)
    return torch.randn(*shape, generator=g, device="cuda")


def tile_shapes(c):
    g = torch.Generator().manual_seed(c["layout"])
    n = (c["hi"] - c["lo"]) // c["step"] + 1
    return [tuple(int(c["lo"] + c["step"] * k) for k in hw)
            for hw in torch.randint(0, n, (c["tiles"], 2), generator=g).tolist()]


# ---- inputs and passes -------------------------------------------------------------------------
def inputs(c, seed):
    """The tensors of a case, from the seed alone."""
    k = c["kind"]
    if k == "batch":
        made = [scene(h, w, 1000 * seed + t, "coherence") for t, (h, w) in enumerate(tile_shapes(c))]
        return {"X": [m[0] for m in made], "coh": [m[1] for m in made]}
    H, W = c["H"], c["W"]
    if k in ("unwrap", "train"):
        X, coh, _ = scene(H, W, seed, c["law"])
        s = {"X": X, "coh": coh}
        if k == "train":   # the gradient that the rest of a model hands back
            s["gU"] = noise(seed, H, W)
        return s
    if k == "precond":   # a residual: noise without its mean
        R = noise(seed, H, W)
        return {"R": R - R.mean()}
    if k == "matvec":    # directions, and the weights D = C^2 / W of an ordinary outer step
        z = noise(seed, 5, H, W)
        d = [0.25 / torch.sqrt(0.25 * v * v + DELTA * DELTA) for v in (z[3], z[4])]
        return {"U": z[0].contiguous(), "Vv": z[1, :-1].contiguous(), "Vh": z[2, :, :-1].contiguous(),
                "Dv": d[0][:-1].contiguous(), "Dh": d[1][:, :-1].contiguous()}
    X, _, ref = scene(H, W, seed, "coherence")   # post: an unwrapped image, its input, a reference
    q = (ref - X.double()) / TWO_PI
    U = (X.double() + TWO_PI * torch.round(q) + 0.02 * noise(seed, H, W) + 1.25).float()
    return {"U": U, "X": X, "ref": ref.float()}


def prepare(case, seed):
    c, s = case, inputs(case, seed)
    k = c["kind"]
    s["kind"] = k
    opts = dict(tau=TAU, delta=DELTA, cg_max_iter=1000)
    if k == "batch":
        s["batch"] = irls.Batch(tile_shapes(c), precision=c["precision"], outer_iters=c["outer"],
                                cg_tol=c["tol"], **opts)
        return s
    if k in ("unwrap", "train"):
        opts |= {"outer_iters": c["outer"], "cg_tol": c["tol"], "system": c.get("system", "full")}
        if k == "train":
            opts["cg_max_iter"] = 3000
    s["plan"] = irls.Plan(c["H"], c["W"], precision=c.get("precision", "fp32"),
                          dct_form=c.get("form", "auto"), **opts)
    if k == "train":
        s["X"].requires_grad_(True)
        s["coh"].requires_grad_(True)
    return s


def run(s):
    k = s["kind"]
    if k == "unwrap":
        return s["plan"].unwrap(s["X"], s["coh"])[0]
    if k == "batch":
        return s["batch"].unwrap(s["X"], s["coh"])[0]
    if k == "train":
        U = irls.unwrap_differentiable(s["X"], s["coh"], s["plan"])
        gX, gC = torch.autograd.grad(U, (s["X"], s["coh"]), grad_outputs=s["gU"])
        return {"U": U.detach(), "gX": gX, "gC": gC}
    if k == "precond":
        return irls.precond_laplacian(s["plan"], s["R"])
    if k == "matvec":
        return irls.apply_A(s["plan"], s["U"], s["Vv"], s["Vh"], s["Dv"], s["Dh"])
    Ur, K, c = irls.round_congruent(s["plan"], s["U"], s["X"])
    E, alpha, rms = irls.best_shift_error(s["plan"], s["U"], s["ref"])
    return {"Ur": Ur, "K": K, "offset": c, "E": E, "alpha": alpha, "rms": rms}


def work(case):
    """Bytes: each input read once, each output written once.  Operations: of the path with the
    preconditioner as fast transforms (about 100 a pixel) and the stencils (about 60); a solve
    takes at least some 20 iterations for each outer step."""
    c = case
    n = sum(h * w for h, w in tile_shapes(c)) if c["kind"] == "batch" else c["H"] * c["W"]
    if c["kind"] in ("unwrap", "batch"):   # phase, coherence; unwrapped phase
        return {"bytes": 12 * n, "flops": 160 * 20 * c["outer"] * n}
    if c["kind"] == "train":               # and the gradients: one handed in, two returned
        return {"bytes": 24 * n, "flops": 2 * 160 * 20 * c["outer"] * n}
    if c["kind"] == "precond":
        return {"bytes": 8 * n, "flops": 100 * n}
    if c["kind"] == "matvec":
        return {"bytes": 32 * n, "flops": 30 * n}
    return {"bytes": 24 * n, "flops": 60 * n}


# ---- the same in 64 bits -----------------------------------------------------------------------
def gradients(X):
    """Wrapped differences, decided in float32 one rounded operation at a time (the wrap decides
    an integer), then in 64 bits."""
    pi, two = (torch.tensor(v, dtype=torch.float32, device=X.device) for v in (math.pi, TWO_PI))

    def wrap(t):
        return (t - two * torch.floor((t + pi) / two)).double()
    return wrap(X[1:] - X[:-1]), wrap(X[:, 1:] - X[:, :-1])


def edge_weights(X, coh):
    if coh is None:
        return torch.ones_like(X[1:]).double(), torch.ones_like(X[:, 1:]).double()
    c = coh.detach().double()
    return 0.5 * (c[1:] + c[:-1]), 0.5 * (c[:, 1:] + c[:, :-1])


def S(U):
    return U[1:] - U[:-1], U[:, 1:] - U[:, :-1]


def St(ev, eh):
    """S^T e_v + e_h T^T."""
    q = ev.new_zeros(eh.shape[0], ev.shape[1])
    q[:-1] -= ev
    q[1:] += ev
    q[:, :-1] -= eh
    q[:, 1:] += eh
    return q


def dct(x):
    """Orthonormal DCT-II along the last dimension, by an FFT of the same length."""
    n = x.shape[-1]
    v = torch.cat([x[..., ::2], x[..., 1::2].flip(-1)], -1)
    k = torch.arange(n, device=x.device, dtype=torch.float64)
    y = (torch.fft.fft(v) * torch.polar(torch.ones_like(k), -math.pi * k / (2 * n))).real
    y *= math.sqrt(2.0 / n)
    y[..., 0] *= math.sqrt(0.5)
    return y


def idct(y):
    n = y.shape[-1]
    y = y * math.sqrt(n / 2.0)
    y[..., 0] *= math.sqrt(2.0)
    k = torch.arange(n, device=y.device, dtype=torch.float64)
    z = torch.zeros_like(y)
    z[..., 1:] = y[..., 1:].flip(-1)
    v = torch.fft.ifft(torch.complex(y, -z) * torch.polar(torch.ones_like(k), math.pi * k / (2 * n))).real
    x = torch.empty_like(y)
    x[..., ::2] = v[..., :(n + 1) // 2]
    x[..., 1::2] = v[..., (n + 1) // 2:].flip(-1)
    return x


class Laplacian:
    """z with S^T S z + z T T^T = tau r and no constant part."""

    def __init__(self, H, W):
        lam = [2 - 2 * torch.cos(math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n)
               for n in (H, W)]
        self.inv = lam[0][:, None] + lam[1][None, :]
        self.inv[0, 0] = 1.0
        self.inv = TAU / self.inv
        self.inv[0, 0] = 0.0

    def __call__(self, r):
        f = dct(dct(r).mT.contiguous()) * self.inv.mT
        return idct(idct(f).mT.contiguous())


def dot(a, b):
    return sum((x * y).sum() for x, y in zip(a, b))


def pcg(x, r, bb, A, M, tol, most):
    """Preconditioned conjugate gradients on lists of arrays, stopped on ||r|| <= tol ||b||."""
    if float(dot(r, r)) <= tol * tol * bb:
        return x
    z = M(r)
    p, rho = z, dot(r, z)
    for _ in range(most):
        q = A(p)
        a = rho / dot(p, q)
        x = [u + a * v for u, v in zip(x, p)]
        r = [u - a * v for u, v in zip(r, q)]
        if float(dot(r, r)) <= tol * tol * bb:
            break
        z = M(r)
        new = dot(r, z)
        p = [u + (new / rho) * v for u, v in zip(z, p)]
        rho = new
    return x


def full_system(L, D):
    """A of the (U, V) system and its block-diagonal preconditioner."""
    def A(p):
        s = S(p[0])
        y = [a - b for a, b in zip(s, p[1:])]
        return [St(*y) / TAU] + [d * v - e / TAU for d, v, e in zip(D, p[1:], y)]
    return A, lambda r: [L(r[0])] + [v / (d + 1 / TAU) for v, d in zip(r[1:], D)]


def schur_system(L, D):
    """The U-only system left after eliminating V, and its preconditioner."""
    om = [d / (1 + TAU * d) for d in D]
    return lambda p: [St(*(o * s for o, s in zip(om, S(p[0]))))], lambda r: [L(r[0])]


def solve(X, coh, outer, tol, system="full", most=1000):
    """The IRLS iteration from U = 0, V = -G; returns U and the slacks V of every step."""
    G, C = gradients(X.detach()), edge_weights(X.detach(), coh)
    L = Laplacian(*X.shape)
    U, V = torch.zeros_like(X, dtype=torch.float64), [-g for g in G]
    b = [St(*G) / TAU] + [-g / TAU for g in G]
    kept = [V]
    for _ in range(outer):
        D = [c * c / torch.sqrt(c * c * v * v + DELTA ** 2) for c, v in zip(C, V)]
        if system == "schur":
            A, M = schur_system(L, D)
            f = [St(*(d / (1 + TAU * d) * g for d, g in zip(D, G)))]
            r = [f[0] - A([U])[0]]
            U, = pcg([U], r, float(dot(f, f)), A, M, tol, most)
            V = [(s - g) / (1 + TAU * d) for s, g, d in zip(S(U), G, D)]
        else:
            A, M = full_system(L, D)
            x = [U] + V
            r = [u - v for u, v in zip(b, A(x))]
            U, *V = pcg(x, r, float(dot(b, b)), A, M, tol, most)
        U = U - U.mean()
        kept.append(V)
    return U, kept, G, C, L


def backward(g, kept, G, C, L, tol, most):
    """Reverse sweep: each step is its converged solve; the cotangent of every solve goes through
    the U-only system, normalised."""
    xU, xV = g - g.mean(), [torch.zeros_like(v) for v in G]
    gG, gC = [torch.zeros_like(v) for v in G], [torch.zeros_like(v) for v in G]
    for k in reversed(range(len(kept) - 1)):
        W = [torch.sqrt(c * c * v * v + DELTA ** 2) for c, v in zip(C, kept[k])]
        D = [c * c / w for c, w in zip(C, W)]
        n = torch.sqrt(dot([xU] + xV, [xU] + xV))
        xU, xV = xU / n, [v / n for v in xV]
        f = [xU + St(*(v / (1 + TAU * d) for v, d in zip(xV, D)))]
        A, M = schur_system(L, D)
        lU, = pcg([torch.zeros_like(xU)], f, float(dot(f, f)), A, M, tol, most)
        lV = [n * (TAU * v + s) / (1 + TAU * d) for v, s, d in zip(xV, S(lU), D)]
        lU = n * lU
        gG = [a + (s - v) / TAU for a, s, v in zip(gG, S(lU), lV)]
        dD = [-v * u for v, u in zip(lV, kept[k + 1])]
        gC = [a + d * (2 * c / w - c ** 3 * v * v / w ** 3) for a, d, c, w, v in zip(gC, dD, C, W, kept[k])]
        xU, xV = torch.zeros_like(xU), [-d * c ** 4 * v / w ** 3 for d, c, w, v in zip(dD, C, W, kept[k])]
    gG = [a - v for a, v in zip(gG, xV)]
    gc = torch.zeros_like(xU)
    gc[1:] += gC[0] / 2
    gc[:-1] += gC[0] / 2
    gc[:, 1:] += gC[1] / 2
    gc[:, :-1] += gC[1] / 2
    return St(*gG), gc


def exact(case, seed):
    c, s = case, inputs(case, seed)
    k = c["kind"]
    if k == "unwrap":
        return solve(s["X"], s["coh"], c["outer"], c["tol"], c["system"])[0]
    if k == "batch":   # about a quarter of a second an image and outer step
        if c["tiles"] * c["outer"] > 64:
            return None
        return [solve(X, q, c["outer"], c["tol"])[0] for X, q in zip(s["X"], s["coh"])]
    if k == "train":
        U, *rest = solve(s["X"], s["coh"], c["outer"], c["tol"], most=3000)
        gX, gC = backward(s["gU"].double(), *rest, c["tol"], 3000)
        return {"U": U, "gX": gX, "gC": gC}
    if k == "precond":
        return Laplacian(c["H"], c["W"])(s["R"].double())
    if k == "matvec":
        U, Vv, Vh, Dv, Dh = (s[n].double() for n in ("U", "Vv", "Vh", "Dv", "Dh"))
        return tuple(full_system(None, (Dv, Dh))[0]([U, Vv, Vh]))
    U, X, ref = (s[n].double() for n in ("U", "X", "ref"))
    off = math.atan2(float(torch.sin(U - X).sum()), float(torch.cos(U - X).sum()))
    K = torch.round((U - off - X) / TWO_PI)
    alpha = float((ref - U).mean())
    E = ref - U - alpha
    return {"Ur": X + TWO_PI * K, "K": None, "offset": off, "E": E, "alpha": alpha,
            "rms": float(torch.sqrt((E * E).mean()))}
