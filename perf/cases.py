"""Performance cases of the reconstruction library: what its users run.

Each case is one call (or one short session of calls) through the package's
public entry points, at the sizes of the reconstruction workloads
(workloads/__init__.py) and around them.  A case's `kind` names the call:

  normal   A^T A on a batch of images (the gradient of every solve)
  pair     A with its adjoint backward, through the autograd wrapper
  sketch   Omega and Y = A^T A Omega (Algorithm 1 steps 1-2), bf16 storage
  factor   Algorithm 1 steps 3-8 and P^{-1} on a few images with its result
  prox     the TV / Hessian prox in the P-metric (20 dual steps)
  solve    some iterations of Algorithm 3 from the start
  unroll   a differentiated unrolled solve, forward and backward

Factors that a solve, prox or unrolled solve takes as given are low-frequency
Fourier modes (orthonormal, what a converged sketch of these operators looks
like) with a spectrum of the operator's kind.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2411_08178_gb300 import api, autograd

EPS32 = 2.0 ** -23
DT = {"f32": torch.float32, "f64": torch.float64}


# ---------------------------------------------------------------- cases ----

def listed() -> list:
    return [
        # the smallest whole solve: 64 x 64 deblurring in float64 with a Haar
        # prior, the setting the method is checked in; launch and latency bound
        dict(name="haar64_solve_f64", kind="solve", op="blur", n1=64, n2=64, dtype="f64", k=9, sigma=1.5,
             reg="wavelet", lam=1e-3, fit="l2", ell=32, sqrt_shift=True, iters=10),
        # learning lambda and a blur kernel through an unrolled solve: one
        # forward and one backward pass of the differentiated workload
        dict(name="unroll_grad_256", kind="unroll", n1=256, n2=256, k=13, sigma=2.0, lam=5e-4, ell=64, K=10),
        # 4 x super-resolution with impulsive noise: Huber fit, Hessian prior,
        # a sketch whose columns are all inactive (P = I)
        dict(name="superres512_hs_solve", kind="solve", op="blur_decim", n1=512, n2=512, dtype="f32", k=7, sigma=2.0,
             decim=4, reg="hs", lam=1e-3, fit="huber", ell=0, sqrt_shift=True, iters=10),
        # the sketch of the 512 x 512 deblurring workload
        dict(name="blur512_sketch", kind="sketch", op="blur", n1=512, n2=512, k=25, sigma=4.0, ell=200),
        # Algorithm 1's factor for that sketch, and one for the CT workload
        dict(name="blur512_factor_l200", kind="factor", spectrum="blur", n1=512, n2=512, k=25, sigma=4.0, ell=200,
             batch=4),
        dict(name="ct512_factor_l400", kind="factor", spectrum="ct", n1=512, n2=512, n_angles=720, ell=400, batch=4),
        # CT as a layer of a learned model: A and its adjoint backward on a
        # small batch of odd-sized images
        dict(name="ct_pair_ragged", kind="pair", op="radon", n1=257, n2=301, dtype="f32", n_angles=363, n_bins=401,
             batch=3),
        # the gradient of the CT workload: A^T A on one image, every iteration
        dict(name="ct512_normal", kind="normal", op="radon", n1=512, n2=512, dtype="f32", n_angles=720, n_bins=736,
             batch=1),
        # the sketch of the CT workload: the largest single call
        dict(name="ct512_sketch", kind="sketch", op="radon", n1=512, n2=512, n_angles=720, n_bins=736, ell=400),
        # the P-metric TV prox of the deblurring workload without the
        # square-root heuristic: 199 active columns, every dual step runs
        dict(name="prox512_tv_l200", kind="prox", reg="tv", n1=512, n2=512, ell=200, sqrt_shift=False, lam_bar=5e-4,
             n_inner=20),
        # iterations of the CT solve with a 400-column preconditioner (without
        # the square-root heuristic, whose weights in the thousands make a
        # float32 iterate after a few steps a matter of rounding)
        dict(name="ct512_solve_l400", kind="solve", op="radon", n1=512, n2=512, dtype="f32", n_angles=720, n_bins=736,
             reg="tv", lam=2e-4, fit="l2", ell=400, sqrt_shift=False, iters=20),
        # the gradient of the fan-beam CT geometry
        dict(name="fan512_normal", kind="normal", op="fanbeam", n1=512, n2=512, dtype="f32", n_angles=720, n_bins=1024,
             src=1000.0, det=2000.0, batch=1),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    """One more case: image sides 64..512 (odd ones among them), angles and
    bins around the workloads', sketch sizes up to 400."""
    kind = rng.choice(["normal", "normal", "pair", "sketch", "factor", "prox", "solve", "solve", "unroll"])
    n1 = _log_int(rng, 64, 512)
    n2 = n1 if rng.random() < 0.4 else max(64, min(512, int(n1 * rng.uniform(0.7, 1.4))))
    n = max(n1, n2)

    def ct(c):
        c.update(n_angles=_log_int(rng, 45, 720), n_bins=max(65, min(736, int(rng.uniform(1.0, 1.45) * n))))
        return c

    def blur(c):
        sigma = rng.uniform(1.0, 4.0)
        c.update(sigma=sigma, k=2 * math.ceil(3 * sigma) + 1)
        return c

    def fan(c):
        c.update(n_angles=_log_int(rng, 45, 720), n_bins=max(65, min(1024, int(rng.uniform(1.2, 2.0) * n))),
                 src=2.0 * n * rng.uniform(0.9, 1.1))
        c["det"] = 2.0 * c["src"]
        return c

    if kind in ("normal", "pair"):
        op = rng.choice(["radon", "radon", "blur", "fanbeam"])
        c = dict(kind=kind, op=op, n1=n1, n2=n2, dtype="f64" if rng.random() < 0.15 else "f32",
                 batch=rng.choice([1, 1, 2, 3, 5, 8]))
        return {"radon": ct, "blur": blur, "fanbeam": fan}[op](c)
    if kind == "sketch":
        op = rng.choice(["radon", "blur"])
        c = dict(kind=kind, op=op, n1=n1, n2=n2, ell=_log_int(rng, 16, 400))
        return (ct if op == "radon" else blur)(c)
    if kind == "factor":
        n1, n2 = max(n1, 128), max(n2, 128)
        c = dict(kind=kind, spectrum=rng.choice(["blur", "ct"]), n1=n1, n2=n2, ell=_log_int(rng, 20, 400),
                 batch=rng.choice([1, 2, 4]))
        return blur(c) if c["spectrum"] == "blur" else dict(c, n_angles=_log_int(rng, 180, 720))
    if kind == "prox":
        return dict(kind=kind, reg=rng.choice(["tv", "tv", "isotv", "hs"]), n1=n1, n2=n2,
                    ell=rng.choice([0, _log_int(rng, 16, 300)]), sqrt_shift=False,
                    lam_bar=math.exp(rng.uniform(math.log(1e-4), math.log(1e-2))), n_inner=20)
    if kind == "unroll":
        n1, n2 = min(n1, 256), min(n2, 256)
        return blur(dict(kind=kind, n1=n1, n2=n2, lam=5e-4, ell=_log_int(rng, 16, 128), K=rng.choice([4, 8, 10])))
    op = rng.choice(["radon", "blur", "blur_decim"])
    c = dict(kind="solve", op=op, n1=n1, n2=n2, dtype="f32", lam=5e-4, fit="l2",
             sqrt_shift=op != "radon" and rng.random() < 0.5,
             reg=rng.choice(["tv", "tv", "isotv", "hs"]), ell=rng.choice([0, _log_int(rng, 16, 300)]), iters=10)
    if op == "radon":
        return ct(dict(c, lam=2e-4))
    if op == "blur_decim":
        c.update(n1=4 * (n1 // 4), n2=4 * (n2 // 4), decim=4, fit="huber", lam=1e-3)
    return blur(c)


# --------------------------------------------------------------- inputs ----

def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed)


def _gauss_kernel(k: int, sigma: float) -> np.ndarray:
    a = np.arange(k, dtype=np.float64) - (k - 1) / 2.0
    g = np.exp(-(a[:, None] ** 2 + a[None, :] ** 2) / (2.0 * sigma * sigma))
    return g / g.sum()


def _phantoms(b: int, n1: int, n2: int, seed: int) -> torch.Tensor:
    """b piecewise-constant phantoms of 12 random ellipses, values in [0, 1], float64."""
    g = _gen(seed)
    r = torch.rand((6, 12, b, 1, 1), generator=g, device="cuda", dtype=torch.float64)
    y = ((torch.arange(n1, device="cuda", dtype=torch.float64) - (n1 - 1) / 2) / (n1 / 2))[None, :, None]
    x = ((torch.arange(n2, device="cuda", dtype=torch.float64) - (n2 - 1) / 2) / (n2 / 2))[None, None, :]
    img = torch.zeros((b, n1, n2), device="cuda", dtype=torch.float64)
    for e in range(12):
        cx, cy = 1.4 * r[0, e] - 0.7, 1.4 * r[1, e] - 0.7
        ax, ay, th = 0.05 + 0.35 * r[2, e], 0.05 + 0.35 * r[3, e], math.pi * r[4, e]
        u = (x - cx) * torch.cos(th) + (y - cy) * torch.sin(th)
        v = (y - cy) * torch.cos(th) - (x - cx) * torch.sin(th)
        img = torch.where((u / ax) ** 2 + (v / ay) ** 2 <= 1.0, r[5, e].expand_as(img), img)
    return img


def _modes(n1: int, n2: int, ell: int) -> torch.Tensor:
    """The ell lowest-frequency real Fourier modes of an n1 x n2 image, orthonormal rows (float64)."""
    a, b = np.meshgrid(np.arange(n1) - n1 // 2, np.arange(n2) - n2 // 2, indexing="ij")
    half = (b > 0) | ((b == 0) & (a >= 0))           # one of each conjugate pair
    half &= (2 * np.abs(a) < n1) & (2 * np.abs(b) < n2)
    a, b = a[half], b[half]
    order = np.lexsort((a, b, a * a + b * b))[:ell]
    i = torch.arange(n1, device="cuda", dtype=torch.float64)[:, None] / n1
    j = torch.arange(n2, device="cuda", dtype=torch.float64)[None, :] / n2
    rows = []
    for p in order:
        ph = 2 * math.pi * (int(a[p]) * i + int(b[p]) * j)
        if a[p] == 0 and b[p] == 0:
            rows.append(torch.full((n1, n2), (n1 * n2) ** -0.5, device="cuda", dtype=torch.float64))
            continue
        rows.append(torch.cos(ph) * math.sqrt(2.0 / (n1 * n2)))
        if len(rows) < ell:
            rows.append(torch.sin(ph) * math.sqrt(2.0 / (n1 * n2)))
        if len(rows) >= ell:
            break
    return torch.stack(rows[:ell]).reshape(ell, -1)


def _norm_bound(c: dict) -> float:
    """An upper bound of the largest eigenvalue of A^T A (and of P^{-1} A^T A, as P >= I)."""
    if c.get("op") == "radon":
        return 1.05 * c["n_angles"] * math.hypot(c["n1"], c["n2"])
    return 1.03 / c.get("decim", 1) ** 2


def _factor_given(c: dict):
    """U and S_hat of the factor that a case takes as given; U in the precision it is stored in."""
    ell, i = c["ell"], torch.arange(c["ell"], device="cuda", dtype=torch.float64)
    U = _modes(c["n1"], c["n2"], ell)
    if c.get("op") == "radon":                       # decays like 1 / |frequency|
        S = _norm_bound(c) / torch.sqrt(1.0 + i)
    else:                                            # a nearly flat top, as the Gaussian blurs'
        S = 0.6 - 0.3 * i / max(1, ell - 1)
    store = torch.float64 if c.get("dtype") == "f64" else torch.bfloat16
    return U.to(store), S


def _huber_delta(c: dict) -> float:
    return 0.01 if c["fit"] == "huber" else 0.0


def _data(c: dict, seed: int) -> torch.Tensor:
    """Noisy measurements of a phantom (float64), by the definitions at the end of this file."""
    A = _Exact(c)
    y = A.apply(_phantoms(1, c["n1"], c["n2"], seed))[0]
    g = _gen(seed + 1)
    if c.get("fit") == "huber":                      # salt and pepper
        r = torch.rand(y.shape, generator=g, device="cuda", dtype=torch.float64)
        return torch.where(r < 0.1, torch.ones_like(y), torch.where(r > 0.9, torch.zeros_like(y), y))
    scale = 0.01 * float(y.abs().max()) if c.get("op") == "radon" else 0.005
    return y + scale * torch.randn(y.shape, generator=g, device="cuda", dtype=torch.float64)


def _operator(ctx, c: dict):
    dt = DT[c.get("dtype", "f32")]
    if c["op"] == "radon":
        return api.Operator(ctx, "radon", c["n1"], c["n2"], dtype=dt, n_angles=c["n_angles"], n_bins=c["n_bins"])
    if c["op"] == "fanbeam":
        return api.Operator(ctx, "fanbeam", c["n1"], c["n2"], dtype=dt, n_angles=c["n_angles"], n_bins=c["n_bins"],
                            src_dist=c["src"], det_dist=c["det"])
    return api.Operator(ctx, c["op"], c["n1"], c["n2"], dtype=dt, kernel=_gauss_kernel(c["k"], c["sigma"]),
                        decim=c.get("decim", 1), haar_levels=3 if c.get("reg") == "wavelet" else 0)


def _alpha(c: dict) -> float:
    return 1.0 / _norm_bound(c)


def _sketch_pair(c: dict, seed: int):
    """A bf16 (Omega, Y): Y = Phi Omega with Phi the blur's normal operator, or the 1 / |frequency| filter
    that a full-angle parallel-beam normal operator approximates."""
    n1, n2, ell = c["n1"], c["n2"], c["ell"]
    Om = torch.randn((ell, n1, n2), generator=_gen(seed), device="cuda").to(torch.bfloat16)
    if c["spectrum"] == "blur":
        mult = _otf(_gauss_kernel(c["k"], c["sigma"]), n1, n2).abs()[:, :n2 // 2 + 1] ** 2
    else:
        f1 = torch.fft.fftfreq(n1, device="cuda", dtype=torch.float64)[:, None]
        f2 = torch.fft.rfftfreq(n2, device="cuda", dtype=torch.float64)[None, :]
        mult = c["n_angles"] / (math.pi * torch.sqrt(f1 * f1 + f2 * f2 + 0.25 / (n1 * n2)))
    Y = torch.empty_like(Om)
    for a in range(0, ell, 50):
        F = torch.fft.rfft2(Om[a:a + 50].float())
        Y[a:a + 50] = torch.fft.irfft2(F * mult.float(), s=(n1, n2)).to(torch.bfloat16)
    return Om, Y


def prepare(case: dict, seed: int) -> dict:
    c = dict(case)
    kind, n1, n2 = c["kind"], c["n1"], c["n2"]
    ctx = api.Context(torch.cuda.current_device())
    st = dict(case=c, ctx=ctx)
    dt = DT[c.get("dtype", "f32")]
    if kind in ("normal", "pair", "sketch", "solve"):
        st["op"] = _operator(ctx, c)
    if kind in ("normal", "pair"):
        st["x"] = _phantoms(c["batch"], n1, n2, seed).to(dt)
        if kind == "pair":
            st["x"].requires_grad_(True)
            st["gy"] = torch.randn((c["batch"],) + st["op"].meas_shape, generator=_gen(seed + 1), device="cuda",
                                   dtype=torch.float64).to(dt)
    elif kind == "sketch":
        st["seed"] = int(seed)
        st["out"] = tuple(torch.empty((c["ell"], n1, n2), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    elif kind == "factor":
        st["Om"], st["Y"] = _sketch_pair(c, seed)
        st["pc"] = api.Precond(ctx, n1 * n2, c["ell"], torch.bfloat16)
        st["z"] = _phantoms(c["batch"], n1, n2, seed + 1).float()
    elif kind in ("prox", "solve", "unroll"):
        st["pc"] = None
        if c["ell"]:
            U, S = _factor_given(c)
            st["pc"] = api.Precond(ctx, n1 * n2, c["ell"], U.dtype)
            st["pc"].import_factor(U, S, 0.0, c.get("sqrt_shift", True))
        if kind == "prox":
            s = _phantoms(1, n1, n2, seed)[0]
            st["s"] = (s + 0.02 * torch.randn(s.shape, generator=_gen(seed + 1), device="cuda",
                                              dtype=torch.float64)).float()
        elif kind == "solve":
            st["solver"] = api.Solver(ctx, st["op"], _data(c, seed).to(dt), c["reg"], c["lam"], pc=st["pc"],
                                      fit=c["fit"], huber_delta=_huber_delta(c), alpha=_alpha(c), n_inner=20)
        else:
            st["op"] = _operator(ctx, dict(c, op="blur"))
            st["unroll"] = api.Unroll(ctx, st["op"], c["lam"], 0.9, c["K"], n_inner=20, ckpt_every=5, pc=st["pc"])
            st["y"] = _data(dict(c, op="blur"), seed).float()
            st["lam"] = torch.tensor(c["lam"], requires_grad=True)
            st["h"] = torch.from_numpy(_gauss_kernel(c["k"], c["sigma"])).float().requires_grad_(True)
            st["xbar"] = torch.randn((n1, n2), generator=_gen(seed + 2), device="cuda")
    return st


# ------------------------------------------------------------------ run ----

def run(st: dict):
    c, ctx = st["case"], st["ctx"]
    kind = c["kind"]
    if kind == "normal":
        return api.op_normal(st["op"], st["x"])
    if kind == "pair":
        y = autograd.op_apply(st["op"], st["x"])
        gx, = torch.autograd.grad(y, st["x"], st["gy"])
        return y, gx
    if kind == "sketch":
        return api.nys_sketch(ctx, st["op"], c["ell"], st["seed"], store_dtype=torch.bfloat16, out=st["out"])
    if kind == "factor":
        # U itself is fixed only up to signs and rotations within close
        # eigenvalues; S_hat and P^{-1} z are what it is for
        pc = api.nys_factor(ctx, st["Om"], st["Y"], EPS32, pc=st["pc"])
        return pc.S_hat, api.precond_apply(ctx, pc, st["z"], True)
    if kind == "prox":
        return api.prox_mixed(ctx, st["pc"], c["reg"], c["lam_bar"], c["n_inner"], st["s"])
    if kind == "solve":
        st["solver"].restart(False)
        st["solver"].step(c["iters"])
        return st["solver"].x()
    x = autograd.unrolled_solve(st["unroll"], st["y"], st["lam"], st["h"])
    gl, gh = torch.autograd.grad(x, (st["lam"], st["h"]), st["xbar"])
    return x, gl, gh


# ----------------------------------------------------------------- work ----

def _op_flops(c: dict) -> float:
    """One application of A (or of A^T): two fused multiply-adds per interpolation sample that falls inside the
    image, or per tap of the two one-dimensional passes."""
    N = c["n1"] * c["n2"]
    if c["op"] == "radon":
        cover = min(1.0, c["n_bins"] / max(c["n1"], c["n2"]))
        return 4.0 * 0.9 * N * c["n_angles"] * cover
    if c["op"] == "fanbeam":
        cover = min(1.0, c["n_bins"] * c["src"] / c["det"] / max(c["n1"], c["n2"]))
        return 4.0 * 0.9 * N * c["n_angles"] * cover * c["det"] / c["src"]
    return 4.0 * c["k"] * N


def _meas(c: dict) -> int:
    if c["op"] in ("radon", "fanbeam"):
        return c["n_angles"] * c["n_bins"]
    return c["n1"] * c["n2"] // c.get("decim", 1) ** 2


def work(case: dict) -> dict:
    c = case
    N, kind = c["n1"] * c["n2"], c["kind"]
    es = 8 if c.get("dtype") == "f64" else 4
    ub = 8 if c.get("dtype") == "f64" else 2
    if kind == "normal":
        return dict(bytes=2.0 * es * N * c["batch"], flops=2.0 * c["batch"] * _op_flops(c))
    if kind == "pair":
        return dict(bytes=2.0 * es * (N + _meas(c)) * c["batch"], flops=2.0 * c["batch"] * _op_flops(c))
    if kind == "sketch":
        return dict(bytes=4.0 * N * c["ell"], flops=2.0 * c["ell"] * _op_flops(c))
    if kind == "factor":
        return dict(bytes=6.0 * N * c["ell"] + 8.0 * N * c["batch"],
                    flops=N * (5.0 * c["ell"] ** 2 + 4.0 * c["ell"] * c["batch"]))
    G = 3 if c.get("reg") == "hs" else 2
    # one dual step: U once, the dual variables and the image read and written
    step_bytes = ub * c["ell"] * N + es * N * (2 * G + 2)
    step_flops = N * (4.0 * c["ell"] + 20.0 * G)
    if kind == "prox":
        return dict(bytes=es * N * (2.0 + G) + c["n_inner"] * step_bytes, flops=c["n_inner"] * step_flops)
    if kind == "solve":
        if c["reg"] == "wavelet":
            return dict(bytes=c["iters"] * (es * 8.0 * N + 2 * ub * c["ell"] * N),
                        flops=c["iters"] * (2 * _op_flops(c) + 8.0 * c["ell"] * N))
        # a strongly weighted dual stops after a few steps: two are counted for CT, all twenty otherwise
        steps = 2 if c["op"] == "radon" else 20
        return dict(bytes=c["iters"] * (es * 8.0 * N + (steps + 1) * step_bytes),
                    flops=c["iters"] * (2 * _op_flops(c) + (steps + 1) * step_flops))
    # unroll: the forward, its recomputation and the reverse pass
    f = c["K"] * (2 * _op_flops(dict(c, op="blur")) + 21 * step_flops)
    return dict(bytes=3.0 * c["K"] * 21 * step_bytes, flops=3.0 * f + 2.0 * c["K"] * 2 * c["k"] ** 2 * N)


# -------------------------------------------- the same results in 64 bits --

def _otf(h: np.ndarray, n1: int, n2: int) -> torch.Tensor:
    """Transfer function of the periodic correlation with h: fft2(H x) = otf * fft2(x)."""
    return _otf_of(torch.from_numpy(h).cuda(), n1, n2)


def _otf_of(h: torch.Tensor, n1: int, n2: int) -> torch.Tensor:
    kh, kw = h.shape
    i = (torch.arange(kh, device=h.device) - (kh - 1) // 2) % n1
    j = (torch.arange(kw, device=h.device) - (kw - 1) // 2) % n2
    z = torch.zeros((n1, n2), dtype=h.dtype, device=h.device)
    z = z.index_put((i[:, None].expand(kh, kw), j[None, :].expand(kh, kw)), h, accumulate=True)
    return torch.fft.fft2(z).conj()


def _filter(x: torch.Tensor, otf: torch.Tensor) -> torch.Tensor:
    return torch.fft.ifft2(torch.fft.fft2(x) * otf).real


class _Exact:
    """A case's operator in float64: periodic blur by FFT, Joseph's ray transform ray by ray."""

    def __init__(self, c: dict, h: torch.Tensor | None = None):
        self.c, self.n1, self.n2 = c, c["n1"], c["n2"]
        self.decim = c.get("decim", 1)
        if c["op"] in ("blur", "blur_decim"):
            self.otf = _otf_of(h, self.n1, self.n2) if h is not None else _otf(_gauss_kernel(c["k"], c["sigma"]),
                                                                               self.n1, self.n2)

    def _rays(self, a: int):
        """(row-step?, bins, position of every (line, bin), weight of every bin) of angle a."""
        c, n1, n2 = self.c, self.n1, self.n2
        c1, c2, A, B = (n1 - 1) / 2.0, (n2 - 1) / 2.0, c["n_angles"], c["n_bins"]
        t = np.arange(B, dtype=np.float64) - (B - 1) / 2.0
        if c["op"] == "radon":
            th = a * math.pi / A
            cs, sn = math.cos(th), math.sin(th)
            if abs(cs) + 1e-9 >= abs(sn):
                u = (t[None, :] - (np.arange(n1)[:, None] - c1) * sn) / cs + c2
                yield True, np.arange(B), u, np.full(B, 1.0 / abs(cs))
            else:
                u = (t[None, :] - (np.arange(n2)[:, None] - c2) * cs) / sn + c1
                yield False, np.arange(B), u, np.full(B, 1.0 / abs(sn))
            return
        th = a * 2.0 * math.pi / A
        cs, sn = math.cos(th), math.sin(th)
        sx, sy = c["src"] * cs, c["src"] * sn
        dx, dy = -c["det"] * cs - t * sn, -c["det"] * sn + t * cs
        nd = np.hypot(dx, dy)
        row = np.abs(dy) >= np.abs(dx)
        if row.any():
            m = np.nonzero(row)[0]
            b = dx[m] / dy[m]
            yield True, m, (sx - (c1 + sy) * b + c2)[None, :] + b[None, :] * np.arange(n1)[:, None], nd[m] / np.abs(dy[m])
        if not row.all():
            m = np.nonzero(~row)[0]
            b = dy[m] / dx[m]
            yield False, m, (sy - (c2 + sx) * b + c1)[None, :] + b[None, :] * np.arange(n2)[:, None], nd[m] / np.abs(dx[m])

    def _samples(self, a: int):
        """Per group of rays: bins, row-step?, flat index pairs into the padded lines, weights."""
        for row, m, u, w in self._rays(a):
            u = torch.from_numpy(u).cuda()
            na = self.n2 if row else self.n1
            lo = torch.floor(u)
            f = u - lo
            e = lo.clamp(-2, na).long() + 1          # padded by one zero on the left, two on the right
            line = torch.arange(u.shape[0], device="cuda")[:, None] * (na + 3)
            e0 = torch.where(e < 0, na + 1, e)
            yield torch.from_numpy(m).cuda(), row, (line + e0).reshape(-1), (line + e + 1).reshape(-1), \
                f, torch.from_numpy(w).cuda()

    def _lines(self, x: torch.Tensor, row: bool) -> torch.Tensor:
        v = x if row else x.transpose(-1, -2)
        return torch.nn.functional.pad(v, (1, 2)).reshape(x.shape[0], -1).T.contiguous()

    def apply(self, x: torch.Tensor) -> torch.Tensor:
        c = self.c
        if c["op"] in ("blur", "blur_decim"):
            return _filter(x, self.otf)[..., ::self.decim, ::self.decim]
        b = x.shape[0]
        out = torch.zeros((c["n_angles"], c["n_bins"], b), dtype=torch.float64, device="cuda")
        by = {True: self._lines(x, True), False: self._lines(x, False)}
        for a in range(c["n_angles"]):
            for m, row, i0, i1, f, w in self._samples(a):
                v = by[row]
                f3 = f[..., None]
                s = torch.lerp(v[i0].reshape(f.shape + (b,)), v[i1].reshape(f.shape + (b,)), f3).sum(0)
                out[a, m] = w[:, None] * s
        return out.permute(2, 0, 1).contiguous()

    def adjoint(self, y: torch.Tensor) -> torch.Tensor:
        c, n1, n2 = self.c, self.n1, self.n2
        if c["op"] in ("blur", "blur_decim"):
            z = y
            if self.decim > 1:
                z = torch.zeros(y.shape[:-2] + (n1, n2), dtype=y.dtype, device=y.device)
                z[..., ::self.decim, ::self.decim] = y
            return _filter(z, self.otf.conj())
        b = y.shape[0]
        acc = {True: torch.zeros((n1 * (n2 + 3), b), dtype=torch.float64, device="cuda"),
               False: torch.zeros((n2 * (n1 + 3), b), dtype=torch.float64, device="cuda")}
        yt = y.permute(1, 2, 0).contiguous()
        for a in range(c["n_angles"]):
            for m, row, i0, i1, f, w in self._samples(a):
                s = (w[:, None] * yt[a, m])[None]
                hi = f[..., None] * s
                acc[row].index_add_(0, i1, hi.reshape(-1, b))
                acc[row].index_add_(0, i0, (s - hi).reshape(-1, b))
        r = acc[True].T.reshape(b, n1, n2 + 3)[:, :, 1:n2 + 1]
        t = acc[False].T.reshape(b, n2, n1 + 3)[:, :, 1:n1 + 1].transpose(1, 2)
        return (r + t).contiguous()

    def normal(self, x: torch.Tensor) -> torch.Tensor:
        return self.adjoint(self.apply(x))


def _exact_inverse(U: torch.Tensor, S: torch.Tensor, sqrt_shift: bool):
    """P^{-1} for P = I + U^T diag(d) U (rows of U), and the rows sqrt(d) U."""
    s_ref = torch.sqrt(S[-1]) if sqrt_shift else S[-1]
    d = torch.clamp(S / s_ref - 1.0, min=0.0)
    Ub = torch.sqrt(d)[:, None] * U
    K = torch.eye(U.shape[0], dtype=U.dtype, device=U.device) + Ub @ Ub.T
    L = torch.linalg.cholesky(K)

    def inv(z):
        f = z.reshape(-1, U.shape[1])
        return (f - torch.cholesky_solve(Ub @ f.T, L).T @ Ub).reshape(z.shape)
    return inv, Ub


def _roll(x, di, dj):
    return torch.roll(x, (-di, -dj), (-2, -1))


def _diff(x, reg):
    if reg in ("tv", "isotv"):
        return torch.stack([x - _roll(x, -1, 0), x - _roll(x, 0, -1)])
    return torch.stack([_roll(x, -1, 0) - 2 * x + _roll(x, 1, 0),
                        0.25 * (_roll(x, 1, 1) - _roll(x, 1, -1) - _roll(x, -1, 1) + _roll(x, -1, -1)),
                        _roll(x, 0, -1) - 2 * x + _roll(x, 0, 1)])


def _diff_t(q, reg):
    if reg in ("tv", "isotv"):
        return (q[0] - _roll(q[0], 1, 0)) + (q[1] - _roll(q[1], 0, 1))
    a, b, c = q
    return (_roll(a, -1, 0) - 2 * a + _roll(a, 1, 0)) + (_roll(c, 0, -1) - 2 * c + _roll(c, 0, 1)) \
        + 0.5 * (_roll(b, 1, 1) - _roll(b, 1, -1) - _roll(b, -1, 1) + _roll(b, -1, -1))


def _ball(q, reg):
    """Projection onto the dual unit ball, pixel by pixel."""
    if reg == "tv":
        return q.clamp(-1.0, 1.0)
    if reg == "isotv":
        return q / torch.sqrt(q[0] ** 2 + q[1] ** 2).clamp(min=1.0)
    a, b, c = q
    m, h = 0.5 * (a + c), 0.5 * (a - c)
    r = torch.sqrt(h * h + b * b)
    l1, l2 = (m + r).clamp(-1.0, 1.0), (m - r).clamp(-1.0, 1.0)
    mp, dp = 0.5 * (l1 + l2), 0.5 * (l1 - l2)
    safe = torch.where(r > 0, r, torch.ones_like(r))
    co, si = torch.where(r > 0, h / safe, torch.ones_like(r)), torch.where(r > 0, b / safe, torch.zeros_like(r))
    return torch.stack([mp + dp * co, dp * si, mp - dp * co])


def _exact_prox(s, reg, lb, inv, n_inner, Q):
    step, t = 1.0 / (lb * (8.0 if reg in ("tv", "isotv") else 32.0)), 1.0
    prev = R = Q
    for _ in range(n_inner):
        Q = _ball(R + step * _diff(s - lb * inv(_diff_t(R, reg)), reg), reg)
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        R = Q + ((t - 1.0) / tn) * (Q - prev)
        prev, t = Q, tn
    return s - lb * inv(_diff_t(prev, reg)), prev


def _haar(n: int, levels: int) -> torch.Tensor:
    """One axis of one pyramid level at a time needs the two-dimensional transform; this is its level matrix."""
    w = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    i = torch.arange(n // 2, device="cuda")
    r = 1.0 / math.sqrt(2.0)
    w[i, 2 * i], w[i, 2 * i + 1] = r, r
    w[n // 2 + i, 2 * i], w[n // 2 + i, 2 * i + 1] = r, -r
    return w


def _haar2(x, levels, inverse=False):
    x = x.clone()
    for lev in (reversed(range(levels)) if inverse else range(levels)):
        h, w = x.shape[-2] >> lev, x.shape[-1] >> lev
        a, b = _haar(h, 1), _haar(w, 1)
        blk = x[..., :h, :w]
        x[..., :h, :w] = a.T @ blk @ b if inverse else a @ blk @ b.T
    return x


def _exact_soft_prox(s, tau, Ub):
    """argmin 1/2 ||x - s||_P^2 + tau ||x||_1, P = I + Ub^T Ub: semi-smooth Newton on the r unknowns."""
    f = s.reshape(-1)

    def soft(z):
        return torch.sign(z) * torch.clamp(z.abs() - tau, min=0.0)

    g = torch.zeros(Ub.shape[0], dtype=torch.float64, device="cuda")
    for _ in range(60):
        z = f - g @ Ub
        F = Ub @ (f - soft(z)) + g
        if float(F.norm()) < 1e-14 * (1.0 + float((Ub @ f).norm())):
            break
        J = torch.eye(Ub.shape[0], dtype=torch.float64, device="cuda") + (Ub * (z.abs() > tau)) @ Ub.T
        g = g - torch.linalg.solve(J, F)
    return soft(f - g @ Ub).reshape(s.shape)


def _exact_solve(c, seed):
    A = _Exact(c)
    dt = DT[c.get("dtype", "f32")]
    y = _data(c, seed).to(dt).double()
    inv, Ub = (lambda z: z), None
    if c["ell"]:
        U, S = _factor_given(c)
        inv, Ub = _exact_inverse(U.double(), S, c["sqrt_shift"])
    alpha, delta, wav = _alpha(c), _huber_delta(c), c["reg"] == "wavelet"
    x = torch.zeros((c["n1"], c["n2"]), dtype=torch.float64, device="cuda")
    u, t = x, 1.0
    Q = torch.zeros((3 if c["reg"] == "hs" else 2,) + x.shape, dtype=torch.float64, device="cuda")
    for _ in range(c["iters"]):
        r = A.apply((_haar2(u, 3, True) if wav else u)[None])[0] - y
        if c["fit"] == "huber":
            r = r.clamp(-delta, delta)
        g = A.adjoint(r[None])[0]
        s = u - alpha * inv(_haar2(g, 3) if wav else g)
        if wav:
            xn = _exact_soft_prox(s, alpha * c["lam"], Ub)
        else:
            xn, Q = _exact_prox(s, c["reg"], alpha * c["lam"], inv, 20, Q)
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        u = xn + ((t - 1.0) / tn) * (xn - x)
        x, t = xn, tn
    return _haar2(x, 3, True) if wav else x


def _exact_unroll(c, seed):
    c = dict(c, op="blur")
    y = _data(c, seed).float().double()
    U, S = _factor_given(c)
    inv, _ = _exact_inverse(U.double(), S, True)
    lam = torch.tensor(float(torch.tensor(c["lam"])), dtype=torch.float64, requires_grad=True)
    h = torch.from_numpy(_gauss_kernel(c["k"], c["sigma"])).float().double().cuda().requires_grad_(True)
    xbar = torch.randn((c["n1"], c["n2"]), generator=_gen(seed + 2), device="cuda").double()
    A = _Exact(c, h)
    x = u = torch.zeros_like(y)
    Q = torch.zeros((2,) + y.shape, dtype=torch.float64, device="cuda")
    t = 1.0
    for _ in range(c["K"]):
        s = u - 0.9 * inv(A.adjoint(A.apply(u) - y))
        xn, Q = _exact_prox(s, "tv", 0.9 * lam, inv, 20, Q)
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        u = xn + ((t - 1.0) / tn) * (xn - x)
        x, t = xn, tn
    gl, gh = torch.autograd.grad(x, (lam, h), xbar)
    return x.detach(), gl, gh


def _philox_gauss(total: int, seed: int) -> torch.Tensor:
    """The first `total` Gaussians of the library's probe generator (Philox4x32-10, Box-Muller), float64."""
    M = 0xFFFFFFFF
    b = torch.arange((total + 3) // 4, device="cuda", dtype=torch.int64)
    c = [b & M, b >> 32, torch.zeros_like(b), torch.zeros_like(b)]
    k0, k1 = seed & M, seed >> 32

    def mul(m, v):                                   # (high, low) words of the 64-bit product
        p, q = m * (v & 0xFFFF), m * (v >> 16)
        return (q + (p >> 16)) >> 16, (p + ((q & 0xFFFF) << 16)) & M
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    u = [((w >> 9).double() + 0.5) * 2.0 ** -23 for w in c]
    z = []
    for a, p in ((u[0], u[1]), (u[2], u[3])):
        rho = torch.sqrt(-2.0 * torch.log(a))
        z += [rho * torch.cos(2 * math.pi * p), rho * torch.sin(2 * math.pi * p)]
    return torch.stack(z, 1).reshape(-1)[:total]


def _exact_factor(c, seed):
    Om, Y = _sketch_pair(c, seed)
    ell = c["ell"]
    Om, Y = Om.reshape(ell, -1).double(), Y.reshape(ell, -1).double()
    v = EPS32 * float(Om.norm())
    for _ in range(9):
        Yv = Y + v * Om
        M = Om @ Yv.T
        C, info = torch.linalg.cholesky_ex(0.5 * (M + M.T))
        if int(info) == 0:
            break
        v *= 10.0
    B = torch.linalg.solve_triangular(C, Yv, upper=False)          # B^T
    _, R = torch.linalg.qr(B.T)
    _, sv, Vh = torch.linalg.svd(R)
    S = torch.clamp(sv * sv - v, min=0.0)
    U = (Vh @ B) / sv[:, None]                                     # rows: left singular vectors of B^T's transpose
    inv, _ = _exact_inverse(U, S, True)
    return S, inv(_phantoms(c["batch"], c["n1"], c["n2"], seed + 1).float().double())


def exact(case: dict, seed: int):
    c = dict(case)
    kind, dt = c["kind"], DT[c.get("dtype", "f32")]
    if kind in ("normal", "pair"):
        A = _Exact(c)
        x = _phantoms(c["batch"], c["n1"], c["n2"], seed).to(dt).double()
        if kind == "normal":
            return A.normal(x)
        y = A.apply(x)
        gy = torch.randn(y.shape, generator=_gen(seed + 1), device="cuda", dtype=torch.float64).to(dt).double()
        return y, A.adjoint(gy)
    if kind == "sketch":
        N = c["n1"] * c["n2"]
        Om = _philox_gauss(N * c["ell"], seed).reshape(c["ell"], c["n1"], c["n2"])
        A = _Exact(c)
        Y = torch.empty_like(Om)
        for a in range(0, c["ell"], 100):                          # A acts on the stored Omega
            Y[a:a + 100] = A.normal(Om[a:a + 100].to(torch.bfloat16).double())
        return Om, Y
    if kind == "factor":
        return _exact_factor(c, seed)
    if kind == "prox":
        s = _phantoms(1, c["n1"], c["n2"], seed)[0]
        s = (s + 0.02 * torch.randn(s.shape, generator=_gen(seed + 1), device="cuda",
                                    dtype=torch.float64)).float().double()
        inv = lambda z: z                                          # noqa: E731
        if c["ell"]:
            U, S = _factor_given(c)
            inv, _ = _exact_inverse(U.double(), S, c["sqrt_shift"])
        Q = torch.zeros((3 if c["reg"] == "hs" else 2,) + s.shape, dtype=torch.float64, device="cuda")
        return _exact_prox(s, c["reg"], c["lam_bar"], inv, c["n_inner"], Q)
    if kind == "solve":
        return _exact_solve(c, seed)
    return _exact_unroll(c, seed)
