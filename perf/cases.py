"""The work that a user of this framework has it do, as cases to time.

Four kinds of call, each through the package's public entry points:

* ``evaluate``: S, f and df/deps of new designs (``Solver.solve_S_grad`` for one design with host arrays, as the
  line-search optimiser calls it; ``solve_S_grad_batch`` for several, device results, as the surrogate's training data
  and multi-start runs call it).  A pass sets the designs and solves them.
* ``scan``: S alone of one design (``Solver.solve_S``), here on a channel subset of an asymmetric grid.
* ``ridges``: ``autograd.ridge_scattering``: ridge edges in, S, and by ``backward`` the gradient of a torch loss.
* ``screen`` and ``train``: the surrogate network's inference on line-search candidates, and its loss and gradients
  on a training batch.

Grids and slabs are those of ``workloads.py`` (64x100, 1024x240, 4096x260, 8192x280) and the sizes between them.
``tol`` is the refinement tolerance of the mixed precision: 1e-10 is the library's default; 1e-12 is for results that
are compared between runs or checked by differences.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_09257_gb300 import apf, autograd, surrogate, workloads

ORDERS = (-2, -1, 0, 1, 2)
TARGET = 0.18
EPS_SUB, EPS_CLAD = 2.25, 1.0
RIDGE_EPS = 13.69  # amorphous silicon


def _grid(nx, ny, nb, nt, lam, h, tol=1e-12):
    return {"nx": nx, "ny": ny, "npml_bot": nb, "npml_top": nt, "lam": lam, "h": h, "tol": tol}


TINY = _grid(64, 100, 20, 20, 16.0, 6)
MID = _grid(1024, 240, 30, 30, 20.0, 12, tol=1e-10)
LARGE = _grid(4096, 260, 30, 30, 24.0, 16, tol=1e-10)
XLARGE = _grid(8192, 280, 30, 30, 32.0, 20)


def listed():
    return [
        # the smallest grid: one call of a design loop, all latency and launches; both precisions
        {"name": "tiny_mixed", "kind": "evaluate", "precision": "mixed", "designs": 1, **TINY},
        {"name": "tiny_fp64", "kind": "evaluate", "precision": "fp64", "designs": 1, **TINY},
        # an irregular problem: odd slab height, unequal PMLs, every third input order; S without a gradient
        {"name": "scan_512_subset", "kind": "scan", "precision": "mixed", "designs": 1, "in_step": 3,
         **_grid(512, 171, 17, 25, 13.7, 7)},
        # one line-search trial of the optimiser on the 103-channel metasurface, mixed and float64
        {"name": "mid_mixed", "kind": "evaluate", "precision": "mixed", "designs": 1, **MID},
        {"name": "mid_fp64", "kind": "evaluate", "precision": "fp64", "designs": 1, **MID},
        # training data for the surrogate, or 16 starts of an optimisation: the largest batch a call takes
        {"name": "mid_mixed_16", "kind": "evaluate", "precision": "mixed", "designs": 16, **MID},
        # high-contrast silicon ridges through torch autograd
        {"name": "ridges_2048", "kind": "ridges", "precision": "mixed", "ridges": 73,
         **_grid(2048, 250, 30, 30, 22.0, 9)},
        # the precision study's grid (343 channels), one design and eight per call
        {"name": "large_mixed", "kind": "evaluate", "precision": "mixed", "designs": 1, **LARGE},
        {"name": "large_mixed_8", "kind": "evaluate", "precision": "mixed", "designs": 8, **LARGE},
        # the largest grid (513 channels)
        {"name": "xlarge_mixed", "kind": "evaluate", "precision": "mixed", "designs": 1, **XLARGE},
        # the surrogate: 64 candidates of one line search; the loss and gradients of one training batch of 128
        {"name": "screen_64", "kind": "screen", "batch": 64, "n": 1024, "in_ch": 12, "width": 48, "modes": 64,
         "layers": 4, "n_out": 5},
        {"name": "train_128", "kind": "train", "batch": 128, "n": 1024, "in_ch": 12, "width": 48, "modes": 64,
         "layers": 4, "n_out": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["evaluate", "evaluate", "evaluate", "fp64", "scan", "ridges", "screen", "train"])
    if kind in ("screen", "train"):
        n = 64 * rng.randint(2, 16)
        return {"kind": kind, "batch": _log_int(rng, 1, 256), "n": n, "in_ch": rng.randint(1, 20),
                "width": rng.randint(12, 54), "modes": rng.randint(8, min(64, n // 2)), "layers": rng.randint(2, 5),
                "n_out": rng.randint(1, 7)}
    precision = "fp64" if kind == "fp64" else "mixed"
    nx = 2 ** rng.randint(5, 10 if precision == "fp64" else 12)
    h = rng.randint(1, 16)
    nb, nt = rng.randint(10, 30), rng.randint(10, 30)
    ny = nb + nt + h + rng.randint(8, 180)
    grid = _grid(nx, ny, nb, nt, round(rng.uniform(12.0, 32.0), 1), h)
    if kind == "scan":
        return {"kind": "scan", "precision": "mixed", "designs": 1, "in_step": rng.randint(1, 4), **grid}
    if kind == "ridges":
        grid["nx"] = max(64, min(2048, nx))
        grid["lam"] = round(rng.uniform(20.0, 32.0), 1)  # over five pixels per wavelength inside the silicon
        ridges = max(1, int(grid["nx"] / (2 * rng.uniform(0.6, 0.9) * grid["lam"])))
        return {"kind": "ridges", "precision": "mixed", "ridges": ridges, **grid}
    designs = 1 if precision == "fp64" else rng.choice([1, 1, rng.randint(2, 8 if nx == 4096 else 16)])
    return {"kind": "evaluate", "precision": precision, "designs": designs, **grid}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _designs(case, seed):
    """Slab permittivities: independent pixels in [1, 3] on grids up to 128 (up to 4 on the 64-pixel one), the
    filtered-threshold pattern above."""
    h, n = case["h"], case["nx"]
    seeds = [1000 * seed + b for b in range(case["designs"])]
    if n > 128:
        return [workloads.filtered_threshold_eps(h, n, s) for s in seeds]
    return [workloads.iid_eps(h, n, s, 1.0, 4.0 if n == 64 and case["lam"] >= 16 else 3.0) for s in seeds]


def _edges(case, seed):
    return workloads.ridge_edges(case["nx"], case["ridges"], seed, mirror=True)


def _orders_in(case):
    """Every in_step-th propagating order as inputs (None: all of them)."""
    step = case.get("in_step", 1)
    return None if step == 1 else [int(m) for m in _propagating(case, EPS_CLAD)[::step]]


def _solver(case):
    s = apf.Solver(device=0, precision=case["precision"])
    s.set_grid(case["nx"], case["ny"], case["npml_bot"], case["npml_top"], case["lam"])
    s.set_refinement(case["tol"], 40)
    return s


def _params(case, seed):
    """Surrogate parameters of a network in training: the initial distribution, with non-zero biases."""
    rng = np.random.default_rng(seed)
    c, m, layers = case["width"], case["modes"], case["layers"]
    parts = [rng.normal(size=(c, case["in_ch"])) / math.sqrt(case["in_ch"]), 0.05 * rng.normal(size=c),
             rng.uniform(-1, 1, size=(layers, c, c, m)) / c, rng.uniform(-1, 1, size=(layers, c, c, m)) / c,
             rng.normal(size=(layers, c, c)) / math.sqrt(c), 0.05 * rng.normal(size=(layers, c)),
             rng.normal(size=(case["n_out"], c)) / math.sqrt(c), 0.05 * rng.normal(size=case["n_out"])]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _slabs(case, seed):
    """Candidate slabs on the device, float32: grey designs in [1, 2.25], smooth along the period."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.randn(case["batch"], case["in_ch"], case["n"], device="cuda", generator=g)
    u = (u + u.roll(1, -1) + u.roll(-1, -1) + u.roll(2, -1) + u.roll(-2, -1)) / 5 ** 0.5
    return torch.clamp(1.625 + 0.8 * u, 1.0, 2.25).contiguous()


def _targets(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    return 0.3 * torch.rand(case["batch"], case["n_out"], device="cuda", generator=g)


def prepare(case, seed):
    st = {"case": case}
    if case["kind"] in ("screen", "train"):
        st["net"] = surrogate.Surrogate(n=case["n"], in_ch=case["in_ch"], width=case["width"], modes=case["modes"],
                                        layers=case["layers"], n_out=case["n_out"], max_batch=256)
        st["net"].set_params(_params(case, seed))
        st["x"], st["t"] = _slabs(case, seed), _targets(case, seed)
        return st
    if case["kind"] == "ridges":
        e = _edges(case, seed)
        s = _solver(case)
        s.set_ridges(e, case["h"], RIDGE_EPS, 1.0, EPS_SUB, EPS_CLAD, eps_out=False)
        s.set_channels()
        mi, mo = s.channels()
        st.update(solver=s, edges=torch.as_tensor(e, device="cuda"),
                  mask=autograd.relative_order_mask(mi, mo, ORDERS, device="cuda"))
        return st
    st["eps"] = _designs(case, seed)
    st["solvers"] = []
    for e in st["eps"]:
        s = _solver(case)
        s.set_eps(e, EPS_SUB, EPS_CLAD)
        s.set_channels(_orders_in(case), None)
        st["solvers"].append(s)
    if case["designs"] > 1:
        mi, mo = st["solvers"][0].channels()
        st["S"] = [torch.empty((len(mo), len(mi)), dtype=torch.complex128, device="cuda") for _ in st["eps"]]
        st["g"] = [torch.empty((case["h"], case["nx"]), dtype=torch.float64, device="cuda") for _ in st["eps"]]
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "screen":
        return {"y": st["net"].forward(st["x"])}
    if kind == "train":
        g, loss = st["net"].gradients(st["x"], st["t"])
        return {"loss": loss, "grads": g}
    if kind == "ridges":
        e = st["edges"].clone().requires_grad_(True)
        S = autograd.ridge_scattering(e, st["solver"], case["h"], RIDGE_EPS, 1.0, EPS_SUB, EPS_CLAD)
        f = autograd.splitter_loss(S, st["mask"], TARGET)
        f.backward()
        return {"S": S.detach(), "f": f.detach(), "grad": e.grad}
    for s, e in zip(st["solvers"], st["eps"]):
        s.set_eps(e, EPS_SUB, EPS_CLAD)
    if kind == "scan":
        return {"S": st["solvers"][0].solve_S()}
    if case["designs"] == 1:
        S, f, g = st["solvers"][0].solve_S_grad("splitter", ORDERS, TARGET)
        return {"S": S, "f": f, "grad": g}
    S, f, g = apf.solve_S_grad_batch(st["solvers"], "splitter", ORDERS, TARGET, out_S=st["S"], out_grad=st["g"])
    return {"S": S, "f": f, "grad": g}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] in ("screen", "train"):
        b, n, c, m = case["batch"], case["n"], case["width"], case["modes"]
        # lift, and per layer: n-to-m analysis, mixing, m-to-n synthesis (as transforms), the position-wise map
        fft = 5.0 * n * math.log2(n)
        fwd = 2.0 * b * n * c * case["in_ch"] + case["layers"] * b * (2 * c * fft + 8.0 * c * c * m + 2.0 * c * c * n)
        nparam = c * case["in_ch"] + case["layers"] * c * c * (2 * m + 1)
        if case["kind"] == "screen":
            return {"bytes": 4.0 * b * (case["in_ch"] * n + case["n_out"]) + 2.0 * nparam, "flops": fwd}
        return {"bytes": 4.0 * b * case["in_ch"] * n + 6.0 * nparam, "flops": 3.0 * fwd}
    n, h, d = case["nx"], case["h"], case.get("designs", 1)
    n_out = len(_propagating(case, EPS_CLAD))
    n_in = -(-n_out // case.get("in_step", 1))
    # one complex multiply-add = 8 flops; a complex-symmetric n x n inverse takes n^3 / 2 of them
    flops = 4.0 * h * n ** 3 + 8.0 * n * n * ((h - 1) * n_in + h * n_in)
    size = 8.0 * n * h + 16.0 * n_in * n_out
    if case["kind"] != "scan":
        flops += 8.0 * n * n * h * n_out + 8.0 * h * n * n_in * n_out
        size += 8.0 * n * h
    return {"bytes": d * size, "flops": d * flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain numpy and torch
# ---------------------------------------------------------------------------
def _propagating(case, eps):
    n, k = case["nx"], 2 * math.pi / case["lam"]
    m = np.arange(-(n // 2), n - n // 2)
    q = k * k * eps / 4 - np.sin(math.pi * m / n) ** 2
    return m[(q > 0) & (q < 1)]


def _nu(case, m, eps):
    k = 2 * math.pi / case["lam"]
    return np.sin(2 * np.arcsin(np.sqrt(k * k * eps / 4 - np.sin(math.pi * m / case["nx"]) ** 2)))


def _outside(case):
    """Per Fourier order (in FFT order): the Schur terms of the rows below and above the slab, and the factors that
    carry the source row to the first slab row and the last slab row to the output row."""
    n, ny, nb, nt, h = (case[v] for v in ("nx", "ny", "npml_bot", "npml_top", "h"))
    k = 2 * math.pi / case["lam"]
    j0 = nb + (ny - nb - nt - h) // 2

    def s(y):
        lo, hi = nb - 0.5, ny - nt - 0.5
        depth, length, eps = (lo - y, nb, EPS_SUB) if y < lo else (y - hi, nt, EPS_CLAD) if y > hi else (0.0, 1, 1.0)
        return 1 + 1j * (-4 * math.log(1e-8) / (2 * k * math.sqrt(eps) * length)) * (depth / length) ** 3

    lam = 4 * np.sin(math.pi * np.fft.fftfreq(n)) ** 2

    def sweep(rows, eps, first, step):
        """Eliminate `rows` in order towards the slab; -> Schur term and the product of couplings over pivots from
        row `first` on."""
        pivot, carry = None, np.ones(n, complex)
        for j in rows:
            d = s(j) * (lam - k * k * eps) + 1 / s(j + 0.5) + 1 / s(j - 0.5)
            if pivot is not None:
                d = d - back * back / pivot
            pivot, back = d, 1 / s(j + 0.5 * step)
            if (j - first) * step >= 0:
                carry = carry * back / pivot
        return -back * back / pivot, carry

    bot, src = sweep(range(0, j0), EPS_SUB, nb, 1)
    top, out = sweep(range(ny - 1, j0 + h - 1, -1), EPS_CLAD, ny - nt - 1, -1)
    return bot, top, src, out


def _fields(case, eps, m_in, m_out):
    """Slab fields of all input columns and all adjoint output columns, (h, columns, nx) complex128, by block
    elimination over the slab rows, refined with 64-bit residuals until they stop falling (the elimination itself is
    in 32 bits on the larger grids)."""
    n, h, dev = case["nx"], case["h"], "cuda"
    k = 2 * math.pi / case["lam"]
    bot, top, src, out = (torch.as_tensor(v, device=dev) for v in _outside(case))
    eps = torch.as_tensor(eps, device=dev)
    d = 4 - k * k * eps
    x = torch.arange(n, device=dev)

    def wave(m, coef):
        t = (torch.as_tensor(m, device=dev)[:, None] * x[None]) % n
        ph = 2 * math.pi * t.double() / n
        return coef[:, None] * torch.complex(torch.cos(ph), torch.sin(ph)) / math.sqrt(n)

    b_in = -2j * torch.as_tensor(np.sqrt(_nu(case, m_in, EPS_SUB)), device=dev) * src[torch.as_tensor(m_in % n, device=dev)]
    w_out = torch.as_tensor(np.sqrt(_nu(case, m_out, EPS_CLAD)), device=dev) * out[torch.as_tensor(m_out % n, device=dev)]
    ni, nc = len(m_in), len(m_in) + len(m_out)
    R = torch.zeros(h, nc, n, dtype=torch.complex128, device=dev)
    R[0, :ni] += wave(m_in, b_in)
    R[h - 1, ni:] += wave(-m_out, w_out)

    def residual(E):
        r = R - d[:, None, :] * E + E.roll(1, -1) + E.roll(-1, -1)
        r[1:] += E[:-1]
        r[:-1] += E[1:]
        r[0] -= torch.fft.ifft(torch.fft.fft(E[0]) * bot)
        r[-1] -= torch.fft.ifft(torch.fft.fft(E[-1]) * top)
        return r

    low = torch.complex128 if n <= 1024 else torch.complex64
    shift = (x[:, None] - x[None, :]) % n
    cb, ct = torch.fft.ifft(bot), torch.fft.ifft(top)
    G = []
    for j in range(h):
        X = torch.zeros(n, n, dtype=torch.complex128, device=dev)
        X[x, x] += d[j]
        X[x, (x + 1) % n] -= 1
        X[x, (x - 1) % n] -= 1
        if j == 0:
            X += cb[shift]
        if j == h - 1:
            X += ct[shift]
        X = X.to(low)
        if G:
            X -= G[-1]
        G.append(torch.linalg.inv(X))
        del X

    def solve(r):
        y = [r[0].to(low)]
        for j in range(1, h):
            y.append(r[j].to(low) + y[-1] @ G[j - 1].T)
        e = [None] * h
        e[-1] = y[-1] @ G[-1].T
        for j in range(h - 2, -1, -1):
            e[j] = (y[j] + e[j + 1]) @ G[j].T
        return torch.stack(e).to(torch.complex128)

    E, best = torch.zeros_like(R), math.inf
    for _ in range(12):
        r = residual(E)
        now = float(torch.linalg.norm(r))
        if now > 0.5 * best:
            break
        best = now
        E = E + solve(r)
    return E, w_out


def _exact_solve(case, eps, m_in, m_out, want_grad):
    E, w_out = _fields(case, eps, m_in, m_out)
    n, h, ni = case["nx"], case["h"], len(m_in)
    spec = torch.fft.fft(E[h - 1, :ni]) / math.sqrt(n)
    S = (w_out[:, None] * spec[:, torch.as_tensor(m_out % n, device="cuda")].T).contiguous()
    if not want_grad:
        return S, None, None
    hit = np.isin(m_out[:, None] - m_in[None, :], ORDERS)
    hit = torch.as_tensor(hit, device="cuda")
    p = S.abs() ** 2
    f = torch.where(hit, (p - TARGET) ** 2, 0.0).sum()
    gam = torch.where(hit, 2 * (p - TARGET), 0.0) * S.conj()
    k = 2 * math.pi / case["lam"]
    g = torch.stack([2 * k * k * (E[j, ni:] * (gam @ E[j, :ni])).sum(0).real for j in range(h)])
    return S, f, g


def _ridge_slab(case, edges):
    n = case["nx"]
    lo = np.arange(n) - n / 2
    fill = np.zeros(n)
    for a, b in edges.reshape(-1, 2):
        for u, v in ((a, b), (-b, -a)):
            fill += np.maximum(0.0, np.minimum(v, lo + 1) - np.maximum(u, lo))
    return np.tile(1.0 + (RIDGE_EPS - 1.0) * fill, (case["h"], 1))


def _exact_net(case, seed):
    c, m, n, layers = case["width"], case["modes"], case["n"], case["layers"]
    p = torch.as_tensor(_params(case, seed), device="cuda").bfloat16().double()  # the weights are applied in bf16
    p.requires_grad_(case["kind"] == "train")
    shapes = [(c, case["in_ch"]), (c,), (layers, c, c, m), (layers, c, c, m), (layers, c, c), (layers, c),
              (case["n_out"], c), (case["n_out"],)]
    W0, b0, Wr, Wi, P, bias, Wh, bh = (t.reshape(s) for t, s in zip(p.split([math.prod(s) for s in shapes]), shapes))
    hcur = torch.einsum("oi,bix->box", W0, _slabs(case, seed).double()) + b0[:, None]
    for l in range(layers):
        X = torch.fft.rfft(hcur)[..., :m]
        Y = torch.einsum("iom,bim->bom", torch.complex(Wr[l], Wi[l]), X)
        # real part of the synthesis: sum_m w_m Re(Y_m e^{i 2 pi m x / n}), w_0 = 1/n, else 2/n
        w = torch.full((m,), 2.0 / n, dtype=torch.float64, device="cuda")
        w[0] = 1.0 / n
        full = torch.zeros(*Y.shape[:2], n, dtype=torch.complex128, device="cuda")
        full[..., :m] = Y * w
        z = (torch.fft.ifft(full) * n).real + torch.einsum("oi,bix->box", P[l], hcur) + bias[l][:, None]
        hcur = torch.nn.functional.gelu(z) if l < layers - 1 else z
    y = hcur.mean(-1) @ Wh.T + bh
    if case["kind"] == "screen":
        return {"y": y}
    loss = ((y - _targets(case, seed).double()) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach(), "grads": p.grad}


def exact(case, seed):
    if case["kind"] in ("screen", "train"):
        return _exact_net(case, seed)
    m_out = _propagating(case, EPS_CLAD)
    m_in = np.array(_orders_in(case) if case.get("in_step", 1) > 1 else m_out)
    if case["kind"] == "ridges":
        e = _edges(case, seed)
        S, f, g = _exact_solve(case, _ridge_slab(case, e), m_in, m_out, True)
        n, col = case["nx"], g.sum(0).cpu().numpy()
        sign = np.where(np.arange(len(e)) % 2 == 0, -1.0, 1.0) * (RIDGE_EPS - 1.0)
        px, pm = np.floor(e + n / 2).astype(int) % n, (np.ceil(n / 2 - e).astype(int) - 1) % n
        return {"S": S, "f": f, "grad": sign * (col[px] + col[pm])}
    out = [_exact_solve(case, e, m_in, m_out, case["kind"] == "evaluate") for e in _designs(case, seed)]
    if case["kind"] == "scan":
        return {"S": out[0][0]}
    if case["designs"] == 1:
        return {"S": out[0][0], "f": out[0][1], "grad": out[0][2]}
    return {"S": [o[0] for o in out], "f": [float(o[1]) for o in out], "grad": [o[2] for o in out]}
