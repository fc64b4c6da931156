"""Timed workloads of the library: what its users call, over the sizes they call it at.

Each case is one pass through the public entry points (operator products, refined
solves, a differentiable solve, building an operator) on seeded synthetic inputs of
the kind the repository's workloads use: standard-normal currents, the tissue-like
contrast in a centred ellipsoid, plane waves and rings of z-dipoles, 5 mm voxels at
298 MHz.  ``exact`` restates each pass with plain torch in 64 bits (uncompressed
Green's spectra, library FFTs).
"""
from __future__ import annotations

import math

import torch

import paper_1811_00484_gb300 as vie

H, FREQ = 5e-3, 298e6                   # voxel edge (m), frequency (Hz)
C0, EPS0 = 299792458.0, 8.8541878128e-12
K0 = 2.0 * math.pi * FREQ / C0
DTYPES = {"c64": torch.complex64, "c128": torch.complex128}
AXES = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))      # components xx, xy, xz, yy, yz, zz
COMP = {(a, b): c for c, ab in enumerate(AXES) for a, b in (ab, ab[::-1])}


def _case(name, kind, n, B=1, tol=1e-6, path="tucker", dtype="c64", adjoint=False):
    c = {"kind": kind, "n1": n[0], "n2": n[1], "n3": n[2], "B": B, "tol": tol, "path": path,
         "dtype": dtype, "adjoint": adjoint}
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # a product inside somebody else's loop on a small grid: latency and launches
        _case("matvec_n16", "matvec", (16, 16, 16), tol=1e-8),
        # the product of the plane-wave workload, one right-hand side
        _case("matvec_n64", "matvec", (64, 64, 64)),
        # the batch of 16 coil right-hand sides
        _case("matvec_n96_b16", "matvec", (96, 96, 96), B=16),
        # a box fitted to a body: edges that are no multiple of 16
        _case("matvec_ragged", "matvec", (50, 72, 60)),
        # the adjoint system operator on such a box with odd edges, four coils
        _case("system_adjoint_ragged_b4", "system", (90, 63, 105), B=4, adjoint=True),
        # the uncompressed operator (spectra in memory), adjoint product, two coils
        _case("adjoint_stored_n128_b2", "matvec", (128, 128, 128), B=2, path="uncompressed", adjoint=True),
        # one operator application of the memory-headline solve: eight coils at 256^3
        _case("system_n256_b8", "system", (256, 256, 256), B=8),
        # FP64 product: refinement residuals, finite-difference checks
        _case("matvec_f64_n64", "matvec", (64, 64, 64), dtype="c128"),
        # refined solves: the plane-wave workload, and four ring dipoles as one batch
        _case("solve_n64", "solve", (64, 64, 64), tol=1e-6),
        _case("solve_n96_b4", "solve", (96, 96, 96), B=4, tol=1e-6),
        # a step of an inverse problem: forward solve, misfit, adjoint solve, gradient
        _case("gradient_n40", "gradient", (40, 40, 40)),
        # a new grid: assembly, FFTs and compression of the six components
        _case("build_n64", "build", (64, 64, 64)),
    ]


def _smooth(n):
    m = 2 * n
    for p in (2, 3, 5, 7):
        while m % p == 0:
            m //= p
    return m == 1


EDGES = [n for n in range(8, 257) if _smooth(n)]


def draw(rng):
    """One more case: any of the kinds, edges over 8 .. 256 (padded edges 7-smooth), no cube in general."""
    kind = rng.choice(("matvec",) * 4 + ("system",) * 3 + ("total",) + ("solve", "gradient", "build"))
    top = {"solve": 80, "gradient": 64, "build": 96}.get(kind, 256)
    base = math.exp(rng.uniform(math.log(8), math.log(top)))
    pick = lambda: min(EDGES, key=lambda n: abs(math.log(n / min(top, max(8, base * 2 ** rng.uniform(-0.6, 0.6))))))
    n = (pick(), pick(), pick())
    op = kind in ("matvec", "system", "total")
    dtype = "c128" if op and rng.random() < 0.25 else "c64"
    path = "uncompressed" if kind != "build" and rng.random() < 0.25 else "tucker"
    room = (2 ** 27 if op else 2 ** 20) // (16 if dtype == "c128" else 1) // (n[0] * n[1] * n[2])
    B = 1 if kind in ("build", "gradient") else max(1, min(rng.choice((1, 1, 2, 3, 4, 8, 16)), room))
    tol = rng.choice((1e-4, 1e-6, 1e-6, 1e-8)) if op else 1e-6
    return _case(None, kind, n, B=B, tol=tol, path=path, dtype=dtype,
                 adjoint=kind in ("matvec", "system") and rng.random() < 0.4)


# --- inputs -------------------------------------------------------------------

def _n(case):
    return case["n1"], case["n2"], case["n3"]


def _normal(g, shape, dtype):
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda", dtype=real))


def _contrast(g, n, dtype):
    u = [((torch.arange(m, device="cuda", dtype=torch.float64) + 0.5 - 0.5 * m) / (0.5 * m)) for m in n]
    q = (u[0][:, None, None] / 0.4) ** 2 + (u[1][None, :, None] / 0.45) ** 2 + (u[2][None, None, :] / 0.5) ** 2
    r = torch.rand(2, *n, generator=g, device="cuda", dtype=torch.float64)
    chi = torch.complex(39.0 + 40.0 * r[0], -(0.3 + 0.7 * r[1]) / (2.0 * math.pi * FREQ * EPS0))
    return torch.where(q <= 1.0, chi, torch.zeros_like(chi)).to(dtype)


def _plane_wave(g, n, dtype):
    z = (torch.arange(n[2], device="cuda", dtype=torch.float64) + 0.5 - 0.5 * n[2]) * H
    amp = torch.rand(1, generator=g, device="cuda", dtype=torch.float64) + 0.5
    e = torch.zeros(1, 3, *n, dtype=torch.complex128, device="cuda")
    e[:, 0] = torch.polar(amp.expand_as(z), -K0 * z)
    return e.to(dtype)


_kept = {}                               # the operator of the grid at work, as a program keeps it


def _operator(case):
    key = (_n(case), case["tol"], case["path"])
    if key not in _kept:
        _kept.clear()
        _kept[key] = vie.Operator(_n(case), H, FREQ, case["tol"],
                                  store_uncompressed=case["path"] == "uncompressed")
    return _kept[key]


def prepare(case, seed):
    n, B, kind, dtype = _n(case), case["B"], case["kind"], DTYPES[case["dtype"]]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s = {"case": case}
    if kind == "build":
        # the first current that the new operator is applied to
        s["J"] = _normal(g, (1, 3) + n, torch.complex128)
        return s
    s["op"] = _operator(case)
    if kind in ("matvec", "system", "total"):
        s["x"] = _normal(g, (B, 3) + n, dtype)
        if kind == "system":
            s["chi"] = _contrast(g, n, dtype)
        if kind == "total":
            s["einc"] = _normal(g, (B, 3) + n, dtype)
        return s
    s["chi"] = _contrast(g, n, dtype)
    if B == 1:
        s["einc"] = _plane_wave(g, n, dtype)
    else:
        turn = float(torch.rand(1, generator=g, device="cuda"))
        src = [[0.15 * math.cos(2 * math.pi * (m + turn) / B), 0.15 * math.sin(2 * math.pi * (m + turn) / B), 0.0]
               for m in range(B)]
        s["einc"] = s["op"].incident_dipole(src, dtype=dtype)
    if kind == "gradient":
        s["target"] = 0.3 * s["einc"] + 0.05 * _normal(g, (1, 3) + n, dtype)   # the measured field
    return s


def run(state):
    case, kind, op = state["case"], state["case"]["kind"], state.get("op")
    path = case["path"]
    if kind == "matvec":
        return op.matvec_adjoint(state["x"], path=path) if case["adjoint"] else op.matvec(state["x"], path=path)
    if kind == "system":
        return op.apply_system(state["chi"], state["x"], adjoint=case["adjoint"], path=path)
    if kind == "total":
        return op.total_field(state["einc"], state["x"], path=path)
    if kind == "solve":
        return op.solve(state["chi"], state["einc"], tol=1e-8, path=path)[0]
    if kind == "gradient":
        chi = state["chi"].detach().requires_grad_(True)
        E = vie.solve_fields(op, chi, state["einc"], tol=1e-8, path=path)
        loss = (E - state["target"]).abs().square().sum()
        loss.backward()
        return {"E": E.detach(), "grad": chi.grad}
    # build: the model's ranks and singular values, and its first product
    new = vie.Operator(_n(case), H, FREQ, case["tol"])
    ranks = torch.tensor(new.info()["ranks"])
    sigma = [s for c in range(6) for s in new.export(c)[2]]
    Y = new.matvec(state["J"])
    new.close()
    return {"ranks": ranks, "sigma": sigma, "Y": Y}


# --- work ---------------------------------------------------------------------

RANK = 15                                # typical multilinear rank of a component


def _product_work(case, B):
    n, es = _n(case), 16 if case["dtype"] == "c128" else 8
    P, h = [2 * m for m in n], [m + 1 for m in n]
    nvox, npad = n[0] * n[1] * n[2], P[0] * P[1] * P[2]
    line = lambda m: 5.0 * m * math.log2(m)
    fft = 6.0 * B * (n[1] * n[2] * line(P[0]) + P[0] * n[2] * line(P[1]) + P[0] * P[1] * line(P[2]))
    flops = fft + 66.0 * B * npad
    bytes_ = 2.0 * 3 * B * nvox * es
    if case["path"] == "tucker":
        flops += 48.0 * h[0] * h[1] * RANK * (RANK + h[2])
        bytes_ += 6.0 * es * RANK * (RANK * RANK + sum(h))
    else:
        bytes_ += 6.0 * npad * es
    if case["kind"] == "system":
        bytes_ += nvox * es
    if case["kind"] == "total":
        bytes_ += 3.0 * B * nvox * es
    return bytes_, flops


def work(case):
    n, B = _n(case), case["B"]
    nvox = n[0] * n[1] * n[2]
    if case["kind"] == "build":
        P, h = [2 * m for m in n], [m + 1 for m in n]
        npad, oct_ = P[0] * P[1] * P[2], float(h[0] * h[1] * h[2])
        flops = 6.0 * (5.0 * npad * math.log2(npad) + 8.0 * oct_ * sum(h))
        return {"bytes": 6.0 * 16 * (RANK ** 3 + RANK * sum(h)) + 2.0 * 3 * nvox * 16, "flops": flops}
    bytes_, flops = _product_work(case, B)
    if case["kind"] in ("solve", "gradient"):
        # about 700 Arnoldi steps per right-hand side, each with 25 basis vectors read twice
        steps = 700 * (2 if case["kind"] == "gradient" else 1)
        return {"bytes": steps * (bytes_ + 2.0 * 25 * B * 3 * nvox * 8),
                "flops": steps * (flops + 2.0 * 25 * 8 * B * 3 * nvox)}
    return {"bytes": bytes_, "flops": flops}


# --- the same passes in 64 bits -------------------------------------------------

def _kernel(n, c):
    """h^3 (k0^2 delta_ab + d_a d_b) g of component c at the circulant offsets of the 2n grid."""
    a, b = AXES[c]
    off, zero = [], []
    for m in n:
        i = torch.arange(2 * m, device="cuda")
        zero.append(i == m)
        off.append(torch.where(i > m, i - 2 * m, i).double() * H)
    X = [off[0][:, None, None], off[1][None, :, None], off[2][None, None, :]]
    r = torch.sqrt(X[0] ** 2 + X[1] ** 2 + X[2] ** 2)
    r[0, 0, 0] = 1.0
    f = torch.complex(3.0 / r ** 2 - K0 ** 2, 3.0 * K0 / r) * ((X[a] / r) * (X[b] / r))
    if a == b:
        f = f + torch.complex(K0 ** 2 - 1.0 / r ** 2, -K0 / r)
    v = H ** 3 * torch.polar(1.0 / (4.0 * math.pi * r), -K0 * r) * f
    q = K0 * H * (3.0 / (4.0 * math.pi)) ** (1.0 / 3.0)
    e = complex(math.cos(q), -math.sin(q))
    v[0, 0, 0] = (2.0 / 3.0) * (1.0 + 1j * q) * e - 1.0 if a == b else 0.0
    v[zero[0]] = 0.0
    v[:, zero[1]] = 0.0
    v[:, :, zero[2]] = 0.0
    return v


def _spectra(n):
    return [torch.fft.fftn(_kernel(n, c)) for c in range(6)]


def _green(G, x):
    """The product with the uncompressed operator, one right-hand side at a time."""
    n = tuple(x.shape[-3:])
    P = tuple(2 * m for m in n)
    out = torch.empty_like(x)
    for b in range(x.shape[0]):
        F = [torch.fft.fftn(x[b, a], s=P) for a in range(3)]
        for a in range(3):
            y = G[COMP[a, 0]] * F[0]
            y.addcmul_(G[COMP[a, 1]], F[1]).addcmul_(G[COMP[a, 2]], F[2])
            out[b, a] = torch.fft.ifftn(y)[: n[0], : n[1], : n[2]]
    return out


def _system(G, chi, x, adjoint):
    if adjoint:
        return x - _green(G, chi * x.conj()).conj().resolve_conj()
    return x - chi * _green(G, x)


def _gmres(apply, b, tol, m=50, cycles=60):
    """Restarted GMRES from zero in b's precision."""
    x, nb = torch.zeros_like(b), torch.linalg.vector_norm(b)
    V = torch.empty(m + 1, b.numel(), dtype=b.dtype, device=b.device)
    for _ in range(cycles):
        r = b - apply(x)
        beta = torch.linalg.vector_norm(r)
        if float(beta / nb) <= tol:
            break
        V[0] = (r / beta).reshape(-1)
        Hm = torch.zeros(m + 1, m, dtype=b.dtype, device=b.device)
        for k in range(m):
            w = apply(V[k].reshape(b.shape)).reshape(-1)
            for _pass in range(2):
                h = V[: k + 1].conj() @ w
                w = w - h @ V[: k + 1]
                Hm[: k + 1, k] += h
            Hm[k + 1, k] = torch.linalg.vector_norm(w)
            V[k + 1] = w / Hm[k + 1, k]
        e = torch.zeros(m + 1, 1, dtype=torch.complex128)
        e[0] = complex(float(beta), 0.0)
        y = torch.linalg.lstsq(Hm.to("cpu", torch.complex128), e).solution[:, 0]
        x = x + (y.to(b.device, b.dtype) @ V[:m]).reshape(b.shape)
    return x


def _solve(G, chi, b, adjoint=False):
    """A w = b to 1e-11 of ||b|| in 64 bits: inner solves in 32 bits, residuals and sums in 64."""
    G32, chi32, out = [g.to(torch.complex64) for g in G], chi.to(torch.complex64), torch.zeros_like(b)
    for i in range(b.shape[0]):
        bi, x = b[i: i + 1], out[i: i + 1]
        for _ in range(12):
            r = bi - _system(G, chi, x, adjoint)
            s = torch.linalg.vector_norm(r)
            if float(s / torch.linalg.vector_norm(bi)) <= 1e-11:
                break
            d = _gmres(lambda v: _system(G32, chi32, v, adjoint), (r / s).to(torch.complex64), 1e-5)
            x += s * d.to(torch.complex128)
    return out


def exact(case, seed):
    n, kind, c128 = _n(case), case["kind"], torch.complex128
    s = prepare(case, seed)
    if kind == "build":
        sigma = []
        for c in range(6):
            T = torch.fft.fftn(_kernel(n, c))
            for q in range(3):
                R = torch.linalg.qr(T.movedim(q, 0).reshape(2 * n[q], -1).conj().T, mode="r")[1]
                sigma.append(torch.linalg.svdvals(R)[: n[q] + 1].cpu().numpy())
        return {"ranks": None, "sigma": sigma, "Y": _green(_spectra(n), s["J"])}
    G = _spectra(n)
    if kind == "matvec":
        x = s["x"].to(c128)
        return _green(G, x.conj()).conj().resolve_conj() if case["adjoint"] else _green(G, x)
    if kind == "system":
        return _system(G, s["chi"].to(c128), s["x"].to(c128), case["adjoint"])
    if kind == "total":
        return s["einc"].to(c128) + _green(G, s["x"].to(c128))
    chi, einc = s["chi"].to(c128), s["einc"].to(c128)
    w = _solve(G, chi, chi * einc)
    if kind == "solve":
        return w
    E = einc + _green(G, w)
    gE = 2.0 * (E - s["target"].to(c128))
    mu = _solve(G, chi, _green(G, gE.conj()).conj().resolve_conj(), adjoint=True)
    return {"E": E, "grad": (mu * E.conj()).sum(dim=(0, 1))}
