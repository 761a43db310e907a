"""The work that is timed: the calls a program makes of this library, from one small deposit to the
ten-equation solve of 512^3 cells, through the public entry points of paper_1905_08890_gb300.gr.

A case is one call (family "solve", "patches", "deposit", "metric", "update", "residual", "guess", "grads") with its
sizes and options.  prepare() draws Zel'dovich particles from the seed on the GPU (a cell-centred lattice displaced
by a P(k) ~ k^-2 Gaussian or lognormal density field, the recipe of the bench) and builds what a program holds
before the call: the context or network, the sources and the fields.  run() makes the call.  exact() is the same
quantity in 64 bits from plain torch: index_add for the deposits, FFT and conjugate-gradient solves of the discrete
equations, and a float64 convolution network.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

from paper_1905_08890_gb300 import gr

RHO_BAR = 1.0 / (24.0 * math.pi)  # K^2 = 24 pi rho = 1
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(gr.__file__)), "weights", "unet128.npz")
FIELDS, SOURCES = gr.FIELDS, gr.SOURCES


def listed():
    return [
        # the smallest whole solve, with the default options (FP64, tol 1e-10): a test problem or a coarse survey
        # of parameters; its time is launches and latency
        dict(name="solve_32", family="solve", n=32, m=32, sigma=0.3, v_rms=0.01, lognormal=False, prec="fp64",
             tol=1e-10, fmg=0),
        # an ordinary solve in the fast precision, as the network's training set is made
        dict(name="solve_128", family="solve", n=128, m=128, sigma=1.0, v_rms=0.003, lognormal=True,
             prec="mixed_df", tol=1e-10, fmg=0),
        # a larger clumpy box with the full multigrid start
        dict(name="solve_256_fmg", family="solve", n=256, m=256, sigma=3.0, v_rms=0.003, lognormal=True,
             prec="mixed_df", tol=1e-8, fmg=1),
        # the headline workload: 512^3 cells, strongly clustered
        dict(name="solve_512", family="solve", n=512, m=512, sigma=5.0, v_rms=0.003, lognormal=True,
             prec="mixed_df", tol=1e-8, fmg=0),
        # a zoom: the base grid and two nested 128^3 patches at 2x and 4x its resolution around one cell
        dict(name="patches_256", family="patches", n=256, m=256, p1=128, p2=128, sigma=3.0, v_rms=0.003,
             lognormal=True, prec="mixed_df", tol=1e-8),
        # the smallest deposit: few particles, an odd number of them
        dict(name="deposit_12345", family="deposit", n=32, npart=12345, sigma=0.3, v_rms=0.3, lognormal=False),
        # the headline workload's sources: 134 million particles
        dict(name="deposit_512", family="deposit", n=512, npart=512 ** 3, sigma=5.0, v_rms=0.003, lognormal=True),
        # a time loop's sources: Lorentz factors in the previous step's metric, particles not a multiple of anything
        dict(name="metric_256", family="metric", n=256, npart=255 ** 3, sigma=3.0, v_rms=0.003, lognormal=True),
        # a time loop's particle update at full size: both kicks and the drift
        dict(name="update_512", family="update", n=512, npart=512 ** 3, sigma=5.0, v_rms=0.003, lognormal=True,
             flags=7),
        # checking a field from elsewhere against the Hamiltonian constraint
        dict(name="residual_256", family="residual", n=256, m=256, sigma=1.0, v_rms=0.003, lognormal=True),
        # the learned initial guess of all ten fields
        dict(name="guess_128", family="guess", n=128, m=128, sigma=1.0, v_rms=0.003, lognormal=True),
        # the backward direction: loss and gradient of the network, as training computes them
        dict(name="grads_64", family="grads", n=64, m=64, sigma=1.0, v_rms=0.003, lognormal=True),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    fam = rng.choice(("solve", "solve", "solve", "solve", "patches", "deposit", "deposit", "metric", "update", "update",
                      "residual", "guess", "grads"))
    c = dict(family=fam, sigma=round(_log(rng, 0.3, 5.0), 4), v_rms=round(_log(rng, 0.001, 0.3), 5), lognormal=True)
    if fam == "solve":
        c["prec"] = rng.choice(("mixed_df", "mixed_df", "mixed_df", "fp64", "mixed"))
        c["n"] = rng.choice((16, 32, 64, 128, 256, 512) if c["prec"] == "mixed_df" else (16, 32, 64, 128))
        c["fmg"] = rng.choice((0, 0, 1)) if c["n"] >= 32 and c["prec"] != "fp64" else 0
        c["tol"] = 1e-10 if c["n"] <= 128 else 1e-8
        c["m"] = c["n"]
    elif fam == "patches":
        c["n"] = rng.choice((32, 64, 128, 256))
        c["p1"] = rng.choice((c["n"] // 2, c["n"] // 4))
        c["p2"] = rng.choice((0, c["p1"]))
        c["prec"], c["tol"], c["m"] = "mixed_df", 1e-8, c["n"]
    elif fam in ("deposit", "metric", "update"):
        c["n"] = rng.choice((32, 64, 128, 256, 512))
        c["npart"] = min(int(c["n"] ** 3 * _log(rng, 0.125, 8.0)), 512 ** 3 - 1) | 1
        if fam == "update":
            c["flags"] = rng.choice((7, 7, 7, 6, 3, 4))
    elif fam == "residual":
        c["n"] = c["m"] = rng.choice((16, 32, 64, 128, 256))
    else:
        c["n"] = c["m"] = rng.choice((32, 64, 128)) if fam == "guess" else rng.choice((32, 64))
        c["v_rms"] = 0.003
        c["sigma"] = round(rng.uniform(0.3, 3.0), 4)
    return c


# ------------------------------------------------------------------ inputs
def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _particles(case, seed):
    """x, u (3, npart) float64 and the particle mass."""
    npart = case["npart"] if "npart" in case else case["m"] ** 3
    m = max(2, math.ceil(npart ** (1.0 / 3.0) - 1e-9))
    w = torch.randn((m, m, m), generator=_rng(seed), device="cuda", dtype=torch.float64)
    kx, ky, kz, k2 = _wave(m)
    wk = torch.fft.rfftn(w) / torch.sqrt(k2)
    wk[0, 0, 0] = 0.0
    g = torch.fft.irfftn(wk, s=(m, m, m))
    g /= g.std()
    sg = case["sigma"]
    if case["lognormal"]:
        lam = math.sqrt(math.log1p(sg * sg))
        delta = torch.clamp(torch.exp(lam * g - 0.5 * lam * lam) - 1.0, min=-0.95)
    else:
        delta = sg * g
    del w, g, wk
    dk = torch.fft.rfftn(delta)
    dk[0, 0, 0] = 0.0
    q = (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) / m
    x = torch.empty((3, npart), device="cuda", dtype=torch.float64)
    u = torch.empty_like(x)
    for d, kd in enumerate((kx, ky, kz)):
        disp = torch.fft.irfftn(1j * kd * dk / k2, s=(m, m, m))
        u[d] = disp.reshape(-1)[:npart]
        shape = [1, 1, 1]
        shape[d] = m
        x[d] = (disp + q.reshape(shape)).reshape(-1)[:npart]
        del disp
    x.remainder_(1.0)
    x[x >= 1.0] = 0.0
    u *= case["v_rms"] / max(float(torch.sqrt(u.square().sum() / npart)), 1e-300)
    return x, u, RHO_BAR / npart


def _wave(n):
    f = torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64) * (2.0 * math.pi)
    fr = torch.fft.rfftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64) * (2.0 * math.pi)
    kx, ky, kz = f[:, None, None], f[None, :, None], fr[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    return kx, ky, kz, k2


def _cloud(n, x):
    """Cloud-in-cell corners of particles x (3, np): yields (flat cell index, weight) eight times."""
    t = x * n - 0.5
    fl = torch.floor(t)
    fr = t - fl
    lo = fl.to(torch.int64)
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                at = [(lo[d] + s) % n for d, s in enumerate((a, b, c))]
                w = 1.0
                for d, s in enumerate((a, b, c)):
                    w = w * (fr[d] if s else 1.0 - fr[d])
                yield (at[0] * n + at[1]) * n + at[2], w


def _chunks(npart, step=1 << 24):
    return [slice(a, min(npart, a + step)) for a in range(0, npart, step)]


def _cic(n, x, u, mass, psi=None):
    """The five sources by index_add; psi: the conformal factor in the Lorentz factor (None: 1)."""
    out = {k: torch.zeros(n ** 3, device="cuda", dtype=torch.float64) for k in SOURCES}
    for sl in _chunks(x.shape[1]):
        xs, us = x[:, sl], u[:, sl]
        u2 = us.square().sum(dim=0)
        if psi is None:
            W = torch.sqrt(1.0 + u2)
        else:
            ps = sum(w * psi.reshape(-1)[at] for at, w in _cloud(n, xs))
            W = torch.sqrt(1.0 + u2 / ps ** 4)
        q = mass * n ** 3
        vals = (q * W, q * us[0], q * us[1], q * us[2], q * u2 / W)
        for at, w in _cloud(n, xs):
            for k, v in zip(SOURCES, vals):
                out[k].index_add_(0, at, v * w)
    return {k: v.reshape(n, n, n) for k, v in out.items()}


# ------------------------------------------------------------------ the discrete equations in 64 bits
def _sh(f, axis, s):
    return torch.roll(f, -s, dims=axis)


def _d(f, axis):
    return (_sh(f, axis, 1) - _sh(f, axis, -1)) * (0.5 * f.shape[0])


def _lap(f):
    n = f.shape[0]
    out = -6.0 * f
    for ax in range(3):
        out += _sh(f, ax, 1)
        out += _sh(f, ax, -1)
    return out * float(n * n)


def _invert(f, shift=0.0):
    """(lap - shift)^-1 f with the seven-point symbol; shift 0: zero-mean solution."""
    n = f.shape[0]
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    s = -4.0 * n * n * torch.sin(math.pi * k / n) ** 2
    sym = s[:, None, None] + s[None, :, None] + s[None, None, : n // 2 + 1] - shift
    if shift == 0.0:
        sym[0, 0, 0] = 1.0
    fk = torch.fft.rfftn(f)
    if shift == 0.0:
        fk[0, 0, 0] = 0.0
    fk /= sym
    return torch.fft.irfftn(fk, s=f.shape)


def _aij(V, U):
    n = U.shape[0]
    div = _d(V[0], 0) + _d(V[1], 1) + _d(V[2], 2)
    A = {}
    for i in range(3):
        A[i, i] = 2.0 * _d(V[i], i) - 0.5 * div + 2.0 * (_sh(U, i, 1) - 2.0 * U + _sh(U, i, -1)) * float(n * n)
        for j in range(i + 1, 3):
            A[i, j] = _d(V[j], i) + _d(V[i], j) + 2.0 * _d(_d(U, i), j)
    AA = sum(A[i, i] ** 2 for i in range(3)) + 2.0 * sum(A[i, j] ** 2 for i in range(3) for j in range(i + 1, 3))
    return A, AA


def _cg(rhs, m, x, tol):
    """lap x - m x = rhs (m > 0) by conjugate gradients preconditioned with (lap - mean m)^-1."""
    mb = float(m.mean())
    r = rhs - (_lap(x) - m * x)
    z = _invert(r, mb)
    p, rz, stop = z, float((r * z).sum()), tol * float(rhs.norm())
    for _ in range(60):
        Ap = _lap(p) - m * p
        a = rz / float((p * Ap).sum())
        x = x + a * p
        r = r - a * Ap
        if float(r.norm()) <= stop:
            break
        z = _invert(r, mb)
        new = float((r * z).sum())
        p, rz = z + (new / rz) * p, new
    return x


def _solution(src, rho):
    """The ten fields that solve the discrete equations for sources src."""
    pi, n = math.pi, src["s0"].shape[0]
    V = [_invert(8.0 * pi * (src[k] - src[k].mean())) for k in ("sx", "sy", "sz")]
    U = _invert(-0.25 * (_d(V[0], 0) + _d(V[1], 1) + _d(V[2], 2)))
    A, AA = _aij(V, U)
    K2, Kdot, s0 = 24.0 * pi * rho, 12.0 * pi * rho, src["s0"]
    w = torch.zeros_like(s0)  # psi - 1
    for _ in range(12):
        ps = 1.0 + w
        N = _lap(w) + 2.0 * pi * s0 / ps + 0.125 * AA / ps ** 7 - 2.0 * pi * rho * ps ** 5
        J = 2.0 * pi * s0 / ps ** 2 + 0.875 * AA / ps ** 8 + 10.0 * pi * rho * ps ** 4
        dw = _cg(-N, J, torch.zeros_like(w), 1e-10)
        w = w + dw
        if float(dw.abs().max()) <= 1e-15 * n:
            break
    ps = 1.0 + w
    m = 2.0 * pi * (s0 + 2.0 * src["sigma"] / ps ** 4) / ps ** 2 + 0.875 * AA / ps ** 8 + (5.0 / 12.0) * K2 * ps ** 4
    f = _cg(m - Kdot * ps ** 5, m, torch.zeros_like(w), 1e-13)
    g = (1.0 + f) / ps ** 7
    out = {"psi": ps, "apsi": 1.0 + f, "U": U}
    B = []
    for i in range(3):
        src_i = 2.0 * sum(_d(g * A[min(i, j), max(i, j)], j) for j in range(3))
        B.append(_invert(src_i - src_i.mean()))
    out["b"] = _invert(-0.25 * (_d(B[0], 0) + _d(B[1], 1) + _d(B[2], 2)))
    for i, c in enumerate("xyz"):
        out["V" + c], out["B" + c] = V[i], B[i]
    return {k: out[k] for k in FIELDS}


def _estimate(src, rho, by=0.9):
    """Fields a program may hold without a solve: V and U from the momentum sources, psi and alpha psi from the
    linearised equations (times `by`), no shift."""
    pi = math.pi
    V = [_invert(8.0 * pi * (src[k] - src[k].mean())) for k in ("sx", "sy", "sz")]
    U = _invert(-0.25 * (_d(V[0], 0) + _d(V[1], 1) + _d(V[2], 2)))
    w = by * _invert(-2.0 * pi * (src["s0"] - rho), 12.0 * pi * rho)
    z = torch.zeros_like(w)
    return {"psi": 1.0 + w, "apsi": 1.0 - w, "Vx": V[0], "Vy": V[1], "Vz": V[2], "U": U, "Bx": 1e-3 * V[1],
            "By": 1e-3 * V[2], "Bz": 1e-3 * V[0], "b": z + 1e-3 * U}


# ------------------------------------------------------------------ the network in 64 bits
_CONVS = [(16, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (192, 64), (64, 64),
          (96, 32), (32, 32), (48, 16), (16, 16)]


def _weights():
    with np.load(WEIGHTS) as z:
        return {k: np.asarray(z[k], dtype=np.float32) for k in ("params", "in_mean", "in_std", "out_mean", "out_std")}


def _net64(params, src, rho, v_rms, wt):
    """Standardised output [10, n, n, n] of the U-Net for flat float64 parameters."""
    F = torch.nn.functional
    off, layers = 0, []
    for cin, cout in _CONVS:
        w = params[off:off + 27 * cout * cin].reshape(27, cout, cin).permute(1, 2, 0).reshape(cout, cin, 3, 3, 3)
        off += 27 * cout * cin
        layers.append((w, params[off:off + cout]))
        off += cout
    hw, hb = params[off:off + 160].reshape(10, 16), params[off + 160:off + 170]
    ch = [torch.log(0.01 + src["s0"] / rho)] + [src[k] / (rho * v_rms) for k in ("sx", "sy", "sz")]
    ch = [(c - float(wt["in_mean"][k])) / float(wt["in_std"][k]) for k, c in enumerate(ch)]
    x = torch.stack(ch + [torch.zeros_like(ch[0])] * 12)[None]

    def conv(v, l):
        # one tap at a time: 27 small matrix products on rolled channels
        w, b = layers[l]
        y = b.reshape(-1, 1)
        for t in range(27):
            s = (t // 9 - 1, (t // 3) % 3 - 1, t % 3 - 1)
            r = torch.roll(v[0], (-s[0], -s[1], -s[2]), dims=(1, 2, 3))
            y = y + w[:, :, t // 9, (t // 3) % 3, t % 3] @ r.reshape(r.shape[0], -1)
        return F.relu(y).reshape((1, -1) + tuple(v.shape[2:]))

    def up(v):
        for ax in (2, 3, 4):
            lo = 0.75 * v + 0.25 * torch.roll(v, 1, dims=ax)
            hi = 0.75 * v + 0.25 * torch.roll(v, -1, dims=ax)
            shape = list(v.shape)
            v = torch.stack((lo, hi), dim=ax + 1).reshape(shape[:ax] + [2 * shape[ax]] + shape[ax + 1:])
        return v

    skips = []
    for lev in range(4):
        x = conv(conv(x, 2 * lev), 2 * lev + 1)
        if lev < 3:
            skips.append(x)
            x = F.avg_pool3d(x, 2)
    for lev in (2, 1, 0):
        x = torch.cat([up(x), skips[lev]], dim=1)
        x = conv(conv(x, 8 + 2 * (2 - lev)), 9 + 2 * (2 - lev))
    return (hw @ x[0].reshape(16, -1) + hb.reshape(-1, 1)).reshape((10,) + tuple(x.shape[2:]))


# ------------------------------------------------------------------ prepare, run
def prepare(case, seed):
    fam, n = case["family"], case["n"]
    x, u, mass = _particles(case, seed)
    st = {"case": case, "rho": mass * x.shape[1]}
    if fam in ("guess", "grads"):
        ctx = gr.Context(n)
        st["src"] = ctx.deposit(x, u, mass)
        ctx.close()
        wt = _weights()
        net = gr.Net(n)
        net.set_params(wt["params"])
        net.set_norm(wt["in_mean"], wt["in_std"], wt["out_mean"], wt["out_std"])
        st["net"] = net
        if fam == "guess":
            st["fld"] = {k: torch.empty((n, n, n), device="cuda", dtype=torch.float64) for k in FIELDS}
        else:
            st["fld"] = _solution(st["src"], st["rho"])
        torch.cuda.synchronize()
        return st
    ctx = st["ctx"] = gr.Context(n)
    if fam in ("solve", "patches"):
        st["src"] = ctx.deposit(x, u, mass)
        if fam == "patches":
            dense = int(torch.argmax(st["src"]["s0"]))
            at = (dense // (n * n), (dense // n) % n, dense % n)
            st["chain"] = gr.centred_chain(n, at, [p for p in (case["p1"], case["p2"]) if p])
            ctx.deposit_patches(st["chain"], x, u, mass)
    elif fam == "residual":
        st["src"] = ctx.deposit(x, u, mass)
        st["fld"] = _estimate(_cic(n, x, u, mass), st["rho"])
        st["eps"] = torch.empty((n, n, n), device="cuda", dtype=torch.float64)
    else:
        st.update(x=x, u=u, mass=mass)
        if fam == "update":
            st["fld"] = _estimate(_cic(n, x, u, mass), st["rho"], 1.0)
            st["dt"] = 0.05 / n / case["v_rms"]  # 0.05 cells at the rms speed
        else:
            st["src"] = ctx.new_sources()
            if fam == "metric":
                st["psi"] = _estimate(_cic(n, x, u, mass), st["rho"], 1.0)["psi"]
    torch.cuda.synchronize()
    if n >= 256:
        torch.cuda.empty_cache()  # the drawing's scratch, for the library's own allocations
    return st


def run(state):
    c = state["case"]
    fam, rho = c["family"], state["rho"]
    if fam == "solve":
        fld = state["ctx"].initial_fields()
        state["ctx"].solve(state["src"], fld, tol=c["tol"], prec=c["prec"], fmg=c["fmg"], rho_hat=rho)
        return fld
    if fam == "patches":
        ctx, chain = state["ctx"], state["chain"]
        fld = ctx.initial_fields()
        ctx.initial_patch_fields(chain)
        ctx.solve(state["src"], fld, tol=c["tol"], prec=c["prec"], rho_hat=rho, patches=chain)
        return {"base": fld, "patches": [q["fld"] for q in chain]}
    if fam == "deposit":
        return state["ctx"].deposit(state["x"], state["u"], state["mass"], state["src"])
    if fam == "metric":
        return state["ctx"].deposit_metric(state["x"], state["u"], state["mass"], state["psi"], state["src"])
    if fam == "update":
        state["ctx"].particle_update(state["x"], state["u"], state["fld"], state["dt"], c["flags"])
        return {"x": state["x"], "u": state["u"]}
    if fam == "residual":
        norm = state["ctx"].residual(gr.GR_PSI, state["src"], state["fld"], state["eps"], rho_hat=rho)
        return {"eps": state["eps"], "norm": norm}
    if fam == "guess":
        state["net"].infer(state["src"], state["fld"], rho, c["v_rms"])
        return state["fld"]
    loss, grads = state["net"].loss_grad(state["src"], state["fld"], rho, c["v_rms"])
    return {"loss": loss, "grads": grads}


def work(case):
    n, fam = case["n"], case["family"]
    N = n ** 3
    if fam in ("solve", "patches"):
        # the sources in, the ten fields out; V(2,2) cycles of ten equations, about seven operations per relaxed
        # cell, four sweeps and as many operations again for the transfers, 8/7 for the coarser levels
        cells = N + (sum(p ** 3 for p in (case["p1"], case["p2"])) if fam == "patches" else 0)
        cyc = math.log10(1.0 / case["tol"]) * 1.1
        return {"bytes": 15.0 * 8 * cells, "flops": 10 * cyc * 8 * 7 * cells * 8 / 7}
    if fam in ("deposit", "metric"):
        # positions and velocities in, five sources out (and psi in); eight corners, five products and sums each
        return {"bytes": 48.0 * case["npart"] + (40.0 + (8.0 if fam == "metric" else 0.0)) * N,
                "flops": 100.0 * case["npart"]}
    if fam == "update":
        # positions and velocities in, the changed ones out, six fields in; 20 gathered values from eight corners
        moved = (24 if case["flags"] & 4 else 0) + (24 if case["flags"] & 3 else 0)
        return {"bytes": (48.0 + moved) * case["npart"] + 48.0 * N, "flops": 400.0 * case["npart"] + 40.0 * N}
    if fam == "residual":
        # s0, psi, V, U in, the residual out
        return {"bytes": 7.0 * 8 * N, "flops": 120.0 * N}
    vox = [N >> (3 * lev) for lev in (0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0)]
    macs = sum(27.0 * a * b * v for (a, b), v in zip(_CONVS, vox)) - 27.0 * 12 * 16 * N  # 4 input channels
    if fam == "guess":
        return {"bytes": (4.0 + 10.0) * 8 * N, "flops": 2.0 * macs}
    return {"bytes": (4.0 + 10.0) * 8 * N, "flops": 6.0 * macs}


# ------------------------------------------------------------------ the same in 64 bits
def exact(case, seed):
    fam, n = case["family"], case["n"]
    if fam == "patches":
        return None  # a composite solve of its own would be needed
    x, u, mass = _particles(case, seed)
    rho = mass * x.shape[1]
    if fam == "deposit":
        return _cic(n, x, u, mass)
    src = _cic(n, x, u, mass)
    if fam == "metric":
        return _cic(n, x, u, mass, _estimate(src, rho, 1.0)["psi"])
    if fam == "solve":
        del x, u
        return _solution(src, rho)
    if fam == "residual":
        fld = _estimate(src, rho)
        ps = fld["psi"]
        AA = _aij([fld["Vx"], fld["Vy"], fld["Vz"]], fld["U"])[1]
        eps = _lap(ps - 1.0) + 2.0 * math.pi * src["s0"] / ps + 0.125 * AA / ps ** 7 - 2.0 * math.pi * rho * ps ** 5
        ref = 2.0 * math.pi * float(src["s0"].square().mean().sqrt())
        return {"eps": eps, "norm": float(eps.square().mean().sqrt()) / ref}
    if fam == "update":
        return _update64(case, x, u, _estimate(src, rho, 1.0), 0.05 / n / case["v_rms"])
    wt = _weights()
    params = torch.from_numpy(wt["params"]).cuda().double()
    if fam == "guess":
        with torch.no_grad():
            y = _net64(params, src, rho, case["v_rms"], wt)
        out = {}
        for k, name in enumerate(FIELDS):
            out[name] = y[k] * float(wt["out_std"][k]) + float(wt["out_mean"][k]) + (1.0 if k < 2 else 0.0)
        return out
    fld = _solution(src, rho)
    params.requires_grad_(True)
    y = _net64(params, src, rho, case["v_rms"], wt)
    t = torch.stack([((fld[name] - (1.0 if k < 2 else 0.0)) - float(wt["out_mean"][k])) / float(wt["out_std"][k])
                     for k, name in enumerate(FIELDS)])
    loss = (y - t).square().mean()
    loss.backward()
    return {"loss": float(loss), "grads": params.grad.cpu().numpy()}


def _update64(case, x, u, fld, dt):
    """Kicks and drift in 64 bits: five substeps per kick, fields and gradients by cloud-in-cell."""
    n, flags = case["n"], case["flags"]
    alpha = fld["apsi"] / fld["psi"]
    beta = [fld["B" + c] + _d(fld["b"], a) for a, c in enumerate("xyz")]
    grid = [alpha, fld["psi"]] + beta + [_d(alpha, a) for a in range(3)] + [_d(fld["psi"], a) for a in range(3)]
    grid += [_d(beta[c], a) for c in range(3) for a in range(3)]
    grid = [g.reshape(-1) for g in grid]
    xo, uo = torch.empty_like(x), torch.empty_like(u)
    for sl in _chunks(x.shape[1]):
        q = [0.0] * 20
        for at, w in _cloud(n, x[:, sl]):
            for k in range(20):
                q[k] = q[k] + w * grid[k][at]
        v = [u[0, sl].clone(), u[1, sl].clone(), u[2, sl].clone()]

        def lorentz():
            g = (v[0] ** 2 + v[1] ** 2 + v[2] ** 2) / q[1] ** 4
            return g, torch.sqrt(1.0 + g)

        def sub(j):
            if j <= 3:
                c = -v[j - 1].clone()
                for i in range(3):
                    v[i] = v[i] - 0.5 * dt * c * q[11 + 3 * (j - 1) + i]
                return
            g, W = lorentz()
            for i in range(3):
                if j == 4:
                    v[i] = v[i] + 0.5 * dt * (g / W) * (q[0] / q[1]) * 2.0 * q[8 + i]
                else:
                    v[i] = v[i] - 0.5 * dt * W * q[5 + i]

        if flags & gr.GR_KICK_SYNC:
            for j in (1, 2, 3, 4, 5):
                sub(j)
        if flags & gr.GR_KICK_OPEN:
            for j in (5, 4, 3, 2, 1):
                sub(j)
        W = lorentz()[1]
        for i in range(3):
            uo[i, sl] = v[i]
            xo[i, sl] = x[i, sl]
            if flags & gr.GR_DRIFT:
                xn = x[i, sl] + dt * (q[0] / q[1] ** 4 * v[i] / W - q[2 + i])
                xo[i, sl] = xn - torch.floor(xn)
    return {"x": xo, "u": uo}
