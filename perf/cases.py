"""Workloads of the correlator library as its users run them, for measuring it.

A case is a dict of plain values.  ``listed()`` gives the fixed ones,
``draw(rng)`` more of the same ranges, ``prepare`` what a program holds before
the call (device or pinned host buffers, plans), ``run`` one pass through the
public entry points, ``work`` the bytes and operations the pass cannot do
without and ``exact`` the result from plain torch in 64 bits.

Kinds of case:
  correlate  one integration on device buffers (Plan.correlate)
  host       one integration from pinned host memory (Plan.correlate_host)
  batch      several sub-arrays in one persistent launch (BatchPlan.correlate)
  calib      gain calibration on visibilities: loss and gradient of one
             optimiser step, or a solve of several sweeps; per-input gains,
             per-channel gains or 2x2 Jones matrices
  grid       gridding of one integration's visibilities (GridPlan.grid)
  stokes     instrumental-polarisation images to Stokes I, Q, U, V
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_0902_0915_gb300 as mw

C_LIGHT = 299792458.0
F0 = 167.04e6    # first channel of the band, Hz
BAND = 30.72e6   # bandwidth the channels divide, Hz
RADIUS = 750.0   # tiles lie in a disc of this radius, metres
N_SOURCES = 20   # sky model of the calibration cases


# ---- the cases ---------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a 32-tile array's short integration, launch-bound
        dict(name="corr4 64in", kind="correlate", bits=4, fp16=False, n_inputs=64, n_chan=64, n_time=1000),
        # the 128-tile array: 0.5 s of the full band in 40 kHz channels, 4+4-bit samples
        dict(name="corr4 256in", kind="correlate", bits=4, fp16=False, n_inputs=256, n_chan=768, n_time=20000),
        # the 512-tile array: 1 s of an eighth of the band in 10 kHz channels, 8+8-bit
        dict(name="corr8 1024in", kind="correlate", bits=8, fp16=False, n_inputs=1024, n_chan=384, n_time=10000),
        # a partly equipped array with 8+8-bit samples: ragged inputs, odd integration
        dict(name="corr8 250in", kind="correlate", bits=8, fp16=False, n_inputs=250, n_chan=384, n_time=4001),
        # four sub-arrays of uneven size correlated together, an eighth of their channels
        dict(name="batch4 48-1024in", kind="batch", bits=4,
             jobs="48x32x2000,128x96x5000,300x192x10000,1024x384x20000"),
        # voltages that arrive in host memory: an eighth of the 128-tile array's band
        dict(name="host4 256in", kind="host", bits=4, n_inputs=256, n_chan=96, n_time=20000),
        # one optimiser step of a small array: forward and backward, launch-bound
        dict(name="calib 64in", kind="calib", gains="input", sweeps=0, n_inputs=64, n_chan=64),
        # one optimiser step at the full array's size: forward and backward
        dict(name="calib 1024in", kind="calib", gains="input", sweeps=0, n_inputs=1024, n_chan=768),
        # gains of every channel solved for on the 128-tile array's integration
        dict(name="calib chan solve 256in", kind="calib", gains="chan", sweeps=10, n_inputs=256, n_chan=768),
        # polarisation leakage of the full array solved for on a third of its channels
        dict(name="calib jones solve 1024in", kind="calib", gains="jones", sweeps=4, n_inputs=1024, n_chan=256),
        # the 128-tile integration gridded for imaging
        dict(name="grid 128t", kind="grid", n_tiles=128, n_chan=768, cells=2048, support=7),
        # the images of that grid converted to Stokes parameters
        dict(name="stokes 2048", kind="stokes", pixels=2048),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _inputs(rng, lo, hi):
    """Array sizes: whole 16-input rows, even and odd ones alike."""
    n = _log_int(rng, lo, hi)
    how = rng.randrange(3)
    return max(lo, n // 16 * 16) if how == 0 else max(lo, n // 2 * 2) if how == 1 else n


def draw(rng):
    kind = rng.choice(["correlate"] * 4 + ["batch", "host"] + ["calib"] * 3 + ["grid", "stokes"])
    if kind in ("correlate", "host"):
        bits = rng.choice([4, 8])
        n = _inputs(rng, 32, 1024 if kind == "correlate" else 512)
        t = _log_int(rng, 500, 20000)
        most = 7e9 if kind == "correlate" else 4e8  # bytes of samples
        c = min(_log_int(rng, 16, 768), max(8, int(most / (n * t * (bits // 4)))),
                max(8, int(1.9e12 / (n * (n + 1) / 2 * t))))
        case = dict(kind=kind, bits=bits, n_inputs=n, n_chan=c, n_time=t)
        if kind == "correlate":
            case["fp16"] = bits == 8 and rng.random() < 0.25
        return case
    if kind == "batch":
        jobs, room = [], 3.5e12
        for _ in range(rng.randint(2, 4)):
            n, t = _inputs(rng, 32, 1024), _log_int(rng, 500, 20000)
            c = min(_log_int(rng, 16, 384), max(4, int(room / 2 / (n * (n + 1) / 2 * t))))
            room -= n * (n + 1) / 2 * t * c
            jobs.append("%dx%dx%d" % (n, c, t))
        return dict(kind=kind, bits=4, jobs=",".join(jobs))
    if kind == "calib":
        gains = rng.choice(["input", "chan", "jones"])
        n = _inputs(rng, 32, 1024)
        if gains == "jones":
            n -= n % 2
        sweeps = rng.choice([0, rng.randint(2, 10)])
        c = min(_log_int(rng, 16, 768), max(8, int(4e8 * 4 / max(4, sweeps) / (n * (n + 1) / 2))))
        return dict(kind=kind, gains=gains, sweeps=sweeps, n_inputs=n, n_chan=c)
    if kind == "grid":
        return dict(kind=kind, n_tiles=_log_int(rng, 16, 128), n_chan=_log_int(rng, 16, 768),
                    cells=2 * _log_int(rng, 128, 1024), support=rng.randint(5, 7))
    return dict(kind=kind, pixels=2 * _log_int(rng, 64, 2048))


# ---- inputs ------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _samples(seed, bits, n_inputs, n_chan, n_time):
    """Packed voltages [n_chan][n_time][n_inputs]: receiver noise (sigma 2 or
    20) and a weak tone common to all inputs, rounded and clipped."""
    gen = _generator(seed)
    sigma, top = (2.0, 7) if bits == 4 else (20.0, 127)
    row = n_inputs * (bits // 4)
    out = torch.empty((n_chan, n_time, row), dtype=torch.uint8, device="cuda")
    step = max(1, int(1.5e8 // (n_time * n_inputs)))
    rate = torch.rand(n_chan, generator=gen, device="cuda") * (2 * math.pi)
    times = torch.arange(n_time, device="cuda", dtype=torch.float32)
    for c0 in range(0, n_chan, step):
        c1 = min(n_chan, c0 + step)
        x = torch.randn((c1 - c0, n_time, n_inputs, 2), generator=gen, device="cuda")
        x *= sigma
        ph = rate[c0:c1, None] * times
        x += (0.15 * sigma * torch.stack([ph.cos(), ph.sin()], -1))[:, :, None]
        x = x.round_().clamp_(-top, top).to(torch.int8)
        if bits == 4:
            out[c0:c1] = ((x[..., 0] & 15) | ((x[..., 1] & 15) << 4)).view(torch.uint8)
        else:
            out[c0:c1] = x.view(torch.uint8).reshape(c1 - c0, n_time, row)
    return out.reshape(-1)


def _unpack(v, bits, n_inputs, n_chan, n_time):
    """The packed samples as complex128 [n_chan, n_time, n_inputs]."""
    if bits == 8:
        x = v.view(torch.int8).reshape(n_chan, n_time, n_inputs, 2).to(torch.float64)
        return torch.view_as_complex(x)
    x = v.view(torch.int8).reshape(n_chan, n_time, n_inputs)
    re = ((x & 15) ^ 8) - 8
    return torch.complex(re.to(torch.float64), (x >> 4).to(torch.float64))


def _positions(seed, n_tiles):
    """Tile positions (metres), uniform in the array's disc."""
    rng = np.random.default_rng(seed)
    r = RADIUS * np.sqrt(rng.uniform(size=n_tiles))
    a = rng.uniform(0, 2 * math.pi, n_tiles)
    return np.ascontiguousarray(np.stack([r * np.cos(a), r * np.sin(a)], 1))


def _tril(n):
    return torch.tril_indices(n, n, device="cuda")


def _sky(seed, case):
    """Calibration data: the model M of point sources, the visibilities V of
    that sky seen through unknown gains plus noise, and starting gains a few
    per cent off.  V, M complex64 [n_chan, N(N+1)/2]."""
    gen = _generator(seed)
    n, n_chan, gains = case["n_inputs"], case["n_chan"], case["gains"]
    tiles = (n + 1) // 2
    pos = torch.from_numpy(_positions(seed, tiles)).cuda()
    lm = (torch.rand((N_SOURCES, 2), generator=gen, device="cuda", dtype=torch.float64) - 0.5)
    flux = torch.exp(torch.rand(N_SOURCES, generator=gen, device="cuda", dtype=torch.float64)
                     * math.log(100.0) + math.log(0.1))
    tau = (pos @ lm.T).repeat_interleave(2, 0)[:n] / C_LIGHT  # [N, sources], seconds

    def crandn(*shape):
        return torch.view_as_complex(torch.randn(shape + (2,), generator=gen, device="cuda"))

    if gains == "jones":
        eye = torch.eye(2, device="cuda").to(torch.complex64)
        true = eye + 0.1 * crandn(n // 2, 2, 2)
        start = true + 0.05 * crandn(n // 2, 2, 2)
    else:
        shape = (n_chan, n) if gains == "chan" else (n,)
        size = 0.8 + 0.4 * torch.rand(shape, generator=gen, device="cuda")
        turn = 2 * math.pi * torch.rand(shape, generator=gen, device="cuda")
        true = torch.polar(size, turn)
        start = true * (1.0 + 0.05 * crandn(*shape))
    i, j = _tril(n)
    nbl = n * (n + 1) // 2
    V = torch.empty((n_chan, nbl), dtype=torch.complex64, device="cuda")
    M = torch.empty((n_chan, nbl), dtype=torch.complex64, device="cuda")
    step = max(1, (1 << 25) // (n * n))
    for c0 in range(0, n_chan, step):
        c1 = min(n_chan, c0 + step)
        nu = F0 + (BAND / n_chan) * torch.arange(c0, c1, device="cuda", dtype=torch.float64)
        turns = tau[None] * nu[:, None, None]
        e = torch.polar(torch.ones_like(turns), 2 * math.pi * (turns - turns.floor())).to(torch.complex64)
        full = (e * flux.to(torch.float32)) @ e.conj().transpose(1, 2)
        if gains == "jones":  # unpolarised sources: no model power in the XY and YX products
            pol = torch.arange(n, device="cuda") % 2
            full = full * (pol[:, None] == pol)
            J = torch.block_diag(*true.unbind(0))
            seen = J @ full @ J.conj().T
        else:
            g = true[c0:c1] if gains == "chan" else true[None]
            seen = g[:, :, None] * full * g[:, None, :].conj()
        M[c0:c1] = full[:, i, j]
        V[c0:c1] = seen[:, i, j]
        V[c0:c1] += 0.1 * crandn(c1 - c0, nbl)
    return V, M, start


def _visibilities(seed, n_inputs, n_chan):
    """One integration's correlator output: noise on the cross products."""
    gen = _generator(seed)
    x = torch.randn((n_chan, n_inputs * (n_inputs + 1) // 2, 2), generator=gen, device="cuda")
    return (x * 1200.0 + 300.0).round_().to(torch.int32)


def _grid_geometry(case):
    """Cell size and kernel width of a grid that the whole array fits."""
    longest = 2 * RADIUS * (F0 + BAND) / C_LIGHT  # wavelengths
    return dict(f0=F0, df=BAND / case["n_chan"], Ng=case["cells"], du=2.1 * longest / case["cells"],
                W=case["support"], sigma=1.0)


def _jobs(case):
    return [tuple(int(k) for k in j.split("x")) for j in case["jobs"].split(",")]


# ---- what a program holds before the call --------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("correlate", "host"):
        shape = (case["n_inputs"], case["n_chan"], case["n_time"])
        v = _samples(seed, case["bits"], *shape)
        plan = mw.Plan(*shape, case["bits"], kind=mw.KIND_FP16 if case.get("fp16") else mw.KIND_EXACT)
        out = plan.empty_out()
        if kind == "host":
            vh = torch.empty(v.shape, dtype=v.dtype, pin_memory=True)
            vh.copy_(v)
            v, out = vh, torch.empty(out.shape, dtype=out.dtype, pin_memory=True)
        return dict(kind=kind, plan=plan, v=v, out=out)
    if kind == "batch":
        jobs = _jobs(case)
        plan = mw.BatchPlan(jobs, sample_bits=case["bits"])
        v = [_samples(seed + 1000003 * k, case["bits"], *j) for k, j in enumerate(jobs)]
        return dict(kind=kind, plan=plan, v=v, out=plan.empty_outs())
    if kind == "calib":
        V, M, start = _sky(seed, case)
        if case["sweeps"] == 0 and case["gains"] != "jones":
            start.requires_grad_(True)
        return dict(kind=kind, gains=case["gains"], sweeps=case["sweeps"], V=V, M=M, g=start)
    if kind == "grid":
        plan = mw.GridPlan(_positions(7, case["n_tiles"]), case["n_chan"], **_grid_geometry(case))
        vis = _visibilities(seed, 2 * case["n_tiles"], case["n_chan"])
        return dict(kind=kind, plan=plan, vis=vis, grids=plan.empty_grids())
    n = case["pixels"]
    inst = torch.view_as_complex(torch.randn((4, n, n, 2), generator=_generator(seed), device="cuda"))
    # the image of a uv grid with cells of one wavelength: one direction cosine wide
    return dict(kind=kind, inst=inst, dl=1.0 / n, chi=0.3, out=torch.empty_like(inst))


# ---- one pass ---------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "correlate" or kind == "batch":
        return state["plan"].correlate(state["v"], state["out"])
    if kind == "host":
        return state["plan"].correlate_host(state["v"], state["out"])
    if kind == "calib":
        V, M, g = state["V"], state["M"], state["g"]
        if state["sweeps"]:
            solve = {"input": mw.calib_solve, "chan": mw.calib_chan_solve,
                     "jones": mw.calib_jones_solve}[state["gains"]]
            gains, losses = solve(V, M, g, state["sweeps"])
            return {"gains": gains, "losses": losses}
        if state["gains"] == "jones":
            loss, grad = mw.calib_jones_loss_grad(V, M, g)
            return {"loss": loss, "grad": grad}
        g.grad = None
        loss = mw.calib_loss(g, V, M)
        loss.backward()
        return {"loss": loss.detach(), "grad": g.grad}
    if kind == "grid":
        return state["plan"].grid(state["vis"], state["grids"])
    return mw.stokes(state["inst"], state["dl"], state["chi"], state["out"])


# ---- what a pass cannot do without --------------------------------------------------
def _correlate_work(bits, n, c, t):
    nbl = n * (n + 1) // 2
    return c * (t * n * (bits // 4) + nbl * 8), 8 * nbl * c * t


def work(case):
    kind = case["kind"]
    if kind in ("correlate", "host"):
        b, f = _correlate_work(case["bits"], case["n_inputs"], case["n_chan"], case["n_time"])
    elif kind == "batch":
        each = [_correlate_work(case["bits"], *j) for j in _jobs(case)]
        b, f = sum(x[0] for x in each), sum(x[1] for x in each)
    elif kind == "calib":
        n, c = case["n_inputs"], case["n_chan"]
        terms, turns = c * n * (n + 1) // 2, max(1, case["sweeps"])
        # frequency-independent gains need every channel before the next sweep;
        # gains of one channel need that channel alone, read once
        passes = 1 if case["gains"] == "chan" else turns
        per = {"input": 34, "chan": 34, "jones": 50}[case["gains"]] + (6 if case["sweeps"] else 0)
        g = {"input": n, "chan": n * c, "jones": 2 * n}[case["gains"]]
        b, f = passes * terms * 16 + 2 * 8 * g, turns * terms * per
    elif kind == "grid":
        t, c, ng, w = case["n_tiles"], case["n_chan"], case["cells"], case["support"]
        b = c * t * (2 * t + 1) * 8 + 4 * ng * ng * 8
        f = t * (t - 1) * c * w * w * 4 * 4
    else:
        n = case["pixels"]
        b, f = n * n * 64, n * n * 150
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits ------------------------------------------------------------
def _exact_correlate(v, bits, n, c, t):
    i, j = _tril(n)
    out = torch.empty((c, n * (n + 1) // 2, 2), dtype=torch.float64, device="cuda")
    per = n * t
    for k in range(c):
        x = _unpack(v[k * per * (bits // 4):(k + 1) * per * (bits // 4)], bits, n, 1, t)[0]
        a, b = x.real.contiguous(), x.imag.contiguous()
        cross = b.T @ a
        out[k, :, 0] = (a.T @ a + b.T @ b)[i, j]
        out[k, :, 1] = (cross - cross.T)[i, j]
    return out


def _pairs(x, n):
    """[c, N(N+1)/2] -> Hermitian complex128 [c, N, N] with a zero diagonal."""
    i, j = _tril(n)
    full = torch.zeros((x.shape[0], n, n), dtype=torch.complex128, device=x.device)
    full[:, i, j] = x.to(torch.complex128)
    full.diagonal(dim1=1, dim2=2).zero_()
    return full + full.conj().transpose(1, 2)


def _blocks(x, n):
    """[c, N(N+1)/2] -> Hermitian tile blocks [c, 2, 2, T, T] ([p][q][a][b])."""
    f = _pairs(x, n).reshape(x.shape[0], n // 2, 2, n // 2, 2).permute(0, 2, 4, 1, 3).contiguous()
    f.diagonal(dim1=3, dim2=4).zero_()
    return f


def _gain_pass(V, M, g, n, step):
    """Loss, half gradient and normal-equation weight of g [N] or [c, N]."""
    chan = g.dim() == 2
    loss, grad, den = 0.0, [], []
    for c0 in range(0, V.shape[0], step):
        v, m = _pairs(V[c0:c0 + step], n), _pairs(M[c0:c0 + step], n)
        gc = g[c0:c0 + step] if chan else g[None].expand(v.shape[0], n)
        r = gc[:, :, None] * gc[:, None, :].conj() * m - v
        loss = loss + 0.5 * (r.abs() ** 2).sum()
        grad.append(torch.einsum("cij,cj->ci", r * m.conj(), gc))
        den.append(torch.einsum("cij,cj->ci", m.abs() ** 2, gc.abs() ** 2))
    grad, den = torch.cat(grad), torch.cat(den)
    return (loss, grad, den) if chan else (loss, grad.sum(0), den.sum(0))


def _jones_pass(V, M, J, n, step):
    """Loss, half gradient [T, 2, 2] and normal matrices [T, 2, 2] of J."""
    loss, G, D = 0.0, 0.0, 0.0
    for c0 in range(0, V.shape[0], step):
        v, m = _blocks(V[c0:c0 + step], n), _blocks(M[c0:c0 + step], n)
        B = torch.einsum("cpqab,brq->cprab", m, J.conj())  # M J_b^H
        r = torch.einsum("apq,cqrab->cprab", J, B) - v
        loss = loss + 0.5 * (r.abs() ** 2).sum()
        G = G + torch.einsum("cpqab,crqab->apr", r, B.conj())
        D = D + torch.einsum("cpqab,crqab->apr", B, B.conj())
    return loss, G, D


def _exact_calib(case, seed):
    V, M, g = _sky(seed, case)
    n, sweeps = case["n_inputs"], case["sweeps"]
    g = g.to(torch.complex128)
    step = max(1, (1 << 25) // (n * n))
    one = _jones_pass if case["gains"] == "jones" else _gain_pass
    if not sweeps:
        loss, grad, _ = one(V, M, g, n, step)
        return {"loss": loss, "grad": 2 * grad}
    losses = []
    for k in range(1, sweeps + 1):
        loss, grad, den = one(V, M, g, n, step)
        losses.append(loss)
        h = g - (grad @ torch.linalg.inv(den) if case["gains"] == "jones" else grad / den)
        g = h if k % 2 else 0.5 * (g + h)
    return {"gains": g, "losses": torch.stack(losses)}


def _exact_grid(case, seed):
    t, geo = case["n_tiles"], _grid_geometry(case)
    ng, w = geo["Ng"], geo["W"]
    vis = _visibilities(seed, 2 * t, case["n_chan"])
    xy = torch.from_numpy(_positions(7, t)).cuda()
    a, b = torch.tril_indices(t, t, -1, device="cuda")
    d = xy[a] - xy[b]
    grid = torch.zeros((ng * ng, 8), dtype=torch.float64, device="cuda")
    for c in range(case["n_chan"]):
        nu = geo["f0"] + c * geo["df"]
        pt = d * nu / C_LIGHT / geo["du"] + 0.5 * ng
        v = torch.view_as_complex(vis[c].to(torch.float64))
        prod = {}
        for p in range(2):
            for q in range(2):
                i = 2 * a + p
                prod[p, q] = v[i * (i + 1) // 2 + 2 * b + q]
        for side in range(2):
            xs = ng - pt if side else pt
            vals = torch.stack([prod[q, p].conj() if side else prod[p, q]
                                for p in range(2) for q in range(2)], 1)
            lo = torch.floor(xs - 0.5 * w).to(torch.int64) + 1
            s = lo[:, :, None] + torch.arange(w + 1, device="cuda")  # [points, (x, y), cells]
            off = s - xs[:, :, None]
            wt = torch.exp(-off * off / (2 * geo["sigma"] ** 2))
            wt = wt * ((off.abs() < 0.5 * w) & (s >= 0) & (s < ng))
            s = s.clamp(0, ng - 1)
            cell = (s[:, 1, :, None] * ng + s[:, 0, None, :]).reshape(-1)
            wts = (wt[:, 1, :, None] * wt[:, 0, None, :]).reshape(len(d), -1, 1)
            rows = (wts * vals[:, None, :]).reshape(-1, 4)
            grid.index_add_(0, cell, torch.view_as_real(rows).reshape(-1, 8))
    return torch.view_as_complex(grid.reshape(ng, ng, 4, 2)).permute(2, 0, 1).contiguous()


def _exact_stokes(inst, n, dl, chi):
    C = inst.to(torch.complex128)
    k = (torch.arange(n, device="cuda", dtype=torch.float64) - n / 2) * dl
    l, m = k[None, :], k[:, None]
    rho2 = l * l + m * m
    up = rho2 < 1
    cth = torch.sqrt((1 - rho2).clamp_min(1e-300))
    ph = torch.atan2(m.expand(n, n), l.expand(n, n)) + chi
    # J = R diag(cos th, 1) with R the rotation by ph: J^-1 = diag(1/cos th, 1) R^T
    c, s = torch.cos(ph), torch.sin(ph)
    inv = [[c / cth, s / cth], [-s, c]]
    B = [[sum(inv[p][r] * C[2 * r + q2] * inv[q][q2] for r in range(2) for q2 in range(2))
          for q in range(2)] for p in range(2)]
    out = torch.stack([B[0][0] + B[1][1], B[0][0] - B[1][1], B[0][1] + B[1][0],
                       -1j * (B[0][1] - B[1][0])])
    return torch.where(up, out, torch.zeros_like(out))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("correlate", "host"):
        n, c, t = case["n_inputs"], case["n_chan"], case["n_time"]
        if 8 * n * n * c * t > (6e12 if case.get("fp16") else 1e12):
            return None
        return _exact_correlate(_samples(seed, case["bits"], n, c, t), case["bits"], n, c, t)
    if kind == "batch":
        jobs = _jobs(case)
        if sum(8 * n * n * c * t for n, c, t in jobs) > 1e12:
            return None
        return [_exact_correlate(_samples(seed + 1000003 * k, case["bits"], *j), case["bits"], *j)
                for k, j in enumerate(jobs)]
    if kind == "calib":
        return _exact_calib(case, seed)
    if kind == "grid":
        return _exact_grid(case, seed)
    n = case["pixels"]
    inst = torch.view_as_complex(torch.randn((4, n, n, 2), generator=_generator(seed), device="cuda"))
    return _exact_stokes(inst, n, 1.0 / n, 0.3)
