"""Performance cases of the random-field library: what its users have it do, through its Python API.

A case names a kind of call and its sizes; the kinds are

  step        one Monte-Carlo step on a fixed mesh with the caller's own modes: pack and upload the mode
              table, then the prepared synthesis (Y and K)
  grid        field, lognormal permeability and porosity on a Cartesian grid from a table on the device
  cells       the same (Y and K) at the centres of an unstructured mesh (a jittered lattice)
  remesh      a new unstructured mesh: plan its cells (handed over in no spatial order), then the field on them
  calibrate   one calibration step on a Cartesian grid: fused field, loss and dL/dY, then the adjoint
  autograd    the same step as a PyTorch user writes it: spectral_mismatch(...).backward(), parameters on the CPU
  adjoint     the adjoint alone on an unstructured mesh, for a dL/dY that the caller's flow solver returned
  ensemble    many realisations of different sizes as one batched launch
  map         permeability, facies and facies values of stored fields
  bimap       the two-field truncation rule on stored fields

Facies labels are asked for in the map cases, where they are an exact function of the stored field.
"""
import math
import random

import numpy as np
import torch

from paper_2212_10961_gb300 import field as F

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # the 64^2 unit square with N = 1000: the smallest field anyone asks for, again and again in a Monte-Carlo
        # loop; latency, launches and host work
        dict(name="step_64x64", kind="step", nx=64, ny=64, nz=0, ex=1.0, ey=1.0, ez=0.0, family="gaussian",
             lx=0.1, ly=0.1, lz=0.0, sigma2=1.0, n_modes=1000),
        # the Horton-Rogers-Lapwood field of the paper's example: 1024 x 512 cells of a 2 x 1 domain
        dict(name="grid_hrl", kind="grid", nx=1024, ny=512, nz=0, ex=2.0, ey=1.0, ez=0.0, family="gaussian",
             lx=0.2, ly=0.05, lz=0.0, sigma2=2.0, n_modes=4096),
        # the headline: a 256^3 cube with a rough (exponential), anisotropic covariance; the largest case
        dict(name="grid_256", kind="grid", nx=256, ny=256, nz=256, ex=1.0, ey=1.0, ez=1.0, family="exponential",
             lx=0.2, ly=0.2, lz=0.05, sigma2=4.0, n_modes=4096),
        # an ordinary reservoir box with ragged sizes and an intermediate smoothness
        dict(name="grid_ragged", kind="grid", nx=252, ny=126, nz=63, ex=2.0, ey=1.0, ez=0.5, family="matern",
             lx=0.13, ly=0.1, lz=0.07, sigma2=1.6, n_modes=2500),
        # an unstructured mesh of 2M cells: the paper's cells of any mesh, with the most modes
        dict(name="cells_2m", kind="cells", nx=252, ny=126, nz=63, ex=2.0, ey=1.0, ez=0.5, family="matern",
             lx=0.1, ly=0.1, lz=0.1, sigma2=2.0, n_modes=8192),
        # a small unstructured 2-D mesh with a rough field
        dict(name="cells_2d", kind="cells", nx=250, ny=130, nz=0, ex=2.0, ey=1.0, ez=0.0, family="exponential",
             lx=0.15, ly=0.1, lz=0.0, sigma2=1.2, n_modes=1000),
        # an adaptive run: every field is on a mesh not seen before
        dict(name="remesh_3d", kind="remesh", nx=126, ny=63, nz=31, ex=2.0, ey=1.0, ez=0.5, family="gaussian",
             lx=0.1, ly=0.1, lz=0.1, sigma2=1.0, n_modes=2048),
        # the 128^3 calibration step (forward and backward)
        dict(name="calibrate_128", kind="calibrate", nx=128, ny=128, nz=128, ex=1.0, ey=1.0, ez=1.0,
             family="gaussian", lx=0.1, ly=0.1, lz=0.1, sigma2=1.0, n_modes=2048),
        # a small calibration in plain PyTorch: parameters and optimiser on the CPU
        dict(name="autograd_40", kind="autograd", nx=40, ny=40, nz=40, ex=1.0, ey=1.0, ez=1.0, family="matern",
             lx=0.2, ly=0.15, lz=0.1, sigma2=1.0, n_modes=512),
        # the backward pass of an unstructured mesh
        dict(name="adjoint_2m", kind="adjoint", nx=252, ny=126, nz=63, ex=2.0, ey=1.0, ez=0.5, family="matern",
             lx=0.1, ly=0.1, lz=0.1, sigma2=2.0, n_modes=2048),
        # a Monte-Carlo ensemble: 64 realisations, 64^3 cubes and squares of 32^2 to 512^2 cells
        dict(name="ensemble_64", kind="ensemble", members=64, recipe=4, edge=512),
        # maps of a stored 256^3 field: bandwidth
        dict(name="map_256", kind="map", nx=256, ny=256, nz=256),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "grid", "grid", "cells", "cells", "remesh", "calibrate", "calibrate", "autograd",
                       "adjoint", "adjoint", "ensemble", "map", "bimap"])
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(16, 64), recipe=rng.randint(1, 10 ** 6), edge=log_int(128, 512))
    if kind in ("map", "bimap"):
        return dict(kind=kind, nx=log_int(64, 256), ny=log_int(64, 256), nz=log_int(16, 256))
    most_cells = {"step": 2 ** 19, "grid": 2 ** 24, "cells": 2 ** 21, "remesh": 2 ** 21, "calibrate": 2 ** 22,
                  "autograd": 2 ** 18, "adjoint": 2 ** 21}[kind]
    fewest = {"step": 2 ** 10, "autograd": 2 ** 12}.get(kind, 2 ** 14)
    most_modes = {"step": 4096, "autograd": 2048, "remesh": 4096, "adjoint": 4096}.get(kind, 8192)
    cells = math.exp(rng.uniform(math.log(fewest), math.log(most_cells)))
    n_modes = log_int(256, most_modes)
    while cells * n_modes > (6.0e10 if kind == "grid" else 1.6e10):
        n_modes = max(256, n_modes // 2)
    dim = rng.choice([2, 3, 3])
    aspect = [math.exp(rng.uniform(-0.7, 0.7)) for _ in range(dim)]
    scale = (cells / math.prod(aspect)) ** (1.0 / dim)
    n = [max(4, int(scale * a)) for a in aspect] + [0] * (3 - dim)
    h = 1.0 / max(n)
    ext = [round(k * h, 4) for k in n]
    ell = [round(math.exp(rng.uniform(math.log(0.04), math.log(0.3))), 4) for _ in range(dim)] + [0.0] * (3 - dim)
    return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], ex=ext[0], ey=ext[1], ez=ext[2],
                family=rng.choice(["gaussian", "matern", "exponential"]), lx=ell[0], ly=ell[1], lz=ell[2],
                sigma2=round(rng.uniform(0.5, 2.5), 3), n_modes=n_modes)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _dim(case):
    return 3 if case["nz"] else 2


def _shape(case):
    return (case["nx"], case["ny"], case["nz"])[:_dim(case)]


def _extent(case):
    return (case["ex"], case["ey"], case["ez"])[:_dim(case)]


def _ell(case):
    return np.array((case["lx"], case["ly"], case["lz"])[:_dim(case)])


def _cell_count(case):
    return math.prod(_shape(case))


def _draw_modes(n, dim, family, seed):
    """Standardised modes as the randomisation method draws them (float64): kappa (n, dim), unit amplitudes rho, psi.
    Gaussian covariance: normal kappa; Matern nu = 1.5 and exponential (nu = 0.5): Student t with 2 nu degrees."""
    rng = np.random.default_rng([seed, 1])
    kappa = rng.standard_normal((n, dim))
    if family == "gaussian":
        kappa *= math.sqrt(math.pi / 2.0)
    else:
        dof = 3.0 if family == "matern" else 1.0
        kappa *= np.sqrt(dof / rng.chisquare(dof, n))[:, None]
    w = rng.standard_normal((2, n))
    return dict(kappa=kappa, rho=np.hypot(w[0], w[1]) / math.sqrt(n), psi=-np.arctan2(w[1], w[0]) / TWO_PI)


def _modes(case, seed):
    m = _draw_modes(case["n_modes"], _dim(case), case["family"], seed)
    m["a"] = m["kappa"] / (TWO_PI * _ell(case))
    m["amp"] = math.sqrt(case["sigma2"]) * m["rho"]
    return m


def _axes(case):
    return [((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * (e / n)).float()
            for n, e in zip(_shape(case), _extent(case))]


def _mesh(axes):
    """Cell centres of the tensor product of the axes, x fastest."""
    grids = torch.meshgrid(*axes[::-1], indexing="ij")
    return [g.reshape(-1).contiguous() for g in grids[::-1]]


def _jittered(case, seed, shuffle=False):
    """Centres of an unstructured mesh: a lattice with every coordinate moved by up to 0.4 cells."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    cells = []
    for c, n, e in zip(_mesh(_axes(case)), _shape(case), _extent(case)):
        u = torch.rand(c.numel(), generator=gen, device="cuda")
        cells.append(c + (u - 0.5) * (0.8 * e / n))
    if shuffle:
        perm = torch.randperm(cells[0].numel(), generator=gen, device="cuda")
        cells = [c[perm].contiguous() for c in cells]
    return cells


def _params(case, mean=0.0):
    return F.FieldParams(family=case["family"], sigma2=case["sigma2"], mean=mean, ell=tuple(_ell(case)),
                         dim=_dim(case), n_modes=case["n_modes"])


def _table(m):
    return F.ModeTable(m["amp"], m["psi"], m["a"], kappa=m["kappa"])


_POROSITY = (0.25, 0.05, 0.05, 0.45)
_MEAN = 0.1


def _parameters32(case, seed):
    """The calibration's parameters as float32 CPU tensors: the trial state, and the ell, sigma2, mu of the truth."""
    m = _draw_modes(case["n_modes"], _dim(case), case["family"], seed)
    t = {k: torch.from_numpy(v).float() for k, v in m.items()}
    t["mu"], t["sigma2"] = torch.tensor(0.0), torch.tensor(case["sigma2"], dtype=torch.float32)
    t["ell"] = torch.from_numpy(_ell(case)).float()
    return t


def _twin(t, n=256):
    """The truth of a twin experiment: the leading modes of the trial state under other mu, sigma2 and ell."""
    n = min(n, t["rho"].numel())
    scale = math.sqrt(1.2 * float(t["sigma2"])) * math.sqrt(t["rho"].numel() / n)
    a = t["kappa"][:n].double() / (TWO_PI * 1.15 * t["ell"].double())
    return 0.05, (scale * t["rho"][:n].double()).cuda(), t["psi"][:n].double().cuda(), a.cuda()


def _residual(case, seed):
    """dL/dY at the cells of an unstructured mesh: a smooth residual between two states of a few modes."""
    m = _modes(case, seed)
    amp, psi, a = (torch.from_numpy(m[k][:64]).float().cuda() for k in ("amp", "psi", "a"))
    cells = torch.stack(_jittered(case, seed))
    g = torch.zeros(cells.shape[1], device="cuda")
    for k in range(64):
        turns = a[k] @ cells
        g += amp[k] * (torch.cos(TWO_PI * (turns + psi[k])) - torch.cos(TWO_PI * (turns / 1.1 + psi[k])))
    return g / g.numel()


def _members(case):
    """The ensemble's realisations: 64^3 cubes (1 in 8) and squares, N modes, covariance family."""
    r = random.Random(case["recipe"])
    out = []
    for _ in range(case["members"]):
        cube = r.random() < 0.125
        n = 64 if cube else int(round(2.0 ** r.uniform(5.0, math.log2(case["edge"]))))
        out.append(dict(nx=n, ny=n, nz=64 if cube else 0, ex=1.0, ey=1.0, ez=1.0 if cube else 0.0,
                        family=r.choice(["gaussian", "exponential"]), lx=0.1, ly=0.1, lz=0.1, sigma2=1.0,
                        n_modes=r.choice([1024, 2048, 4096])))
    return out


def _stored(n, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, generator=gen, device="cuda")


_THRESHOLDS = (-0.861454, 0.861454)
_RULE = [[0, 1], [2, 1], [2, 3]]


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind)
    if kind in ("map", "bimap"):
        n = _cell_count(case)
        s["Y"] = _stored(n, seed)
        if kind == "bimap":
            s["Y2"] = _stored(n, seed + 1)
        else:
            s["maps"] = F.MapSpec(y=False, lognormal=True, thresholds=_THRESHOLDS, facies=True,
                                  values=(0.0183, 0.27, 3.99))
            s["out"] = s["maps"].allocate(n, s["Y"].device)
        return s
    if kind == "ensemble":
        members = _members(case)
        cells = [_mesh(_axes(m)) for m in members]
        sizes = [c[0].numel() for c in cells]
        zeros = torch.zeros(max(sizes), device="cuda")
        x, y, z = (torch.cat([c[k] if k < len(c) else zeros[:n] for c, n in zip(cells, sizes)]) for k in range(3))
        s["plan"] = F.CellPlan(x, y, z, dim=3, segments=sizes)
        s["Y"], s["K"] = (torch.empty(sum(sizes), device="cuda") for _ in range(2))
        maps = F.MapSpec(y=True, lognormal=True)
        items, at = [], 0
        for i, (m, n) in enumerate(zip(members, sizes)):
            out = {"Y": s["Y"][at:at + n], "K": s["K"][at:at + n]}
            items.append((_table(_modes(m, seed * 1000 + i)), _params(m), i, maps, out))
            at += n
        s["batch"] = F.Batch(s["plan"], items, tile_cells=512)
        return s
    if kind in ("calibrate", "autograd"):
        t = _parameters32(case, seed)
        axes = _axes(case)
        mu, amp, psi, a = _twin(t)
        s["plan"] = F.CellPlan(*_mesh(axes))
        s["target"] = _grid64(axes, mu, amp, psi, a).exp().float()
        if kind == "autograd":
            s["t"] = {k: v.clone().requires_grad_() for k, v in t.items()}
        else:
            m = {k: t[k].double().numpy() for k in ("kappa", "rho", "psi")}
            m["a"] = m["kappa"] / (TWO_PI * t["ell"].double().numpy())
            s["params"] = F.FieldParams(family=case["family"], sigma2=float(t["sigma2"]), mean=0.0,
                                        ell=tuple(t["ell"].double().tolist()), dim=_dim(case),
                                        n_modes=case["n_modes"])
            s["table"] = F.ModeTable(s["params"].sigma * m["rho"], m["psi"], m["a"], kappa=m["kappa"])
        return s
    m = _modes(case, seed)
    s["params"] = _params(case, _MEAN)
    if kind == "step":
        s["modes"] = m
        s["plan"] = F.CellPlan(*_mesh(_axes(case)))
        s["table"] = _table(m)
        s["synth"] = F.PreparedSynth(s["params"], s["plan"], maps=F.MapSpec(y=True, lognormal=True))
        return s
    s["table"] = _table(m)
    if kind == "remesh":
        s["cells"] = _jittered(case, seed, shuffle=True)
        return s
    if kind == "grid":
        s["plan"] = F.CellPlan(*_mesh(_axes(case)))
        s["maps"] = F.MapSpec(y=True, lognormal=True, porosity=_POROSITY)
    else:
        s["plan"] = F.CellPlan(*_jittered(case, seed))
        s["maps"] = F.MapSpec(y=True, lognormal=True)
    if kind == "adjoint":
        s["gY"] = _residual(case, seed)
    else:
        s["out"] = s["maps"].allocate(_cell_count(case), s["plan"].buf.device)
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
_GRADS = ("dmu", "dsigma2", "dell", "drho", "dpsi", "dkappa")


def _gradients(g):
    """The gradients as the caller's float32 optimiser takes them."""
    return {k: g[k].float() for k in _GRADS}


def run(state):
    s, kind = state, state["kind"]
    if kind == "step":
        m = s["modes"]
        s["table"].update(m["amp"], m["psi"], m["a"], kappa=m["kappa"])
        return s["synth"](s["table"])
    if kind in ("grid", "cells"):
        return F.synth(s["table"], s["params"], s["plan"], maps=s["maps"], out=s["out"])
    if kind == "remesh":
        plan = F.CellPlan(*s["cells"])
        return F.synth(s["table"], s["params"], plan, maps=F.MapSpec(y=True))
    if kind == "calibrate":
        loss, gY, _ = F.synth_mismatch(s["table"], s["params"], s["plan"], s["target"])
        g = F.backward(s["table"], s["params"], s["plan"], gY)
        return dict(_gradients(g), loss=loss.float(), gY=gY)
    if kind == "autograd":
        t = s["t"]
        for v in t.values():
            v.grad = None
        loss = F.spectral_mismatch(t["mu"], t["sigma2"], t["ell"], t["rho"], t["psi"], t["kappa"], s["plan"],
                                   s["target"])
        loss.backward()
        return dict({k: v.grad for k, v in t.items()}, loss=loss.detach().float())
    if kind == "adjoint":
        return _gradients(F.backward(s["table"], s["params"], s["plan"], s["gY"]))
    if kind == "ensemble":
        s["batch"].launch()
        return {"Y": s["Y"], "K": s["K"]}
    if kind == "map":
        return F.map_property(s["Y"], s["maps"], 0.0, 1.0, out=s["out"])
    facies, prop = F.map_bitruncated(s["Y"], s["Y2"], _THRESHOLDS, (0.0,), _RULE, (0.0183, 0.27, 3.99, 58.9))
    return {"facies": facies, "prop": prop}


def work(case):
    """Inputs and outputs once; per cell and mode one complex multiply-add's real part (4 flops) forward, the sine
    and the cosine product with dL/dY (4) and, of the coordinate sums, no more than the same again (4) backward."""
    kind = case["kind"]
    if kind in ("map", "bimap"):
        n = _cell_count(case)
        return {"bytes": n * (4 + 4 + 1 + 4) if kind == "map" else n * (8 + 1 + 4), "flops": 0}
    if kind == "ensemble":
        ms = _members(case)
        cells = [_cell_count(m) for m in ms]
        return {"bytes": sum(c * 8 + 48 * m["n_modes"] for c, m in zip(cells, ms)),
                "flops": sum(4.0 * c * m["n_modes"] for c, m in zip(cells, ms))}
    n, modes = _cell_count(case), case["n_modes"]
    xyz = 4 * _dim(case) * n
    per_cell = {"step": 8, "grid": 12, "cells": 8 + xyz // n, "remesh": 4 + xyz // n, "calibrate": 8 + 4,
                "autograd": 8 + 4, "adjoint": 4 + xyz // n}[kind]
    flops = {"calibrate": 12.0, "autograd": 12.0, "adjoint": 8.0}.get(kind, 4.0)
    return {"bytes": per_cell * n + 48 * modes, "flops": flops * n * modes}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _phasor(a, x):
    """exp(2 pi i a x) as (cos, sin), modes by cells, in float64."""
    t = torch.outer(a, x.double())
    t = TWO_PI * (t - torch.round(t))
    return torch.cos(t), torch.sin(t)


def _columns(axes, psi, a):
    """Over blocks of the (y, z) cells: (first, last, cos, sin) of 2 pi (psi + a_y y + a_z z), modes by cells."""
    psi_turns = psi - torch.round(psi)
    ys, zs = axes[1], axes[2] if len(axes) > 2 else axes[1].new_zeros(1)
    az = a[:, 2] if len(axes) > 2 else torch.zeros_like(psi)
    per = max(1, 2 ** 24 // (a.shape[0] * ys.numel()))
    cy, sy = _phasor(a[:, 1], ys)
    for l0 in range(0, zs.numel(), per):
        z = zs[l0:l0 + per]
        t = torch.outer(az, z.double()) + psi_turns[:, None]
        t = TWO_PI * (t - torch.round(t))
        cz, sz = torch.cos(t)[:, :, None], torch.sin(t)[:, :, None]
        c = (cz * cy[:, None, :] - sz * sy[:, None, :]).reshape(a.shape[0], -1)
        s = (sz * cy[:, None, :] + cz * sy[:, None, :]).reshape(a.shape[0], -1)
        yield l0 * ys.numel(), (l0 + z.numel()) * ys.numel(), c, s


def _grid64(axes, mu, amp, psi, a):
    """mu + sum_j A_j cos(2 pi (a_j . x + psi_j)) on a grid (x fastest), float64: the sum regrouped per axis."""
    nx = axes[0].numel()
    out = torch.empty(math.prod(x.numel() for x in axes), dtype=torch.float64, device=axes[0].device)
    cx, sx = _phasor(a[:, 0], axes[0])
    for c0, c1, c, s in _columns(axes, psi, a):
        out[c0 * nx:c1 * nx] = ((c * amp[:, None]).T @ cx - (s * amp[:, None]).T @ sx).reshape(-1) + mu
    return out


def _cells64(cells, mu, amp, psi, a):
    """The same sum at any cells."""
    x = torch.stack([c.double() for c in cells], dim=1)
    out = torch.empty(x.shape[0], dtype=torch.float64, device=x.device)
    for i in range(0, x.shape[0], 2 ** 26 // a.shape[0]):
        j = i + 2 ** 26 // a.shape[0]
        t = x[i:j] @ a.T + psi
        out[i:j] = torch.cos(TWO_PI * (t - torch.round(t))) @ amp + mu
    return out


def _sums_grid64(axes, g, psi, a):
    """Per mode sum_i g cos, sum_i g sin and sum_i g x_c sin of theta_ij, on a grid."""
    nx, d = axes[0].numel(), len(axes)
    cx, sx = _phasor(a[:, 0], axes[0])
    x = axes[0].double()
    ys, zs = axes[1].double(), axes[2].double() if d > 2 else axes[1].double().new_zeros(1)
    yz = [ys.repeat(zs.numel()), zs.repeat_interleave(ys.numel())]
    cos, sin = torch.zeros_like(psi), torch.zeros_like(psi)
    lever = torch.zeros_like(a)
    for c0, c1, c, s in _columns(axes, psi, a):
        rows = g[c0 * nx:c1 * nx].reshape(-1, nx)
        re, im = (rows @ cx.T).T, (rows @ sx.T).T
        xre, xim = ((rows * x) @ cx.T).T, ((rows * x) @ sx.T).T
        cos += (re * c - im * s).sum(1)
        both = re * s + im * c
        sin += both.sum(1)
        lever[:, 0] += (xre * s + xim * c).sum(1)
        for k in range(1, d):
            lever[:, k] += both @ yz[k - 1][c0:c1]
    return cos, sin, lever


def _sums_cells64(cells, g, psi, a):
    x = torch.stack([c.double() for c in cells], dim=1)
    cos, sin = torch.zeros_like(psi), torch.zeros_like(psi)
    lever = torch.zeros_like(a)
    step = 2 ** 26 // a.shape[0]
    for i in range(0, x.shape[0], step):
        t = x[i:i + step] @ a.T + psi
        t = TWO_PI * (t - torch.round(t))
        gi, s = g[i:i + step], torch.sin(t)
        cos += gi @ torch.cos(t)
        sin += gi @ s
        lever += s.T @ (gi[:, None] * x[i:i + step])
    return cos, sin, lever


def _grads64(sums, g, sigma2, ell, rho, kappa, a):
    """dL/d(mu, sigma2, ell, rho, psi, kappa) from the per-mode sums."""
    cos, sin, lever = sums
    sigma = math.sqrt(sigma2)
    amp = sigma * rho
    da = -TWO_PI * amp[:, None] * lever
    return dict(dmu=g.sum().reshape(1), dsigma2=(rho @ cos / (2.0 * sigma)).reshape(1),
                dell=-(a * da).sum(0) / ell, drho=sigma * cos, dpsi=-TWO_PI * amp * sin,
                dkappa=da / (TWO_PI * ell))


def exact(case, seed):
    kind = case["kind"]
    if kind == "map":
        y = _stored(_cell_count(case), seed).double()
        return {"K": y.exp(), "facies": None, "prop": None}
    if kind == "bimap":
        return None
    if kind == "ensemble":
        ys = []
        for i, c in enumerate(_members(case)):
            m = {k: torch.from_numpy(v).cuda() for k, v in _modes(c, seed * 1000 + i).items()}
            ys.append(_grid64(_axes(c), 0.0, m["amp"], m["psi"], m["a"]))
        y = torch.cat(ys)
        return {"Y": y, "K": y.exp()}
    if kind in ("calibrate", "autograd"):
        t = _parameters32(case, seed)
        axes = _axes(case)
        target = _grid64(axes, *_twin(t)).exp().float().double()
        d = {k: v.double().cuda() for k, v in t.items()}
        a = d["kappa"] / (TWO_PI * d["ell"])
        sigma2 = float(d["sigma2"])
        k = _grid64(axes, 0.0, math.sqrt(sigma2) * d["rho"], d["psi"], a).exp()
        n = k.numel()
        g = 2.0 / n * (k - target) * k
        out = _grads64(_sums_grid64(axes, g, d["psi"], a), g, sigma2, d["ell"], d["rho"], d["kappa"], a)
        loss = ((k - target) ** 2).mean()
        if kind == "calibrate":
            return dict(out, loss=loss.reshape(1), gY=g)
        return dict({k[1:]: v.reshape(()) if k in ("dmu", "dsigma2") else v for k, v in out.items()}, loss=loss)
    m = {k: torch.from_numpy(v).cuda() for k, v in _modes(case, seed).items()}
    if kind == "adjoint":
        g = _residual(case, seed).double()
        sums = _sums_cells64(_jittered(case, seed), g, m["psi"], m["a"])
        return _grads64(sums, g, case["sigma2"], torch.from_numpy(_ell(case)).cuda(), m["rho"], m["kappa"], m["a"])
    if kind in ("step", "grid"):
        y = _grid64(_axes(case), _MEAN, m["amp"], m["psi"], m["a"])
    else:
        y = _cells64(_jittered(case, seed, shuffle=kind == "remesh"), _MEAN, m["amp"], m["psi"], m["a"])
    if kind == "remesh":
        return {"Y": y}
    out = {"Y": y, "K": y.exp()}
    if kind == "grid":
        phi0, phi1, lo, hi = _POROSITY
        out["prop"] = (phi0 + phi1 * (y - _MEAN) / math.sqrt(case["sigma2"])).clamp(lo, hi)
    return out
