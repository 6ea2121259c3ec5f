"""GPU tests of the band-limited path (csrc/band.cuh): modes of low frequency
summed on a coarse node lattice and interpolated to the cells.

The fields are checked against the FP64 oracle at sampled cells with the
forward tolerance of the other paths (1e-5 sigma): the interpolation's own
error is at most 1.7e-7 per mode amplitude and adds incoherently over modes.
The path is taken by size, so the cases are as large as it needs; that it was
taken shows in the number of kernels launched.
"""
import math

import numpy as np
import pytest

from helpers import GRAD_TOL, check_forward, check_lognormal, gpu_env, oracle_field, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = gpu_env()
    from paper_2212_10961_gb300 import field as F
    from paper_2212_10961_gb300 import workloads as W
    return torch, F, W


def _modes(n, dim, ell, law, seed):
    """Modes with normal ("gaussian") or Student t (1 degree: "rough") kappa."""
    rng = np.random.default_rng(seed)
    kappa = rng.standard_normal((n, dim)) * math.sqrt(math.pi / 2)
    if law == "rough":
        kappa = rng.standard_normal((n, dim)) / np.sqrt(rng.chisquare(1, n))[:, None]
    a = kappa / (2 * math.pi * np.asarray(ell))
    return {"a": a, "amp": rng.rayleigh(1.0, n) * math.sqrt(1.0 / n), "psi": rng.uniform(-0.5, 0.5, n), "kappa": kappa}


def _mesh(axes):
    m = np.meshgrid(*axes[::-1], indexing="ij")
    return [np.ascontiguousarray(v.ravel().astype(np.float32)) for v in m[::-1]]


def _uniform(shape, extent):
    return [((np.arange(n) + 0.5) * (e / n)).astype(np.float32) for n, e in zip(shape, extent)]


def _params(F, n, dim, ell):
    return F.FieldParams(family="gaussian", sigma2=1.0, mean=0.25, ell=ell, dim=dim, n_modes=n)


def _check_grid(env, axes, ell, n, law, seed=3, modes=None):
    torch, F, W = env
    dim = len(axes)
    cells = _mesh(axes)
    plan = F.CellPlan(*to_dev(torch, cells))
    assert plan.grid_shape()[:dim] == tuple(len(a) for a in axes)
    m = modes or _modes(n, dim, ell, law, seed)
    table = F.ModeTable(m["amp"], m["psi"], m["a"])
    l0 = F.launch_count()
    out = F.synth(table, _params(F, n, dim, ell), plan, maps=F.MapSpec(y=True, lognormal=True))
    torch.cuda.synchronize()
    assert plan.status() == 0
    launches = F.launch_count() - l0
    idx = np.unique(np.concatenate([np.random.default_rng(1).choice(len(cells[0]), 6000), np.arange(300),
                                    np.arange(len(cells[0]) - 300, len(cells[0]))]))
    y_or = oracle_field(m, 0.25, cells, idx)
    check_forward(out["Y"].cpu().numpy()[idx], y_or, 1.0, "band %s" % [len(a) for a in axes])
    check_lognormal(out["K"].cpu().numpy()[idx], y_or, 1.0)
    return launches


# every route of the grid path: 2-D of few and of many tiles, 3-D of few tiles
# (partial sums), 3-D of many (the light modes as chunks of the product), with
# modes left for the direct sum and without
@pytest.mark.parametrize("shape,extent,ell,n,law", [
    ((701, 499), (1.4, 1.0), (0.2, 0.1), 6000, "gaussian"),
    ((701, 499), (1.4, 1.0), (0.2, 0.1), 6001, "rough"),
    ((1537, 1025), (1.5, 1.0), (0.1, 0.2), 2500, "rough"),
    ((100, 81, 61), (1.0, 0.8, 0.6), (0.2, 0.2, 0.2), 6000, "gaussian"),
    ((129, 101, 90), (1.29, 1.0, 0.9), (0.2, 0.15, 0.2), 4097, "rough"),
    ((257, 131, 65), (1.0, 0.5, 0.25), (0.1, 0.1, 0.1), 3000, "gaussian"),
    ((33, 40, 301), (0.1, 0.13, 1.0), (0.1, 0.1, 0.1), 4000, "rough"),
    ((640, 9, 130), (4.0, 0.05, 0.9), (0.1, 0.1, 0.1), 3000, "rough"),
])
def test_band_grid_against_oracle(env, shape, extent, ell, n, law):
    assert _check_grid(env, _uniform(shape, extent), ell, n, law) >= 6


def test_band_grid_axes_in_any_order_and_far_away(env):
    # rectilinear axes: random spacings far from the origin, one axis running
    # down and one in random order (its cells' nodes lie far apart, so the
    # staged loads give way to plain ones)
    rng = np.random.default_rng(5)
    axes = [np.float32(900.0) + np.cumsum(rng.uniform(0.002, 0.006, 400)).astype(np.float32),
            np.ascontiguousarray((np.float32(-70.0) + np.cumsum(rng.uniform(0.004, 0.012, 120)).astype(np.float32))[::-1]),
            rng.permutation(np.linspace(0.0, 1.0, 90).astype(np.float32))]
    assert _check_grid(env, axes, (0.1, 0.1, 0.1), 3000, "rough") >= 6
    axes[0] = rng.permutation(axes[0])
    assert _check_grid(env, axes, (0.1, 0.1, 0.1), 3000, "gaussian") >= 6
    axes2 = [rng.permutation(np.linspace(0.0, 2.0, 1400).astype(np.float32)), np.linspace(0, 1, 900).astype(np.float32)]
    assert _check_grid(env, axes2, (0.1, 0.1), 4000, "gaussian") >= 5


def test_band_grid_degenerate_frequencies(env):
    # modes that do not vary along an axis, modes of frequency 0, equal phases
    # (the light sum far larger than any amplitude) and one very fast mode
    n = 4000
    m = _modes(n, 3, (0.2, 0.2, 0.2), "gaussian", 8)
    m["a"][:, 2] = 0.0
    m["a"][::7] = 0.0
    m["a"][11] = (3.0e4, -2.0e5, 17.0)
    m["psi"][: n // 2] = 0.0
    m["amp"] = m["amp"] / math.sqrt(n)  # the coherent half would sum to tens of sigma
    axes = _uniform((180, 160, 70), (1.0, 0.9, 0.4))
    assert _check_grid(env, axes, (0.2, 0.2, 0.2), n, "gaussian", modes=m) >= 6


def test_band_grid_fused_mismatch(env):
    # the fused loss sees the field of the synthesis (same kernels), on the
    # routes that finalize and on the one that writes from the product
    torch, F, W = env
    for shape, law, n in (((128, 128, 80), "gaussian", 2000), ((160, 128, 90), "rough", 3000), ((900, 700), "rough", 3000)):
        dim = len(shape)
        ell = (0.2,) * dim
        plan = F.CellPlan(*to_dev(torch, _mesh(_uniform(shape, (1.0, 0.9, 0.8)[:dim]))))
        m = _modes(n, dim, ell, law, 4)
        table = F.ModeTable(m["amp"], m["psi"], m["a"])
        p = _params(F, n, dim, ell)
        ref = F.synth(table, p, plan, maps=F.MapSpec(y=True, lognormal=True))
        T = torch.full_like(ref["K"], 1.5)
        loss_u, gY_u = F.mismatch_grad(ref["K"], T)
        loss, gY, out = F.synth_mismatch(table, p, plan, T, want_Y=True, want_K=True)
        torch.cuda.synchronize()
        assert torch.equal(out["Y"], ref["Y"]) and torch.equal(out["K"], ref["K"]) and torch.equal(gY, gY_u)
        assert loss.item() == pytest.approx(loss_u.item(), rel=1e-12)
        again = F.synth(table, p, plan, maps=F.MapSpec(y=True))["Y"]
        assert torch.equal(again, ref["Y"])  # deterministic


# ---------------------------------------------------------------------------
# Cells of any plan
# ---------------------------------------------------------------------------
def _cloud(kind, n, dim, seed):
    """Cell centres: "lattice" (jittered), "even" (independent uniform),
    "clusters" (dense blobs far apart: groups that spread over many nodes)."""
    rng = np.random.default_rng(seed)
    if kind == "lattice":
        side = int(round(n ** (1.0 / dim)))
        grid = np.stack(np.meshgrid(*[np.arange(side)] * dim, indexing="ij"), -1).reshape(-1, dim)
        c = (grid + 0.5 + rng.uniform(-0.4, 0.4, grid.shape)) / side
    elif kind == "even":
        c = rng.random((n, dim))
    else:
        centre = rng.random((40, dim)) * 3.0 - 1.0
        c = centre[rng.integers(0, 40, n)] + 0.004 * rng.standard_normal((n, dim))
    return [np.ascontiguousarray(c[:, k].astype(np.float32)) for k in range(dim)]


def _check_cells(env, cells, ell, n, law, segments=None, segment=0, seed=6, maps=None):
    torch, F, W = env
    dim = len(ell)
    plan = F.CellPlan(*to_dev(torch, cells), segments=segments)
    m = _modes(n, dim, ell, law, seed)
    table = F.ModeTable(m["amp"], m["psi"], m["a"])
    l0 = F.launch_count()
    out = F.synth(table, _params(F, n, dim, ell), plan, segment, F.MapSpec(y=True, lognormal=True))
    torch.cuda.synchronize()
    launches = F.launch_count() - l0
    o0 = int(plan.offsets[segment])
    count = plan.segment_size(segment)
    idx = np.unique(np.concatenate([np.random.default_rng(1).choice(count, 6000), np.arange(300),
                                    np.arange(count - 300, count)]))
    y_or = oracle_field(m, 0.25, [c[:] for c in cells[:dim]], o0 + idx)
    check_forward(out["Y"].cpu().numpy()[idx], y_or, 1.0, "cells %d" % count)
    check_lognormal(out["K"].cpu().numpy()[idx], y_or, 1.0)
    return launches, plan


@pytest.mark.parametrize("kind,cells,dim,n,law", [
    ("lattice", 300_000, 2, 4000, "gaussian"), ("lattice", 300_001, 2, 4100, "rough"),
    ("even", 150_333, 3, 4000, "gaussian"), ("lattice", 262_144, 3, 5003, "rough"),
    ("clusters", 400_000, 3, 3000, "gaussian"), ("clusters", 300_000, 2, 4000, "rough"),
])
def test_band_cells_against_oracle(env, kind, cells, dim, n, law):
    launches, plan = _check_cells(env, _cloud(kind, cells, dim, 3), (0.2, 0.25, 0.2)[:dim], n, law)
    assert launches >= 6 and plan.status() == 0


def test_band_cells_segments_and_lower_dimension(env):
    # the second of three segments, and a 2-D field on the cells of a 3-D plan
    torch, F, W = env
    parts = [_cloud("even", k, 3, 10 + k % 7) for k in (1000, 600_000, 37)]
    cells = [np.concatenate([p[c] for p in parts]) for c in range(3)]
    launches, _ = _check_cells(env, cells, (0.2, 0.2, 0.2), 6000, "gaussian", segments=[1000, 600_000, 37], segment=1)
    assert launches >= 6
    launches, _ = _check_cells(env, cells, (0.2, 0.2), 6000, "gaussian")
    assert launches >= 6


def test_band_cells_not_finite(env):
    # a cell that is not finite: the plan says so, the path stays with the
    # direct sum and every other cell keeps its value
    torch, F, W = env
    for bad in (np.nan, np.inf):
        cells = _cloud("even", 200_000, 3, 4)
        cells[1][77] = bad
        plan = F.CellPlan(*to_dev(torch, cells))
        m = _modes(4000, 3, (0.2, 0.2, 0.2), "gaussian", 2)
        y = F.synth(F.ModeTable(m["amp"], m["psi"], m["a"]), _params(F, 4000, 3, (0.2, 0.2, 0.2)), plan)["Y"]
        torch.cuda.synchronize()
        assert plan.status() == 1
        idx = np.setdiff1d(np.random.default_rng(1).choice(200_000, 4000), [77])
        check_forward(y.cpu().numpy()[idx], oracle_field(m, 0.25, cells, idx), 1.0, "beside a cell at %s" % bad)


def test_band_cells_fused_mismatch_and_workspace(env):
    # the fused loss and gradient are those of the synthesis; without room for
    # the lattice (workspace=False) all modes are summed at the cells
    torch, F, W = env
    for law, n in (("gaussian", 4000), ("rough", 6000)):
        cells = _cloud("lattice", 262_144, 3, 3)
        plan = F.CellPlan(*to_dev(torch, cells))
        m = _modes(n, 3, (0.2, 0.2, 0.2), law, 4)
        table = F.ModeTable(m["amp"], m["psi"], m["a"])
        p = _params(F, n, 3, (0.2, 0.2, 0.2))
        ref = F.synth(table, p, plan, maps=F.MapSpec(y=True, lognormal=True))
        T = torch.full_like(ref["K"], 1.5)
        loss_u, gY_u = F.mismatch_grad(ref["K"], T)
        loss, gY, out = F.synth_mismatch(table, p, plan, T, want_Y=True)
        direct = F.synth(table, p, plan, workspace=False)["Y"]
        torch.cuda.synchronize()
        assert torch.equal(out["Y"], ref["Y"]) and torch.equal(gY, gY_u)
        assert loss.item() == pytest.approx(loss_u.item(), rel=1e-12)
        assert not torch.equal(direct, ref["Y"])
        assert (direct - ref["Y"]).abs().max().item() <= 2e-5


# ---------------------------------------------------------------------------
# The adjoint: g spread onto the lattice, the modes summed there
# ---------------------------------------------------------------------------
def _check_adjoint(env, cells, ell, n, law, g=None, segments=None, segment=0, seed=6, modes=None, scale=1.0):
    """Gradients of a sample of modes (every light/direct class is in it)
    against the oracle's FP64 sums, sums over all modes against the modes'."""
    torch, F, W = env
    from oracle import field as of
    from oracle import native
    dim = len(ell)
    plan = F.CellPlan(*to_dev(torch, cells), segments=segments)
    o0, count = int(plan.offsets[segment]), plan.segment_size(segment)
    if g is None:
        g = np.random.default_rng(seed + 1).standard_normal(count).astype(np.float32)
    m = modes or _modes(n, dim, ell, law, seed)
    table = F.ModeTable(m["amp"], m["psi"], m["a"])
    gd = torch.from_numpy(g).cuda() * scale
    l0 = F.launch_count()
    gr = F.backward(table, _params(F, n, dim, ell), plan, gd, segment)
    torch.cuda.synchronize()
    launches = F.launch_count() - l0
    again = F.backward(table, _params(F, n, dim, ell), plan, gd, segment)
    assert plan.status() == 0
    for k in ("dA", "dpsi", "da", "dell", "dsigma"):
        assert torch.equal(gr[k], again[k]), "%s differs from one run to the next" % k
    fast = np.argsort(np.abs(m["a"] / np.sqrt(np.abs(m["a"])).mean(0).clip(1e-30) ** 2).max(1))
    idx = np.unique(np.concatenate([fast[:20], fast[-40:], np.random.default_rng(2).choice(n, 200)]))
    c = np.stack([c[o0:o0 + count] for c in cells[:dim]], axis=-1)
    g64 = g.astype(np.float64) * scale
    sums = native.mode_sums(m["a"][idx], m["psi"][idx], c, g64)
    ref = of.grads_from_sums(*sums, m["amp"][idx], m["a"][idx], 1.0, ell, g64)
    for k in ("dA", "dpsi", "da"):
        got = gr[k].cpu().numpy()[idx]
        for col in ([...],) if got.ndim == 1 else [(slice(None), q) for q in range(dim)]:
            top = np.abs(ref[k][tuple(col)]).max()
            err = np.abs(got[tuple(col)] - ref[k][tuple(col)]).max()
            assert err <= GRAD_TOL * top, "%s %s: %.3e of %.3e" % (k, col, err, top)
    assert gr["dmu"].item() == pytest.approx(g64.sum(), rel=1e-9, abs=1e-9 * np.abs(g64).sum())
    dell = -(gr["da"].cpu().numpy() * m["a"]).sum(0) / np.asarray(ell)
    np.testing.assert_allclose(gr["dell"].cpu().numpy()[:dim], dell, rtol=1e-9, atol=1e-9 * np.abs(dell).max())
    return launches, {k: v.cpu().numpy() for k, v in gr.items()}


# grids: 2-D of few and of many tiles, 3-D with and without modes left for
# the product, thin grids, an axis that is not interpolated
@pytest.mark.parametrize("shape,extent,ell,n,law", [
    ((1401, 999), (1.4, 1.0), (0.2, 0.1), 4001, "rough"),
    ((1024, 1025), (1.0, 1.0), (0.2, 0.2), 6000, "gaussian"),
    ((129, 101, 90), (1.29, 1.0, 0.9), (0.2, 0.2, 0.2), 4097, "gaussian"),
    ((160, 141, 130), (1.6, 1.4, 1.3), (0.2, 0.15, 0.2), 3000, "rough"),
    ((33, 40, 601), (0.1, 0.13, 2.0), (0.1, 0.1, 0.1), 5000, "rough"),
    ((640, 9, 260), (4.0, 0.05, 1.8), (0.1, 0.1, 0.1), 3000, "rough"),
    ((2003, 8, 90), (4.0, 0.05, 0.9), (0.1, 0.1, 0.1), 3000, "gaussian"),
])
def test_band_grid_adjoint_against_oracle(env, shape, extent, ell, n, law):
    launches, _ = _check_adjoint(env, _mesh(_uniform(shape, extent)), ell, n, law)
    assert launches >= 8


def test_band_grid_adjoint_axes_in_any_order_and_far_away(env):
    # axes in random order and far from the origin, one with a wide gap (the
    # nodes inside it are read by no cell); modes that do not vary
    rng = np.random.default_rng(5)
    axes = [np.float32(900.0) + np.cumsum(rng.uniform(0.002, 0.006, 400)).astype(np.float32),
            np.ascontiguousarray((np.float32(-70.0) + np.cumsum(rng.uniform(0.004, 0.012, 120)).astype(np.float32))[::-1]),
            rng.permutation(np.linspace(0.0, 1.0, 90).astype(np.float32))]
    launches, _ = _check_adjoint(env, _mesh(axes), (0.1, 0.1, 0.1), 3000, "gaussian")
    assert launches >= 8
    axes[0] = rng.permutation(np.where(axes[0] > 900.8, axes[0] + np.float32(3.0), axes[0]))
    m = _modes(3000, 3, (0.1, 0.1, 0.1), "gaussian", 8)
    m["a"][::7] = 0.0
    m["a"][11] = (3.0e3, -2.0e4, 17.0)
    launches, _ = _check_adjoint(env, _mesh(axes), (0.1, 0.1, 0.1), 3000, "gaussian", modes=m)
    assert launches >= 8


@pytest.mark.parametrize("kind,cells,dim,n,law", [
    ("lattice", 300_000, 2, 4000, "gaussian"), ("lattice", 300_001, 2, 4100, "rough"),
    ("even", 250_333, 3, 4000, "gaussian"), ("lattice", 262_144, 3, 5003, "rough"),
    ("clusters", 400_000, 3, 3000, "gaussian"), ("clusters", 300_000, 2, 4000, "rough"),
])
def test_band_cells_adjoint_against_oracle(env, kind, cells, dim, n, law):
    launches, _ = _check_adjoint(env, _cloud(kind, cells, dim, 3), (0.2, 0.25, 0.2)[:dim], n, law)
    assert launches >= 7


def test_band_cells_adjoint_segment_and_coherent_g(env):
    # the second of three segments, and a g of one sign (the largest sums of
    # the fixed-point lattice)
    parts = [_cloud("even", k, 3, 10 + k % 7) for k in (1000, 600_000, 37)]
    cells = [np.concatenate([p[c] for p in parts]) for c in range(3)]
    g = np.random.default_rng(3).uniform(0.5, 1.0, 600_000).astype(np.float32)
    launches, _ = _check_adjoint(env, cells, (0.2, 0.2, 0.2), 6000, "gaussian", g=g, segments=[1000, 600_000, 37],
                                 segment=1)
    assert launches >= 7


@pytest.mark.parametrize("grid", [False, True])
def test_band_adjoint_scales_and_carries_what_is_not_finite(env, grid):
    # g times a power of two gives the same digits times it; a g that holds an
    # infinity or a NaN gives gradients that are not finite; g = 0 gives 0
    torch, F, W = env
    cells = _mesh(_uniform((160, 141, 130), (1.6, 1.4, 1.3))) if grid else _cloud("even", 250_000, 3, 4)
    ell, n = (0.2, 0.2, 0.2), 4000
    _, one = _check_adjoint(env, cells, ell, n, "gaussian")
    for e in (-90, 70):
        _, big = _check_adjoint(env, cells, ell, n, "gaussian", scale=2.0 ** e)
        for k in ("dA", "dpsi", "da"):
            assert np.array_equal(one[k] * 2.0 ** e, big[k])
    plan = F.CellPlan(*to_dev(torch, cells))
    m = _modes(n, 3, ell, "gaussian", 6)
    table = F.ModeTable(m["amp"], m["psi"], m["a"])
    for bad in (float("nan"), float("inf"), -float("inf")):
        g = torch.ones(len(cells[0]), device="cuda")
        g[12345] = bad
        gr = F.backward(table, _params(F, n, 3, ell), plan, g)
        assert not torch.isfinite(gr["dA"]).any() and not torch.isfinite(gr["dpsi"]).any()
    gr = F.backward(table, _params(F, n, 3, ell), plan, torch.zeros(len(cells[0]), device="cuda"))
    assert all(not v.any() for k, v in gr.items())


@pytest.mark.parametrize("grid", [False, True])
def test_band_captured_with_changing_table(env, grid):
    # a captured call keeps nothing of the table it was captured with: the
    # lattice is chosen on the device at every replay, forward and adjoint
    torch, F, W = env
    cells = _mesh(_uniform((160, 141, 130), (1.6, 1.4, 1.3))) if grid else _cloud("even", 250_000, 3, 4)
    ell, n = (0.2, 0.2, 0.2), 4000
    plan = F.CellPlan(*to_dev(torch, cells))
    g = torch.from_numpy(np.random.default_rng(2).standard_normal(len(cells[0])).astype(np.float32)).cuda()
    p = _params(F, n, 3, ell)
    tables = []
    for law, seed in (("gaussian", 3), ("rough", 4)):
        m = _modes(n, 3, ell, law, seed)
        tables.append(F.ModeTable(m["amp"], m["psi"], m["a"]))
    call = F.PreparedSynth(p, plan)
    want = []
    for t in tables:
        y = call(t)["Y"].clone()
        want.append((y, F.backward(t, p, plan, g)["da"].clone()))
    ws = F.Workspace()
    F.backward(tables[0], p, plan, g, workspace=ws)
    torch.cuda.synchronize()
    table, graph, s = tables[0], torch.cuda.CUDAGraph(), torch.cuda.Stream()
    keep = table.dev.clone()
    with torch.cuda.stream(s):
        with torch.cuda.graph(graph, stream=s):
            out = call(table, stream=s)
            da = F.backward(table, p, plan, g, stream=s, workspace=ws)["da"]
    for k, content in ((0, keep), (1, tables[1].dev), (0, keep)):
        table.dev.copy_(content)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out["Y"], want[k][0]) and torch.equal(da, want[k][1])
