"""GPU tests of the node lattice near the limits of its tables: cells of any
plan whose field varies much faster along one axis than along the others, so
that one axis takes as many nodes as the selection allows."""
import numpy as np
import pytest

from helpers import check_forward, oracle_field, to_dev
from test_gpu_band import _check_adjoint, _check_grid, _modes, _params, env  # noqa: F401

pytestmark = pytest.mark.gpu

GUARD = 1 << 20


class _Guarded:
    """A workspace of exactly the bytes asked for, inside a larger allocation
    whose other bytes must stay as they are."""

    def __init__(self, torch):
        self.torch, self.all = torch, None

    def get(self, nbytes, device):
        n = (int(nbytes) + 255) // 256 * 256
        self.all = self.torch.full((n + 2 * GUARD,), 0xa5, dtype=self.torch.uint8, device=device)
        return self.all[GUARD:GUARD + n]

    def untouched(self):
        return bool((self.all[:GUARD] == 0xa5).all()) and bool((self.all[-GUARD:] == 0xa5).all())


@pytest.mark.parametrize("fine", [0, 1, 2])
@pytest.mark.parametrize("cells", [100_000, 262_144])
def test_one_fine_axis(env, cells, fine):  # noqa: F811
    torch, F, W = env
    ell = [0.3, 0.3, 0.3]
    ell[fine] = 0.01
    c = [np.ascontiguousarray(v) for v in np.random.default_rng(5).random((cells, 3)).astype(np.float32).T]
    n = 4096
    _check_adjoint(env, c, tuple(ell), n, "gaussian")
    plan = F.CellPlan(*to_dev(torch, c))
    m = _modes(n, 3, tuple(ell), "gaussian", 6)
    table, p = F.ModeTable(m["amp"], m["psi"], m["a"]), _params(F, n, 3, tuple(ell))
    g = torch.randn(cells, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    ws = _Guarded(torch)
    guarded = F.backward(table, p, plan, g, workspace=ws)
    assert ws.untouched()
    plain = F.backward(table, p, plan, g)
    assert all(torch.equal(guarded[k], plain[k]) for k in ("dA", "dpsi", "da"))
    ws = _Guarded(torch)
    y = F.synth(table, p, plan, workspace=ws)["Y"].cpu().numpy()
    assert ws.untouched()
    idx = np.random.default_rng(2).choice(cells, 6000, replace=False)
    check_forward(y[idx], oracle_field(m, 0.25, c, idx), 1.0, "fine axis %d" % fine)


def test_frequencies_whose_scale_underflows(env):  # noqa: F811
    # one mode of 2e-36 turns per unit among constant ones, over 3e38 units: the
    # squared mean of the roots underflows, so that every mode looks constant
    # and the selection's estimate is 9 nodes an axis; the mode needs 2000
    torch, F, W = env
    cells, n = 300_000, 60_000
    c = [np.ascontiguousarray(v) for v in (np.random.default_rng(5).random((cells, 3)) * 3e38).astype(np.float32).T]
    ell = (1e35,) * 3
    m = _modes(n, 3, ell, "gaussian", 6)
    m["a"][:] = 0.0
    m["a"][17, 0] = 2e-36
    m["amp"][17] = 1.0
    plan = F.CellPlan(*to_dev(torch, c))
    ws = _Guarded(torch)
    y = F.synth(F.ModeTable(m["amp"], m["psi"], m["a"]), _params(F, n, 3, ell), plan, workspace=ws)["Y"].cpu().numpy()
    assert ws.untouched() and plan.status() == 0
    idx = np.random.default_rng(2).choice(cells, 6000, replace=False)
    check_forward(y[idx], oracle_field(m, 0.25, c, idx), 1.0, "underflowing frequencies")


@pytest.mark.parametrize("order", ["running", "random"])
def test_long_x_axis(env, order):  # noqa: F811
    # 32,768 x cells: the light modes' chunks get part of what an axis in no
    # order would need (each tile of it reads nearly all nodes)
    axes = [np.linspace(0.0, 400.0, 32_768).astype(np.float32), np.linspace(0.0, 0.4, 32).astype(np.float32),
            np.linspace(0.0, 0.2, 16).astype(np.float32)]
    if order == "random":
        axes[0] = np.random.default_rng(3).permutation(axes[0])
    _check_grid(env, axes, (0.3, 0.3, 0.3), 1000, "rough")


@pytest.mark.parametrize("order", ["running", "back", "random", "gap", "crowd"])
def test_long_x_axis_adjoint(env, order):  # noqa: F811
    # rows of several staged pieces: each 32 nodes take the cells that they
    # weigh, ordered by node on an axis in no order (unless they crowd at few
    # nodes), none for nodes inside a gap
    x = np.linspace(0.0, 40.0, 5003).astype(np.float32)
    if order == "back":
        x = np.ascontiguousarray(x[::-1])
    if order == "crowd":
        x[::2] *= np.float32(1e-3)
        x = np.random.default_rng(3).permutation(x)
    if order == "random":
        x = np.random.default_rng(3).permutation(x)
    if order == "gap":
        x = np.where(x > 20.0, x + np.float32(30.0), x)
    axes = [x, np.linspace(0.0, 0.4, 37).astype(np.float32), np.linspace(0.0, 0.2, 31).astype(np.float32)]
    m = np.meshgrid(*axes[::-1], indexing="ij")
    cells = [np.ascontiguousarray(v.ravel()) for v in m[::-1]]
    _check_adjoint(env, cells, (0.3, 0.3, 0.3), 2000, "gaussian")


def test_adjoint_with_every_axis_in_random_order(env):  # noqa: F811
    rng = np.random.default_rng(7)
    axes = [rng.permutation(np.linspace(0.0, e, n).astype(np.float32)) for n, e in ((300, 1.0), (141, 0.9), (130, 0.8))]
    m = np.meshgrid(*axes[::-1], indexing="ij")
    cells = [np.ascontiguousarray(v.ravel()) for v in m[::-1]]
    for law in ("gaussian", "rough"):
        _check_adjoint(env, cells, (0.15, 0.2, 0.2), 3000, law)


@pytest.mark.parametrize("law", ["gaussian", "rough"])
def test_wide_random_x_axis(env, law):  # noqa: F811
    # 2-D: a block's cells read more x nodes than it stages at a time
    axes = [np.random.default_rng(3).permutation(np.linspace(0.0, 60.0, 3001).astype(np.float32)),
            np.linspace(0.0, 0.4, 400).astype(np.float32)]
    _check_grid(env, axes, (0.3, 0.3), 2000, law)


def _launches(F, torch, table, p, plan):
    n = F.launch_count()
    F.synth(table, p, plan)
    torch.cuda.synchronize()
    return F.launch_count() - n


@pytest.mark.parametrize("shape,ell,n,law,offset,lattice", [
    ((128, 128), 0.2, 5600, "gaussian", 0.0, False),       # 47 us directly, 51 with the lattice
    ((250, 130), 0.2, 3700, "gaussian", 0.0, False),       # 50 and 52
    ((250, 130), 0.2, 5600, "gaussian", 0.0, True),        # 68 and 51
    ((64, 60, 50), 0.2, 1400, "gaussian", 0.0, True),      # 111 and 62
    ((64, 60, 50), 0.2, 1400, "gaussian", 2.0e4, False),   # nodes beyond 2^16 spacings from 0: the device refuses
    ((96, 80, 70), 0.2, 4000, "grid", 2.0e4, False),       # the same on a grid
])
def test_calls_that_cannot_gain_are_not_tried(env, shape, ell, n, law, offset, lattice):  # noqa: F811
    torch, F, W = env
    dim = len(shape)
    rng = np.random.default_rng(4)
    h = 1.0 / max(shape)
    axes = np.meshgrid(*[(np.arange(k) + 0.5) * h for k in shape[::-1]], indexing="ij")[::-1]
    cells = [(v.ravel() + offset + (0.0 if law == "grid" else 0.4 * h) * rng.uniform(-1, 1, v.size)).astype(np.float32) for v in axes]
    plan = F.CellPlan(*to_dev(torch, [np.ascontiguousarray(c) for c in cells]))
    m = _modes(n, dim, (ell,) * dim, "gaussian", 6)
    table, p = F.ModeTable(m["amp"], m["psi"], m["a"]), _params(F, n, dim, (ell,) * dim)
    taken = _launches(F, torch, table, p, plan)
    try:
        F.grid_path("always" if law == "grid" else False)
        direct = _launches(F, torch, table, p, plan)
    finally:
        F.grid_path(True)
    assert (taken > direct) == lattice


def test_adjoint_of_the_largest_finite_gradient(env):  # noqa: F811
    # max |g| just below the largest float is finite
    c = [np.ascontiguousarray(v) for v in np.random.default_rng(5).random((250_000, 3)).astype(np.float32).T]
    g = np.zeros(250_000, dtype=np.float32)
    g[1234] = 3.1e38
    _check_adjoint(env, c, (0.2, 0.2, 0.2), 4000, "gaussian", g=g)


@pytest.mark.parametrize("ell,lattice", [(0.08, False), (0.2, True)])  # 254 us directly, 318 with the lattice; 244 and 143
def test_adjoints_that_cannot_gain_are_not_tried(env, ell, lattice):  # noqa: F811
    torch, F, W = env
    rng = np.random.default_rng(3)
    axes = np.stack(np.meshgrid(np.arange(24), np.arange(26), np.arange(27), indexing="ij"), 0).reshape(3, -1)
    c = ((axes + 0.5 + rng.uniform(-0.4, 0.4, axes.shape)) / 27).astype(np.float32)
    plan = F.CellPlan(*to_dev(torch, list(c)))
    m = _modes(4000, 3, (ell,) * 3, "gaussian", 6)
    table, p = F.ModeTable(m["amp"], m["psi"], m["a"]), _params(F, 4000, 3, (ell,) * 3)
    g = torch.ones(c.shape[1], device="cuda")
    counts = []
    for setting in (True, False):
        F.grid_path(setting)
        try:
            n = F.launch_count()
            F.backward(table, p, plan, g)
            counts.append(F.launch_count() - n)
        finally:
            F.grid_path(True)
    assert (counts[0] > counts[1]) == lattice
