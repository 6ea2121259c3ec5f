"""CPU checks of the node lattice's workspace (csrc/band.cuh): the tables hold
every lattice that the device's selection may choose, whatever the cells'
shape and the number of modes."""
import ctypes

import pytest

from paper_2212_10961_gb300 import _abi

CELLS, CELLS_ADJOINT, GRID, GRID_ADJOINT = range(4)
FIELDS = ("limit_x", "limit_y", "limit_z", "held_x", "held_y", "held_z", "nodes", "nodes_held", "bytes", "base")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def room(kind, dim, cells, n_modes):
    cells = (list(cells) + [1, 1, 1])[:3]
    out = (ctypes.c_int64 * 10)()
    _abi.check(_abi.lib().grf_debug_lattice_room(kind, dim, (ctypes.c_int64 * 3)(*cells), n_modes, out))
    return dict(zip(FIELDS, out))


CASES = [(kind, dim, (n,), modes)
         for kind in (CELLS, CELLS_ADJOINT) for dim in (2, 3)
         for n in (30_000, 65_537, 100_000, 262_144, 2_000_376, 2 ** 24) for modes in (1000, 4096, 60_000)]
CASES += [(kind, 3 if len(shape) > 2 else 2, shape, modes)
          for kind in (GRID, GRID_ADJOINT)
          for shape in ((256, 256, 256), (2003, 8, 90), (33, 40, 601), (1401, 999), (70_000, 40), (65_536, 16, 16))
          for modes in (1000, 6000)]


@pytest.mark.parametrize("kind,dim,cells,modes", CASES)
def test_tables_hold_every_lattice_the_selection_accepts(kind, dim, cells, modes):
    r = room(kind, dim, cells, modes)
    if r["bytes"] == 0:
        assert not any(r.values())
        return
    for c in "xyz"[:dim]:
        assert r["limit_" + c] <= r["held_" + c], c
    assert r["nodes"] <= r["nodes_held"]


@pytest.mark.parametrize("shape,modes", [((66_000, 16_384), 65_000), ((70_000, 30_000), 40_000), ((16, 70_000, 500), 50_000),
                                         ((9, 900, 70_000), 33_000), ((32_768, 2048), 65_536), ((16_384, 2048), 65_536)])
def test_adjoint_tables_stay_within_32_bit_indices(shape, modes):
    r = room(GRID_ADJOINT, len(shape), shape, modes)
    n_pad = (modes + 127) // 128 * 128
    assert all(r["held_" + c] * n_pad < 2 ** 31 for c in "xyz")


BIG = [(GRID, 3, s, 1024) for s in ((32_768, 32, 16), (65_536, 16, 16), (262_144, 16, 16), (1_000_000, 32, 16))]
BIG += [(k, len(s), s, m) for k in (GRID, GRID_ADJOINT) for s in ((256, 256, 256), (70_000, 40), (65_536, 16, 16))
        for m in (4096, 60_000)]
BIG += [(k, d, (n,), m) for k in (CELLS, CELLS_ADJOINT) for d in (2, 3) for n in (70_000, 2_000_376, 2 ** 26)
        for m in (8192, 65_536)]


@pytest.mark.parametrize("kind,dim,cells,modes", BIG)
def test_workspace_stays_within_its_bound(kind, dim, cells, modes):
    # 1 GB, or 64 bytes per cell where that is more (grids: with the grid path's own tables)
    r = room(kind, dim, cells, modes)
    n = 1
    for c in cells:
        n *= c
    assert r["bytes"] + r["base"] <= max(2 ** 30, 64 * n)


@pytest.mark.parametrize("shape,modes", [((256, 256, 256), 8192), ((65_536, 16, 16), 1024), ((262_144, 16, 16), 1024)])
def test_long_grids_keep_the_lattice(shape, modes):
    assert room(GRID, 3, shape, modes)["bytes"] > 0


def test_large_calls_are_offered_the_lattice():
    # so that the cases above are not all empty
    assert all(room(k, 3, c, 4096)["bytes"] > 0
               for k, c in ((CELLS, (2_000_000,)), (CELLS_ADJOINT, (2_000_000,)), (GRID, (256,) * 3), (GRID_ADJOINT, (256,) * 3)))
