"""GPU tests that the node lattice (csrc/band.cuh) is what the large calls run
on: their results differ from those of the direct sums in rounding, and only in
rounding, on every route; and the checked library (index checks on the device)
takes the same routes and skips nothing."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from helpers import to_dev
from test_gpu_band import _cloud, _mesh, _modes, _params, _uniform, env  # noqa: F401

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

ROUTES = [("grid 2-D", _uniform((701, 499), (1.4, 1.0)), (0.2, 0.1), 6000),
          ("grid 2-D, many tiles", _uniform((1537, 1025), (1.5, 1.0)), (0.1, 0.2), 8000),
          ("grid 3-D, few tiles", _uniform((100, 81, 61), (1.0, 0.8, 0.6)), (0.2, 0.2, 0.2), 6000),
          ("grid 3-D", _uniform((257, 131, 65), (1.0, 0.5, 0.25)), (0.1, 0.1, 0.1), 3000),
          ("cells 2-D", None, (0.2, 0.25), 4000), ("cells 3-D", None, (0.2, 0.25, 0.2), 4000)]


# "rough" leaves modes for the direct sum on every route, "gaussian" none
@pytest.mark.parametrize("law", ["gaussian", "rough"])
@pytest.mark.parametrize("name,axes,ell,n", ROUTES, ids=[r[0] for r in ROUTES])
def test_large_calls_run_on_the_lattice(env, name, axes, ell, n, law):  # noqa: F811
    torch, F, W = env
    dim = len(ell)
    cells = _mesh(axes) if axes else _cloud("lattice", 300_000, dim, 3)
    plan = F.CellPlan(*to_dev(torch, cells))
    m = _modes(n, dim, ell, law, 3)
    table, p = F.ModeTable(m["amp"], m["psi"], m["a"]), _params(F, n, dim, ell)
    g = torch.randn(len(cells[0]), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")

    ws, wb = F.Workspace(), F.Workspace()

    def call():
        return F.synth(table, p, plan, workspace=ws)["Y"], F.backward(table, p, plan, g, workspace=wb)["dA"]

    y, da = call()
    chosen = [F.lattice_choice("synth", plan, p, ws)]
    if name not in ("grid 2-D", "grid 3-D, few tiles"):  # their adjoints keep the products
        chosen.append(F.lattice_choice("backward", plan, p, wb))
    for c in chosen:
        assert c["light"] > 0 and c["light"] + c["direct"] == n
        assert (c["direct"] > 0) == (law == "rough")
        assert all(k >= 8 for k in c["nodes"][:dim])
    try:
        F.grid_path("always" if axes else False)
        y0, da0 = call()
    finally:
        F.grid_path(True)
    torch.cuda.synchronize()
    assert not torch.equal(y, y0)
    assert (y - y0).abs().max().item() <= 2e-5  # twice the forward tolerance of either
    if len(chosen) == 1:
        return
    assert not torch.equal(da, da0)
    assert (da - da0).abs().max().item() <= 2e-4 * da0.abs().max().item()


CHILD = r'''
import ctypes, json, sys
import numpy as np
import torch
sys.path.insert(0, ROOT)
sys.path.insert(0, ROOT + "/tests")
from paper_2212_10961_gb300 import _abi, field as F
import test_gpu_band as B

L = _abi.lib()
assert L.grf_checked_build() == 1
env = (torch, F, None)
faults = ctypes.c_int64(-1)
_abi.check(L.grf_take_index_faults(ctypes.byref(faults)))
for law in ("gaussian", "rough"):
    B._check_grid(env, B._uniform((257, 131, 65), (1.0, 0.5, 0.25)), (0.1, 0.1, 0.1), 3000, law)
    B._check_grid(env, B._uniform((701, 499), (1.4, 1.0)), (0.2, 0.1), 6000, law)
    B._check_adjoint(env, B._mesh(B._uniform((129, 101, 90), (1.29, 1.0, 0.9))), (0.2, 0.2, 0.2), 4097, law)
    B._check_cells(env, B._cloud("lattice", 262_144, 3, 3), (0.2, 0.25, 0.2), 5003, law)
    B._check_adjoint(env, B._cloud("clusters", 300_000, 3, 3), (0.2, 0.25, 0.2), 4000, law)
_abi.check(L.grf_take_index_faults(ctypes.byref(faults)))
print("RESULT " + json.dumps(faults.value))
'''


def test_checked_library_on_the_lattice():
    import __graft_entry__
    __graft_entry__.build()
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + CHILD], env=dict(os.environ, GRF_LIBRARY="checked"),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert [ln for ln in r.stdout.splitlines() if ln.startswith("RESULT ")] == ["RESULT 0"]
