"""Programmatic dependent launch changes when a kernel may start, never what
it computes, on the paths whose kernels read ahead of their wait: the mixed
march on grids that leave no room beside them (the next launch enters as
CTAs leave) and that do, with both loaders, the mixed direct stages before
the step control, the next-nearest-neighbour pass, periodic z, and the
reverse step.  Ordinary launches (GLEMUR_PDL=0, read once per process, so in
a child process) give the same bits."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# name: nx, ny, nz, precision, curl, periodic_z, adjoint
CASES = {
    "march-tma-large": (128, 128, 96, 1, 0, 0, 0),
    "march-copies-large": (129, 120, 90, 1, 0, 0, 0),
    "march-tma-small": (64, 24, 20, 1, 0, 0, 0),
    "mixed-direct": (70, 40, 33, 1, 1, 0, 0),
    "nnn": (33, 30, 29, 0, 2, 0, 0),
    "periodic": (32, 30, 28, 0, 0, 1, 0),
    "adjoint": (34, 31, 30, 0, 0, 0, 1),
    "adjoint-mixed": (36, 31, 30, 1, 0, 0, 1),
}

CHILD = r"""
import json, sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1])
import paper_1405_0942_gb300 as G
import glemur_inputs as gi
out = {}
for name, (nx, ny, nz, prec, curl, per, adj) in json.loads(sys.argv[2]).items():
    if per:
        g, x0, B0 = gi.periodic_case(nx, ny, nz)
    else:
        g = gi.Grid(nx, ny, nz)
        X = gi.nodes(g)
        x0 = gi.predistort(X, 2)
        B0 = gi.braid_field(X, gi.braid_regions(6, None, True))
    r = G.Relaxation(g.nx, g.ny, g.nz, g.lo, g.hi, precision=prec, curl=curl, periodic_z=per,
                     diag_each_attempt=1, dt0=1e-4)
    xs = torch.from_numpy(x0).cuda()
    r.set_x(xs)
    r.set_B0(torch.from_numpy(B0).cuda())
    if adj:
        value, mu, lam = r.adjoint_segment(xs, [1e-4] * 5, 0, 2)
        np.save(sys.argv[3] + f"_{name}.npy", np.stack([mu.cpu().numpy(), lam.cpu().numpy()]))
        out[name] = value
    else:
        r.attempts(8)
        np.save(sys.argv[3] + f"_{name}.npy", r.get_x().cpu().numpy())
        st = r.stats()
        out[name] = [st[k] for k in ("accepted", "rejected", "dt", "t", "lam", "energy", "xi",
                                     "status")]
print(json.dumps(out))
"""


@pytest.fixture(scope="module")
def runs(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("pdl")
    out = {}
    for pdl in ("1", "0"):
        res = subprocess.run([sys.executable, "-c", CHILD, ROOT, json.dumps(CASES),
                              str(tmp / pdl)], env=dict(os.environ, GLEMUR_PDL=pdl),
                             capture_output=True, text=True, timeout=600)
        assert res.returncode == 0, res.stderr[-2000:]
        out[pdl] = json.loads(res.stdout.strip().splitlines()[-1])
    return tmp, out


@pytest.mark.parametrize("name", list(CASES))
def test_same_bits_as_ordinary_launches(runs, name):
    tmp, out = runs
    # NaN fields (the direct current has no energy) compare by their text
    assert json.dumps(out["1"][name]) == json.dumps(out["0"][name])
    a, b = (np.load(tmp / f"{p}_{name}.npy") for p in ("1", "0"))
    assert np.isfinite(a).all() and np.array_equal(a, b)
    if not CASES[name][-1]:
        assert out["1"][name][0] >= 1 and out["1"][name][-1] == 0
