"""The mixed-precision mimetic stages on long, thin grids: more z-slabs of
the schedule's usual length than a launch's z extent may count (65535).  A
step's displacements at the far end of the grid against the FP64 oracle on a
cut of it (a step reaches two planes per stage, twelve in all).  Tolerance:
that of the FP32 stencils in test_gpu_march.py, 3e-4 of the largest move plus
2e-7 of the largest displacement, plus the rounding of positions stored at
labels up to 2^19, 2^-33."""
import numpy as np
import pytest

import glemur_inputs as gi
import oracle as ora

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

H = 0.125                     # node spacing; exact labels
NZ = 40 * 65535 + 3           # one slab of 40 planes too many, and a ragged one
CUT, REACH = 48, 12


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1405_0942_gb300 as pkg
    pkg.lib()
    return pkg


@pytest.mark.parametrize("kz", ["0", "1"], ids=["schedule", "one plane"])
@pytest.mark.parametrize("nx", [3, 4], ids=["copies", "tma"])
def test_more_slabs_than_a_launch_counts(G, nx, kz, monkeypatch):
    monkeypatch.setenv("GLEMUR_KZ", kz)
    ny = 3
    r = G.Relaxation(nx, ny, NZ, lo=(0, 0, 0), hi=((nx - 1) * H, (ny - 1) * H, (NZ - 1) * H),
                     precision=G.MIXED)
    dev = dict(dtype=torch.float64, device="cuda")
    k = torch.arange(NZ, **dev).view(NZ, 1, 1)
    z, y, x = torch.broadcast_tensors(k * H, torch.arange(ny, **dev).view(1, ny, 1) * H,
                                      torch.arange(nx, **dev).view(1, 1, nx) * H)
    X = torch.stack([x, y, z])
    d = torch.zeros_like(X)
    for c in range(3):        # single precision, as the mixed state stores it
        d[c, 1:-1, 1:-1, 1:-1] = (0.02 * torch.sin(0.7 * k + 1.1 * c)).float().double()[1:-1]
    B0 = torch.stack([0.3 * torch.sin(z + y), 0.3 * torch.cos(z - x), 1.0 + 0.2 * torch.sin(x + y)])
    r.set_x(X + d)
    r.set_B0(B0)
    dt = 0.1 * H * H
    assert r.step_fixed(dt)["accepted"] == 1
    cut = slice(NZ - CUT, NZ)
    got = (r.get_x()[:, cut] - X[:, cut]).cpu().numpy()
    g = gi.Grid(nx, ny, CUT, lo=(0.0, 0.0, 0.0), hi=((nx - 1) * H, (ny - 1) * H, (CUT - 1) * H))
    Xc = gi.nodes(g)
    d0 = d[:, cut].cpu().numpy()
    x1, _, rc = ora.step_fixed(g, Xc + d0, B0[:, cut].cpu().numpy().copy(), dt, 0)
    assert rc == ora.OK
    want = x1 - Xc
    far = slice(REACH + 1, None)
    move = np.abs(want - d0)[:, far].max()
    tol = 3e-4 * move + 2e-7 * np.abs(d0).max() + 2.0 ** -33
    assert move > 100 * tol
    assert np.abs(got - want)[:, far].max() <= tol
