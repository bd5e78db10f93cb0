"""A mixed-precision raw state keeps its boundary entries bit for bit over a
step: line-tied nodes do not move, whatever their displacement's bits (a
negative zero among them)."""
import numpy as np
import pytest

import glemur_inputs as gi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1405_0942_gb300 as pkg
    pkg.lib()
    return pkg


@pytest.mark.parametrize("tma", ["1", "0"], ids=["tma", "copies"])
@pytest.mark.parametrize("curl", [0, 1], ids=["mimetic", "direct"])
@pytest.mark.parametrize("dims", [(12, 9, 8), (13, 9, 8), (68, 10, 7)],
                         ids=lambda d: "x".join(map(str, d)))
def test_boundary_bits(G, dims, curl, tma, monkeypatch):
    monkeypatch.setenv("GLEMUR_TMA", tma)
    nx, ny, nz = dims
    X = gi.nodes(gi.Grid(*dims))
    r = G.Relaxation(*dims, precision=G.MIXED, curl=curl)
    h = 2.0 / (max(dims) - 1)
    d0 = 0.05 * h * np.random.default_rng(3).uniform(-1, 1, X.shape)
    r.set_x(torch.from_numpy(X + d0).cuda())
    r.set_B0(torch.from_numpy(gi.braid_field(X, gi.braid_regions(6, None, True))).cuda())
    raw = r.get_state()
    d = raw.view(torch.float32)[:3 * nx * ny * nz].view(3, nz, ny, nx)
    inner = torch.zeros(nz, ny, nx, dtype=torch.bool, device=d.device)
    inner[1:-1, 1:-1, 1:-1] = True
    d[:, ~inner] = -0.0
    before = d.view(torch.int32).clone()
    r.set_state(raw)
    for n in (1, 2):          # both displacement buffers
        assert r.step_fixed(0.05 * h * h)["accepted"] == n
        after = r.get_state().view(torch.float32)[:3 * nx * ny * nz].view(3, nz, ny, nx)
        after = after.view(torch.int32)
        assert torch.equal(after[:, ~inner], before[:, ~inner])
        assert not torch.equal(after[:, inner], before[:, inner])
