"""The mixed-precision mimetic stage kernel at the edges of its tiles (64 x 8
columns, pairs of nodes along x, kz planes per CTA): grids of a pair, one
node less and more than a tile, odd and even row lengths, slabs of one and
two planes, with the TMA tiles (nx a multiple of 4) and the plain copies,
against the FP64 oracle.  Tolerances are those of the FP32 stencils in
test_gpu_parity.py: 2e-4 of the largest velocity; a step's positions to 3e-4
of the largest move plus FP32 rounding of the displacement (a step beyond the
explicit scheme's stability limit would amplify the stages' rounding)."""
import numpy as np
import pytest

import glemur_inputs as gi
import oracle as ora

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1405_0942_gb300 as pkg
    pkg.lib()
    return pkg


DIMS = [(3, 3, 3), (4, 3, 5), (5, 8, 4), (62, 7, 6), (63, 9, 7), (64, 8, 3), (65, 10, 9),
        (66, 11, 5), (67, 17, 6), (68, 16, 8), (128, 9, 4), (129, 8, 5), (132, 18, 7)]


@pytest.mark.parametrize("kz", ["0", "1", "2", "3"])
@pytest.mark.parametrize("dims", DIMS, ids=lambda d: "x".join(map(str, d)))
def test_tile_edges(G, dims, kz, monkeypatch):
    monkeypatch.setenv("GLEMUR_KZ", kz)
    g = gi.Grid(*dims)
    X = gi.nodes(g)
    x0 = gi.predistort(X, 2)
    B0 = gi.braid_field(X, gi.braid_regions(6, None, True))
    u_ref, rc = ora.velocity(g, x0, B0, 0)
    assert rc == ora.OK
    dt = 0.1 * min(g.h) ** 2      # inside the explicit scheme's stability limit
    x_ref, _, rc = ora.step_fixed(g, x0, B0, dt, 0)
    assert rc == ora.OK
    E_ref, _ = ora.energy(g, x_ref, B0)
    move = np.abs(x_ref - x0).max()
    for tma in ("1", "0") if dims[0] % 4 == 0 else ("0",):
        monkeypatch.setenv("GLEMUR_TMA", tma)
        r = G.Relaxation(*dims, precision=G.MIXED)
        r.set_x(torch.from_numpy(x0).cuda())
        r.set_B0(torch.from_numpy(B0).cuda())
        u = r.velocity().cpu().numpy()
        assert np.abs(u - u_ref).max() <= 2e-4 * np.abs(u_ref).max(), tma
        ub = u.copy()
        ub[:, 1:-1, 1:-1, 1:-1] = 0
        assert np.all(ub == 0)                         # line-tied boundary
        st = r.step_fixed(dt)
        assert st["accepted"] == 1
        x = r.get_x().cpu().numpy()
        assert np.abs(x - x_ref).max() <= 3e-4 * move + 2e-7 * np.abs(x_ref - X).max(), tma
        keep = x.copy()
        keep[:, 1:-1, 1:-1, 1:-1] = x0[:, 1:-1, 1:-1, 1:-1]
        assert np.abs(keep - x0).max() <= 1e-8         # boundary positions (FP32 displacement)
        assert abs(r.energy() - E_ref) <= 1e-6 * E_ref
