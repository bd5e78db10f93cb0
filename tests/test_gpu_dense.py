"""The dense FP64 passes at the edges of their shares: grids of a single
interior row along each axis, boundary groups (faces, edges, corners) of one
node less and more than a warp, fewer node warps than SMs and a few rounds of
them, for the three currents against the FP64 oracle.  Tolerances are those of
test_gpu_parity.py for the same quantities: 1e-11 of the largest velocity,
1e-13 of the energy, 1e-12 of the largest position after a step (at a step
inside the explicit scheme's stability limit)."""
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


DIMS = [(3, 3, 40), (41, 3, 3), (3, 37, 4), (34, 34, 3), (35, 6, 5), (10, 4, 6), (18, 18, 3),
        (50, 33, 18), (61, 47, 44)]


@pytest.mark.parametrize("curl", [0, 1, 2], ids=["mimetic", "direct", "nnn"])
@pytest.mark.parametrize("dims", DIMS, ids=lambda d: "x".join(map(str, d)))
def test_dense_passes(G, dims, curl):
    g = gi.Grid(*dims)
    X = gi.nodes(g)
    x0 = gi.predistort(X, 2)
    B0 = gi.braid_field(X, gi.braid_regions(6, None, True))
    r = G.Relaxation(*dims, curl=curl)
    r.set_x(torch.from_numpy(x0).cuda())
    r.set_B0(torch.from_numpy(B0).cuda())
    u_ref, rc = ora.velocity(g, x0, B0, curl)
    assert rc == ora.OK
    u = r.velocity().cpu().numpy()
    assert np.abs(u - u_ref).max() <= 1e-11 * np.abs(u_ref).max()
    E_ref, _ = ora.energy(g, x0, B0)
    assert abs(r.energy() - E_ref) <= 1e-13 * E_ref
    dt = 0.1 * min(g.h) ** 2
    x_ref, _, rc = ora.step_fixed(g, x0, B0, dt, curl)
    assert rc == ora.OK
    assert r.step_fixed(dt)["accepted"] == 1
    x = r.get_x().cpu().numpy()
    assert np.abs(x - x_ref).max() <= 1e-12 * np.abs(x_ref).max()
