"""Mixed-precision mimetic stages on grids whose rows take an odd, small
number of 32-node tiles, where 32-wide tiles replace the march's 64-wide
ones: one, three and five tiles to a row with the last one of a single node,
part full and full, rows with and without a 16-byte pitch, and neighbours on
the other side of the rule, against the FP64 oracle and against the march (a
context with planes per CTA given takes it).  Tolerances as in
test_gpu_march.py; two contexts differ by at most twice those, and the reverse
step's change of the adjoint, a product with Jacobians of the same stages, by
the velocity's tolerance."""
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


DIMS = [(3, 70, 90), (5, 64, 64), (16, 130, 66), (24, 64, 64), (25, 64, 64), (32, 150, 80),
        (33, 64, 64), (65, 64, 64), (66, 31, 200), (68, 64, 64), (93, 61, 63), (96, 64, 64),
        (97, 64, 64), (129, 63, 65), (130, 31, 120)]


@pytest.mark.parametrize("dims", DIMS, ids=lambda d: "x".join(map(str, d)))
def test_stages(G, dims, monkeypatch):
    g = gi.Grid(*dims)
    X = gi.nodes(g)
    x0 = gi.predistort(X, 2)
    B0 = gi.braid_field(X, gi.braid_regions(6, None, True))
    u_ref, rc = ora.velocity(g, x0, B0, 0)
    assert rc == ora.OK
    dt = 0.1 * min(g.h) ** 2
    x_ref, _, rc = ora.step_fixed(g, x0, B0, dt, 0)
    assert rc == ora.OK
    E_ref, _ = ora.energy(g, x_ref, B0)
    umax, move = np.abs(u_ref).max(), np.abs(x_ref - x0).max()
    tol_x = 3e-4 * move + 2e-7 * np.abs(x_ref - X).max()
    lam_next = torch.from_numpy(np.random.default_rng(7).standard_normal(x0.shape)).cuda()
    out = []
    for kz in ("0", "8"):
        monkeypatch.setenv("GLEMUR_KZ", kz)
        r = G.Relaxation(*dims, precision=G.MIXED)
        r.set_x(torch.from_numpy(x0).cuda())
        r.set_B0(torch.from_numpy(B0).cuda())
        u = r.velocity().cpu().numpy()
        assert np.abs(u - u_ref).max() <= 2e-4 * umax
        lam, mu = torch.zeros_like(lam_next), torch.zeros_like(lam_next)
        r.vjp_step(dt, lam_next, lam, mu)
        assert r.step_fixed(dt)["accepted"] == 1
        x = r.get_x().cpu().numpy()
        assert np.abs(x - x_ref).max() <= tol_x
        assert abs(r.energy() - E_ref) <= 1e-6 * E_ref
        out.append((u, x, (lam - lam_next).cpu().numpy(), mu.cpu().numpy()))
    (u0, a0, l0, m0), (u1, a1, l1, m1) = out
    assert np.abs(u0 - u1).max() <= 4e-4 * umax and np.abs(a0 - a1).max() <= 2 * tol_x
    assert np.abs(l0 - l1).max() <= 2e-4 * np.abs(l1).max()
    assert np.abs(m0 - m1).max() <= 2e-4 * np.abs(m1).max()
