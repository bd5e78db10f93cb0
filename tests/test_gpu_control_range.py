"""The step control at error norms below the smallest normal double: an
accepted attempt whose Lambda is positive but subnormal grows the step by
grow_max (eq. "time stepping" with the ratio lambda0 / Lambda beyond the
double range), as one with Lambda = 0 does, and the run goes on.

The norm is made subnormal by the field's strength: the displacements of an
attempt are of the order of dt |B|^2, so with |B| near 1e-147 every stage
input rounds to the state, the six k agree, and the embedded error is the
rounding of sum_j e_j k_j, about 1e-17 dt max |k|, here placed near 1e-315.
The step sizes are exact: dt0 times a power of grow_max."""
import numpy as np
import pytest

import glemur_inputs as gi
import oracle as ora

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
SMALLEST_NORMAL = 2.2250738585072014e-308


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1405_0942_gb300 as pkg
    pkg.lib()
    return pkg


@pytest.mark.parametrize("persist", ["0", "1"], ids=["launches", "persistent"])
def test_subnormal_error_norm_grows_the_step(G, persist, monkeypatch):
    monkeypatch.setenv("GLEMUR_PERSIST", persist)
    g = gi.Grid(12, 11, 13)
    X = gi.nodes(g)
    x0 = gi.predistort(X, 2)
    B1 = gi.braid_field(X, gi.braid_regions(6, None, True))
    u, rc = ora.velocity(g, x0, B1, 0)
    assert rc == ora.OK
    dt0, grow = 1e-3, 5.0
    B0 = B1 * np.sqrt(1e-315 / (1e-17 * dt0 * np.abs(u).max()))
    r = G.Relaxation(12, 11, 13, dt0=dt0, grow_max=grow)
    r.set_x(torch.from_numpy(x0).cuda())
    r.set_B0(torch.from_numpy(B0).cuda())
    x_start = r.get_x()
    r.attempts(1)
    st = r.stats()
    assert st["accepted"] == 1 and 0.0 < st["lam"] < SMALLEST_NORMAL
    assert st["dt"] == dt0 * grow
    r.attempts(1)
    st = r.stats()
    assert st["status"] == 0 and st["accepted"] == 2 and st["t"] == dt0 + dt0 * grow
    assert st["dt"] == dt0 * grow * grow
    assert torch.equal(r.get_x(), x_start)
