"""The field conversions at the boundary (set_x, get_x, the raw state) at the
edges of their work split (256 nodes of the plane and 1, 2, 4 or 8 planes per
CTA, by the grid's size) and for every class of double: on grids whose labels are exact, so
that FP32 displacements are the rounding of an exact difference, bit for bit.
And set_x after a state of NaNs: only the boundary of the second state buffer
and of the stage inputs is written, so a step's results must not depend on
what their interiors held."""
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


SPECIAL = np.array([0.0, -0.0, 1.0 + 2.0**-24, 1.0 + 3 * 2.0**-24, 1.0 + 2.0**-24 + 2.0**-52,
                    -1.0 - 2.0**-25, 2.0 - 2.0**-25, 2.0**-126, -(2.0**-126) * (1 - 2.0**-25),
                    2.0**-127, 2.0**-149, 2.0**-150, 3e-46, 5e-324, -1e-310,
                    2.0**128 - 2.0**103, np.nextafter(2.0**128 - 2.0**103, 0.0), -1e39, 1e300,
                    np.inf, -np.inf, np.nan])


@pytest.mark.parametrize("precision,periodic", [(0, 0), (0, 1), (1, 0)],
                         ids=["fp64", "fp64-periodic", "mixed"])
@pytest.mark.parametrize("dims", [(3, 3, 3), (17, 15, 8), (16, 16, 9), (43, 6, 12), (17, 9, 33),
                                  (101, 99, 10), (101, 99, 21), (200, 130, 11)],
                         ids=lambda d: "x".join(map(str, d)))
def test_conversions_are_exact(G, dims, precision, periodic):
    lo = [-(n // 2) / 8 for n in dims]
    hi = [l + (n - 1) / 8 for l, n in zip(lo, dims)]      # h = 1/8: labels are exact
    lab = [l + np.arange(n) / 8 for l, n in zip(lo, dims)]
    X = np.stack(np.broadcast_arrays(lab[0][None, None, :], lab[1][None, :, None],
                                     lab[2][:, None, None])).copy()
    rng = np.random.default_rng(3)
    x = X + 0.1 * rng.standard_normal(X.shape)
    for c in range(3):                                    # label 0 along axis c: x is d
        zero = np.broadcast_to(X[c] == 0.0, X[c].shape)
        x[c][zero] = np.resize(SPECIAL, zero.sum())
    r = G.Relaxation(*dims, lo=lo, hi=hi, precision=precision, periodic_z=periodic or None)
    r.set_x(torch.from_numpy(x).cuda())
    t = np.float64 if precision == 0 else np.float32
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        d = (x - X).astype(t)
    if periodic:
        d[:, 0], d[:, -1] = (x[:, -2] - X[:, -2]).astype(t), (x[:, 1] - X[:, 1]).astype(t)
    got = r.get_state().cpu().numpy().view(t).reshape(d.shape)
    np.testing.assert_array_equal(got, d)
    assert np.array_equal(np.signbit(got[d == 0]), np.signbit(d[d == 0]))
    np.testing.assert_array_equal(r.get_x().cpu().numpy(), X + d.astype(np.float64))


@pytest.mark.parametrize("precision,curl,periodic",
                         [(0, 0, 0), (0, 1, 0), (0, 2, 0), (1, 0, 0), (1, 1, 0), (0, 0, 1),
                          (0, 2, 1)])
@pytest.mark.parametrize("dims", [(20, 11, 13), (33, 16, 9)], ids=lambda d: "x".join(map(str, d)))
def test_set_x_after_any_state(G, dims, precision, curl, periodic):
    g = gi.Grid(*dims)
    X = gi.nodes(g)
    x0 = torch.from_numpy(gi.predistort(X, 2)).cuda()
    B0 = torch.from_numpy(gi.braid_field(X, gi.braid_regions(6, None, True))).cuda()
    out = []
    for poison in (False, True):
        r = G.Relaxation(*dims, precision=precision, curl=curl, dt0=0.1 * min(g.h) ** 2,
                         periodic_z=periodic or None)
        r.set_B0(B0)
        if poison:
            r.set_state(torch.full_like(r.get_state(), 255))
        r.set_x(x0)
        u = r.velocity()
        r.step(3)
        res = [u, r.get_state(), r.get_x(), r.energy()]
        if curl == 0 and not periodic:
            res += list(r.adjoint_segment(x0, [1e-4, 2e-4, 1e-4], G.LOSS_ENERGY, 2))
        out.append([np.asarray(a.cpu() if torch.is_tensor(a) else a) for a in res])
    for a, b in zip(*out):
        assert np.isfinite(a.astype(np.float64)).all()
        assert a.tobytes() == b.tobytes()
