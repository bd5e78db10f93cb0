"""glemur_alpha_line at the edges of its work split (36 nodes per CTA, the
pairs' CTA of 64 or 256 threads from 67 nodes on) and glemur_convexity on a
grid scrambled so that every neighbour octant decides some node, against the
FP64 oracle.  alpha* to 1e-10 (FP64) or 1e-3 (FP32 state) of its largest value
on the line, as in test_gpu_diagnostics.py; epsilon* is a_r times a difference
of two of them over at least h_z, hence to 2 a_r / h_z of that bound.  kappa
is the sign of FP64 determinants, none of them near zero: equal node for
node."""
import math

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


def relaxation(G, g, x, B0, precision, curl=0):
    r = G.Relaxation(g.nx, g.ny, g.nz, g.lo, g.hi, precision=precision, curl=curl)
    r.set_x(torch.from_numpy(np.ascontiguousarray(x)).cuda())
    r.set_B0(torch.from_numpy(np.ascontiguousarray(B0)).cuda())
    return r


LINES = [(0, 4), (0, 36), (0, 37), (0, 66), (0, 67), (0, 72), (0, 73), (0, 300), (1, 36), (1, 37)]


# (three planes only with the mimetic current: the direct one's alpha* on the
# single middle plane is zero by symmetry, which leaves no scale)
@pytest.mark.parametrize("curl,precision,nz", [(0, 0, 3), (0, 1, 3)]
                         + [(c, p, nz) for c in (0, 1) for p, nz in LINES])
def test_line_split(G, curl, precision, nz):
    g = gi.Grid(9, 7, nz)
    X = gi.nodes(g)
    B0 = gi.braid_field(X, gi.braid_regions(6, None, True))
    r = relaxation(G, g, gi.predistort(X, 2), B0, precision, curl)
    x = r.get_x().cpu().numpy()
    a_r = math.sqrt(2.0)
    for (i, j) in [(4, 3), (1, 1), (7, 5)]:
        a, e = r.alpha_line(i, j, a_r)
        a_o, e_o, rc = ora.alpha_line(g, x, B0, i, j, a_r, curl)
        assert rc == ora.OK
        assert np.isnan(a[0]) and np.isnan(a[-1])
        tol = (1e-10 if precision == 0 else 1e-3) * np.abs(a_o[1:-1]).max()
        assert np.abs(a[1:-1] - a_o[1:-1]).max() <= tol, (i, j)
        assert abs(e - e_o) <= 2 * a_r / g.h[2] * tol, (i, j, e, e_o)


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("dims", [(3, 3, 3), (17, 9, 11), (33, 20, 14)],
                         ids=lambda d: "x".join(map(str, d)))
def test_convexity_scrambled(G, dims, precision):
    g = gi.Grid(*dims)
    X = gi.nodes(g)
    rng = np.random.default_rng(7)
    h = np.array(g.h).reshape(3, 1, 1, 1)
    x0 = X + 0.3 * h * rng.uniform(-1.0, 1.0, X.shape)
    r = relaxation(G, g, x0, gi.uniform_field(g), precision)
    n, kap = r.convexity(with_field=True)
    k_o, n_o = ora.convexity(g, r.get_x().cpu().numpy())
    assert n == n_o
    assert np.array_equal(kap.cpu().numpy().astype(np.int32), k_o)
    if dims[0] > 3:
        assert 0 < n_o < np.prod(dims)
