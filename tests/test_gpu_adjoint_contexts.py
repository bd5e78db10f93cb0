"""The reverse step beside its context: in FP64 contexts whose stages are
single kernels (GLEMUR_F64_FUSED=1, no stage data kept) as in the two-pass
ones, against the complex-step oracle; and without a trace in the forward run
that goes on afterwards.  Tolerance of the products: 1e-9, as in
test_gpu_adjoint.py."""
import numpy as np
import pytest

import glemur_inputs as gi
import oracle as ora

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
H = ora.CSTEP_H


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1405_0942_gb300 as pkg
    pkg.lib()
    return pkg


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def case(nx, ny, nz):
    g = gi.Grid(nx, ny, nz)
    X = gi.nodes(g)
    B0 = gi.braid_field(X, gi.braid_regions(6, None, True, l=0.35, L=0.3))
    mask = np.zeros((3, nz, ny, nx))
    mask[:, 1:-1, 1:-1, 1:-1] = 1.0
    return g, gi.predistort(X, 2), B0, mask


@pytest.mark.parametrize("fused", ["0", "1"], ids=["two-pass", "fused"])
@pytest.mark.parametrize("dims", [(12, 11, 13), (3, 9, 5), (33, 6, 4)],
                         ids=lambda d: "x".join(map(str, d)))
def test_reverse_step(G, dims, fused, monkeypatch):
    monkeypatch.setenv("GLEMUR_F64_FUSED", fused)
    g, x0, B0, mask = case(*dims)
    dt = 0.1 * min(g.h) ** 2
    rng = np.random.default_rng(5)
    lam_next = rng.standard_normal(x0.shape) * mask
    v = rng.standard_normal(x0.shape) * mask
    w = rng.standard_normal(B0.shape)
    _, x1v, rc = ora.cs_relax_loss(g, x0 + 1j * H * v, B0, [dt])
    assert rc == ora.OK
    _, x1w, _ = ora.cs_relax_loss(g, x0, B0 + 1j * H * w, [dt])
    r = G.Relaxation(*dims)
    r.set_x(cuda(x0))
    r.set_B0(cuda(B0))
    lam = torch.zeros_like(cuda(x0))
    mu = torch.zeros_like(lam)
    r.vjp_step(dt, cuda(lam_next), lam, mu)
    want_x = (lam_next * (x1v.imag / H)).sum()
    want_b = (lam_next * (x1w.imag / H)).sum()
    assert abs((lam.cpu().numpy() * v).sum() - want_x) < 1e-9 * abs(want_x)
    assert abs((mu.cpu().numpy() * w).sum() - want_b) < 1e-9 * abs(want_b)


@pytest.mark.parametrize("precision,fused", [(0, "0"), (0, "1"), (1, "0")],
                         ids=["two-pass", "fused", "mixed"])
def test_forward_run_goes_on_unchanged(G, precision, fused, monkeypatch):
    monkeypatch.setenv("GLEMUR_F64_FUSED", fused)
    g, x0, B0, mask = case(14, 13, 15)
    out = []
    for reverse in (False, True):
        r = G.Relaxation(14, 13, 15, precision=precision)
        r.set_x(cuda(x0))
        r.set_B0(cuda(B0))
        r.step(2)
        if reverse:
            lam, mu = torch.zeros_like(cuda(x0)), torch.zeros_like(cuda(x0))
            r.vjp_step(1e-3, cuda(mask), lam, mu)
            r.loss_grad(0, lam, mu)
            r.loss_grad(1, lam, mu)
        for _ in range(2):
            r.step_fixed(1e-3)
        out.append((r.get_x(), r.velocity(), r.energy()))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]
