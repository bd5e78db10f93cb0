"""Size of the reverse step's workspace (a host function, no GPU): a gradient
on a grid of N nodes takes no more device memory than the 101 float64 values a
node that a reverse step with the stages' inputs, B and 1/det G takes.  The
largest grid whose gradient fits on a device depends on it."""
import pytest

import paper_1405_0942_gb300.glemur as glemur


@pytest.mark.parametrize("dims", [(3, 3, 3), (12, 11, 13), (64, 64, 64), (65, 33, 47), (384, 384, 384)],
                         ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("precision,per_node", [(glemur.FP64, 101 * 8), (glemur.MIXED, 62 * 8 - 12)],
                         ids=["fp64", "mixed"])
def test_bytes_per_node(dims, precision, per_node):
    nx, ny, nz = dims
    n = int(glemur.lib().glemur_adjoint_workspace_bytes(nx, ny, nz, precision))
    fixed = 64 * 1024          # partials, pointer tables, and each buffer rounded up to 256 bytes
    assert 0 < n <= per_node * nx * ny * nz + fixed
