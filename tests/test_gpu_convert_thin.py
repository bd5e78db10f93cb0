"""The field conversions on thin grids, whose planes have fewer nodes than a
CTA has threads and share it (256 // (nx ny) columns of planes to a CTA):
planes of 9 nodes to a CTA's 256 and one more, as many columns as planes and a
ragged last one, each number of planes per thread.  Exact, as the cases of
test_gpu_convert.py, whose check this is."""
import pytest

import test_gpu_convert as convert
from test_gpu_convert import G  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,periodic", [(0, 0), (0, 1), (1, 0)],
                         ids=["fp64", "fp64-periodic", "mixed"])
@pytest.mark.parametrize("dims", [(3, 3, 28), (3, 3, 29), (3, 3, 4000), (3, 3, 9001),
                                  (3, 3, 40001), (5, 7, 3), (7, 5, 2200), (11, 12, 1300),
                                  (16, 8, 305), (16, 16, 1217), (4, 64, 77), (257, 3, 9)],
                         ids=lambda d: "x".join(map(str, d)))
def test_thin_grids(G, dims, precision, periodic):  # noqa: F811
    convert.test_conversions_are_exact(G, dims, precision, periodic)
