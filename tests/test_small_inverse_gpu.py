"""FP64 inverses on both sides of the size up to which k_gj takes them instead of the split products
(dense_inverse.cu): log|det|, sign, ratios and energies against numpy, within the tolerance of the other
sizes (cond(Phi) x 1e3 x 2^-53)."""
import pytest

from tests.test_fp64_split_gpu import test_block_edges as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ne", [3, 10, 19, 20, 21, 22])
def test_around_the_line(ne):
    check(ne)
