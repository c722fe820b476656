"""The elastic solve on grids of few columns and long lines along z, which take a line to a
block (fewer columns than a block has lines) or just not, against the FP64 oracle within the
bounds of the other shapes."""
import pytest

from tests.test_gpu_elastic_shapes import test_solve_shapes as check_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 256), (1, 1, 512), (1, 1, 1024), (2, 2, 512), (8, 1, 256), (16, 1, 256),
                                   (4, 1, 1024), (4, 2, 1024)])
@pytest.mark.parametrize("fixed", [False, True])
def test_few_columns(shape, fixed):
    check_shape(shape, fixed)
