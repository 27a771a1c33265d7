"""The explicit passes change their form at 77,824 rows (two blocks of 256 on each of 152 SMs): the
last size below it, the size itself and one beyond give the bits of a batch of one, whose passes have
one form."""
import pytest

from test_gpu_ssp_forms import afc, test_step_equals_a_batch_of_one as _same  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("elem,n", [("q1", (41, 33, 57)), ("q1", (38, 32, 64)), ("q1", (38, 32, 65)), ("p1", (38, 32, 64))])
def test_bits_at_the_switch(afc, elem, n, precision):  # noqa: F811
    _same(afc, elem, n, precision, "ssp3")
