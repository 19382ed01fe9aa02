"""How many blocks of a GMRES on a few SMs (max_blocks) hold rows."""
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sms", [2, 3, 9, 12])
def test_few_sms_in_fp64_all_hold_rows(sms):
    """Rows cost an SM more in fp64 than the rotations do: up to 12 SMs none is set aside for them."""
    B = lib()
    assert B.gmres_plan(2000 * sms, "fp64", sms)["blocks"] == sms
    assert B.gmres_plan(2000 * 19, "fp64", 20)["blocks"] == 19
