"""Trend tiles, their validity words, the core lists and the live lists at patch sides 8 and 16
(the parity tests of this repository run on side 4), on an adapted grid whose patches are
partly live: masks bit for bit and fields and trends against the FP64 oracle over two
adaptive steps, with the persistent stage and with one launch per phase, and in the
viscous form.  The tolerances are those of the parity tests."""
import pytest

from test_gpu_parity import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [0.0, 2.0e5])
@pytest.mark.parametrize("persistent", [True, False])
@pytest.mark.parametrize("patch", [8, 16])
def test_sides_match_oracle(patch, persistent, nu):
    P = Pair(3, 6, kind="jet", seed=3, patch=patch, persistent=persistent, nu=nu)
    P.adapt()
    P.check_masks()
    P.rhs()
    P.check_fields(which="trend")
    for _ in range(2):
        dt = P.ora.dt_cfl()
        P.ora.step(dt)
        P.lib.step(-1.0, 1, True)
        P.check_masks()
        P.check_fields()
