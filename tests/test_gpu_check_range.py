"""The input check where squares leave the range of double: cells whose E^2
and |M|^2 overflow (both infinite: refused) or fall among the subnormals (equal
after rounding: refused), and their neighbours inside the range, are decided
as the plain double expressions E < 0, M^2 >= E^2 > 0 decide them, by single
contexts and by the batches' own call of the check."""
import numpy as np
import pytest

from paper_1206_0919_gb300 import shasta as S
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

SCALES = [1e160, 1e155, 2.0 ** 512, 2.0 ** 511, 2.0 ** 510, 1e150, 2.0 ** -499, 2.0 ** -500, 2.0 ** -501, 2.0 ** -520,
          1e-157, 1e-160, 3e-162, 1e-162, 1e-200, 1e-310]


def refused(call):
    try:
        call()
        return False
    except S.ShastaError as e:
        assert e.status == S.EUNPHYSICAL
        return True


@pytest.mark.parametrize("scale", SCALES)
def test_check_where_squares_leave_the_range(scale):
    require_gpu()
    shape = (5, 2, 1)
    answers = []
    with S.Solver(shape, precision="fp64") as s, S.Batch(1000) as b, np.errstate(over="ignore", under="ignore"):
        for f in (0.0, 0.1, 0.9, 0.99, 1 - 2.0 ** -15, 1 - 2.0 ** -17, np.nextafter(1, 0), 1.0, 1.5):
            for d in ((1.0, 0.0, 0.0), (0.0, 0.6, -0.8), (0.48, 0.6, 0.64)):
                U = [np.ones((1, 2, 5)) for _ in range(5)]
                for k in (1, 2, 3):
                    U[k][:] = 0.0
                E = np.float64(scale) * 1.25
                M = [E * f * c for c in d]
                for k, v in enumerate((E, *M)):
                    U[k].flat[7] = v
                M2 = (M[0] * M[0] + M[1] * M[1]) + M[2] * M[2]
                bad = bool(M2 >= E * E and M2 > 0.0)
                answers.append(bad)
                assert refused(lambda: s.set_conserved(U)) == bad, (f, d)
                assert refused(lambda: b.remove(b.add_conserved(shape, U))) == bad, (f, d)
    assert any(answers) or scale < 1e-163
