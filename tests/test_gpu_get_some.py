"""Getting some of the conserved fields: the bits of a full get, the arrays left
out untouched, and the time of the fields asked for (one field of five read
and written: a fifth of an FP64 get's bytes, two fifths of a float one's, whose
quads are read whole; the bounds leave half and a fifth for the call itself)."""
import time

import pytest

from paper_1206_0919_gb300 import shasta as S
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,bound", [("fp32", 0.6), ("fp64", 0.5)])
def test_single_fields_cost_a_single_field(precision, bound):
    require_gpu()
    import torch
    n = 288
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    U = [torch.rand((n, n, n), generator=g, device="cuda", dtype=torch.float64) for _ in range(5)]
    with S.Solver((n, n, n), precision=precision, check_input=False) as s:
        s.set_conserved(U)

        def us(out):
            best = 1e9
            for _ in range(8):
                torch.cuda.synchronize()
                t = time.perf_counter()
                s.get_conserved(out)
                best = min(best, time.perf_counter() - t)
            return best * 1e6

        full = [torch.empty_like(u) for u in U]
        whole = us(full)
        for k in range(5):
            out = [torch.full_like(U[0], -7.0) for _ in range(5)]
            one = us([out[j] if j == k else None for j in range(5)])
            assert torch.equal(out[k], full[k])
            assert all(bool((out[j] == -7.0).all()) for j in range(5) if j != k)
            assert one < bound * whole, (k, one, whole)
