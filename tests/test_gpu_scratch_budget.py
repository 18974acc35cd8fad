"""A call accepted at one memory budget is accepted at every larger one: where the scratch of the
FP64 corrections just does not fit, the FP64 solve alone does."""
import pytest

from paper_2312_13051_gb300 import inputs as I
from tests.gpu_common import lib  # noqa: F401

pytestmark = pytest.mark.gpu


def _accepted(lib, model, p, budget):
    c = lib.Context(0, mem_budget_bytes=budget)
    try:
        lib.wilson_loop(model, I.Plane(3, 1), p, precision="fp64", ctx=c, gap_tol=0.0)
        return True
    except lib.BWError as e:
        assert e.code == 2, e  # BW_ENOMEM
        return False
    finally:
        c.close()


@pytest.mark.parametrize("p", [1, 16])
def test_no_gap_in_the_accepted_budgets(lib, p):
    model = I.random_hermitian_model(34, 2)
    lo, hi = 1 << 12, 1 << 22
    assert _accepted(lib, model, p, hi) and not _accepted(lib, model, p, lo)
    while hi - lo > 256:
        mid = (lo + hi) // 2
        if _accepted(lib, model, p, mid):
            hi = mid
        else:
            lo = mid
    refused = [b for b in range(hi, 3 * hi, 1024) if not _accepted(lib, model, p, b)]
    assert not refused, (hi, refused)
