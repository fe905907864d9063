"""The float32 apply sums the terms on the coarse grid that the rule names: one pair batch launches two GEMMs and one
expansion more than without."""
import pytest

from _helpers import to_gpu
from test_gpu_term_split import CASES, system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


def launches(case):
    import paper_2401_04189_gb300 as P
    n, r, theta, uniform = CASES[case]
    s = system(n, r, theta, uniform=uniform)
    ctx = P.Context.from_system(s, precision="fp32")
    occ = to_gpu(s.psi)
    P.tx_exchange_apply(ctx, occ)
    P.tx_reset_launch_count()
    P.tx_exchange_apply(ctx, occ)
    return P.tx_launch_count()


def test_launches_of_the_split():
    plain = launches("sharp")
    assert launches("mixed") == plain + 3 and launches("graded") == plain + 3
    assert launches("smooth") == plain + 3 and launches("two") == plain + 3
