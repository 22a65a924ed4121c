"""lelbm_stats.disp_max, the largest |c_i| streamed, at drifts of thousands of cells a step."""
import math

import pytest

from paper_2508_06911_gb300 import build, lelbm as L, workloads as W
from paper_2508_06911_gb300.solver import Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


# RT 0.6: R_ac 3, not refined; the set is every integer velocity within 3.5 of u.  On both sides of the limit of
# the 32-bit tally (the gather of deterministic streaming searches a window of the drift's width: kept short)
@pytest.mark.parametrize("u,deterministic", [(10.0, 0), (4000.0, 0), (5000.0, 0), (20000.0, 0), (10.0, 1), (40.0, 1)])
def test_disp_max(u, deterministic):
    w = W.hot_box(2, 8, 0.6, u=u)
    s = Solver.grid2d(w, precision=L.LELBM_FP64, deterministic=deterministic)
    s.step(1)
    st = s.stats()
    s.close()
    far = max((u + i) ** 2 + (u + j) ** 2 for i in range(-4, 5) for j in range(-4, 5) if i * i + j * j <= 12.25)
    assert st.fallback_mx == 0 and st.q_max == 37
    assert st.disp_max == pytest.approx(math.sqrt(far), rel=1e-14)
