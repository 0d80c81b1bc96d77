"""The trace of small rings on grids of many rows, against the oracle's tables element by element with
the bounds of the parity tests. A block of the trace keeps the mask's rows in shared memory beside
its queues, so the lanes per ray that fit depend on the rows: 2,173 is the most with eight lanes,
2,558 with four. The ring lies at the lower end of the grid."""
import pytest

from paper_2211_00316_gb300 import phantoms as P
from test_gpu_parity_small import Case, check_tables

pytestmark = pytest.mark.gpu


class Tall(P.Geometry):
    """A grid whose rows all lie above -35 dx."""

    @property
    def y0(self) -> float:
        return -35 * self.dx


@pytest.mark.parametrize("n,ny", [(64, 2173), (64, 2174), (64, 2558), (51, 2559), (95, 2623), (96, 2558), (128, 2559),
                                  (151, 2623), (192, 2623)])
def test_tables(oracle_mod, n, ny):
    w = P.custom(n, 64, 1e-3, 28e-3, kind="discs", ny=71, freqs=(3e5,))
    w.geom = Tall(nx=64, ny=ny, dx=1e-3, n_xducers=n, ring_radius=28e-3)
    ct = P.two_disc_phantom(w.geom, centres_mm=((-9.0, -3.0), (9.0, 6.0)), radius_mm=5.0)
    w.c_true, w.c_init = ct, P.blur(ct, w.geom.dx)
    case = Case(oracle_mod, w, 3e5)
    check_tables(case)
    case.job.close()
