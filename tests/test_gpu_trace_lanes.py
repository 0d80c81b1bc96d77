"""The trace with one, two, four and eight lanes per ray (the transducer count decides), against the
oracle's tables element by element with the bounds of the parity tests; the last 32 rays of a fan are
all there, one short or nearly all missing."""
import pytest

from paper_2211_00316_gb300 import phantoms as P
from test_gpu_parity_small import Case, check_tables

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [48, 51, 83, 96, 107, 128, 151, 152, 182, 211, 250, 251])
def test_tables(oracle_mod, n):
    w = P.custom(n, 64, 1e-3, 28e-3, kind="discs", ny=71, freqs=(3e5,))
    case = Case(oracle_mod, w, 3e5)
    check_tables(case)
    case.job.close()
