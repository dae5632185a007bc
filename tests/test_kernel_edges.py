"""Kernels at the sizes where their tiling can go wrong, against the CPU oracle and LAPACK."""
import numpy as np
import pytest

from oracle import amg_oracle as O
from paper_1503_08462_gb300 import amgeig as ae

from helpers import eig_rel_tol, lam_max, problem_and_blob

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("q,qe,modes", [(60, 5, 0), (80, 15, 100), (80, 16, 101), (80, 17, 0), (100, 27, 131),
                                        (100, 28, 128)])
def test_dense_pencil_border_edges(q, qe, modes):
    """Dense pencils with borders around multiples of 32 columns (65, 95, 96, 97, 127, 128: the columns of the
    standard form and of the back-map live in 32-row register slots, one warp each) and odd mode counts, against
    the oracle's iterates after one finest correction (float64 path; bounds of the iteration parity tests)."""
    p, blob, _ = problem_and_blob("square", 64, 400, 1)
    oh = O.read_blob(blob)
    kw = dict(q_extra=qe, fixed_corrections=1, coarse_modes=modes)
    lam_o, U_o, _ = O.solve(oh, q, tol=0.0, opts=O.Options(**kw))
    with ae.Hierarchy(blob) as h:
        lam, U, info, _ = h.solve(q, tol=0.0, opt=ae.options(**kw))
    assert info.dense_fallbacks > 0
    tol = eig_rel_tol(lam_o, lam_max(p))
    assert np.all(np.abs(lam - lam_o) / lam_o < tol)
    assert np.max(np.abs(U.T @ (oh.M[0] @ U) - np.eye(q))) < 1e-10
