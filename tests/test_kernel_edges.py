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


@pytest.mark.parametrize("width", [1, 4, 5, 20, 31, 33, 61, 64, 65, 97, 128])
@pytest.mark.parametrize("tune", [0, 1])
def test_block_per_row_sweeps(width, tune):
    """The float32 V-cycle on a 3D hierarchy whose coarse levels keep over 96 nonzeros a row (one block per row in
    the smoothing sweeps: 32, 16 or 8 nonzero streams of ceil(width / 4) lanes), on every level against the
    oracle's V-cycle, with the rule's launch shapes and with the tuner's; 2e-5 of each column's largest entry (a few
    units of 2^-24 per level, the bound of the V-cycle tests)."""
    p, blob, hh = problem_and_blob("cube", 20, 60, 4)
    assert any(lv.col_idx.shape[0] >= 96 * lv.n for lv in hh.levels[:-1])
    oh = O.read_blob(blob)
    rng = np.random.default_rng(width)
    with ae.Hierarchy(blob) as h:
        if tune:  # a solve tunes the operators at its width
            h.solve(1, tol=0.0, opt=ae.options(precision=ae.AMGEIG_MIXED_FP32, q_extra=width - 1, fixed_corrections=1,
                                               coarse_modes=20), vectors=False)
        for level in range(oh.n_levels - 1):
            b = rng.standard_normal((oh.sizes[level], width))
            ref = O.vcycle(oh, level, b, np.zeros_like(b))
            x = ae.amgeig_apply_vcycle(h.handle, level, b, ae.options(precision=ae.AMGEIG_MIXED_FP32, autotune=tune))
            err = np.abs(x - ref).max(axis=0) / np.abs(ref).max(axis=0)
            assert np.all(err <= 2e-5), (level, err.max())
