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


@pytest.mark.parametrize("n,nwant", [(39, 7), (40, 7), (41, 41), (63, 5), (64, 64), (65, 9), (127, 33), (129, 20), (255, 40),
                                     (257, 16), (511, 24), (512, 31), (513, 12)])
def test_sym_eigh_cluster_sizes(n, nwant):
    """The dense eigensolver around the sizes where its tridiagonalisation changes form or distribution (one
    block below 40 rows and above 512, rows dealt over 16 CTAs in between, one lane per own row) and where the
    shifts, vectors and reflector chunks have remainders, against LAPACK (bounds of the eigensolver tests)."""
    rng = np.random.default_rng(n)
    c = rng.standard_normal((n, n))
    H = np.diag(5.0 + 3.0 * np.arange(n)) + c + c.T
    w, V = ae.amgeig_sym_eigh(H, nwant)
    full = np.linalg.eigvalsh(H)
    scale = np.abs(full).max()
    assert np.all(np.abs(w - full[:nwant]) <= 1e-12 * scale)
    assert np.abs(V.T @ V - np.eye(nwant)).max() < 1e-12
    assert np.abs(H @ V - V * w).max() <= 1e-11 * scale


@pytest.mark.parametrize("n,nwant", [(1, 1), (3, 2), (16, 16), (39, 12), (40, 12), (127, 64), (128, 64)])
def test_noalloc_gives_the_allocating_entrys_bits(n, nwant):
    """Both entry points run the same kernels: the same bits, also on a diagonal and a decoupled matrix."""
    import torch

    rng = np.random.default_rng(n)
    c = rng.standard_normal((n, n))
    dense = np.diag(5.0 + 3.0 * np.arange(n)) + c + c.T
    split = dense.copy()
    split[: n // 2, n // 2:] = 0.0
    split[n // 2:, : n // 2] = 0.0
    for H in (dense, split, np.diag(1.0 + np.arange(n))):
        w, V = ae.amgeig_sym_eigh(H, nwant)
        Hd = torch.tensor(H, dtype=torch.float64, device="cuda")
        wd = torch.empty(nwant, dtype=torch.float64, device="cuda")
        Vd = torch.empty((n, nwant), dtype=torch.float64, device="cuda")
        ae.amgeig_sym_eigh_noalloc(Hd, wd, Vd)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(wd.cpu().numpy(), w)
        np.testing.assert_array_equal(Vd.cpu().numpy(), V)
        full = np.linalg.eigvalsh(H)
        assert np.all(np.abs(w - full[:nwant]) <= 1e-12 * np.abs(full).max())
        assert np.abs(V.T @ V - np.eye(nwant)).max() < 1e-12
