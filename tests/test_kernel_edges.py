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


@pytest.mark.parametrize("kind", ["dense", "decoupled", "diagonal", "close"])
@pytest.mark.parametrize("n,nwant", [(1, 1), (3, 2), (39, 7), (40, 7), (41, 41), (63, 5), (64, 64), (65, 9), (127, 33),
                                     (129, 20), (255, 40), (257, 16), (328, 64), (511, 24), (512, 31), (513, 12)])
def test_coarse_eigensolver_sizes(n, nwant, kind):
    """The solve path's dense eigensolver around the sizes where its tridiagonalisation changes form or distribution
    (one block below 40 rows and above 512, rows dealt over 16 CTAs in between, one lane per own row) and where the
    shifts, vectors and reflector chunks have remainders: a one-level hierarchy, whose solve is the dense
    eigenproblem of its pencil, against LAPACK.  decoupled, diagonal: reflections with nothing to reflect and zero
    off-diagonals; close: all wanted values within 1e-4 ||H|| (one clean-up group; needs values beyond them that
    make ||H||)."""
    from paper_1503_08462_gb300.inputs import hierarchy

    if kind == "close" and nwant == n:
        pytest.skip("no values beyond the wanted ones")

    rng = np.random.default_rng(n)
    c = rng.standard_normal((n, n))
    H = np.diag(50.0 + 3.0 * np.arange(n)) + c + c.T
    if kind == "decoupled":
        H[: n // 2, n // 2:] = 0.0
        H[n // 2:, : n // 2] = 0.0
    elif kind == "diagonal":
        H = np.diag(1.0 + rng.permutation(n))
    elif kind == "close":
        Q, _ = np.linalg.qr(c)
        spec = np.concatenate([rng.uniform(1.0, 1.5, nwant), rng.uniform(10.0, 2.0e4, n - nwant)])
        H = (Q * np.sort(spec)) @ Q.T
        H = 0.5 * (H + H.T)
    H[np.abs(H) == 0.0] = 0.0
    H = H + np.diag(np.full(n, max(0.0, 1.0 - np.linalg.eigvalsh(H)[0])))  # SPD
    rp = np.arange(0, n * n + 1, n)
    ci = np.tile(np.arange(n), n)
    hh = hierarchy.build_hierarchy(rp, ci, H.ravel(), np.eye(n).ravel(), coarse_cap=n)
    assert hh.sizes == [n]
    with ae.Hierarchy(hierarchy.to_blob(hh)) as h:
        lam, U, _, _ = h.solve(nwant, tol=1.0, opt=ae.options(coarse_modes=nwant))
    full = np.linalg.eigvalsh(H)
    scale = np.abs(full).max()
    assert np.all(np.abs(lam - full[:nwant]) <= 1e-12 * scale)
    assert np.abs(U.T @ U - np.eye(nwant)).max() < (1e-12 if kind != "dense" else 2e-12)
    assert np.abs(H @ U - U * lam).max() <= 1e-11 * scale


def _one_level(rp, ci, vals, n):
    """A one-level hierarchy of the pencil (A, I): its solve is the dense eigenproblem of A."""
    from paper_1503_08462_gb300.inputs import hierarchy

    mass = np.where(np.repeat(np.arange(n), np.diff(rp)) == ci, 1.0, 0.0)
    hh = hierarchy.build_hierarchy(rp, ci, vals, mass, coarse_cap=n)
    assert hh.sizes == [n]
    return ae.Hierarchy(hierarchy.to_blob(hh))


@pytest.mark.parametrize("a,b,nwant", [(43, 51, 6), (45, 50, 6), (50, 64, 5), (53, 61, 5)])
def test_coarse_eigensolver_large_levels(a, b, nwant):
    """One-level hierarchies of 2193, 2250, 3200 and 3233 rows: the back-transformation's columns and reflectors no
    longer fit a CTA's shared memory eight and four at a time beyond 2215 rows, nor four and four beyond 3200.  The
    a x b Dirichlet Laplacian has the eigenvalues 4 sin^2(pi i / (2a + 2)) + 4 sin^2(pi j / (2b + 2))."""
    import scipy.sparse as sp

    def line(n):
        return sp.diags([-np.ones(n - 1), 2.0 * np.ones(n), -np.ones(n - 1)], [-1, 0, 1])

    n = a * b
    A = (sp.kron(line(a), sp.identity(b)) + sp.kron(sp.identity(a), line(b))).tocsr()
    A.sort_indices()
    with _one_level(A.indptr, A.indices, A.data, n) as h:
        lam, U, _, _ = h.solve(nwant, tol=1.0, opt=ae.options(coarse_modes=nwant))
    si, sj = (4.0 * np.sin(np.pi * np.arange(1, k + 1) / (2 * k + 2)) ** 2 for k in (a, b))
    ref = np.sort((si[:, None] + sj[None, :]).ravel())[:nwant]
    # as test_coarse_eigensolver_sizes, in units of ||A|| < 8; rounding of the n reflections grows with sqrt(n)
    assert np.all(np.abs(lam - ref) <= 1e-11)
    assert np.abs(U.T @ U - np.eye(nwant)).max() < 1e-11
    assert np.abs(A @ U - U * lam).max() <= 1e-10


def test_dense_pencil_beyond_the_largest_chunk():
    """A correction whose pencil (2144 coarse modes and 90 columns, 2234 rows) passes 2215 rows while its coarsest
    level does not, against the oracle's iterate (float64 path)."""
    p, blob, hh = problem_and_blob("square", 66, 2230, 1)
    assert hh.sizes[-1] <= 2215 < hh.sizes[-1] + 90
    oh = O.read_blob(blob)
    q, kw = 80, dict(q_extra=10, fixed_corrections=1, coarse_modes=0)
    lam_o, _, _ = O.solve(oh, q, tol=0.0, opts=O.Options(**kw))
    with ae.Hierarchy(blob) as h:
        lam, U, info, _ = h.solve(q, tol=0.0, opt=ae.options(**kw))
    assert info.dense_fallbacks > 0
    assert np.all(np.abs(lam - lam_o) / lam_o < eig_rel_tol(lam_o, lam_max(p)))
    assert np.max(np.abs(U.T @ (oh.M[0] @ U) - np.eye(q))) < 1e-10


@pytest.mark.parametrize("lam,repeated", [(0.25, "0x1.00006daf5b7p-2"), (0.2718281828, "0x1.165a8baf5b7p-2"),
                                          (0.3141592653, "0x1.41b365af5b7p-2")])
def test_shift_beside_repeated_decoupled_values(lam, repeated):
    """A diagonal matrix whose eight equal leading entries lie exactly on a counting point of the shift search for
    the eigenvalue just below them (1.6e-6 ||H||, the spacing of the first float-float round) while its other
    neighbour is outside its clean-up group: a count that stops at a run of vanishing minors loses the entries after
    it, puts the shift on the repeated value and leaves the neighbour's vector in the result."""
    n, nwant = 64, 16
    d = 0.5 + 0.5 * (np.arange(n) + 1) / n
    d[:8] = float.fromhex(repeated)
    d[n - 9:n - 3] = 0.175 - 0.01 * np.arange(6)
    d[n - 3], d[n - 2], d[n - 1] = lam - 2.4e-4, lam, 1.0
    with _one_level(np.arange(n + 1), np.arange(n), d, n) as h:
        w, U, _, _ = h.solve(nwant, tol=1.0, opt=ae.options(coarse_modes=nwant))
    assert np.all(np.abs(w - np.sort(d)[:nwant]) <= 1e-12)
    assert np.abs(U.T @ U - np.eye(nwant)).max() < 1e-12
    assert np.abs(d[:, None] * U - U * w).max() <= 1e-11


@pytest.mark.parametrize("n,nwant", [(5, 5), (24, 9), (65, 20), (200, 40), (512, 33)])
@pytest.mark.parametrize("run", [2, 3])
def test_coarse_eigensolver_repeated_values(n, nwant, run):
    """Diagonal matrices whose values come in runs of 2 and 3: zero off-diagonals and groups of equal shifts."""
    d = 1.0 - (np.arange(n) // run) / 512.0
    with _one_level(np.arange(n + 1), np.arange(n), d, n) as h:
        w, U, _, _ = h.solve(nwant, tol=1.0, opt=ae.options(coarse_modes=nwant))
    assert np.all(np.abs(w - np.sort(d)[:nwant]) <= 1e-12)
    assert np.abs(U.T @ U - np.eye(nwant)).max() < 1e-12
    assert np.abs(d[:, None] * U - U * w).max() <= 1e-11


@pytest.mark.parametrize("q,qe", [(1, 0), (2, 0), (1, 2), (6, 1), (11, 9), (20, 11)])
@pytest.mark.parametrize("modes", [33, 0])
def test_back_map_row_runs(q, qe, modes):
    """Accepted corrections on an odd coarsest level whose rows the back-map splits into 37 to 8 runs for 1 to 31
    columns, the last run short, against the oracle's iterates after one finest correction (float64 path; bounds of
    the iteration parity tests)."""
    p, blob, hh = problem_and_blob("square", 48, 300, 3)
    oh = O.read_blob(blob)
    kw = dict(q_extra=qe, fixed_corrections=1, coarse_modes=modes)
    lam_o, _, _ = O.solve(oh, q, tol=0.0, opts=O.Options(**kw))
    with ae.Hierarchy(blob) as h:
        lam, U, _, _ = h.solve(q, tol=0.0, opt=ae.options(**kw))
    assert np.all(np.abs(lam - lam_o) / lam_o < eig_rel_tol(lam_o, lam_max(p)))
    assert np.max(np.abs(U.T @ (oh.M[0] @ U) - np.eye(q))) < 1e-10


@pytest.mark.parametrize("width", [4, 20, 33, 128])
def test_block_per_row_sweeps_bf16(width):
    """The same sweeps on operators held in bfloat16, against the oracle's V-cycle on a hierarchy with the same
    rounded values (bound of the bfloat16 V-cycle test)."""
    import copy

    import torch

    def rounded(v):
        return torch.from_numpy(v.astype(np.float32)).bfloat16().double().numpy()

    _, blob, hh = problem_and_blob("cube", 20, 60, 4)
    oh = O.read_blob(blob)
    last = oh.n_levels - 1
    assert any(oh.A[l].nnz >= 96 * oh.sizes[l] for l in range(last))
    ob = copy.copy(oh)
    ob.A, ob.P = [a.copy() for a in oh.A], [m.copy() for m in oh.P]
    for l in range(last):
        ob.A[l].data, ob.P[l].data = rounded(oh.A[l].data), rounded(oh.P[l].data)
    ob.A[last] = oh.A[last]
    ob.R = [m.T.tocsr() for m in ob.P]
    ob.colour_cache = {}
    rng = np.random.default_rng(width)
    with ae.Hierarchy(blob) as h:
        for level in range(last):
            b = rng.standard_normal((oh.sizes[level], width))
            ref = O.vcycle(ob, level, b, np.zeros_like(b))
            x = ae.amgeig_apply_vcycle(h.handle, level, b, ae.options(precision=ae.AMGEIG_MIXED_BF16))
            assert np.abs(x - ref).max() <= 2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("q,qe", [(1, 0), (10, 7), (20, 12)])
def test_recombination_by_the_prolongation_chain(q, qe):
    """The mixed path on a cube whose finest level (15,625 rows) recombines by the prolongation chain and whose next
    (7,813 rows) by the composite, against the oracle's iterates after two finest corrections; bounds of the other
    mixed iteration tests, the subspace up to its last gap of 1e-3."""
    from helpers import m_subspace_angle

    p, blob, _ = problem_and_blob("cube", 26, 400, 4)
    oh = O.read_blob(blob)
    composite = abs(oh.P[0])
    for pl in oh.P[1:]:
        composite = composite @ abs(pl)
    assert oh.sizes[0] >= 8192 > oh.sizes[1] and composite.nnz > 4 * sum(pl.nnz for pl in oh.P)
    kw = dict(q_extra=qe, fixed_corrections=2, v_cycles=2)
    lam_o, U_o, _ = O.solve(oh, q, tol=0.0, opts=O.Options(**kw))
    with ae.Hierarchy(blob) as h:
        lam, U, _, _ = h.solve(q, tol=0.0, opt=ae.options(precision=ae.AMGEIG_MIXED_FP32, **kw))
    gaps = np.append(np.diff(lam_o) / lam_o[1:], 1.0 if q == 1 else 0.0)
    k = int(np.nonzero(gaps > 1e-3)[0].max()) + 1
    assert np.max(np.abs(lam - lam_o) / lam_o) <= 1e-6
    assert m_subspace_angle(U[:, :k], U_o[:, :k], oh.M[0]) <= 1e-4
    assert np.abs(U.T @ (oh.M[0] @ U) - np.eye(q)).max() < 1e-10
