"""The work that the eigensolver is used for, as timed and compared cases.

Each case is one call sequence of a user's program on seeded problems: complete
solves (Algorithm 3.2) of 2D and 3D P1 finite-element pencils from a thousand to
784,385 unknowns, loads with a solve, a burst of served requests, and the dense
symmetric eigensolver on its own.

The pencils are -Laplace + V on the meshes of inputs/meshes.py (jittered grids on
the square, the L-shape and the cube), V a smooth positive potential made from the
seed, and -div(kappa grad) with the 4 x 4 checkerboard coefficient.  The potential
takes the place of the plain Laplacian because the symmetric domains have nearly
double eigenvalues there (relative gaps below 1e-7), whose single eigenvectors no
float64 computation determines to more than a few digits; it grows with the wanted
pairs so that it stays comparable to their eigenvalues and keeps them apart.  The
mesh of a domain and size is made once; the potential (on the checkerboard:
coefficients and mesh) is what the seed changes.
"""
import functools
import math
import time

import numpy as np
import torch

from paper_1503_08462_gb300 import amgeig as ae
from paper_1503_08462_gb300.inputs import hierarchy, meshes

SERVE_POOL = (("square", 181), ("lshape", 104), ("checker", 128))  # 32,400 / 32,033 / 16,129 unknowns


def listed():
    """The twelve cases, from the smallest call to the largest."""
    bench = dict(precision="mixed", v_cycles=2)
    return [
        # the allocation-free dense eigensolver on device buffers: a caller's own small projected problem
        dict(name="eigh_device_n64", kind="eigh_device", n=64, nwant=20),
        # the dense eigensolver on host buffers, the size of the L-shape's coarsest level and its 64 modes
        dict(name="eigh_host_n328", kind="eigh_host", n=328, nwant=64),
        # the smallest configuration, unit square h = 1/32, q = 4, solved tightly: latency and launches count
        dict(name="square_h32_q4", kind="solve", domain="square", m=32, q=4, q_extra=2, cap=50, modes=0, tol=1e-9,
             max_corrections=60, refine=0, **bench),
        # the same with the default precision of the interface
        dict(name="square_h32_q4_f64", kind="solve", domain="square", m=32, q=4, q_extra=2, cap=50, modes=0,
             tol=1e-9, max_corrections=60, refine=0, precision="f64", v_cycles=1),
        # one request of the serving stream, alone: an L-shape of 32,033 unknowns, odd q
        dict(name="lshape_h104_q11", kind="solve", domain="lshape", m=104, q=11, q_extra=9, cap=400, modes=64,
             tol=1e-6, max_corrections=60, refine=0, **bench),
        # a burst of served requests on three hierarchies (host buffers, four workers, no shared solves)
        dict(name="serve_8_requests", kind="serve", requests=8, q_max=12, tol=1e-6),
        # the default precision at an ordinary size
        dict(name="lshape_h128_q10_f64", kind="solve", domain="lshape", m=128, q=10, q_extra=4, cap=400, modes=64,
             tol=1e-6, max_corrections=60, refine=0, precision="f64", v_cycles=1),
        # a fresh problem end to end: load of the host blob, coarse modes, solve, eigenvectors to the host, release
        dict(name="load_solve_lshape_h256_q20", kind="load_solve", domain="lshape", m=256, q=20, q_extra=8, cap=400,
             modes=64, tol=1e-4, max_corrections=60, refine=0, **bench),
        # the benchmark's workload: L-shape h = 1/512, 784,385 unknowns, q = 20 with 8 buffer vectors
        dict(name="lshape_h512_q20", kind="solve", domain="lshape", m=512, q=20, q_extra=8, cap=400, modes=64,
             tol=1e-4, max_corrections=60, refine=0, **bench),
        # a 3D problem: cube, 250,047 unknowns of 15 nonzeros, q = 10 with 7 buffer vectors
        dict(name="cube_m64_q10", kind="solve", domain="cube", m=64, q=10, q_extra=7, cap=400, modes=64, tol=1e-6,
             max_corrections=60, refine=0, **bench),
        # many pairs: q = 50 with 22 buffer vectors (the checkerboard configuration's block) and compensated
        # Rayleigh quotients, 261,121 unknowns
        dict(name="square_h512_q50", kind="solve", domain="square", m=512, q=50, q_extra=22, cap=400, modes=112,
             tol=1e-6, max_corrections=60, refine=2, **bench),
        # the widest block: q = 100 with 28 buffer vectors (the cube configuration's block) on 103,823 unknowns
        dict(name="cube_m48_q100", kind="solve", domain="cube", m=48, q=100, q_extra=28, cap=400, modes=128,
             tol=1e-6, max_corrections=120, refine=0, **bench),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds: dense problems of 16 to 700 rows, solves of 400 to 784,385 unknowns for
    1 to 100 pairs, loads, bursts."""
    kind = rng.choice(["eigh_device", "eigh_host", "solve", "solve", "solve", "solve", "solve", "load_solve", "serve"])
    if kind == "eigh_device":
        n = _log_int(rng, 12, 128)
        return dict(kind=kind, n=n, nwant=rng.randint(1, min(n, 64)))
    if kind == "eigh_host":
        n = _log_int(rng, 16, 700)
        return dict(kind=kind, n=n, nwant=rng.randint(1, min(n, 96)))
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(2, 12), q_max=rng.randint(2, 16), tol=1e-6)
    domain = rng.choice(["square", "square", "lshape", "lshape", "cube", "checker"])
    wide = kind == "solve" and domain in ("square", "cube") and rng.random() < 0.3
    lo, hi = {"square": (24, 512), "lshape": (24, 512), "cube": (12, 64), "checker": (24, 256)}[domain]
    if wide:  # the widest blocks on the smaller meshes: no more than the largest listed case
        lo, hi = (64, 320) if domain == "square" else (20, 44)
    precision = "f64" if not wide and domain != "checker" and rng.random() < 0.25 else "mixed"
    if precision == "f64":
        hi = 160 if domain != "cube" else 24
    m = _log_int(rng, lo, hi)
    if domain == "checker":
        m = 4 * max(6, m // 4)
    q = rng.randint(33, 100) if wide else rng.randint(1, 8 if domain == "checker" else 24)
    q_extra = rng.randint(16, 28) if wide else 4 + q // 2
    return dict(kind=kind, domain=domain, m=m, q=q, q_extra=q_extra, cap=400,
                modes=128 if wide else 64, tol=rng.choice([1e-4, 1e-6]), max_corrections=60,
                refine=rng.choice([0, 0, 1, 2]), precision=precision, v_cycles=1 if precision == "f64" else 2)


# ------------------------------------------------------------------ problems


@functools.lru_cache(maxsize=3)
def _mesh(domain, m):
    if domain == "square":
        return meshes.square_2d(m, seed=1)
    if domain == "lshape":
        return meshes.lshape_2d(m, seed=2)
    return meshes.cube_3d(m, seed=4)


def _problem(domain, m, seed, q):
    """The pencil (A, M): the checkerboard of `seed`, or the domain's mesh with the potential of `seed`, made for
    about q wanted pairs."""
    if domain == "checker":
        return meshes.square_2d(m, checker=4, seed=seed)
    p = _mesh(domain, m)
    rng = np.random.default_rng(seed)
    v = np.zeros(p.n)
    for _ in range(12):  # a random smooth field: twelve plane waves of up to three periods across the unit length
        k = rng.uniform(-3.0, 3.0, p.coords.shape[1]) * 2 * math.pi
        v += rng.uniform(0.5, 1.0) * np.cos(p.coords @ k + rng.uniform(0, 2 * math.pi))
    v = max(25.0, 4.0 * q) * (v - v.min()) / (v.max() - v.min())
    rows = np.repeat(np.arange(p.n), np.diff(p.row_ptr))
    a = p.a_vals + 0.5 * (v[rows] + v[p.col_idx]) * p.m_vals
    return meshes.Problem(p.name, p.n, p.row_ptr, p.col_idx, a, p.m_vals, p.coords, p.h)


def _blob(domain, m, seed, q, cap):
    return hierarchy.problem_blob(_problem(domain, m, seed, q), coarse_cap=cap)[0]


def _options(case, coarse_rows):
    return ae.options(q_extra=case["q_extra"], max_corrections=case["max_corrections"], v_cycles=case["v_cycles"],
                      precision=ae.AMGEIG_FP64 if case["precision"] == "f64" else ae.AMGEIG_MIXED_FP32,
                      coarse_modes=min(case["modes"], coarse_rows), refine=case["refine"])


def _dense(case, seed):
    """A projected operator: graded positive diagonal (Ritz values) under a dense symmetric coupling."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    c = rng.standard_normal((n, n))
    return np.diag(10.0 + 12.0 * np.arange(n)) + 2.0 * (c + c.T)


def _requests(case):
    """(problem, q) of each request of a burst: the same for every seed, whose pencils differ.  Requests on the
    checkerboard, whose low spectrum is dense, stay at up to 8 pairs."""
    rng = np.random.default_rng([case["requests"], case["q_max"]])
    reqs = [(int(rng.integers(0, len(SERVE_POOL))), int(rng.integers(1, case["q_max"] + 1)))
            for _ in range(case["requests"])]
    return [(k, min(q, 8) if SERVE_POOL[k][0] == "checker" else q) for k, q in reqs]


def _serve_options(q, coarse_rows):
    return ae.options(q_extra=4 + q // 2, max_corrections=60, precision=ae.AMGEIG_MIXED_FP32, v_cycles=2,
                      coarse_modes=min(64, coarse_rows), batch=0)


# ------------------------------------------------------------------ the calls


def prepare(case, seed):
    kind = case["kind"]
    if kind == "eigh_device":
        n, w = case["n"], case["nwant"]
        f = dict(dtype=torch.float64, device="cuda")
        return dict(case=case, H=torch.tensor(_dense(case, seed), **f), values=torch.empty(w, **f),
                    vectors=torch.empty((n, w), **f))
    if kind == "eigh_host":
        return dict(case=case, H=_dense(case, seed))
    if kind == "serve":
        pool = [ae.Hierarchy(_blob(d, m, seed, case["q_max"], 400)) for d, m in SERVE_POOL]
        reqs = _requests(case)
        return dict(case=case, pool=pool, reqs=reqs,
                    out=[(np.empty(q), np.empty((pool[k].sizes[0], q))) for k, q in reqs],
                    opts=[_serve_options(q, pool[k].sizes[-1]) for k, q in reqs])
    blob = _blob(case["domain"], case["m"], seed, case["q"], case["cap"])
    if kind == "load_solve":
        return dict(case=case, blob=blob)
    h = ae.Hierarchy(blob)
    return dict(case=case, h=h, opt=_options(case, h.sizes[-1]), values=np.empty(case["q"]),
                vectors=torch.empty((h.sizes[0], case["q"]), dtype=torch.float64, device="cuda"))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "eigh_device":
        stream = torch.cuda.current_stream().cuda_stream
        ae.amgeig_sym_eigh_noalloc(state["H"], state["values"], state["vectors"], stream)
        return {"values": state["values"], "vectors": state["vectors"]}
    if kind == "eigh_host":
        values, vectors = ae.amgeig_sym_eigh(state["H"], case["nwant"])
        return {"values": values, "vectors": vectors}
    if kind == "serve":
        ids = {}
        for i, (k, q) in enumerate(state["reqs"]):
            ids[ae.amgeig_submit(state["pool"][k].handle, q, case["tol"], state["opts"][i])] = i
        while ids:
            for rid in list(ids):
                done, code = ae.amgeig_poll(rid, *state["out"][ids[rid]])
                if done:
                    if code not in (ae.AMGEIG_OK, ae.AMGEIG_ENOCONV):
                        raise RuntimeError(ae.strerror(code))
                    del ids[rid]
            time.sleep(0.0002)
        return [{"values": v, "vectors": u} for v, u in state["out"]]
    if kind == "load_solve":
        with ae.Hierarchy(state["blob"], modes=case["modes"]) as h:
            values, vectors, _, _ = h.solve(case["q"], case["tol"], _options(case, h.sizes[-1]))
        return {"values": values, "vectors": vectors}
    ae.amgeig_solve(state["h"].handle, case["q"], case["tol"], state["opt"], state["values"], state["vectors"], True)
    return {"values": state["values"], "vectors": state["vectors"]}


def _size(domain, m):
    """(unknowns, nonzeros of A) of a mesh, to a percent."""
    n = {"square": (m - 1) ** 2, "checker": (m - 1) ** 2, "lshape": 3 * m * m - 4 * m + 1, "cube": (m - 1) ** 3}[domain]
    return n, n * (15 if domain == "cube" else 7)


def _solve_work(domain, m, q, q_extra):
    """The finest pencil read once and the pairs written once; the operations of a single correction (a defect, one
    V-cycle's sweeps and residual, the projection and the recombination), which no solve can do without."""
    n, nnz = _size(domain, m)
    w = q + q_extra
    return 20.0 * nnz + 4.0 * n + 8.0 * n * q, 14.0 * nnz * w + 6.0 * n * w * w


def work(case):
    if case["kind"] in ("eigh_device", "eigh_host"):
        n, w = case["n"], case["nwant"]
        return {"bytes": 8.0 * (n * n + n * w + w), "flops": 4.0 / 3.0 * n ** 3 + 2.0 * n * n * w}
    if case["kind"] == "serve":
        each = [_solve_work(*SERVE_POOL[k], q, 4 + q // 2) for k, q in _requests(case)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    b, f = _solve_work(case["domain"], case["m"], case["q"], case["q_extra"])
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ 64-bit values


def _lines(domain, m):
    """Unknowns of each grid line (2D) or plane (3D), in node order: elements couple neighbouring ones only."""
    if domain == "cube":
        return [(m - 1) ** 2] * (m - 1)
    if domain == "lshape":
        return [m - 1] * m + [2 * m - 1] * (m - 1)
    return [m - 1] * (m - 1)


class _LineCholesky:
    """A = L L^T over the blocks of grid lines, dense float64 blocks on the GPU."""

    def __init__(self, p, lines):
        dev = "cuda"
        off = np.concatenate([[0], np.cumsum(lines)])
        self.off, self.diag, self.low = off, [], []
        line_of = np.repeat(np.arange(len(lines)), lines)
        rows = np.repeat(np.arange(p.n), np.diff(p.row_ptr))
        for b, size in enumerate(lines):
            s, e = p.row_ptr[off[b]], p.row_ptr[off[b + 1]]
            r, c, a = rows[s:e] - off[b], p.col_idx[s:e], p.a_vals[s:e]
            here = line_of[c] == b
            d = torch.zeros((size, size), dtype=torch.float64, device=dev)
            d[torch.from_numpy(r[here]).to(dev), torch.from_numpy(c[here].astype(np.int64) - off[b]).to(dev)] = \
                torch.from_numpy(a[here]).to(dev)
            w = None
            if b:
                back = line_of[c] == b - 1
                w = torch.zeros((size, lines[b - 1]), dtype=torch.float64, device=dev)
                w[torch.from_numpy(r[back]).to(dev),
                  torch.from_numpy(c[back].astype(np.int64) - off[b - 1]).to(dev)] = torch.from_numpy(a[back]).to(dev)
                w = torch.linalg.solve_triangular(self.diag[-1], w.T, upper=False).T.contiguous()
                d -= w @ w.T
            self.diag.append(torch.linalg.cholesky(d))
            self.low.append(w)

    def solve(self, x):
        x, o = x.clone(), self.off
        last = len(self.diag) - 1
        for b in range(last + 1):
            part = x[o[b]:o[b + 1]]
            if b:
                part -= self.low[b] @ x[o[b - 1]:o[b]]
            part.copy_(torch.linalg.solve_triangular(self.diag[b], part, upper=False))
        for b in range(last, -1, -1):
            part = x[o[b]:o[b + 1]]
            if b < last:
                part -= self.low[b + 1].T @ x[o[b + 1]:o[b + 2]]
            part.copy_(torch.linalg.solve_triangular(self.diag[b].T, part, upper=True))
        return x


def _pairs(domain, m, seed, q, q_potential):
    """The q smallest eigenpairs by subspace iteration with A^-1 and a Rayleigh-Ritz step, all in float64; vectors
    M-orthonormal, largest entry positive.  None where the factorisation or the iteration would be long."""
    lines = _lines(domain, m)
    width = min(sum(lines), q + max(16, q))
    cost = sum(lines) * max(lines) ** 2 * 2.4 + 45 * 4.0 * sum(lines) * max(lines) * width
    if cost > 1.2e13 or width > sum(lines) // 2:
        return None
    p = _problem(domain, m, seed, q_potential)
    crow, col = torch.from_numpy(p.row_ptr.astype(np.int64)), torch.from_numpy(p.col_idx.astype(np.int64))
    mass = torch.sparse_csr_tensor(crow, col, torch.from_numpy(p.m_vals), (p.n, p.n)).cuda()
    f = _LineCholesky(p, lines)
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn((p.n, width), dtype=torch.float64, device="cuda", generator=g)
    old = None
    for _ in range(60):
        mx = mass @ x
        y = f.solve(mx)  # A y = M x: y^T A y = y^T M x
        s, t = y.T @ mx, y.T @ (mass @ y)
        chol = torch.linalg.cholesky((s + s.T) / 2)
        half = torch.linalg.solve_triangular(chol, (t + t.T) / 2, upper=False)
        h = torch.linalg.solve_triangular(chol, half.T, upper=False)
        mu, z = torch.linalg.eigh((h + h.T) / 2)  # mu = 1 / lambda, ascending
        z = torch.linalg.solve_triangular(chol.T, z, upper=True).flip(1)
        mu = mu.flip(0)
        x = (y @ z) / mu.sqrt()  # M-orthonormal
        top = x[:, :q]
        sign = torch.sign(top.gather(0, top.abs().argmax(0, keepdim=True)))
        top = top * sign
        if old is not None and float((top - old).norm() / top.norm()) < 1e-12:
            break
        old = top
    return (1.0 / mu[:q]).cpu().numpy(), top.cpu().numpy()


def exact(case, seed):
    if case["kind"] in ("eigh_device", "eigh_host"):
        # an eigenvector of the dense solver has no sign of its own
        return {"values": np.linalg.eigvalsh(_dense(case, seed))[:case["nwant"]], "vectors": None}
    if case["kind"] == "serve":
        reqs = _requests(case)
        best = {k: _pairs(*SERVE_POOL[k], seed, max(q for j, q in reqs if j == k), case["q_max"])
                for k in {k for k, _ in reqs}}
        return [{"values": best[k][0][:q], "vectors": best[k][1][:, :q]} for k, q in reqs]
    pairs = _pairs(case["domain"], case["m"], seed, case["q"], case["q"])
    return None if pairs is None else {"values": pairs[0], "vectors": pairs[1]}
