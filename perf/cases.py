"""The work that programs have this library do, as cases that can be timed and compared.

A case is a dict of plain values.  ``kind`` says which public call a pass makes:

product      y = A x on a handle that is kept (the inner step of every solver and time step)
multi        Y = A X for k right-hand sides
chain        y = B (C x), two rectangular operators of an operator-based time step
solve        one linear system on a handle that is kept (a time step's pressure solve)
solve_multi  k systems that share one matrix
setup        a new matrix: handle from host CSR with reordering, a vector and the cells' numbers
             taken into the new numbering, one product, and the handle's release
serve        a burst of independent requests (matrix, right-hand side) through the solve server,
             host memory to host memory

Matrices are the finite-volume Laplacians of jittered tetrahedral meshes (``kuhn``: 6 size^3
cells, five entries a row) and of mixed hexahedron / prism / tetrahedron meshes (``mixed``: rows
of 4 to 13 entries), cells in random order, Dirichlet boundaries (positive definite), as in
this repository's workloads.  For ``kuhn`` the seed makes the mesh's jitter, its cell order and
the vectors.  The number of cells of a mixed mesh depends on its random elements, so these come
from the size, and the seed makes its coefficients: a_ij d_i d_j with random d (as of a varying
diffusivity; positive definite like the original), and the vectors.
"""
import functools
import time

import numpy as np
import torch

from paper_2107_12371_gb300 import capi, meshgen

RCM = capi.SPMV_REORDER_RCM


def listed():
    return [
        # the smallest mesh of the paper's size range, cells in file order: one product of a
        # small system, where a launch and the latency of its loads are what counts
        {"name": "product_f64_48k", "kind": "product", "mesh": "kuhn", "size": 20,
         "dtype": "f64", "reorder": 0, "index_bits": 0},
        # the benchmark's matrix (6M cells after RCM): larger than the L2, the steady state of
        # a big solver
        {"name": "product_f64_6m", "kind": "product", "mesh": "kuhn", "size": 100,
         "dtype": "f64", "reorder": 1, "index_bits": 0},
        # single precision on a mixed-element mesh of an odd size, int32 columns (the smoother
        # or inner iteration of a single-precision code; ragged rows)
        {"name": "product_f32_mixed_400k", "kind": "product", "mesh": "mixed", "size": 51,
         "dtype": "f32", "reorder": 1, "index_bits": 32},
        # divergence of a gradient (cells x faces times faces x cells), the operator-based
        # formulation's basic chain
        {"name": "chain_f64_300k", "kind": "chain", "size": 37, "dtype": "f64"},
        # 32 right-hand sides (a block method), double precision, rows sorted by length
        {"name": "multi_f64_k32", "kind": "multi", "mesh": "mixed", "size": 40, "dtype": "f64",
         "k": 32, "sigma": 1024},
        # five right-hand sides in single precision: velocity, temperature and one scalar
        # advanced together; a k that is no power of two
        {"name": "multi_f32_k5", "kind": "multi", "mesh": "mixed", "size": 47, "dtype": "f32",
         "k": 5, "sigma": 0},
        # a small pressure solve with the default options (one of many in a time loop)
        {"name": "solve_f64_48k", "kind": "solve", "mesh": "kuhn", "size": 20, "mixed": 0,
         "persistent": 0, "reorder": 0, "rtol": 1e-10},
        # an ordinary solve as one cooperative kernel (an option the library offers for it)
        {"name": "solve_f64_300k_persistent", "kind": "solve", "mesh": "kuhn", "size": 37,
         "mixed": 0, "persistent": 1, "reorder": 1, "rtol": 1e-10},
        # a large solve by FP32 inner iterations and FP64 refinement, the fastest way to a
        # double-precision answer on this card
        {"name": "solve_mixed_3m", "kind": "solve", "mesh": "kuhn", "size": 80, "mixed": 1,
         "persistent": 0, "reorder": 1, "rtol": 1e-10},
        # eight systems that share a mixed-element matrix, in lock-step
        {"name": "solve_multi_f64_k8", "kind": "solve_multi", "mesh": "mixed", "size": 40, "k": 8,
         "mixed": 0, "persistent": 0, "sigma": 1024, "rtol": 1e-10},
        # a new matrix with reverse Cuthill-McKee: what every new mesh costs before its first
        # product
        {"name": "setup_rcm_800k", "kind": "setup", "mesh": "kuhn", "size": 51, "reorder": 1,
         "sigma": 0},
        # sixteen requests of 10 to 200 thousand cells, half of them mixed precision, in flight
        # together
        {"name": "serve_16", "kind": "serve", "count": 16, "lo": 10000, "hi": 200000,
         "slots": 8, "rtol": 1e-8},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["product", "product", "multi", "multi", "chain", "solve", "solve",
                       "solve", "solve_multi", "setup", "serve"])
    mesh = rng.choice(["kuhn", "kuhn", "mixed"])
    # sizes by the cube's edge: a factor of five in the edge is 125 in the rows
    size = _log(rng, 12, 72) if mesh == "kuhn" else _log(rng, 10, 52)
    if kind == "product":
        return {"kind": kind, "mesh": mesh, "size": size, "dtype": rng.choice(["f64", "f32"]),
                "reorder": rng.choice([0, 1]), "index_bits": rng.choice([0, 0, 32])}
    if kind == "multi":
        return {"kind": kind, "mesh": mesh, "size": min(size, 48),
                "dtype": rng.choice(["f64", "f32"]), "k": _log(rng, 2, 48),
                "sigma": rng.choice([0, 256, 1024])}
    if kind == "chain":
        return {"kind": kind, "size": _log(rng, 8, 40), "dtype": rng.choice(["f64", "f32"])}
    if kind == "solve":
        return {"kind": kind, "mesh": mesh, "size": size, "mixed": rng.choice([0, 1]),
                "persistent": rng.choice([0, 1]), "reorder": rng.choice([0, 1]), "rtol": 1e-10}
    if kind == "solve_multi":
        return {"kind": kind, "mesh": mesh, "size": min(size, 44), "k": _log(rng, 2, 24),
                "mixed": rng.choice([0, 1]), "persistent": rng.choice([0, 1]),
                "sigma": rng.choice([0, 1024]), "rtol": 1e-10}
    if kind == "setup":
        return {"kind": kind, "mesh": mesh, "size": size, "reorder": rng.choice([1, 1, 2]),
                "sigma": rng.choice([0, 0, 1024])}
    return {"kind": kind, "count": rng.choice([6, 9, 12, 16]), "lo": _log(rng, 8000, 20000),
            "hi": _log(rng, 60000, 250000), "slots": rng.choice([4, 8]), "rtol": 1e-8}


# ---- inputs -----------------------------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _mixed_mesh(size):
    return meshgen.mixed_matrix(size, seed=1, dirichlet=True)[0]


def _matrix(case, seed):
    """Host CSR of the case's mesh."""
    if case["mesh"] == "mixed":
        m = _mixed_mesh(case["size"])
        d = np.random.default_rng(seed).uniform(0.8, 1.25, m.n)
        values = m.values * np.repeat(d, np.diff(m.row_ptr)) * d[m.col_idx]
        return meshgen.CsrMatrix(m.n, m.row_ptr, m.col_idx, values)
    return meshgen.kuhn_tet_matrix_fast(case["size"], seed=seed, dirichlet=True)[0]


def _vectors(seed, shape, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64).mul_(2).sub_(1).to(
        dtype).contiguous()


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _requests(case, seed):
    """The burst's requests: cell counts spread evenly over the logarithm of the range, in a
    fixed mixed-up order; every other one in mixed precision."""
    count = case["count"]
    out = []
    for i in range(count):
        at = ((i * 7) % count + 0.5) / count
        nx, ny, nz = meshgen.box_for_cells(case["lo"] * (case["hi"] / case["lo"]) ** at)
        m, rng = meshgen.kuhn_tet_matrix_fast(nx, ny, nz, seed=int(seed) * 1000 + i,
                                              dirichlet=True)
        out.append((m, meshgen.uniform_vectors(rng, m.n), i % 2))
    return out


class _Server:
    def __init__(self, slots):
        self.handle = capi.spmv_server_create(8 << 30, slots)

    def __del__(self):
        capi.spmv_server_destroy(self.handle)


def prepare(case, seed):
    capi.load()
    s = dict(case)
    kind = case["kind"]
    if kind == "serve":
        s["server"] = _Server(case["slots"])
        s["requests"] = _requests(case, seed)
        s["opts"] = [capi.cg_default_options(rtol=case["rtol"], mixed=mixed)
                     for _, _, mixed in s["requests"]]
        return s
    if kind == "chain":
        M, G, L, _ = meshgen.kuhn_tet_operators(case["size"], seed=seed)
        prec = capi.SPMV_PREC_FP32 if case["dtype"] == "f32" else capi.SPMV_PREC_FP64
        s["B"] = capi.Matrix(M.n, M.row_ptr, M.col_idx, M.values, n_cols=M.n_cols, precision=prec)
        s["C"] = capi.Matrix(G.n, G.row_ptr, G.col_idx, G.values, n_cols=G.n_cols, precision=prec)
        s["x"] = _vectors(seed, L.n, _dtype(case))
        s["y"] = torch.empty(M.n, dtype=_dtype(case), device="cuda")
        return s
    m = _matrix(case, seed)
    if kind == "setup":
        s["m"] = m
        s["x"] = _vectors(seed, m.n)
        s["ids"] = torch.arange(m.n, dtype=torch.float64, device="cuda")
        return s
    if kind in ("solve", "solve_multi"):
        prec = capi.SPMV_PREC_DUAL if case["mixed"] else capi.SPMV_PREC_FP64
    else:
        prec = capi.SPMV_PREC_FP32 if case["dtype"] == "f32" else capi.SPMV_PREC_FP64
    s["A"] = capi.Matrix(m.n, m.row_ptr, m.col_idx, m.values, precision=prec,
                         reorder=RCM if case.get("reorder", 1) else 0,
                         sigma=case.get("sigma", 0), index_bits=case.get("index_bits", 0))
    shape = (m.n, case["k"]) if "k" in case else (m.n,)
    dtype = _dtype(case) if "dtype" in case else torch.float64
    s["x"] = _vectors(seed, shape, dtype)  # the vector that is multiplied, or the right-hand side
    s["y"] = torch.zeros(shape, dtype=dtype, device="cuda")
    return s


# ---- one pass ---------------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "product":
        if s["dtype"] == "f32":
            s["A"].apply_f32(s["x"], s["y"])
        else:
            s["A"].apply(s["x"], s["y"])
        return s["y"]
    if kind == "multi":
        s["A"].apply_multi(s["x"], s["y"])
        return s["y"]
    if kind == "chain":
        f = capi.spmv_apply_chain_f32 if s["dtype"] == "f32" else capi.spmv_apply_chain
        f(s["B"].handle, s["C"].handle, s["x"], s["y"])
        return s["y"]
    if kind == "solve":
        s["A"].solve(s["x"], s["y"], rtol=s["rtol"], mixed=s["mixed"], persistent=s["persistent"])
        return s["y"]
    if kind == "solve_multi":
        s["A"].solve_multi(s["x"], s["y"], rtol=s["rtol"], mixed=s["mixed"],
                           persistent=s["persistent"])
        return s["y"]
    if kind == "setup":
        m = s["m"]
        A = capi.Matrix(m.n, m.row_ptr, m.col_idx, m.values, reorder=s["reorder"],
                        sigma=s["sigma"])
        x, y, ids = (torch.empty_like(s["x"]) for _ in range(3))
        A.permute(0, s["x"], x)
        A.permute(0, s["ids"], ids)
        A.apply(x, y)
        A.close()
        return {"y": y, "ids": ids.long()}
    srv = s["server"].handle
    pending, out = {}, [None] * len(s["requests"])
    for i, (m, b, _) in enumerate(s["requests"]):
        t = capi.spmv_server_submit(srv, m.n, m.row_ptr, m.col_idx, m.values, b, s["opts"][i])
        pending[t] = (i, np.empty(m.n))
    while pending:
        for t in list(pending):
            i, x = pending[t]
            r = capi.spmv_server_poll(srv, t, x)
            if r is not None:
                if r["status"] != capi.SPMV_OK:
                    raise RuntimeError("request %d ended with status %d" % (i, r["status"]))
                out[i] = x
                del pending[t]
        if pending:
            time.sleep(0.0002)
    return out


# ---- what a pass cannot do without --------------------------------------------------------------

def _counts(case):
    """Rows and entries of the case's mesh (within a per cent for the mixed ones)."""
    n = case["size"]
    if case.get("mesh") == "mixed":
        rows = 3.0 * n ** 3
        return rows, 5.85 * rows
    rows = 6.0 * n ** 3
    return rows, (5.0 - 2.0 / n) * rows


def _iterations(edge, rtol):
    """Jacobi-CG iterations on a cube of edge^3 hexahedra (234 at edge 20, 1,107 at 100, to
    1e-10)."""
    return 11.3 * edge * np.log10(1.0 / rtol) / 10.0


def work(case):
    kind = case["kind"]
    if kind == "serve":
        total, flops = 0.0, 0.0
        for i in range(case["count"]):
            at = (i + 0.5) / case["count"]
            rows = case["lo"] * (case["hi"] / case["lo"]) ** at
            it = _iterations((rows / 6.0) ** (1.0 / 3.0), case["rtol"])
            # FP64 and mixed requests alternate; per iteration the matrix once and the vectors
            # (x, r, p read and written, the diagonal read)
            total += it * rows * (0.5 * (12 * 5 + 56) + 0.5 * (8 * 5 + 28))
            flops += it * rows * 26
        return {"bytes": total, "flops": flops}
    if kind == "chain":
        n = case["size"]
        cells = 6.0 * n ** 3
        faces = 12.0 * n ** 3
        e = 4 if case["dtype"] == "f32" else 8
        return {"bytes": (e + 4) * 4 * cells + (e + 4) * 2 * faces + 2 * e * cells,
                "flops": 2 * (4 * cells + 2 * faces)}
    rows, nnz = _counts(case)
    if kind == "setup":
        # the CSR in, the handle's CSR and sliced copies out (10 B an entry), the vectors
        return {"bytes": 12 * nnz + 4 * rows + 12 * nnz + 10 * nnz + 48 * rows, "flops": 2 * nnz}
    if kind in ("product", "multi"):
        k = case.get("k", 1)
        e = 4 if case["dtype"] == "f32" else 8
        return {"bytes": (e + 4) * nnz + 2 * e * k * rows, "flops": 2 * nnz * k}
    k = case.get("k", 1)
    e = 4 if case["mixed"] else 8
    edge = case["size"] if case.get("mesh") != "mixed" else 0.76 * case["size"]
    it = _iterations(edge, case["rtol"])
    # per iteration: the matrix once, x, r, p read and written and the diagonal read
    return {"bytes": it * ((e + 4) * nnz + (6 * k + 1) * e * rows),
            "flops": it * k * (2 * nnz + 14 * rows)}


def tolerance(case):
    """About four times the distance from exact() that was measured (relative, over the norm):
    1.2e-7 for requests to rtol 1e-8, 2.6e-9 for solves to rtol 1e-10 (another order of the
    sums can stop a solve an iteration earlier or later), 5e-8 for FP32 products, 1.2e-16 for
    FP64 ones."""
    kind = case["kind"]
    if kind == "serve":
        return {"rel": 5e-7, "max": 5e-5}
    if kind in ("solve", "solve_multi"):
        return {"rel": 1.2e-8, "max": 1.2e-6}
    if kind in ("product", "multi", "chain") and case["dtype"] == "f32":
        return {"rel": 2e-7, "max": 8e-6}
    return {"rel": 5e-16, "max": 2e-14}


# ---- the same in 64 bits, without this library ---------------------------------------------------

def _csr(m, n_cols=None):
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    return torch.sparse_csr_tensor(t(np.asarray(m.row_ptr, np.int64)),
                                   t(np.asarray(m.col_idx, np.int64)), t(m.values),
                                   size=(m.n, n_cols or m.n))


def _diagonal(m):
    rows = np.repeat(np.arange(m.n), np.diff(m.row_ptr))
    d = np.zeros(m.n)
    at = m.col_idx == rows
    d[rows[at]] = m.values[at]
    return torch.from_numpy(d).cuda()


def _solution(m, b, tol=1e-13):
    """Jacobi-CG of all columns of b to a recurrence residual of tol."""
    A, d = _csr(m), _diagonal(m)[:, None]
    B = b.double().reshape(m.n, -1)
    x, r = torch.zeros_like(B), B.clone()
    z = r / d
    p, rho = z.clone(), (r * z).sum(0)
    bb = (B * B).sum(0)
    for it in range(20000):
        q = A @ p
        alpha = rho / (p * q).sum(0)
        x += alpha * p
        r -= alpha * q
        z = r / d
        new = (r * z).sum(0)
        p = z + (new / rho) * p
        rho = new
        if it % 25 == 24 and bool(((r * r).sum(0) <= tol * tol * bb).all()):
            break
    return x.reshape(b.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = []
        for m, b, _ in _requests(case, seed):
            out.append(_solution(m, torch.from_numpy(b).cuda()).cpu().numpy())
        return out
    if kind == "chain":
        M, G, L, _ = meshgen.kuhn_tet_operators(case["size"], seed=seed)
        x = _vectors(seed, L.n, _dtype(case)).double()
        return _csr(M, M.n_cols) @ (_csr(G, G.n_cols) @ x)
    m = _matrix(case, seed)
    # Vectors of a reordered handle live in its numbering.  Which one that is says the handle
    # (the setup case compares the numbering itself); the values come from plain torch.
    sigma = case.get("sigma", 0)
    reorder = case["reorder"] if kind == "setup" else (RCM if case.get("reorder", 1) else 0)
    A = capi.Matrix(m.n, m.row_ptr, m.col_idx, m.values, reorder=reorder, sigma=sigma)
    perm = torch.from_numpy(A.permutation().astype(np.int64)).cuda()
    A.close()
    if kind == "setup":
        return {"y": (_csr(m) @ _vectors(seed, m.n))[perm], "ids": None}
    shape = (m.n, case["k"]) if "k" in case else (m.n,)
    x = _vectors(seed, shape, _dtype(case) if "dtype" in case else torch.float64).double()
    own = torch.empty_like(x)
    own[perm] = x
    if kind in ("solve", "solve_multi"):
        return _solution(m, own)[perm]
    return (_csr(m) @ own)[perm]
