"""The stored matrix in stream order, on the GPU: every form of a step (even,
padded, compact, empty, two lanes per row, a warp per row), both column widths,
the edges of chunks and the sums through accumulators, each against the oracle.

Products use integers, so every order of summation gives the oracle's bits.
Solves are held to their tolerance by the oracle's product.
"""
import re

import numpy as np
import pytest

import fe_inputs as fi
import oracle
from gpu_util import cg_mod, handle

pytestmark = pytest.mark.gpu

TOL = 1e-10


def _rows(kind, n, rng):
    """Entries per row: the edges of chunks (9; 14 in FP32), of lanes (32), of lane pairs (64)."""
    if kind == "even":
        return np.full(n, 27)
    if kind == "edges":  # runs of 40 rows of one length
        return np.resize(np.repeat([0, 1, 8, 9, 10, 14, 15, 18, 19, 27, 28, 29, 32], 40), n)
    if kind == "uneven":  # little padding, half of it, and steps too uneven to pad
        return np.where(np.arange(n) % 96 < 32, rng.integers(25, 29, n),
                        np.where(np.arange(n) % 96 < 64, rng.integers(8, 25, n), rng.integers(0, 32, n)))
    if kind == "pairs":
        return np.resize([33, 34, 63, 64, 5, 0, 47], n)
    return np.resize(np.array([65, 96, 97, 700, 0, 3] + [7] * 30), n)  # "long"


def _matrix(kind, n, span, seed):
    """Integer values; the columns of a row lie within `span` of its middle."""
    rng = np.random.default_rng(seed)
    ln = np.minimum(_rows(kind, n, rng), n)
    rp = np.zeros(n + 1, np.int32)
    np.cumsum(ln, out=rp[1:])
    ci = np.empty(rp[-1], np.int32)
    for i in range(n):
        k = int(ln[i])
        lo, hi = max(0, i - max(span, 2 * k)), min(n, i + max(span, 2 * k) + 1)
        ci[rp[i]:rp[i + 1]] = np.sort(rng.choice(hi - lo, k, replace=False) + lo) if k else []
    return fi.CSR(rp, ci, rng.integers(-50, 51, rp[-1]).astype(np.float64), n)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("span", [300, 10 ** 6])
@pytest.mark.parametrize("kind", ["even", "edges", "uneven", "pairs", "long"])
def test_product_of_every_step_form(kind, span, mixed):
    """Exactly the oracle's product, whatever the layout (a span beyond 65535
    takes 32-bit columns), the CTA count and the lanes per row (n small: two)."""
    import torch
    cg = cg_mod()
    for n, ctas in ((1, 0), (33, 0), (1500, 3), (1500, 0), (70000, 0)):
        if span > 65535 and n < 70000:
            continue
        A = _matrix(kind, n, span, n + len(kind))
        x = np.random.default_rng(5).integers(-20, 21, n).astype(np.float64)
        with handle(A, ctas=ctas, precision=int(mixed)) as h:
            y = torch.full((n,), np.nan, dtype=torch.float64, device="cuda")
            cg.cg_spmv(h, torch.from_numpy(x).cuda(), y)
        assert np.array_equal(y.cpu().numpy(), oracle.spmv(A, x)), (n, ctas)


def _spd(kind, n, span, seed):
    """Symmetric, diagonally dominant, with the row lengths' pattern of `kind`."""
    import scipy.sparse as sp
    B = _matrix(kind, n, span, seed)
    S = sp.csr_matrix((B.val, B.col_idx, B.row_ptr), shape=(n, n))
    S = S + S.T
    S.setdiag(0)
    S.eliminate_zeros()
    S = (S + sp.diags(np.asarray(abs(S).sum(axis=1)).ravel() + 1.0)).tocsr()
    S.sort_indices()
    return fi.CSR(S.indptr.astype(np.int32), S.indices.astype(np.int32), S.data.astype(np.float64), n)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("kind,n,span", [("edges", 60000, 200), ("uneven", 60000, 200), ("uneven", 70000, 10 ** 6),
                                         ("long", 3000, 200), ("pairs", 1200, 200)])
def test_solve_over_every_step_form(kind, n, span, mixed):
    """The rings of a solve over the same forms, plain and Jacobi: the true
    residual within tol, and in FP64 the oracle's steps."""
    cg = cg_mod()
    A = _spd(kind, n, span, 3)
    b = oracle.spmv(A, fi.xstar(1, n))
    for jacobi in (0, 1):
        x = np.zeros(n)
        with handle(A, precision=int(mixed), preconditioner=jacobi, ctas=152) as h:
            res = cg.cg_solve(h, b, x, tol=TOL)
        assert res.status == cg.CG_OK, res
        assert np.linalg.norm(b - oracle.spmv(A, x)) <= 1.0000001 * TOL * np.linalg.norm(b)
        if not mixed and not jacobi:
            assert abs(res.iters - oracle.cg(A, b, tol=TOL).iters) <= 2


@pytest.mark.parametrize("values", [(1.0, 1.0 + 1e-7), (1.0, 1e4, 1e8), (1e-8, 1.0, 3.0), (1e-150, 1e-149)])
def test_sums_that_leave_the_accumulators_range(values):
    """Few distinct eigenvalues: r.r and p.q fall or rise by orders of magnitude
    from one step to the next, so the accumulators' exponent does not fit and the
    general sum takes over.  CG needs a step per eigenvalue (a few more by
    rounding); diagonal systems have the solution b / d."""
    cg = cg_mod()
    n = 40000
    d = np.resize(np.array(values), n)
    A = fi.CSR(np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), d, n)
    b = np.ones(n)
    x = np.zeros(n)
    with handle(A, ctas=152) as h:
        res = cg.cg_solve(h, b, x, tol=TOL, maxit=40)
    assert res.status == cg.CG_OK, res
    assert np.linalg.norm(b - d * x) <= 1.0000001 * TOL * np.linalg.norm(b)
    assert abs(res.iters - oracle.cg(A, b, tol=TOL, maxit=40).iters) <= 2


@pytest.mark.parametrize("mixed", [False, True])
def test_batch_layout_from_host_and_device_and_at_the_budget(mixed):
    """A request's host arrays pass in runs through the staging buffer (more than
    its 4 M entries here), device arrays are read in place: the same bits.  With
    the smallest budget that submit accepts, the request is solved too."""
    import torch
    cg = cg_mod()
    A = _spd("uneven", 160000, 300, 7)
    assert A.nnz > (4 << 20)
    b = oracle.spmv(A, fi.xstar(2, A.n))
    arrays = (A.row_ptr, A.col_idx, A.val)

    def solved(budget, on_device):
        x = np.zeros(A.n)
        if on_device:
            dev = [torch.from_numpy(a).cuda() for a in arrays]
            xd = torch.zeros(A.n, dtype=torch.float64, device="cuda")
            req = cg.Request(*dev, torch.from_numpy(b).cuda(), xd, tol=TOL)
        else:
            req = cg.Request(*arrays, b.copy(), x, tol=TOL)
        with cg.Batch(precision=int(mixed), group_override=5, budget_bytes=budget) as bt:
            res = bt.wait_all(bt.submit([req]), 60000)[0]
        assert res.done and res.status == cg.CG_OK, res
        return xd.cpu().numpy() if on_device else x

    xh = solved(0, False)
    assert np.linalg.norm(b - oracle.spmv(A, xh)) <= 1.0000001 * TOL * np.linalg.norm(b)
    assert np.array_equal(xh, solved(0, True))
    with pytest.raises(cg.CGError) as refused:
        solved(1 << 20, False)
    need = int(re.search(r"needs up to (\d+) bytes", str(refused.value)).group(1))
    assert np.array_equal(xh, solved(need, False))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("span", [300, 10 ** 6])
@pytest.mark.parametrize("kind", ["even", "edges", "uneven", "pairs", "long"])
def test_ring_product_of_every_step_form(kind, span, precision):
    """The product of a solve's steps, which in mixed precision is the FP32 ring's:
    one step from x = 0 with integers (products and sums exact in FP32, dot products
    in FP64) gives x = (b.b / b.Ab) b to the last bit."""
    cg = cg_mod()
    for n, ctas in ((533, 0), (1500, 3), (1500, 0), (70000, 0), (70000, 7)):
        if span > 65535 and n < 70000:
            continue
        A = _matrix(kind, n, span, 2 * n + len(kind))
        rng = np.random.default_rng(6)
        b = rng.integers(1, 21, n) * rng.choice([-1.0, 1.0], n)
        gamma = float(b @ oracle.spmv(A, b))
        assert gamma != 0.0
        if gamma < 0:
            A = fi.CSR(A.row_ptr, A.col_idx, -A.val, n)
        x = np.zeros(n)
        with handle(A, ctas=ctas, precision=precision) as h:
            res = cg.cg_solve(h, b, x, tol=0.0, maxit=1)
        assert res.status == cg.CG_ENOTCONV and res.iters == 1, (n, ctas, res)
        assert np.array_equal(x, (float(b @ b) / abs(gamma)) * b), (n, ctas)
