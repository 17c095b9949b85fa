"""Calls at their limits, on the GPU: the step limit at the step that converges,
a wait limit shorter than a pass over the matrix, the smallest budget that takes a
request and one near the card's memory."""
import re

import numpy as np
import pytest

import fe_inputs as fi
import oracle
from gpu_util import cg_mod, handle

pytestmark = pytest.mark.gpu

TOL = 1e-10


def _system(N, seed):
    A = fi.q1(N, 1.0, seed)
    return A, oracle.spmv(A, fi.xstar(seed, A.n))


@pytest.mark.parametrize("ctas", [3, 0])  # the large-share kernel and the small-share one
@pytest.mark.parametrize("jacobi", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
def test_step_limit_at_the_converging_step(precision, jacobi, ctas):
    """A solve whose limit is the step that converges has converged (in mixed
    precision the residual replacement behind that step tells), with the same
    bits; with one step less it has not."""
    cg = cg_mod()
    A, b = _system(22, 81)
    with handle(A, ctas=ctas, precision=precision, preconditioner=jacobi) as h:
        assert h.partition_info()[1] == (cg.CG_SOLVE_KERNEL_LARGE_SHARE if ctas else cg.CG_SOLVE_KERNEL_SMALL_SHARE)
        xs, res = [], []
        for maxit in (10 * A.n, None, -1):
            x = np.zeros(A.n)
            limit = maxit if not res else res[0].iters + (maxit or 0)
            res.append(cg.cg_solve(h, b, x, tol=TOL, maxit=limit))
            xs.append(x)
    assert [r.status for r in res] == [cg.CG_OK, cg.CG_OK, cg.CG_ENOTCONV], res
    assert res[1].iters == res[0].iters == res[2].iters + 1
    assert np.array_equal(xs[0], xs[1]) and res[1].relres == res[0].relres <= TOL


@pytest.mark.parametrize("chunk", [0, 7])
@pytest.mark.parametrize("jacobi", [0, 1])
def test_step_limit_of_a_mixed_batch(jacobi, chunk):
    """The same in a batch, alone and in a group of CTAs, in one round and in many."""
    cg = cg_mod()
    A, b = _system(12, 82)
    for group in (1, 3):
        with cg.Batch(precision=cg.CG_PREC_MIXED, preconditioner=jacobi, chunk_iters=chunk, group_override=group) as bt:
            def solve(maxit):
                x = np.zeros(A.n)
                return bt.wait(bt.submit([cg.Request(A.row_ptr, A.col_idx, A.val, b, x, tol=TOL, maxit=maxit)])[0]), x
            r0, x0 = solve(10 * A.n)
            r1, x1 = solve(r0.iters)
            r2, _ = solve(r0.iters - 1)
        assert [r.status for r in (r0, r1, r2)] == [cg.CG_OK, cg.CG_OK, cg.CG_ENOTCONV], (r0, r1, r2)
        assert r1.iters == r0.iters and np.array_equal(x0, x1)



def test_wait_limit_is_no_limit_on_a_pass():
    """A mixed solve whose direct pass (one row of 2 M entries, one warp's work)
    takes several times the wait limit, in a handle and in a batch: no wait on
    another CTA or on a copy is that long, so nothing times out."""
    import torch
    cg = cg_mod()
    n, long_row = 4096, 2 << 20
    rp = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    rp[1:] += long_row - 1
    ci = torch.cat([torch.arange(long_row, dtype=torch.int32, device="cuda") % 1024,
                    torch.arange(1, n, dtype=torch.int32, device="cuda")])
    va = torch.ones(ci.numel(), dtype=torch.float64, device="cuda")
    b = torch.ones(n, dtype=torch.float64, device="cuda")
    mixed = cg.CG_PREC_MIXED
    with cg.Batch(precision=mixed, group_override=1, wait_limit_ms=1, validate=False) as bt:
        reqs = [cg.Request(rp, ci, va, b, torch.zeros_like(b), tol=TOL, maxit=1) for _ in range(3)]
        systems = [_system(8, 90 + i) for i in range(3)]
        reqs += [cg.Request(A.row_ptr, A.col_idx, A.val, c, np.zeros(A.n), tol=TOL) for A, c in systems]
        res = bt.wait_all(bt.submit(reqs), 60000)
        assert bt.stats()["last_round_ms"] > 4  # two passes of the long row
    assert [r.status for r in res] == 3 * [cg.CG_ENOTCONV] + 3 * [cg.CG_OK], res
    with cg.cg_create(rp, ci, va, precision=mixed, ctas=1, wait_limit_ms=1) as h:
        r = cg.cg_solve(h, b, torch.zeros_like(b), tol=TOL, maxit=1)
    assert r.status == cg.CG_ENOTCONV, r


@pytest.mark.parametrize("base", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
def test_device_arrays_that_are_not_this_gpus(precision, base):
    """Arrays declared to be on the device that are not this GPU's own memory
    (here pinned host memory; another GPU's is another case) are copied, not read
    in place: the bits of the same arrays on this GPU, from a handle and a batch,
    in several runs through the batch's staging buffer."""
    import ctypes
    import torch
    from paper_2112_10823_gb300 import _binding as bd
    cg = cg_mod()
    A, b = _system(60, 83)
    assert A.nnz > (4 << 20)
    ref = np.zeros(A.n)
    with handle(A, precision=precision) as h:
        cg.cg_solve(h, b, ref, tol=TOL)
    rp, ci, va = (torch.from_numpy(a).pin_memory() for a in (A.row_ptr + np.int32(base), A.col_idx + np.int32(base), A.val))
    csr = bd.cg_csr(rp.data_ptr(), ci.data_ptr(), va.data_ptr(), base, 1)
    o = bd.cg_opts()
    bd.lib.cg_opts_default(ctypes.byref(o))
    o.precision = precision
    out = ctypes.c_void_p(0)
    assert bd.lib.cg_create(ctypes.byref(out), ctypes.byref(csr), A.n, A.nnz, ctypes.byref(o)) == cg.CG_OK
    x = np.zeros(A.n)
    it, rr = ctypes.c_int64(0), ctypes.c_double(0)
    assert bd.lib.cg_solve(out, b.ctypes.data, x.ctypes.data, TOL, 10 * A.n, ctypes.byref(it), ctypes.byref(rr)) == cg.CG_OK
    bd.lib.cg_destroy(out)
    assert np.array_equal(x, ref)
    xs = [np.zeros(A.n), np.zeros(A.n)]
    with cg.Batch(precision=precision, group_override=8) as bt:
        r = bt.wait(bt.submit([cg.Request(A.row_ptr, A.col_idx, A.val, b, xs[0], tol=TOL)])[0])
        req = bd.cg_request()
        req.csr, req.n, req.nnz = csr, A.n, A.nnz
        req.b, req.x, req.tol, req.maxit = b.ctypes.data, xs[1].ctypes.data, TOL, 10 * A.n
        t = ctypes.c_uint64(0)
        assert bd.lib.cg_batch_submit(bt._b, ctypes.byref(req), 1, ctypes.byref(t)) == cg.CG_OK
        r2 = bt.wait(t.value)
    assert r.status == r2.status == cg.CG_OK and r.iters == r2.iters
    assert np.array_equal(xs[0], xs[1])


def _banded(n, length, seed):
    """Symmetric, diagonally dominant; `length` (odd) entries in an inner row."""
    import scipy.sparse as sp
    rng = np.random.default_rng(seed)
    h = length // 2
    S = sp.diags([rng.uniform(-1, 0, n - d) for d in range(1, h + 1)], range(1, h + 1), shape=(n, n))
    S = S + S.T
    S = (S + sp.diags(np.asarray(abs(S).sum(axis=1)).ravel() + 1.0)).tocsr()
    S.sort_indices()
    return fi.CSR(S.indptr.astype(np.int32), S.indices.astype(np.int32), S.data.astype(np.float64), n)


@pytest.mark.parametrize("host", [True, False])
@pytest.mark.parametrize("precision,jacobi", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("n,length,opts", [(20000, 65, {}), (5000, 97, {}), (300, 7, {"step_shape": 3}),
                                           (20000, 3, {"step_shape": 3}), (500, 5, {"group_override": 1 << 20})])
def test_smallest_accepted_budget_takes_the_request(n, length, opts, precision, jacobi, host):
    """A budget of exactly the bytes that submit asks for takes a request whose
    steps are single rows, or whose CTAs' tables outweigh the matrix; with the bits
    of an ample budget."""
    import torch
    cg = cg_mod()
    A = _banded(n, length, n)
    b = oracle.spmv(A, fi.xstar(4, n))

    def solved(budget):
        arrays = [A.row_ptr, A.col_idx, A.val, b, np.zeros(n)]
        if not host:
            arrays = [torch.from_numpy(a).cuda() for a in arrays]
        with cg.Batch(precision=precision, preconditioner=jacobi, budget_bytes=budget, **opts) as bt:
            r = bt.wait(bt.submit([cg.Request(*arrays, tol=TOL)])[0], 60000)
            assert bt.stats()["bytes_in_use"] == 0
        assert r.done and r.status == cg.CG_OK, r
        return arrays[4] if host else arrays[4].cpu().numpy()

    with pytest.raises(cg.CGError) as refused:
        solved(4096)
    need = int(re.search(r"needs up to (\d+) bytes", str(refused.value)).group(1))
    assert np.array_equal(solved(need), solved(1 << 30))


def test_host_arrays_beside_a_budget_near_the_cards_memory():
    """With 200 MB left beside the budget, a one-CTA request with host arrays of
    more than that is admitted as before, through a small staging buffer, with the
    bits of device arrays."""
    import torch
    cg = cg_mod()
    A = fi.q1(100, 1.0, 84)
    assert 12 * A.nnz > (250 << 20)
    b = np.ones(A.n)
    dev = [torch.from_numpy(a).cuda() for a in (A.row_ptr, A.col_idx, A.val, b, np.zeros(A.n))]
    x = np.zeros(A.n)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    with cg.Batch(group_override=1, budget_bytes=free - (200 << 20)) as bt:
        rd = bt.wait(bt.submit([cg.Request(*dev, tol=TOL, maxit=3)])[0], 60000)
        rh = bt.wait(bt.submit([cg.Request(A.row_ptr, A.col_idx, A.val, b, x, tol=TOL, maxit=3)])[0], 60000)
    assert rd.status == rh.status == cg.CG_ENOTCONV, (rd, rh)
    assert np.array_equal(x, dev[4].cpu().numpy())
