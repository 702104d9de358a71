"""Solves whose vectors stay on the chip (one cluster or one cooperative grid):
block counts and row splits at their edges, reaches longer than a block's rows,
more slots than the unrolled products take, and reaches too long for the chip,
which take the streaming kernels.

Matrices are symmetric with 1 <= a_ii <= 2 and off-diagonal row sums of at most
a_ii / 2, so A has its eigenvalues in [1/2, 3] and condition number at most 6: a
solution with relative residual 1e-12 lies within 6e-12 of the exact one."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spl
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _spd(n, offsets, rng):
    """Diagonally dominant symmetric matrix with entries at +-offsets."""
    offs = [o for o in offsets if 0 < o < n]
    bands = [rng.uniform(-1, 1, n - o) * 0.25 / max(len(offs), 1) for o in offs]
    return sp.diags([rng.uniform(1, 2, n)] + bands + bands, [0] + offs + [-o for o in offs],
                    format="csr")


def _dev(A, b):
    import paper_2309_02156_gb300 as sa
    A.sort_indices()
    t = lambda a, d: torch.from_numpy(np.ascontiguousarray(a, dtype=d)).to(DEV)
    return sa.CSR(t(A.indptr, np.int32), t(A.indices, np.int32), t(A.data, np.float64)), \
        t(b, np.float64)


def _solve(A, b, tol, max_iters=2000, **kw):
    import paper_2309_02156_gb300 as sa
    n = A.shape[0]
    seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", max_iters=max_iters, **kw)
    Ad, bd = _dev(A, b)
    x = torch.zeros(n, dtype=torch.float64, device=DEV)
    infos = [seq.solve(Ad, bd, tol, x.zero_()) for _ in range(2)]
    seq.close()
    assert infos[0] == infos[1]           # the same solve again gives the same bits
    return infos[0], x.cpu().numpy()


# n: below a warp, ragged, the last cluster sizes and the first grid sizes of
# both precisions (16,384 and 57,344 rows), several slices per warp
@pytest.mark.parametrize("precision", ["f64", "mixed_krylov"])
@pytest.mark.parametrize("n,offsets", [
    (1, []), (31, [1, 7]), (33, [1, 7]), (700, [1, 300]), (4097, [1, 64]), (16384, [1, 128]),
    (16385, [1, 128]), (57344, [1, 239]), (57345, [1, 239]), (131071, [1, 362]),
    (5000, list(range(1, 5))), (5000, list(range(1, 12))), (20011, list(range(1, 12))),
    (20000, [1, 9999]), (200003, [1, 100001])])
def test_cg_matches_direct_solve(n, offsets, precision):
    rng = np.random.default_rng(n + len(offsets))
    A = _spd(n, offsets, rng)
    b = rng.standard_normal(n)
    info, x = _solve(A, b, 1e-12, krylov="cg", precision=precision)
    assert info["status"] == 0 and info["final_relres"] <= 1e-12
    assert np.linalg.norm(b - A @ x) <= 1.01e-12 * np.linalg.norm(b)
    if n <= 60000:
        ref = spl.spsolve(A.tocsc(), b) if n > 1 else b / A.toarray()[0]
        assert np.linalg.norm(x - ref) <= 6e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [500, 30000])
def test_cg_status_codes(n):
    """Iteration cap, breakdown and a NaN right-hand side on cluster and grid."""
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(n)
    A = _spd(n, [1, 50], rng)
    b = rng.standard_normal(n)
    info, _ = _solve(A, b, 1e-12, max_iters=3, krylov="cg")
    assert info["status"] == 1 and info["iters"] == 3
    assert 1e-12 < info["final_relres"] < 1.0
    for bad, code in ((-A, -4), (A, -5)):
        seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", krylov="cg")
        bb = b.copy()
        if code == -5:
            bb[n // 2] = np.nan
        Ad, bd = _dev(bad.tocsr(), bb)
        with pytest.raises(sa.SeqError) as e:
            x = torch.zeros(n, dtype=torch.float64, device=DEV)
            info = seq.solve(Ad, bd, 1e-10, x)
        assert e.value.code == code
        seq.close()


@pytest.mark.parametrize("schedule", [(1, 256), (1, 1024), (2, 512), (4, 1024), (8, 512)])
def test_batch_on_every_form(schedule):
    """One batch of all forms (offset slots, nine and 24 of them, columns out of
    order, a reach of half the rows), sizes around the 32-row slices and past the
    sketch's flush of 33 tiles per team, guesses from a three-column history."""
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(sum(schedule))
    mats = [_spd(n, o, rng) for n, o in [(1, []), (31, [1, 7]), (33, [1, 7]), (5000, [1, 2, 70, 140]),
                                         (4100, list(range(1, 12))), (3000, [1, 1499]),
                                         (20011, [1, 141]), (2500, [1, 50])]]
    arrays = []
    for k, A in enumerate(mats):
        A.sort_indices()
        ptr, ci, v = A.indptr, A.indices.copy(), A.data.copy()
        if k == len(mats) - 1:
            for i in range(A.shape[0]):
                ci[ptr[i]:ptr[i + 1]] = ci[ptr[i]:ptr[i + 1]][::-1]
                v[ptr[i]:ptr[i + 1]] = v[ptr[i]:ptr[i + 1]][::-1]
        arrays.append((ptr, ci, v))
    t = lambda a, d: torch.from_numpy(np.ascontiguousarray(a, dtype=d)).to(DEV)
    bt = sa.Batch([(t(p, np.int32), t(c, np.int32)) for p, c, _ in arrays], M=3, s=12, zeta=4)
    if schedule[0] > 1:
        bt.set_cluster(*schedule)
    else:
        bt.set_schedule(schedule[1], 1, 0)
    bs = [rng.standard_normal(A.shape[0]) for A in mats]
    for _ in range(3):
        for k, A in enumerate(mats):
            bt.push(k, t(rng.standard_normal(A.shape[0]), np.float64))
    xs = [torch.empty(A.shape[0], dtype=torch.float64, device=DEV) for A in mats]
    infos = bt.step([t(v, np.float64) for _, _, v in arrays], [t(b, np.float64) for b in bs], xs, 1e-11)
    for A, b, x, f in zip(mats, bs, xs, infos):
        assert f["status"] == 0 and f["history_cols"] == 3
        ref = spl.spsolve(A.tocsc(), b) if A.shape[0] > 1 else b / A.toarray()[0]
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 6e-11 * np.linalg.norm(ref)
    bt.close()


# rows per block from one slice up, restarts around the pass widths (8, 16, 24,
# 32 columns) and past the longest resident one (33), each preconditioner
@pytest.mark.parametrize("opts", [
    dict(restart=1), dict(restart=9), dict(restart=17), dict(restart=25), dict(restart=32),
    dict(restart=33), dict(precond_sweeps=1), dict(precond_sweeps=2),
    dict(precond_sweeps=3, precond_kind="chebyshev"), dict(precond_sweeps=4, precond_kind="chebyshev")])
@pytest.mark.parametrize("precision", ["f64", "mixed_krylov"])
@pytest.mark.parametrize("n,offsets", [(1, []), (33, [1, 7]), (1000, [1, 31]), (1000, [1, 2, 31, 62]),
                                       (20011, [1, 141]), (6000, [1, 2900]), (92161, [1, 303])])
def test_gmres_matches_direct_solve(n, offsets, precision, opts):
    rng = np.random.default_rng(n + len(offsets))
    A = _spd(n, offsets, rng)
    b = rng.standard_normal(n)
    info, x = _solve(A, b, 1e-12, krylov="gmres", precision=precision, **opts)
    assert info["status"] == 0 and info["final_relres"] <= 1e-12
    assert np.linalg.norm(b - A @ x) <= 1.01e-12 * np.linalg.norm(b)


@pytest.mark.parametrize("n", [500, 30000])
@pytest.mark.parametrize("precision", ["f64", "mixed_krylov"])
def test_gmres_status_codes(n, precision):
    """Iteration cap, a zero and a NaN right-hand side, a start at the solution."""
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(n)
    A = _spd(n, [1, 50], rng)
    b = rng.standard_normal(n)
    info, _ = _solve(A, b, 1e-12, max_iters=4, krylov="gmres", precision=precision)
    assert info["status"] == 1 and info["iters"] == 4
    info, x = _solve(A, 0 * b, 1e-12, krylov="gmres", precision=precision)
    assert info["status"] == 0 and info["iters"] == 0 and not x.any()
    seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", krylov="gmres", precision=precision)
    bad = b.copy()
    bad[n // 2] = np.nan
    Ad, bd = _dev(A, bad)
    with pytest.raises(sa.SeqError) as e:
        seq.solve(Ad, bd, 1e-10, torch.zeros(n, dtype=torch.float64, device=DEV))
    assert e.value.code == -5
    seq.close()
