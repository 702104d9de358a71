"""Resident solves at the edges of what the entry points take: vectors that start
at any element, and solves of several sizes at once.

Matrices are symmetric with 1 <= a_ii <= 2 and off-diagonal row sums of at most
a_ii / 2: eigenvalues in [1/2, 3]."""
import threading

import numpy as np
import pytest
import scipy.sparse as sp
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _spd(n, offsets, rng):
    offs = [o for o in offsets if 0 < o < n]
    bands = [rng.uniform(-1, 1, n - o) * 0.25 / max(len(offs), 1) for o in offs]
    A = sp.diags([rng.uniform(1, 2, n)] + bands + bands, [0] + offs + [-o for o in offs], format="csr")
    A.sort_indices()
    return A


def _dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).to(DEV)


def _csr(A):
    import paper_2309_02156_gb300 as sa
    return sa.CSR(_dev(A.indptr, np.int32), _dev(A.indices, np.int32), _dev(A.data, np.float64))


def _view(t, start):
    """A copy of t that starts `start` elements into a 16-byte aligned buffer."""
    buf = torch.zeros(t.numel() + 2, dtype=t.dtype, device=DEV)
    assert buf.data_ptr() % 16 == 0
    out = buf[start:start + t.numel()]
    out.copy_(t)
    return out


# x in shared memory; x outside it because of its size, and because of the reach
@pytest.mark.parametrize("krylov", ["cg", "gmres"])
@pytest.mark.parametrize("precision", ["f64", "mixed_krylov"])
@pytest.mark.parametrize("n,offsets", [(5001, [1, 70]), (1001 * 1001, [1, 1001]), (30000, [1, 14000])])
def test_vectors_at_any_element(n, offsets, precision, krylov):
    """x and b that start at an odd element give the same bits: every element is
    computed alike, whatever the width of an access."""
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(n)
    A = _spd(n, offsets, rng)
    b = rng.standard_normal(n)
    Ad, bd = _csr(A), _dev(b, np.float64)
    seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", max_iters=500, krylov=krylov, precision=precision)
    got = []
    for start in (0, 1):
        x = _view(torch.zeros_like(bd), start)
        info = seq.solve(Ad, _view(bd, start), 1e-12, x)
        assert info["status"] == 0
        got.append((info, x.cpu().numpy()))
    seq.close()
    assert got[0][0] == got[1][0] and np.array_equal(got[0][1], got[1][1])
    assert np.linalg.norm(b - A @ got[1][1]) <= 1.01e-12 * np.linalg.norm(b)


@pytest.mark.parametrize("start", [0, 1])
def test_batch_vectors_at_any_element(start):
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(7)
    mats = [_spd(n, o, rng) for n, o in [(33, [1, 7]), (5001, [1, 70]), (20011, [1, 141])]]
    bt = sa.Batch([(_dev(A.indptr, np.int32), _dev(A.indices, np.int32)) for A in mats], M=2, s=8, zeta=2)
    bt.set_cluster(4, 512, 0)
    for k, A in enumerate(mats):
        bt.push(k, _view(_dev(rng.standard_normal(A.shape[0]), np.float64), start))
    bs = [rng.standard_normal(A.shape[0]) for A in mats]
    xs = [_view(torch.zeros(A.shape[0], dtype=torch.float64, device=DEV), start) for A in mats]
    bt.step([_view(_dev(A.data, np.float64), start) for A in mats],
            [_view(_dev(b, np.float64), start) for b in bs], xs, 1e-11)
    for A, b, x in zip(mats, bs, xs):
        assert np.linalg.norm(b - A @ x.cpu().numpy()) <= 1.01e-11 * np.linalg.norm(b)
    bt.close()


# sizes whose launches need different amounts of shared memory, in one kernel
@pytest.mark.parametrize("krylov,sizes", [("cg", (90000, 28900)), ("gmres", (60025, 3600))])
def test_two_threads_of_different_sizes(krylov, sizes):
    """A thread per context, each with a stream of its own: every solve of either
    succeeds and has the bits that it has alone."""
    import paper_2309_02156_gb300 as sa
    wrong = []

    def work(n, alone, reps):
        rng = np.random.default_rng(n)
        A = _spd(n, [1, int(np.sqrt(n))], rng)
        with torch.cuda.stream(torch.cuda.Stream()):
            Ad, bd = _csr(A), _dev(rng.standard_normal(n), np.float64)
            seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", max_iters=3, krylov=krylov)
            for _ in range(reps):
                x = torch.zeros_like(bd)
                try:
                    seq.solve(Ad, bd, 1e-12, x)
                except sa.SeqError as e:
                    wrong.append((n, str(e)))
                if alone.setdefault(n, x) is not x and not torch.equal(alone[n], x):
                    wrong.append((n, "other bits"))
            seq.close()

    alone = {}
    for n in sizes:
        work(n, alone, 1)
    threads = [threading.Thread(target=work, args=(n, alone, 3000)) for n in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, (len(wrong), wrong[:3])


@pytest.mark.parametrize("krylov", ["cg", "gmres"])
def test_resident_solve_counts_its_launches(krylov):
    """Two launches for the matrix's offsets, one for its copy, one for the solve."""
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(3)
    n = 5001
    seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", krylov=krylov)
    info = seq.solve(_csr(_spd(n, [1, 70], rng)), _dev(rng.standard_normal(n), np.float64), 1e-10,
                     torch.zeros(n, dtype=torch.float64, device=DEV))
    seq.close()
    assert info["launches"] == 4


def _irregular(kind, n, rng):
    """CSR arrays of a symmetric matrix without the slot form."""
    if kind == "offsets25":
        A = _spd(n, list(range(1, 13)), rng)
    elif kind == "scattered":
        A = _spd(n, [1], rng)
        i, j = rng.integers(0, n, (2, 3 * n))
        S = sp.coo_matrix((rng.uniform(-0.01, 0.01, 3 * n), (i, j)), shape=(n, n)).tocsr()
        A = (A + S + S.T).tocsr()
        A.sort_indices()
    else:
        A = _spd(n, [1, 70], rng)
    ptr, ci, v = A.indptr, A.indices.copy(), A.data.copy()
    if kind == "unsorted":
        for i in range(n):
            ci[ptr[i]:ptr[i + 1]] = ci[ptr[i]:ptr[i + 1]][::-1]
            v[ptr[i]:ptr[i + 1]] = v[ptr[i]:ptr[i + 1]][::-1]
    if kind == "repeated":                   # every diagonal entry in two halves
        rows = np.repeat(np.arange(n), np.diff(ptr))
        half = np.where(ci == rows, 0.5, 1.0)
        order = np.argsort(np.concatenate([rows, np.arange(n)]), kind="stable")
        ci = np.concatenate([ci, np.arange(n)])[order]
        v = np.concatenate([v * half, 0.5 * A.diagonal()])[order]
        ptr = ptr + np.arange(n + 1)
    return A, (ptr, ci, v)


# the largest size of the one-block form and the smallest of the grid's kernels,
# which read the general layout; a long reach has the slot form and no room
@pytest.mark.parametrize("n,kind", [(n, k) for n in (1000, 65535, 65536) for k in
                                    ("unsorted", "repeated", "offsets25", "scattered", "far")
                                    if n > 1000 or k != "far"])
@pytest.mark.parametrize("precision", ["f64", "mixed_krylov"])
def test_cg_without_a_resident_form(n, kind, precision):
    """CG on matrices that no resident team takes: right, and below the grid's
    sizes without a copy of the matrix (two launches look at its offsets, one
    solves)."""
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(n)
    if kind == "far":
        A = _spd(n, [1, n - 5000], rng)
        arrays = A.indptr, A.indices, A.data
    else:
        A, arrays = _irregular(kind, n, rng)
    b = rng.standard_normal(n)
    seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", max_iters=500, krylov="cg", precision=precision)
    Ad = sa.CSR(_dev(arrays[0], np.int32), _dev(arrays[1], np.int32), _dev(arrays[2], np.float64))
    x = torch.zeros(n, dtype=torch.float64, device=DEV)
    info = seq.solve(Ad, _dev(b, np.float64), 1e-12, x)
    seq.close()
    assert info["status"] == 0
    assert np.linalg.norm(b - A @ x.cpu().numpy()) <= 1.01e-12 * np.linalg.norm(b)
    if n < 65536 and precision == "f64":
        assert info["launches"] == 3


def test_sketch_with_row_pointers_that_decrease():
    """Rows of entries that lie outside the span of their warp's first and last
    row (an invalid matrix): read where the row pointers say, as elsewhere."""
    import paper_2309_02156_gb300 as sa
    from oracle import sketch
    n, M, s, zeta, seed = 100, 3, 16, 4, 9
    rng = np.random.default_rng(1)
    A = _spd(n, [1, 7], rng)
    ptr = A.indptr.copy()
    ptr[4] += 100                # rows 3 and 61 run past their neighbours,
    ptr[62] += 90
    ptr[20] -= 60                # row 20 starts before them
    cols = [rng.standard_normal(n) for _ in range(M)]
    b = rng.standard_normal(n)
    Y = np.zeros((n, M))
    for i in range(n):
        for e in range(ptr[i], max(ptr[i], ptr[i + 1])):
            Y[i] += A.data[e] * np.array([c[A.indices[e]] for c in cols])
    seq = sa.Sequence(n, M, s, zeta=zeta, seed=seed)
    for c in cols:
        seq.push(_dev(c, np.float64))
    Ad = sa.CSR(_dev(ptr, np.int32), _dev(A.indices, np.int32), _dev(A.data, np.float64))
    seq.guess(Ad, _dev(b, np.float64), torch.empty(n, dtype=torch.float64, device=DEV))
    W, _ = seq.last_sketch()
    seq.close()
    S = sketch.sparse_sign_matrix(n, s, zeta, seed)
    ref = S @ np.column_stack([Y, b])
    assert np.all(np.abs(W.reshape(s, M + 1) - ref) <= 1e-11 * np.linalg.norm(ref, axis=0))


@pytest.mark.parametrize("regular", [True, False])
def test_batch_reports_the_threads_that_run(regular):
    """Patterns that share their column offsets run at most 512 threads per SM."""
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(5)
    arrays = []
    for n in (33, 3000, 5001):
        A = _spd(n, [1, 70], rng)
        arrays.append((A.indptr, A.indices, A.data) if regular else _irregular("unsorted", n, rng)[1])
    bt = sa.Batch([(_dev(a[0], np.int32), _dev(a[1], np.int32)) for a in arrays], M=4, s=16)
    for threads, per_sm in ((256, 1), (512, 1), (1024, 1), (512, 2), (1024, 2)):
        bt.set_schedule(threads, per_sm, 0)
        got = bt.schedule()
        assert got["threads"] == (min(threads, 512 // per_sm) if regular else threads)
        assert got["blocks_per_sm"] == per_sm
    bt.set_cluster(4, 1024, 0)
    assert bt.schedule()["threads"] == (512 if regular else 1024)
    xs = [torch.zeros(len(a[0]) - 1, dtype=torch.float64, device=DEV) for a in arrays]
    chosen = bt.autotune([_dev(a[2], np.float64) for a in arrays],
                         [_dev(rng.standard_normal(len(a[0]) - 1), np.float64) for a in arrays], xs, 1e-8)
    assert chosen["threads"] * chosen["blocks_per_sm"] <= (512 if regular else 1024)
    bt.close()


# both sides of every line in the choice of CG's form: cluster and grid (FP64 22,528
# rows, FP32 131,072), one block and the grid's kernels (65,536), and the reach from
# which FP64 takes the streaming kernels (4,524 at 70,000 rows)
@pytest.mark.parametrize("n,offsets,precision", [
    (22528, [1, 150], "f64"), (22529, [1, 150], "f64"), (131072, [1, 362], "mixed_krylov"),
    (131073, [1, 362], "mixed_krylov"), (136900, [1, 370], "mixed_krylov"), (65535, [1, 5000], "f64"),
    (65536, [1, 5000], "f64"), (70000, [1, 4523], "f64"), (70000, [1, 4524], "f64"),
    (70000, [1, 4524], "mixed_krylov"), (262144, [1, 64, 4096], "f64"), (200000, [1, 10000], "f64")])
def test_cg_at_the_lines_of_its_forms(n, offsets, precision):
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(n)
    A = _spd(n, offsets, rng)
    b = rng.standard_normal(n)
    Ad, bd = _csr(A), _dev(b, np.float64)
    for bad, status in ((None, 0), ("cap", 1), ("nan", -5), ("indefinite", -4)):
        seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", krylov="cg", precision=precision,
                          max_iters=3 if bad == "cap" else 500)
        M, c = (_csr((-A).tocsr()), bd) if bad == "indefinite" else (Ad, bd.clone())
        if bad == "nan":
            c[n // 2] = float("nan")
        x = torch.zeros_like(bd)
        if status < 0:
            with pytest.raises(sa.SeqError) as e:
                seq.solve(M, c, 1e-12, x)
            assert e.value.code == status
        else:
            info = seq.solve(M, c, 1e-12, x)
            r = np.linalg.norm(b - A @ x.cpu().numpy()) / np.linalg.norm(b)
            assert info["status"] == status
            assert r <= 1.01e-12 if status == 0 else info["iters"] == 3
        seq.close()


@pytest.mark.parametrize("schedule", [(1, 1024), (2, 512), ("cluster", 4)])
@pytest.mark.parametrize("regular", [True, False])
def test_batch_guess_of_the_largest_sketch(schedule, regular):
    """M = 16, s = 64, the largest workspace: solutions within the span of the
    history are found by the guess (64 random rows of 16 random columns: condition
    of a few, so to a thousand roundings), and by one sketch column less."""
    import paper_2309_02156_gb300 as sa
    for M, s in ((16, 64), (15, 63)):
        rng = np.random.default_rng(M)
        arrays, hist, bs = [], [], []
        for n in (64, 1000, 5001):
            A = _spd(n, [1, 7], rng)
            X = rng.standard_normal((n, M))
            arrays.append((A.indptr, A.indices, A.data) if regular else _irregular("unsorted", n, rng)[1])
            if not regular:
                p, c, v = arrays[-1]
                A = sp.csr_matrix((v, c, p), shape=(n, n))
            hist.append(X)
            bs.append(A @ (X @ rng.standard_normal(M)))
        bt = sa.Batch([(_dev(a[0], np.int32), _dev(a[1], np.int32)) for a in arrays], M=M, s=s)
        if schedule[0] == "cluster":
            bt.set_cluster(schedule[1], 512, 0)
        else:
            bt.set_schedule(schedule[1], schedule[0], 0)
        for k, X in enumerate(hist):
            for j in range(M):
                bt.push(k, _dev(X[:, j], np.float64))
        xs = [_dev(np.zeros(len(b)), np.float64) for b in bs]
        infos = bt.step([_dev(a[2], np.float64) for a in arrays], [_dev(b, np.float64) for b in bs], xs, 1e-8)
        bt.close()
        for i in infos:
            assert i["status"] == 0 and i["iters"] == 0 and i["guess_relres"] <= 1e3 * 2.0 ** -52


# both sides of every line between the resident GMRES and the cycle graph (the last
# column: one launch per solve)
@pytest.mark.parametrize("n,reach,sweeps,precision,resident", [
    (92160, 303, 0, "f64", True), (92161, 303, 0, "f64", False), (38913, 3000, 0, "f64", True),
    (38913, 3001, 0, "f64", False), (77825, 1000, 0, "f64", True), (77825, 1001, 0, "f64", False),
    (30000, 1000, 8, "f64", True), (30000, 1001, 8, "f64", False), (40000, 333, 8, "f64", True),
    (40000, 334, 8, "f64", False), (77824, 277, 8, "f64", True), (77825, 277, 8, "f64", False),
    (20000, 1800, 0, "mixed_krylov", True), (20000, 1801, 0, "mixed_krylov", False),
    (196608, 443, 0, "mixed_krylov", True), (196609, 443, 0, "mixed_krylov", False),
    (20000, 277, 8, "mixed_krylov", True), (20000, 278, 8, "mixed_krylov", False),
    (73728, 271, 8, "mixed_krylov", True), (73729, 271, 8, "mixed_krylov", False)])
@pytest.mark.parametrize("kind", ["jacobi", "chebyshev"])
def test_gmres_at_the_lines_of_its_forms(n, reach, sweeps, precision, resident, kind):
    import paper_2309_02156_gb300 as sa
    if not sweeps and kind == "chebyshev":
        pytest.skip("no sweeps")
    rng = np.random.default_rng(n + reach)
    A = _spd(n, [1, reach], rng)
    b = rng.standard_normal(n)
    Ad, bd = _csr(A), _dev(b, np.float64)
    for bad, status in ((None, 0), ("cap", 1), ("nan", -5)):
        seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", krylov="gmres", precision=precision,
                          max_iters=3 if bad == "cap" else 500, precond_sweeps=sweeps, precond_kind=kind)
        c = bd.clone()
        if bad == "nan":
            c[n // 2] = float("nan")
        x = torch.zeros_like(bd)
        if status < 0:
            with pytest.raises(sa.SeqError) as e:
                seq.solve(Ad, c, 1e-12, x)
            assert e.value.code == status
        else:
            info = seq.solve(Ad, c, 1e-12, x)
            r = np.linalg.norm(b - A @ x.cpu().numpy()) / np.linalg.norm(b)
            assert (info["launches"] < 100) == resident
            if bad == "cap" and info["status"] == 0:      # three iterations were enough
                status = 0
            assert info["status"] == status
            assert r <= 1.01e-12 if status == 0 else r > 1e-12 and info["iters"] == 3
        seq.close()


@pytest.mark.parametrize("ctas,reaches", [(8, (600, 1280, 1281, 5000)), (4, (2560, 2561)), (1, (9999, 10001))])
def test_batch_with_long_reaches(ctas, reaches):
    """Reaches at both sides of half a CTA's rows (20,480 rows: 2,560 a CTA of 8)."""
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(ctas)
    n = 20480
    for r in reaches:
        A = _spd(n, [1, r], rng)
        bs = [rng.standard_normal(n) for _ in range(3)]
        bt = sa.Batch([(_dev(A.indptr, np.int32), _dev(A.indices, np.int32))] * 3, M=2, s=8, zeta=2)
        if ctas > 1:
            bt.set_cluster(ctas, 512, 0)
        else:
            bt.set_schedule(512, 1, 0)
        xs = [_dev(np.zeros(n), np.float64) for _ in bs]
        infos = bt.step([_dev(A.data, np.float64)] * 3, [_dev(b, np.float64) for b in bs], xs, 1e-11)
        bt.close()
        for b, x, i in zip(bs, xs, infos):
            assert i["status"] == 0
            assert np.linalg.norm(b - A @ x.cpu().numpy()) <= 1.01e-11 * np.linalg.norm(b)


@pytest.mark.parametrize("offsets,threads", [([1, 264], 512), ([1, 2, 264], 1024), (list(range(1, 12)), 1024)])
def test_batch_threads_of_sequences_off_the_chip(offsets, threads):
    """70,000 rows do not fit one block's shared memory: five common offsets run 512
    threads, wider rows the threads that were set."""
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(len(offsets))
    n = 70000
    A = _spd(n, offsets, rng)
    b = rng.standard_normal(n)
    bt = sa.Batch([(_dev(A.indptr, np.int32), _dev(A.indices, np.int32))], M=2, s=8, zeta=2)
    bt.set_schedule(1024, 1, 0)
    assert bt.schedule()["threads"] == threads
    x = _dev(np.zeros(n), np.float64)
    info = bt.step([_dev(A.data, np.float64)], [_dev(b, np.float64)], [x], 1e-11)[0]
    bt.close()
    assert info["status"] == 0 and np.linalg.norm(b - A @ x.cpu().numpy()) <= 1.01e-11 * np.linalg.norm(b)
