"""Products with the solve's copy of the matrix, over the forms a matrix can
take: rows that share their column offsets (stored by offset), up to the most
offsets a slice may have and past it, rows with holes, odd sizes around the
32-row slices, and rows the offset form refuses (columns out of order, repeated
columns), which take the general layout.

Every matrix is strictly diagonally dominant with ||I - D^-1 A||_inf <= 1/2, so
||A^-1||_inf ||A||_inf <= 3 max|a_ii| / min|a_ii| <= 6: a solution with relative
residual 1e-12 lies within 6e-12 sqrt(n) of the exact one (2-norm; the infinity
norm bounds cost at most a factor sqrt(n) each way)."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spl
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _matrix(kind, n, rng):
    """CSR arrays of a diagonally dominant matrix of the named form."""
    offs = {"penta": [-7, -1, 0, 1, 7], "wide": [-14, -7, -2, -1, 0, 1, 2, 7, 14],
            "holes": [-7, -1, 0, 1, 7], "slots24": list(range(-12, 12)),
            "slots25": list(range(-12, 13)), "unsorted": [-7, -1, 0, 1, 7],
            "repeated": [-7, -1, 0, 1, 7], "scattered": [0]}[kind]
    rows = []
    for i in range(n):
        cols = [i + o for o in offs if 0 <= i + o < n]
        if kind == "holes":
            cols = [c for c in cols if c == i or rng.random() < 0.6]
        if kind == "scattered":
            cols = sorted(set(cols) | set(rng.integers(0, n, 6).tolist()))
        if kind == "unsorted":
            cols = cols[::-1]
        if kind == "repeated" and len(cols) > 1:
            cols = sorted(cols + [c for c in cols if c != i][:1])
        vals = rng.uniform(-1, 1, len(cols))
        off = sum(abs(v) for c, v in zip(cols, vals) if c != i)
        scale = 0.5 / off if off > 0 else 0.0
        d = rng.uniform(1, 2)
        rows.append((cols, [d if c == i else v * scale * d for c, v in zip(cols, vals)]))
    rowptr = np.cumsum([0] + [len(c) for c, _ in rows]).astype(np.int32)
    colind = np.concatenate([c for c, _ in rows]).astype(np.int32)
    return rowptr, colind, np.concatenate([v for _, v in rows])


FORMS = ["penta", "wide", "holes", "slots24", "slots25", "unsorted", "repeated", "scattered"]


@pytest.mark.parametrize("opts", [dict(), dict(precision="mixed_krylov"),
                                  dict(precond_sweeps=3),
                                  dict(precision="mixed_krylov", precond_sweeps=2)],
                         ids=["f64", "mixed", "f64_jacobi", "mixed_jacobi"])
@pytest.mark.parametrize("kind", FORMS)
@pytest.mark.parametrize("n", [1, 31, 33, 1000, 5025])
def test_gmres_on_every_form(kind, n, opts):
    import paper_2309_02156_gb300 as sa
    rng = np.random.default_rng(1000 * FORMS.index(kind) + n)
    rowptr, colind, vals = _matrix(kind, n, rng)
    A = sp.csr_matrix((vals, colind, rowptr), shape=(n, n))
    b = rng.standard_normal(n)
    ref = spl.spsolve(A.tocsc(), b)
    seq = sa.Sequence(n, 2, 8, zeta=2, guess="zero", krylov="gmres", max_iters=2000, **opts)
    Ad = sa.CSR(*(torch.from_numpy(t).to(DEV) for t in (rowptr, colind, vals)))
    x = torch.zeros(n, dtype=torch.float64, device=DEV)
    info = seq.solve(Ad, torch.from_numpy(b).to(DEV), 1e-12, x)
    assert info["status"] == 0
    err = np.linalg.norm(x.cpu().numpy() - np.ravel(ref)) / np.linalg.norm(ref)
    assert err <= 6e-12 * np.sqrt(n)
    seq.close()
