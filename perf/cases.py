"""The work that a user of this package has it do, as cases that can be timed.

Each case is one call sequence of a time-stepping program: the guess for the
next system of a sequence from the history of solutions, the solve that starts
from it, one time step of a batch of sequences, or the training of the
coefficient predictor.  Operators and sizes are those of the sequences the
package is used on: the five-point variable-coefficient operator on the unit
square (symmetric, or with advection), and the fourth-order plus-shaped stencil
of width two (up to nine entries per row).

The systems are manufactured: the solution x(t) is a sum of smooth modes that
move in time, b(t) = A(t) x(t), and the history holds the earlier solutions as a
solver would have left them, with smooth errors of relative size `eta`.  So the
solution is known without a solve, and inputs are quick to make.

A solve that ends at its tolerance returns x near that solution (`exact`).  The
unpreconditioned restarted solves on large grids need a thousand iterations, and
how many moves with the last bit of every sum; they run here with the iteration
budget that a time stepper sets per step (`cap`), which fixes the work.
"""
import math

import torch

import paper_2309_02156_gb300 as sa

DEV = "cuda"
SEED = 0x5EEDBA5E


def listed():
    return [
        # A small SPD sequence, CG to 1e-10 from the sketched guess: the call
        # where latency counts (64 x 64, M = 10, s = 40).
        dict(name="cg_f64_64", kind="solve", grid=64, stencil=5, v0=0.0, krylov="cg",
             precision="f64", M=10, s=40, dt=0.01, tol=1e-10, eta=1e-9, cap=0,
             sweeps=0, pc="jacobi"),
        # A mid-size SPD sequence with an odd number of rows, FP32 CG inside
        # FP64 refinement.
        dict(name="cg_mixed_181", kind="solve", grid=181, stencil=5, v0=0.0, krylov="cg",
             precision="mixed_krylov", M=12, s=48, dt=0.01, tol=1e-10, eta=1e-9, cap=0,
             sweeps=0, pc="jacobi"),
        # A larger SPD sequence in FP64 (262,144 rows), CG to 1e-10.
        dict(name="cg_f64_512", kind="solve", grid=512, stencil=5, v0=0.0, krylov="cg",
             precision="f64", M=20, s=80, dt=0.01, tol=1e-10, eta=1e-9, cap=0,
             sweeps=0, pc="jacobi"),
        # The fourth-order scheme on 100 x 100, nonsymmetric: GMRES(30) in FP64.
        dict(name="gmres_f64_100_wide", kind="solve", grid=100, stencil=9, v0=20.0,
             krylov="gmres", precision="f64", M=20, s=80, dt=0.005, tol=1e-9, eta=1e-8, cap=60,
             sweeps=0, pc="jacobi"),
        # The main sequence: advection-diffusion on 1024 x 1024, FP64 GMRES(30)
        # without a preconditioner, four restart cycles.
        dict(name="gmres_f64_1024", kind="solve", grid=1024, stencil=5, v0=20.0,
             krylov="gmres", precision="f64", M=20, s=80, dt=0.005, tol=1e-10, eta=1e-8, cap=120,
             sweeps=0, pc="jacobi"),
        # The same with FP32 inner solves in FP64 refinement, eight cycles.
        dict(name="gmres_mixed_1024", kind="solve", grid=1024, stencil=5, v0=20.0,
             krylov="gmres", precision="mixed_krylov", M=20, s=80, dt=0.005, tol=1e-10,
             eta=1e-8, cap=240, sweeps=0, pc="jacobi"),
        # The same sequence with the degree-8 Chebyshev preconditioner, to 1e-10,
        # with the history, the sketch and the inner solves in FP32.
        dict(name="cheb8_mixed_1024", kind="solve", grid=1024, stencil=5, v0=20.0,
             krylov="gmres", precision="mixed", M=20, s=80, dt=0.005, tol=1e-10,
             eta=1e-8, cap=0, sweeps=8, pc="chebyshev"),
        # The largest grid, 2048 x 2048: FP64 history, preconditioned FP32 inner
        # solves, FP64 refinement to 1e-10.
        dict(name="cheb8_mixed_2048", kind="solve", grid=2048, stencil=5, v0=20.0,
             krylov="gmres", precision="mixed_krylov", M=20, s=80, dt=0.005, tol=1e-10,
             eta=1e-8, cap=0, sweeps=8, pc="chebyshev"),
        # A guess alone over the POD basis of the 1024 x 1024 history.
        dict(name="guess_pod_1024", kind="guess", grid=1024, stencil=5, v0=20.0, M=20, s=80,
             dt=0.005, eta=1e-8, guess="pod", basis_m=10),
        # 64 independent SPD sequences, a cluster of eight CTAs for each.
        dict(name="batch_64", kind="batch", count=64, gmin=48, gmax=384, M=12, s=48, dt=0.01,
             tol=1e-10, eta=1e-8, ctas=8),
        # 512 independent SPD sequences; clusters of four were the fastest of the
        # fixed schedules on these inputs (four 402 ms a step, one block 412).
        dict(name="batch_512", kind="batch", count=512, gmin=48, gmax=384, M=12, s=48, dt=0.01,
             tol=1e-10, eta=1e-8, ctas=4),
        # Training of the coefficient predictor: the normalisation and two epochs
        # over the samples of a sequence, forward, backward and Adam.
        dict(name="mlp_train", kind="mlp", M=20, s=80, hidden=256, count=384, batch=32,
             epochs=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["cg", "cg", "cg_mixed", "gmres", "gmres_mixed", "precond", "guess",
                       "batch", "mlp"])
    M = rng.randint(8, 24)
    s = rng.randint(2 * M, min(4 * M, 96))
    if what in ("cg", "cg_mixed"):
        return dict(kind="solve", grid=_log_int(rng, 32, 512 if what == "cg" else 255),
                    stencil=5, v0=0.0, krylov="cg",
                    precision="f64" if what == "cg" else "mixed_krylov", M=M, s=s, dt=0.01,
                    tol=1e-10, eta=1e-9, cap=0, sweeps=0, pc="jacobi")
    if what in ("gmres", "gmres_mixed"):
        grid = _log_int(rng, 64, 1024)
        return dict(kind="solve", grid=grid, stencil=rng.choice([5, 5, 9]), v0=20.0,
                    krylov="gmres", precision="f64" if what == "gmres" else "mixed_krylov",
                    M=M, s=s, dt=0.005, tol=1e-10, eta=1e-8,
                    cap=30 * rng.randint(1, 4), sweeps=0, pc="jacobi")
    if what == "precond":
        return dict(kind="solve", grid=_log_int(rng, 96, 1024), stencil=5, v0=20.0,
                    krylov="gmres", precision=rng.choice(["f64", "mixed_krylov", "mixed"]),
                    M=M, s=s, dt=0.005, tol=1e-10, eta=1e-8, cap=0,
                    sweeps=rng.choice([4, 8]), pc=rng.choice(["jacobi", "chebyshev", "chebyshev"]))
    if what == "guess":
        return dict(kind="guess", grid=_log_int(rng, 100, 1024), stencil=rng.choice([5, 9]),
                    v0=20.0, M=M, s=s, dt=0.005, eta=1e-8, guess="pod",
                    basis_m=rng.randint(4, M // 2))
    if what == "batch":
        count = _log_int(rng, 8, 256)
        M = rng.randint(8, 16)
        return dict(kind="batch", count=count, gmin=48, gmax=rng.randint(160, 384), M=M,
                    s=rng.randint(2 * M, min(4 * M, 64)), dt=0.01, tol=1e-10, eta=1e-8,
                    ctas=rng.choice([4, 8] if count <= 96 else [1, 4]))
    return dict(kind="mlp", M=M, s=s, hidden=rng.choice([64, 128, 256]),
                count=rng.randint(64, 512), batch=rng.choice([8, 16, 32]), epochs=2)


# ---------------------------------------------------------------------------
# Operators and solutions, made on the device.

def _points(grids):
    """Grid columns i, j = 1..N, step h and grid number of every unknown."""
    ii, jj, hh, kk = [], [], [], []
    for k, N in enumerate(grids):
        a = torch.arange(1, N + 1, device=DEV, dtype=torch.float64)
        ii.append(a.repeat(N))
        jj.append(a.repeat_interleave(N))
        hh.append(torch.full((N * N,), 1.0 / (N + 1), device=DEV, dtype=torch.float64))
        kk.append(torch.full((N * N,), k, device=DEV, dtype=torch.int64))
    return torch.cat(ii), torch.cat(jj), torch.cat(hh), torch.cat(kk)


def _pattern(N, stencil):
    """CSR rowptr, colind (int32, columns sorted); per row all stencil columns
    (dropped ones pointing at the row itself) and the mask of kept entries."""
    r = torch.arange(N * N, device=DEV)
    i, j = r % N, r // N
    steps = [(0, -1), (-1, 0), (0, 0), (1, 0), (0, 1)]
    if stencil == 9:
        steps = [(0, -2), (0, -1), (-2, 0), (-1, 0), (0, 0), (1, 0), (2, 0), (0, 1), (0, 2)]
    cols, mask = [], []
    for di, dj in steps:
        mask.append((i + di >= 0) & (i + di < N) & (j + dj >= 0) & (j + dj < N))
        cols.append(r + di + dj * N)
    mask = torch.stack(mask, 1)
    rowptr = torch.zeros(N * N + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(mask.sum(1), 0)
    cols = torch.where(mask, torch.stack(cols, 1), r[:, None])
    return rowptr.to(torch.int32), cols[mask].to(torch.int32), cols, mask


def _values5(i, j, h, phi, v0, t):
    """Entries S, W, P, E, N of -div(k grad u) + v . grad u + u (first-order
    upwind), k = 1 + sin(2 pi (x + t) + phi) cos(2 pi y) / 2 at face midpoints."""
    def k(x, y):
        return 1.0 + 0.5 * torch.sin(2 * math.pi * (x + t) + phi) * torch.cos(2 * math.pi * y)
    c = 1.0 / (h * h)
    ke, kw = k((i + 0.5) * h, j * h) * c, k((i - 0.5) * h, j * h) * c
    kn, ks = k(i * h, (j + 0.5) * h) * c, k(i * h, (j - 0.5) * h) * c
    vx, vy = v0 * math.cos(t), v0 * math.sin(t)
    diag = ke + kw + kn + ks + 1.0 + (abs(vx) + abs(vy)) / h
    return torch.stack([-ks - max(vy, 0.0) / h, -kw - max(vx, 0.0) / h, diag,
                        -ke + min(vx, 0.0) / h, -kn + min(vy, 0.0) / h], 1)


def _values9(i, j, h, phi, v0, t):
    """Entries of -k (u_xx + u_yy) + v . grad u + u, fourth-order centred."""
    k = 1.0 + 0.5 * torch.sin(2 * math.pi * (i * h + t) + phi) * torch.cos(2 * math.pi * j * h)
    d2, d1 = k / (12 * h * h), 1.0 / (12 * h)
    vx, vy = v0 * math.cos(t), v0 * math.sin(t)
    far, near = d2, -16.0 * d2
    return torch.stack([far + vy * d1, near - 8 * vy * d1, far + vx * d1, near - 8 * vx * d1,
                        60.0 * d2 + 1.0, near + 8 * vx * d1, far - vx * d1, near + 8 * vy * d1,
                        far - vy * d1], 1)


def _apply(entries, cols, mask, x):
    """A x, summed over each row's entries in column order."""
    y = torch.zeros_like(x)
    for k in range(entries.shape[1]):
        y += torch.where(mask[:, k], entries[:, k] * x[cols[:, k]], 0.0)
    return y


class _Modes:
    """x(t) = sum_k c_k(t) sin(a_k pi x) sin(b_k pi y), c_k a cosine in t, for
    every grid of a case; `noise` adds other modes of relative size eta."""

    def __init__(self, gen, i, j, h, which, grids, top=6):
        self.top = top
        self.which = which
        a = torch.arange(1, top + 1, device=DEV, dtype=torch.float64) * math.pi
        self.sx = torch.sin(torch.outer(i * h, a))
        self.sy = torch.sin(torch.outer(j * h, a))
        k = torch.arange(1, top + 1, dtype=torch.float64)
        shape = (grids, top, top)
        self.amp = torch.randn(shape, generator=gen, dtype=torch.float64) / \
            (k[:, None] ** 2 + k[None, :] ** 2)
        self.freq = 2.0 + 28.0 * torch.rand(shape, generator=gen, dtype=torch.float64)
        self.phase = 2 * math.pi * torch.rand(shape, generator=gen, dtype=torch.float64)
        self.gen = gen

    def _sum(self, c):
        c = c.to(DEV)
        if c.shape[0] == 1:
            return ((self.sy @ c[0]) * self.sx).sum(1)
        out = torch.empty(self.sx.shape[0], device=DEV, dtype=torch.float64)
        lo = 0
        for k, m in enumerate(torch.bincount(self.which).tolist()):
            out[lo:lo + m] = ((self.sy[lo:lo + m] @ c[k]) * self.sx[lo:lo + m]).sum(1)
            lo += m
        return out

    def at(self, t):
        return self._sum(self.amp * torch.cos(self.freq * t + self.phase))

    def noise(self, eta):
        return self._sum(eta * 0.1 * torch.randn(self.amp.shape, generator=self.gen,
                                                 dtype=torch.float64))


def _system(case, seed):
    """(CSR, b, x, history oldest first) of the next system of a sequence."""
    gen = torch.Generator().manual_seed(seed)
    N = case["grid"]
    u = torch.rand(2, generator=gen, dtype=torch.float64)
    phi, t = float(2 * math.pi * u[0]), float(u[1])
    i, j, h, which = _points([N])
    modes = _Modes(gen, i, j, h, which, 1)
    rowptr, colind, cols, mask = _pattern(N, case["stencil"])
    entries = (_values5 if case["stencil"] == 5 else _values9)(i, j, h, phi, case["v0"], t)
    x = modes.at(t)
    b = _apply(entries, cols, mask, x)
    M = case["M"]
    hist = [modes.at(t - (M - k) * case["dt"]) + modes.noise(case["eta"]) for k in range(M)]
    return sa.CSR(rowptr, colind, entries[mask]), b, x, hist


def _batch_grids(case, seed):
    """Grid sides, uniform in gmin..gmax (the same for every seed, so that the
    work does not change with the inputs)."""
    gen = torch.Generator().manual_seed(1234 + case["count"])
    return torch.randint(case["gmin"], case["gmax"] + 1, (case["count"],), generator=gen).tolist()


def _batch_system(case, seed, with_history=True):
    gen = torch.Generator().manual_seed(seed)
    grids = _batch_grids(case, seed)
    i, j, h, which = _points(grids)
    phi = (2 * math.pi * torch.rand(len(grids), generator=gen, dtype=torch.float64)).to(DEV)[which]
    t = float(torch.rand(1, generator=gen, dtype=torch.float64))
    modes = _Modes(gen, i, j, h, which, len(grids))
    entries = _values5(i, j, h, phi, 0.0, t)
    x = modes.at(t)
    pats = {N: _pattern(N, 5) for N in set(grids)}
    patterns, values, bs = [], [], []
    lo = 0
    for N in grids:
        rp, ci, cols, mask = pats[N]
        bs.append(_apply(entries[lo:lo + N * N], cols, mask, x[lo:lo + N * N]))
        patterns.append((rp, ci))
        values.append(entries[lo:lo + N * N][mask])
        lo += N * N
    M = case["M"]
    hist = [modes.at(t - (M - k) * case["dt"]) + modes.noise(case["eta"])
            for k in range(M)] if with_history else []
    return grids, patterns, values, bs, x, hist


# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "guess"):
        A, b, _, hist = _system(case, seed)
        if kind == "solve":
            opts = dict(precision=case["precision"], krylov=case["krylov"],
                        precond_sweeps=case["sweeps"], precond_kind=case["pc"])
            if case["cap"]:
                opts["max_iters"] = case["cap"]
        else:
            opts = dict(guess=case["guess"], basis_m=case["basis_m"])
        seq = sa.Sequence(A.n, case["M"], case["s"], seed=SEED, **opts)
        for x in hist:
            seq.push(x)
        return dict(case=case, seq=seq, A=A, b=b, x=torch.empty_like(b))
    if kind == "batch":
        grids, patterns, values, bs, _, hist = _batch_system(case, seed)
        bt = sa.Batch(patterns, case["M"], case["s"], seed=SEED)
        n = [N * N for N in grids]
        for x in hist:
            for k, xk in enumerate(torch.split(x, n)):
                bt.push(k, xk)
        bt.set_autopush(False)      # the same step again: the history stays
        if case["ctas"] > 1:
            bt.set_cluster(case["ctas"], 1024, 0)
        else:
            bt.set_schedule(1024, 1, 0)
        out = torch.empty(sum(n), device=DEV, dtype=torch.float64)
        return dict(case=case, batch=bt, values=values, b=bs, out=out,
                    x=list(torch.split(out, n)))
    samples, params = _mlp_inputs(case, seed)
    net = sa.MLP(case["M"], case["s"], hidden=case["hidden"], max_batch=case["batch"])
    return dict(case=case, net=net, samples=samples, params=params)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        state["seq"].guess(state["A"], state["b"], state["x"])
        state["seq"].solve(state["A"], state["b"], case["tol"], state["x"])
        return state["x"]
    if kind == "guess":
        state["seq"].guess(state["A"], state["b"], state["x"])
        return state["x"]
    if kind == "batch":
        state["batch"].step(state["values"], state["b"], state["x"], case["tol"])
        return state["out"]
    net = state["net"]
    net.set_params(state["params"])
    net.fit_normalization(state["samples"])
    losses = net.train(state["samples"], case["epochs"], case["batch"])
    params, norm = net.get_params()
    return [losses, params, norm]


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve" and not case["cap"]:
        return _system(case, seed)[2]
    if kind == "batch":
        return _batch_system(case, seed, with_history=False)[4]
    if kind == "mlp":
        return _mlp_exact(case, seed)
    return None     # a capped solve's or a guess's x depends on the sketch and the iterations


def work(case):
    """Bytes read and written at least once, and the floating-point operations
    of the work that the case fixes; for solves to a tolerance one iteration
    per decade is counted beyond the inputs and outputs."""
    kind = case["kind"]
    if kind == "mlp":
        inp = 4 * case["M"] + case["s"]
        H, M = case["hidden"], case["M"]
        npar = H * inp + H + H * H + H + M * H + M
        steps = case["epochs"] * (case["count"] // case["batch"])
        stride = inp + M + M * M + 1
        return {"bytes": 4.0 * case["count"] * stride * case["epochs"] + 8.0 * npar,
                "flops": 6.0 * npar * case["batch"] * steps}
    if kind == "batch":
        rows = sum(N * N for N in _batch_grids(case, 0))
        nnz = 5 * rows
        its = 10
    else:
        rows = case["grid"] ** 2
        nnz = case["stencil"] * rows
        its = 0 if kind == "guess" else (case["cap"] or 10)
    M = case["M"]
    elem = 4.0 if case.get("precision") == "mixed" else 8.0
    need = 12.0 * nnz + 4.0 * rows + elem * rows * M + 16.0 * rows
    flops = 2.0 * nnz * M + 2.0 * rows * M
    if kind == "solve" and case["krylov"] == "gmres" and case["cap"]:
        # The basis does not fit on the chip: each CGS2 step reads it twice.
        e = 8.0 if case["precision"] == "f64" else 4.0
        for c in range(its):
            k = c % 30 + 1
            need += e * rows * (2 * k + 2)
            flops += 2.0 * nnz + 8.0 * rows * k
    else:
        flops += its * (2.0 * nnz + 10.0 * rows)
    return {"bytes": need, "flops": flops}


# ---------------------------------------------------------------------------
# The coefficient predictor's samples: features, target, Gram matrix, ||S b||.

def _mlp_inputs(case, seed):
    gen = torch.Generator().manual_seed(seed)
    M, s, H, count = case["M"], case["s"], case["hidden"], case["count"]
    inp = 4 * M + s
    W = torch.randn(count, s, M, generator=gen, dtype=torch.float64)
    base = torch.randn(count, 4 * M, generator=gen, dtype=torch.float64)
    res = 0.1 * torch.randn(count, s, generator=gen, dtype=torch.float64)
    y = base[:, :M] + 0.3 * torch.tanh(base[:, M:2 * M]) + \
        0.05 * torch.randn(count, M, generator=gen, dtype=torch.float64)
    gram = W.transpose(1, 2) @ W
    nb = torch.linalg.vector_norm((W @ y[:, :, None])[:, :, 0] +
                                  torch.randn(count, s, generator=gen, dtype=torch.float64), dim=1)
    samples = torch.cat([base, res, y, gram.reshape(count, M * M), nb[:, None]], 1)

    def he(rows, cols):
        bound = math.sqrt(6.0 / cols)
        return (2 * torch.rand(rows * cols, generator=gen, dtype=torch.float64) - 1) * bound
    zero = torch.zeros
    params = torch.cat([he(H, inp), zero(H, dtype=torch.float64), he(H, H),
                        zero(H, dtype=torch.float64), he(M, H), zero(M, dtype=torch.float64)])
    return samples.to(torch.float32).to(DEV).contiguous(), params.to(torch.float32).numpy()


def _mlp_exact(case, seed):
    """Only the normalisation has a 64-bit value that the training's bfloat16
    weights do not decide: feature mean and deviation, output scale."""
    samples, _ = _mlp_inputs(case, seed)
    M, inp = case["M"], 4 * case["M"] + case["s"]
    f = samples.double()
    mu = f[:, :inp].mean(0)
    sd = f[:, :inp].var(0, unbiased=False).sqrt().clamp_min(1e-6)
    sig = (f[:, inp:inp + M] - f[:, :M]).square().mean(0).sqrt().clamp_min(1e-6)
    return [None, None, torch.cat([mu, sd, sig]).cpu().numpy()]
