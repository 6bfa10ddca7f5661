"""The work that users of this framework have it do, as cases that can be timed.

Every case goes through the Python binding (``paper_1302_5010_gb300.mpl``) and has one of
four kinds:

  solve      ``Solver.solve`` of a batch of LASSO problems to the KKT tolerance 1e-6, on a
             handle that has solved an earlier batch (its dictionary copies, Q = A^T A and
             captured graphs are what a program keeps between batches);
  correlate  ``Solver.correlate``, the worst-case analysis product A^T R alone;
  noalloc    ``mpl_correlate_noalloc``, the same product for programs that own the device
             memory themselves;
  train      ``Solver.train_proposal``, the training of the warm-start proposal network.

Inputs are drawn on the GPU by torch's seeded generator: the recipes of
``paper_1302_5010_gb300.synth`` (Gaussian unit-norm dictionaries with planted sparse codes;
face-shaped dictionaries [D I] with partly replaced pixels).
"""
import math

import numpy as np
import torch

from paper_1302_5010_gb300 import mpl

TOL = 1e-6
DEV = "cuda"


def _solve(name, n, m, p, kmin, kmax, lam_frac, rho, precision=1, qgram=0, smax=0, omega=1, values="gaussian",
           warm=False, sync_every=2, gemm_tile=128):
    return dict(kind="solve", data="gauss", name=name, n=n, m=m, p=p, kmin=kmin, kmax=kmax, lam_frac=lam_frac,
                rho=rho, precision=precision, qgram=qgram, smax=smax, omega=omega, values=values, sigma=1e-3,
                warm=warm, sync_every=sync_every, gemm_tile=gemm_tile)


def listed():
    return [
        # one signal on a small dictionary, default options: an interactive call, where
        # launches and the host's part count
        dict(_solve("one_256x1024_f32", 256, 1024, 1, 10, 10, 0.05, 2, precision=0), sigma=0.01),
        # a batch on the shape of the paper's Table I/II dictionary: mixed precision, Gram rows
        # from Q and the learned warm start, as a tuned service runs it
        _solve("batch256_1024x8192_bf16", 1024, 8192, 256, 20, 60, 0.02, 15, qgram=1, values="signed_uniform",
               warm=True, sync_every=1),
        # the same batch with every option at its default: plain FP32, computed Gram rows
        _solve("batch256_1024x8192_f32", 1024, 8192, 256, 20, 60, 0.02, 15, precision=0, values="signed_uniform"),
        # odd sizes in every dimension (rows that are no multiple of 4, so only FP32 applies)
        # with subspace exploratory matching (Algorithm 2)
        _solve("odd99_777x6001_f32_smpl", 777, 6001, 99, 10, 40, 0.03, 8, precision=0, omega=2),
        # a mid-sized batch whose sizes fill no tile
        _solve("batch75_1496x20011_bf16", 1496, 20011, 75, 30, 110, 0.015, 30, smax=512),
        # face-recognition-shaped batch: coherent class atoms and an identity block
        dict(kind="solve", data="face", name="face2048_1024x10024_bf16", n=1024, m=10024, p=2048, classes=100,
             per_class=90, rank=9, corrupt=0.10, noise=0.05, lam_frac=0.01, rho=10, precision=1, qgram=1, smax=512,
             omega=1, warm=False, sync_every=1, gemm_tile=256),
        # one batch of the streaming workload, mixed and plain
        _solve("stream512_2048x32768_bf16", 2048, 32768, 512, 50, 200, 0.01, 50, qgram=1, smax=512, sync_every=4,
               gemm_tile=256),
        _solve("stream512_2048x32768_f32", 2048, 32768, 512, 50, 200, 0.01, 50, precision=0, smax=512),
        # the largest batch: the benchmark's workload
        _solve("batch1024_4096x65536_bf16", 4096, 65536, 1024, 100, 400, 0.01, 100, qgram=1, smax=1024, sync_every=1,
               gemm_tile=256),
        # one signal on a big dictionary, where every correlation reads the whole dictionary
        _solve("one_1024x262144_bf16", 1024, 262144, 1, 60, 60, 0.02, 20, smax=256),
        # the correlation alone in FP32 for a program that owns its memory, ragged sizes
        dict(kind="noalloc", name="noalloc500_2044x32771_f32", n=2044, m=32771, p=500),
        # training of the proposal network on a solved stream
        dict(kind="train", name="train4096_1024x8192", n=1024, m=8192, p=4096, kmin=20, kmax=60, lam_frac=0.02,
             rho=15, values="signed_uniform", sigma=1e-3, epochs=4, batch=2048),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.random()
    if what < 0.62:
        n = _logint(rng, 200, 2200)
        precision = 1 if rng.random() < 0.6 else 0
        if precision == 1:
            n = max(8, n // 8 * 8)  # the mixed path wants rows of whole 16-byte units
        m = int(n * rng.uniform(4.0, 14.0))
        p = _logint(rng, 1, 512)
        frac = rng.uniform(0.01, 0.04)
        kmax = max(3, int(n * rng.uniform(0.03, 0.08)))
        rho = max(2, int(kmax * rng.uniform(0.2, 0.4)))
        case = _solve("", n, m, p, max(1, kmax // 3), kmax, frac, rho, precision=precision,
                      qgram=int(m <= 24000 and rng.random() < 0.5), smax=min(512, n), omega=rng.choice([1, 1, 1, 2]),
                      values=rng.choice(["gaussian", "signed_uniform"]), sync_every=rng.choice([1, 2, 4]),
                      gemm_tile=rng.choice([64, 128, 256]))
        del case["name"]
        return case
    if what < 0.72:
        n = rng.choice([512, 768, 1024])
        classes = rng.randint(20, 100)
        return dict(kind="solve", data="face", n=n, m=classes * 90 + n, p=_logint(rng, 16, 2048), classes=classes,
                    per_class=90, rank=9, corrupt=0.10, noise=0.05, lam_frac=rng.uniform(0.01, 0.03), rho=10,
                    precision=rng.randint(0, 1), qgram=rng.randint(0, 1), smax=512, omega=1, warm=False,
                    sync_every=rng.choice([1, 2, 4]), gemm_tile=rng.choice([64, 128, 256]))
    if what < 0.79:
        n = 8 * _logint(rng, 64, 250)
        case = _solve("", n, _logint(rng, 40000, 300000), rng.randint(1, 8), n // 60, n // 25, 0.02, n // 100 + 2,
                      precision=rng.randint(0, 1), smax=256)
        del case["name"]
        return case
    if what < 0.87:
        precision = rng.randint(0, 1)
        n = _logint(rng, 100, 4096)
        if precision == 1:
            n = max(8, n // 8 * 8)
        return dict(kind="correlate", n=n, m=_logint(rng, 500, 65536), p=_logint(rng, 1, 1024), precision=precision)
    if what < 0.95:
        return dict(kind="noalloc", n=_logint(rng, 100, 4096), m=_logint(rng, 500, 65536), p=_logint(rng, 1, 1024))
    n = 8 * _logint(rng, 32, 128)
    return dict(kind="train", n=n, m=8 * n, p=_logint(rng, 256, 4096), kmin=n // 50 + 1, kmax=n // 17, lam_frac=0.02,
                rho=max(2, n // 68), values="signed_uniform", sigma=1e-3, epochs=rng.randint(1, 4),
                batch=rng.choice([1024, 2048, 4096]))


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _gauss_dictionary(case, g):
    At = torch.randn((case["m"], case["n"]), generator=g, device=DEV)
    At /= torch.linalg.vector_norm(At, dim=1, keepdim=True)
    return At


def _gauss_signals(case, At, p, g):
    """b_i = A x_i + e_i with planted sparse codes, lambda_i a fraction of ||A^T b_i||_inf."""
    n, m = case["n"], case["m"]
    kmin, kmax = case["kmin"], case["kmax"]
    B = torch.empty((p, n), device=DEV)
    lam = torch.empty(p, device=DEV)
    step = max(1, min(p, (1 << 28) // m))
    for i in range(0, p, step):
        q = min(step, p - i)
        supp = torch.rand((q, m), generator=g, device=DEV).topk(kmax, dim=1).indices
        k = torch.randint(kmin, kmax + 1, (q, 1), generator=g, device=DEV)
        if case["values"] == "gaussian":
            v = torch.randn((q, kmax), generator=g, device=DEV)
        else:  # +-1 times U(0.5, 1.5)
            v = 0.5 + torch.rand((q, kmax), generator=g, device=DEV)
            v = torch.where(torch.rand((q, kmax), generator=g, device=DEV) < 0.5, -v, v)
        v = torch.where(torch.arange(kmax, device=DEV) < k, v, torch.zeros_like(v))
        X = torch.zeros((q, m), device=DEV).scatter_(1, supp, v)
        B[i:i + q] = X @ At + case["sigma"] * torch.randn((q, n), generator=g, device=DEV)
        lam[i:i + q] = case["lam_frac"] * (B[i:i + q] @ At.T).abs().amax(dim=1)
    return B, lam


def _pixels(img):
    """Shifted to be nonnegative and scaled to [0, 1], row by row."""
    img = img - img.amin(dim=1, keepdim=True)
    return img / img.amax(dim=1, keepdim=True)


def _unit(v):
    return v / torch.linalg.vector_norm(v, dim=1, keepdim=True)


def _face_dictionary(case, g):
    n, classes, per, rank = case["n"], case["classes"], case["per_class"], case["rank"]
    bases = torch.randn((classes, n, rank), generator=g, device=DEV) / math.sqrt(n)
    W = torch.randn((classes, rank, per), generator=g, device=DEV)
    noise = torch.randn((classes * per, n), generator=g, device=DEV) / math.sqrt(n)
    img = (bases @ W).transpose(1, 2).reshape(classes * per, n) + case["noise"] * noise
    return torch.cat([_unit(_pixels(img)), torch.eye(n, device=DEV)]).contiguous(), bases


def _face_signals(case, At, bases, p, g):
    """Fresh points of a class's subspace, a fraction of their pixels replaced by U(0, 1)."""
    n, classes, rank = case["n"], case["classes"], case["rank"]
    c = torch.randint(classes, (p,), generator=g, device=DEV)
    img = torch.bmm(bases[c], torch.randn((p, rank, 1), generator=g, device=DEV))[:, :, 0]
    img = _pixels(img + case["noise"] * torch.randn((p, n), generator=g, device=DEV) / math.sqrt(n))
    ncor = int(round(case["corrupt"] * n))
    at = torch.rand((p, n), generator=g, device=DEV).topk(ncor, dim=1).indices
    img.scatter_(1, at, torch.rand((p, ncor), generator=g, device=DEV))
    B = _unit(img).contiguous()
    return B, case["lam_frac"] * (B @ At.T).abs().amax(dim=1)


def _solve_inputs(case, seed):
    """The dictionary, an earlier batch of the stream (as large as this one) and this batch."""
    g = _generator(seed)
    if case["data"] == "face":
        At, bases = _face_dictionary(case, g)
        draw_signals = lambda p: _face_signals(case, At, bases, p, g)  # noqa: E731
    else:
        At = _gauss_dictionary(case, g)
        draw_signals = lambda p: _gauss_signals(case, At, p, g)  # noqa: E731
    return At, draw_signals(case["p"]), draw_signals(case["p"])


def _correlate_inputs(case, seed):
    g = _generator(seed)
    At = _gauss_dictionary(case, g)
    return At, torch.randn((case["p"], case["n"]), generator=g, device=DEV) * 0.3


# ---------------------------------------------------------------- state and pass
def prepare(case, seed):
    n, m, p = case["n"], case["m"], case["p"]
    if case["kind"] == "solve":
        At, (B0, lam0), (B, lam) = _solve_inputs(case, seed)
        opts = dict(omega=case["omega"], sync_every=case["sync_every"], qgram=case["qgram"])
        if case["smax"]:
            opts["smax"] = case["smax"]
        if case["precision"] == 1:
            opts["gemm_tile"] = case["gemm_tile"]
        solver = mpl.Solver(At, rho=case["rho"], precision=case["precision"], **opts)
        del At  # the handle keeps its own copy
        X = torch.empty((p, m), device=DEV)
        # the batch before this one: Q, the BF16 copy, the workspace and the graphs are in place
        solver.solve(B0, lam0, X, TOL)
        if case["warm"]:
            solver.train_proposal(B0, lam0, X, epochs=1)
            solver.set(mpl.MPL_OPT_WARM_START, 2)
            solver.solve(B0, lam0, X, TOL)
        return dict(case=case, solver=solver, B=B, lam=lam, X=X)
    if case["kind"] == "train":
        g = _generator(seed)
        At = _gauss_dictionary(case, g)
        B, lam = _gauss_signals(case, At, p, g)
        solver = mpl.Solver(At, rho=case["rho"], precision=1, qgram=1)
        Xref = torch.empty((p, m), device=DEV)
        for i in range(0, p, 1024):
            solver.solve(B[i:i + 1024], lam[i:i + 1024], Xref[i:i + 1024], TOL)
        return dict(case=case, solver=solver, B=B, lam=lam, Xref=Xref)
    At, R = _correlate_inputs(case, seed)
    C = torch.empty((p, m), device=DEV)
    if case["kind"] == "correlate":
        return dict(case=case, solver=mpl.Solver(At, precision=case["precision"]), R=R, C=C)
    return dict(case=case, At=At, R=R, C=C)


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        res = state["solver"].solve(state["B"], state["lam"], state["X"], TOL)
        return {"X": state["X"], "status": res.stats["status"], "nnz": res.stats["nnz"],
                "objective": res.stats["objective"]}
    if case["kind"] == "train":
        losses = state["solver"].train_proposal(state["B"], state["lam"], state["Xref"], epochs=case["epochs"],
                                                batch=case["batch"])
        return {"losses": losses, "weights": mpl.mpl_proposal_get_weights(state["solver"].h)}
    if case["kind"] == "correlate":
        state["solver"].correlate(state["R"], state["C"])
        return state["C"]
    rc = mpl.mpl_correlate_noalloc(state["At"], case["n"], case["m"], state["R"], case["p"], state["C"])
    if rc != mpl.MPL_OK:
        raise mpl.MplError(rc, "mpl_correlate_noalloc")
    return state["C"]


def work(case):
    n, m, p = case["n"], case["m"], case["p"]
    if case["kind"] == "solve":
        # the dictionary in the precision of the correlation, the signals and the solutions once
        # each; a first worst-case analysis and the one that certifies
        elem = 2 if case["precision"] == 1 else 4
        return {"bytes": elem * n * m + 4 * p * (n + 1) + 4 * p * m, "flops": 2 * 2.0 * n * m * p}
    if case["kind"] == "train":
        # one correlation for the examples (64 candidates a signal), then forward and backward
        # of 3 -> 64 -> 64 -> 1 for each of them in every epoch
        examples = 64 * p
        return {"bytes": 2 * n * m + 4 * p * (n + 1) + 4 * p * m + 16 * examples * case["epochs"],
                "flops": 2.0 * n * m * p + 6.0 * (3 * 64 + 64 * 64 + 64) * examples * case["epochs"]}
    elem = 2 if case["kind"] == "correlate" and case["precision"] == 1 else 4
    return {"bytes": elem * n * m + 4 * p * n + 4 * p * m, "flops": 2.0 * n * m * p}


# ---------------------------------------------------------------- exact values
def _restricted(G, h, lam, valid, x):
    """min lam ||x||_1 + x^T G x / 2 - h^T x for a batch of padded positive definite blocks, by
    an active-set method from x: sign-fixed solves, cut at the first sign change.  Returns the
    minimisers, or None where the method does not end."""
    q, s = h.shape
    eye = torch.eye(s, dtype=G.dtype, device=G.device)
    for _ in range(40 * 8):
        grad = h - torch.bmm(G, x[:, :, None])[:, :, 0]
        zero = valid & (x == 0)
        worst = torch.where(zero, grad.abs(), torch.zeros_like(grad))
        on = valid & (x != 0)
        sign = torch.sign(x)
        # the free variables are stationary: let in the zero that violates most
        stationary = torch.where(on, (grad - lam[:, None] * sign).abs(), torch.zeros_like(grad)).amax(1) <= 1e-11 * lam
        best, j = worst.max(dim=1)
        enter = stationary & (best > lam * (1 + 1e-10))
        if bool((stationary & ~enter).all()):
            return x
        rows = torch.nonzero(enter)[:, 0]
        on[rows, j[rows]] = True
        sign[rows, j[rows]] = torch.sign(grad[rows, j[rows]])
        M = G * (on[:, :, None] & on[:, None, :]) + eye * (~on).to(G.dtype)[:, None, :]
        rhs = torch.where(on, h - lam[:, None] * sign, torch.zeros_like(h))
        L, info = torch.linalg.cholesky_ex(M)
        if bool((info != 0).any()):
            return None
        y = torch.cholesky_solve(rhs[:, :, None], L)
        y = (y + torch.cholesky_solve(rhs[:, :, None] - torch.bmm(M, y), L))[:, :, 0]
        # the step ends where a free variable first loses its sign, which then becomes zero
        flip = on & (y * sign < 0)
        t = torch.where(flip, x / (x - y), torch.full_like(x, 2.0))
        tmin, jm = t.min(dim=1)
        full = tmin >= 1.0
        step = torch.where(full, torch.ones_like(tmin), tmin)[:, None]
        x = torch.where(on, x + step * (y - x), torch.zeros_like(x))
        cut = torch.nonzero(~full)[:, 0]
        x[cut, jm[cut]] = 0.0
    return None


def _lasso64(At, B, lam):
    """The LASSO solutions in 64 bits: active sets grown by the largest violators until no
    correlation off the set exceeds lambda.  None where a solve does not end."""
    p, m = B.shape[0], At.shape[0]
    cap, grow = 64, 24
    B, lam = B.double(), lam.double()
    S = torch.full((p, cap), -1, dtype=torch.int64, device=DEV)
    x = torch.zeros((p, cap), dtype=torch.float64, device=DEV)
    count = torch.zeros(p, dtype=torch.int64, device=DEV)
    X = torch.zeros((p, m), dtype=torch.float64, device=DEV)
    G = torch.zeros((p, cap, cap), dtype=torch.float64, device=DEV)
    h = torch.zeros((p, cap), dtype=torch.float64, device=DEV)
    part = max(1, (1 << 27) // At.shape[1])
    for _ in range(100):
        R = B.clone()
        g = torch.empty((p, m), dtype=torch.float64, device=DEV)
        for j in range(0, m, part):
            R -= X[:, j:j + part] @ At[j:j + part].double()
        for j in range(0, m, part):
            g[:, j:j + part] = R @ At[j:j + part].double().T
        g.abs_()
        inside = S >= 0
        g.scatter_(1, S.clamp(min=0), torch.where(inside, 0.0, g.gather(1, S.clamp(min=0))))
        top, idx = g.topk(min(grow, m), dim=1)
        take = top > lam[:, None] * (1 + 1e-9)
        new = take.sum(dim=1)
        if int(new.max()) == 0:
            return X
        need = int((count + new).max())
        if need > cap:
            if need > At.shape[1]:
                return None
            more = max(need, cap * 3 // 2) - cap
            S = torch.nn.functional.pad(S, (0, more), value=-1)
            x, h = (torch.nn.functional.pad(v, (0, more)) for v in (x, h))
            G = torch.nn.functional.pad(G, (0, more, 0, more))
            cap += more
        for i in range(0, p, max(1, (1 << 27) // (cap * At.shape[1]))):
            e = min(p, i + max(1, (1 << 27) // (cap * At.shape[1])))
            where = count[i:e, None] + torch.arange(top.shape[1], device=DEV)
            r, c = torch.nonzero(take[i:e], as_tuple=True)
            S[i + r, where[r, c]] = idx[i + r, c]
            A = At[S[i:e].clamp(min=0)].double() * (S[i:e] >= 0)[:, :, None]
            G[i:e] = torch.bmm(A, A.transpose(1, 2))
            h[i:e] = torch.bmm(A, B[i:e, :, None])[:, :, 0]
        count += new
        live = torch.nonzero(new > 0)[:, 0]
        for i in range(0, live.numel(), max(1, (1 << 27) // (cap * cap))):
            at = live[i:i + max(1, (1 << 27) // (cap * cap))]
            y = _restricted(G[at], h[at], lam[at], S[at] >= 0, x[at])
            if y is None:
                return None
            x[at] = y
        X.zero_()
        r, c = torch.nonzero(S >= 0, as_tuple=True)
        X[r, S[r, c]] = x[r, c]
    return None


def exact(case, seed):
    n, m, p = case["n"], case["m"], case["p"]
    if case["kind"] in ("correlate", "noalloc"):
        At, R = _correlate_inputs(case, seed)
        C = torch.empty((p, m), dtype=torch.float64, device=DEV)
        step = max(1, (1 << 27) // n)
        for j in range(0, m, step):
            C[:, j:j + step] = R.double() @ At[j:j + step].double().T
        return C
    # the weights after a training depend on its order of examples, which is the library's own
    if case["kind"] == "train":
        return None
    # hundreds of active atoms in each of hundreds of signals take minutes in 64 bits
    if 1.0 * n * m * p > 6e9 or case["data"] == "face" and p > 256:
        return None
    At, _, (B, lam) = _solve_inputs(case, seed)
    X = _lasso64(At, B, lam)
    if X is None:
        return None
    obj = torch.empty(p, dtype=torch.float64)
    for i in range(p):
        s = torch.nonzero(X[i])[:, 0]
        r = B[i].double() - X[i, s] @ At[s].double()
        obj[i] = float(lam[i].double() * X[i].abs().sum() + 0.5 * (r @ r))
    return {"X": X, "status": None, "nnz": None, "objective": np.asarray(obj)}
