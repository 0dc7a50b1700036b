"""Performance cases of the equality-constrained LQR solver.

A case is one call sequence of a user's program on a batch of problems of one
kind, through ``eclqr.Batch`` or ``autograd.solve``:

  kind "run"      build, solve, multipliers and refinement of a batch (Batch.run)
  kind "graph"    the same pass, captured once and replayed (a fixed-rate loop)
  kind "resolve"  a new initial state on factors that are already built (Batch.solve)
  kind "grad"     forward and backward pass of the differentiable solve

The data follow the workload generator of this package (``synth``): random
stage matrices, a random feasible trajectory that fixes every offset, seeded.
They are drawn on the device, because drawing them is not what is measured.
Mixed rows number at most m - 1 per stage unless the case says otherwise: with
a random square D_i single problems come out nearly singular, and their
multipliers are then not determined to the digits that outputs are compared at.
"""
import math

import numpy as np
import torch

from paper_2407_05433_gb300 import autograd, eclqr, synth

OUTPUTS = ("x", "u", "lam", "mu", "eta", "alpha")


def _case(name, kind, problems, horizons, dims, rows, state_rows=0, end_rows=0, orthogonal=False, cross=False,
          degenerate=0.0):
    """problems: how many; horizons: (shortest, longest), uniform between; dims: "NxM NxM ...", taken in
    turn; rows: (fewest, most) mixed rows a stage, -1 as the most meaning m - 1; state_rows: state-only rows
    of every stage but the last; end_rows: terminal rows, -1 meaning uniform in 0..n/2; orthogonal: A_i
    orthogonal instead of I + 0.1 randn; cross: nonzero M_i; degenerate: the share of stages with
    duplicated mixed rows or mixed rows without controls."""
    c = {"kind": kind, "problems": problems, "n_short": horizons[0], "n_long": horizons[1], "dims": dims,
         "rows_min": rows[0], "rows_max": rows[1], "state_rows": state_rows, "end_rows": end_rows,
         "orthogonal": orthogonal, "cross": cross, "degenerate": degenerate}
    return {"name": name, **c} if name else c


def listed():
    return [
        # one small controller with a path constraint and a terminal set, solved once: the smallest call
        _case("single_n4", "run", 1, (64, 64), "4x2", (1, 1), end_rows=2),
        # the same controller in a fixed-rate loop, the pass captured once
        _case("single_n4_graph", "graph", 1, (64, 64), "4x2", (1, 1), end_rows=2),
        # state-only rows on every stage, one problem: the method's published timing shape
        _case("state_rows_n8", "run", 1, (1024, 1024), "8x4", (0, 0), state_rows=2),
        # one trajectory with redundant rows, rows without controls, more rows than controls and a fixed end
        _case("degenerate_n12", "run", 1, (1024, 1024), "12x6", (0, 8), end_rows=12, degenerate=0.2),
        # one long trajectory, cut into chunks and scanned
        _case("long_n16", "run", 1, (16384, 16384), "16x8", (4, 4), end_rows=8, orthogonal=True),
        # a handful of problems of odd sizes with cross costs: fewer tasks than the chip has SMs
        _case("few_odd", "run", 24, (37, 211), "13x5 9x4 21x7", (0, -1), end_rows=-1, cross=True),
        # the largest dimensions that the solver takes
        _case("wide_n32", "run", 160, (48, 96), "32x16", (0, 14), end_rows=8),
        # a fleet of unequal problems, over four per SM and group: the serving batch
        _case("fleet", "run", 2560, (32, 128), "8x4 12x6 16x8 24x12", (0, -1), end_rows=-1),
        # the same kind of fleet replanned from new initial states on the factors it holds
        _case("fleet_resolve", "resolve", 1024, (32, 128), "8x4 16x8", (0, -1), end_rows=-1),
        # the differentiable batch: solve, loss, and the gradient of every input
        _case("grad_n16", "grad", 256, (256, 256), "16x8", (4, 4), end_rows=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _weight(problems, stages, n, m):
    return problems * stages * (n + m) ** 3


def draw(rng):
    """Another case of the same kinds: sizes over the logarithm of their ranges, no dearer than the fleet."""
    most = sum(_weight(640, 80, n, m) for n, m in ((8, 4), (12, 6), (16, 8), (24, 12)))
    while True:
        what = rng.choice(["single", "single", "state", "long", "few", "fleet", "resolve", "grad"])
        n = rng.randint(3, 32)
        m = rng.randint(max(2, n // 4), max(2, min(16, n // 2 + 1)))
        end = rng.choice([0, -1, max(1, n // 4)])
        cross = rng.random() < 0.25
        if what == "single":
            N = _log(rng, 24, 2048)
            c = _case("", rng.choice(["run", "graph"]), 1, (N, N), f"{n}x{m}", (0, -1), end_rows=end, cross=cross)
        elif what == "state":
            N, n, m = _log(rng, 256, 8192), rng.randint(6, 14), rng.randint(4, 7)
            c = _case("", "run", 1, (N, N), f"{n}x{m}", (0, 0), state_rows=rng.randint(1, 2))
        elif what == "long":
            N, n = _log(rng, 4096, 16384), rng.randint(8, 18)
            m = (n + 1) // 2
            r = rng.randint(1, m - 1)
            c = _case("", "run", 1, (N, N), f"{n}x{m}", (r, r), end_rows=n // 2, orthogonal=True)
        elif what == "few":
            N = _log(rng, 48, 400)
            dims = " ".join(f"{k}x{rng.randint(max(2, k // 4), max(2, k // 2))}" for k in (rng.randint(4, 28) for _ in range(rng.randint(1, 3))))
            c = _case("", "run", _log(rng, 4, 96), (N // 2, N), dims, (0, -1), end_rows=end, cross=cross)
        elif what in ("fleet", "resolve"):
            N = _log(rng, 32, 160)
            dims = " ".join(f"{k}x{max(2, k // 2)}" for k in (rng.randint(4, 26) for _ in range(rng.randint(1, 4))))
            c = _case("", "run" if what == "fleet" else "resolve", _log(rng, 128, 2560), (N // 2, N), dims, (0, -1), end_rows=end, cross=cross)
        else:
            N, n = _log(rng, 24, 256), rng.randint(4, 20)
            m = max(2, n // 2)
            c = _case("", "grad", _log(rng, 8, 256), (N, N), f"{n}x{m}", (0, m - 1), end_rows=n // 4)
        dims = _dims(c)
        if sum(_weight(c["problems"] / len(dims), (c["n_short"] + c["n_long"]) / 2, n, m) for n, m in dims) <= most / (4 if c["kind"] == "grad" else 1):
            return c


def _dims(case):
    return [tuple(int(v) for v in d.split("x")) for d in case["dims"].split()]


# ---------------------------------------------------------------- data
def _spd(g, count, k, device):
    L = torch.randn(count, k, k, generator=g, device=device, dtype=torch.float64)
    H = L @ L.transpose(1, 2)
    H.diagonal(dim1=1, dim2=2).add_(1e-3)
    return H


def _problems(case, seed):
    """The batch's problems as synth.ECLQRProblem, with the distributions of synth.make_problem.  Horizons
    and row counts belong to the case, all values to the seed."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    rng = np.random.default_rng([case["problems"], case["n_short"], case["n_long"]])
    dims = _dims(case)
    got = [None] * case["problems"]
    for k, (n, m) in enumerate(dims):
        ids = list(range(k, case["problems"], len(dims)))
        if not ids:
            continue
        g = torch.Generator(device=dev).manual_seed(seed * 64 + k)
        rn = lambda *s: torch.randn(*s, generator=g, device=dev, dtype=torch.float64)  # noqa: E731
        N = rng.integers(case["n_short"], case["n_long"] + 1, size=len(ids))
        S, P = int(N.sum()), len(ids)
        most = case["rows_max"] if case["rows_max"] >= 0 else m - 1
        p = rng.integers(case["rows_min"], most + 1, size=S)
        q = np.full(S + P, case["state_rows"], dtype=np.int64)
        ends = np.cumsum(N + 1) - 1
        q[ends] = rng.integers(0, n // 2 + 1, size=P) if case["end_rows"] < 0 else case["end_rows"]
        if case["orthogonal"]:
            A, R = torch.linalg.qr(rn(S, n, n).cpu())
            A = (A * torch.sign(R.diagonal(dim1=1, dim2=2))[:, None, :]).to(dev)
        else:
            A = torch.eye(n, device=dev, dtype=torch.float64) + 0.1 * rn(S, n, n)
        B = rn(S, n, m)
        if case["cross"]:
            H = _spd(g, S, n + m, dev)
            Qs, M, R = H[:, :n, :n], H[:, :n, n:], H[:, n:, n:]
        else:
            Qs, M, R = _spd(g, S, n, dev), torch.zeros(S, n, m, device=dev, dtype=torch.float64), _spd(g, S, m, dev)
        stage = torch.from_numpy(np.delete(np.arange(S + P), ends)).to(dev)  # stages 0..N-1 of every problem
        Q = torch.empty(S + P, n, n, device=dev, dtype=torch.float64)
        Q[stage] = Qs
        Q[torch.from_numpy(ends).to(dev)] = _spd(g, P, n, dev)
        C, D, E = rn(int(p.sum()), n), rn(int(p.sum()), m), rn(int(q.sum()), n)
        lo = np.concatenate([[0], np.cumsum(p)])
        for s in rng.choice(S, size=int(round(case["degenerate"] * S)), replace=False):
            if p[s] >= 2 and rng.integers(0, 2) == 0:
                j = int(rng.integers(lo[s], lo[s + 1] - 1))
                C[j + 1], D[j + 1] = C[j], D[j]
            elif p[s] > 0:
                rows = lo[s] + rng.choice(p[s], size=max(1, (p[s] + 1) // 2), replace=False)
                D[torch.from_numpy(rows).to(dev)] = 0.0
        xs, us = rn(S + P, n), rn(S, m)
        xi, xn = xs[stage], xs[stage + 1]
        c = xn - torch.einsum("sij,sj->si", A, xi) - torch.einsum("sij,sj->si", B, us)
        of_p = torch.from_numpy(np.repeat(np.arange(S), p)).to(dev)
        of_q = torch.from_numpy(np.repeat(np.arange(S + P), q)).to(dev)
        d = -(C * xi[of_p]).sum(1) - (D * us[of_p]).sum(1)
        e = -(E * xs[of_q]).sum(1)
        a = {k2: v.contiguous().cpu().numpy() for k2, v in dict(A=A, B=B, c=c, C=C, D=D, d=d, E=E, e=e, Q=Q, M=M, R=R,
                                                                qv=rn(S + P, n), rv=rn(S, m), xs=xs).items()}
        lq = np.concatenate([[0], np.cumsum(q)])
        s0 = 0
        for t, j in enumerate(ids):
            s1, z0 = s0 + int(N[t]), s0 + t
            z1 = z0 + int(N[t]) + 1
            st, sz, sp, sq = slice(s0, s1), slice(z0, z1), slice(lo[s0], lo[s1]), slice(lq[z0], lq[z1])
            got[j] = synth.ECLQRProblem(
                N=int(N[t]), n=n, m=m, p=p[st].astype(np.int32), q=q[sz].astype(np.int32), A=a["A"][st], B=a["B"][st],
                c=a["c"][st], C=a["C"][sp], D=a["D"][sp], d=a["d"][sp], E=a["E"][sq], e=a["e"][sq], Q=a["Q"][sz],
                M=a["M"][st], R=a["R"][st], qv=a["qv"][sz], rv=a["rv"][st], s0=a["xs"][z0].copy())
            s0 = s1
    return got


def _new_s0(pbs, seed):
    rng = np.random.default_rng([seed, 2])
    return [rng.standard_normal(pb.n) for pb in pbs]


def _targets(pbs, seed):
    rng = np.random.default_rng([seed, 3])
    return [rng.standard_normal((pb.N + 1, pb.n)) for pb in pbs]


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    pbs = _problems(case, seed)
    batch = eclqr.Batch(pbs)
    state = {"kind": case["kind"], "batch": batch}
    if case["kind"] == "graph":
        batch.capture()
    elif case["kind"] == "resolve":
        batch.build()
        state["s0"] = torch.from_numpy(np.concatenate(_new_s0(pbs, seed))).to(batch.device)
    elif case["kind"] == "grad":
        state["params"] = autograd.batch_params(batch)
        state["target"] = torch.from_numpy(np.concatenate([t.ravel() for t in _targets(pbs, seed)])).to(batch.device)
    return state


def run(state):
    batch = state["batch"]
    if state["kind"] == "grad":
        x, u = autograd.solve(batch, *state["params"])
        loss = ((x - state["target"]) ** 2).sum() + (u ** 2).sum()
        grads = torch.autograd.grad(loss, state["params"], allow_unused=True)
        return {"x": x.detach(), "u": u.detach(), **{"d" + k: v for k, v in zip(autograd.PARAM_KEYS, grads)}}
    if state["kind"] == "graph":
        batch.replay()
    elif state["kind"] == "resolve":
        batch.solve(state["s0"])
        return {"x": batch.x, "u": batch.u, "status": batch.status}
    else:
        batch.run()
    return {**{k: getattr(batch, k) for k in OUTPUTS}, "status": batch.status}


def work(case):
    """Bytes: every input and output once.  Flops: the sequential method's, for the mean stage."""
    by = fl = 0.0
    dims = _dims(case)
    for k, (n, m) in enumerate(dims):
        P = len(range(k, case["problems"], len(dims)))
        S = P * (case["n_short"] + case["n_long"]) / 2
        p = (case["rows_min"] + (case["rows_max"] if case["rows_max"] >= 0 else m - 1)) / 2
        q = case["state_rows"]
        mb = max(0.0, m - min(m, p))
        data = 2 * n * n + 2 * n * m + m * m + 2 * n + m + (p + q) * (n + 1) + p * m
        out = 2 * n + m + p + q
        # backward recursion on the reduced problem: [A B]'P[A B], the control block's factor and gains
        k2 = n + mb
        riccati = 2 * n * n * k2 + n * k2 * k2 + mb ** 3 / 3 + 2 * mb * mb * n
        # stage elimination: QR of the control rows, Y and Z, and the products with them
        elim = 4 * m * m * min(m, p + q) + 2 * (n * n * m + n * m * mb) + 2 * (m * m * n + 2 * n * n * m + n * m * mb)
        # one residual pass, rollout and multipliers
        passes = 6 * (2 * n * n + 2 * n * m + m * m)
        if case["kind"] == "resolve":
            by += 8 * S * (n * n + 2 * n * m + 3 * n + 2 * m + out)
            fl += S * passes
        else:
            by += 8 * S * (data + out) * (2 if case["kind"] == "grad" else 1)
            fl += S * (riccati + elim + passes * (3 if case["kind"] == "grad" else 1))
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------- 64-bit values
def exact(case, seed):
    """The KKT system by block elimination from the last stage to the first, LU inside a block, refined
    on its own residual; batched over problems of equal (n, m).  None where it would take long."""
    pbs = _problems(case, seed)
    if sum(pb.N for pb in pbs) * max(pb.n + pb.m for pb in pbs) ** 3 > 3e9 or max(pb.N for pb in pbs) > 20000:
        return None
    unique = case["degenerate"] == 0  # rows that repeat others leave the multipliers to a choice
    s0 = _new_s0(pbs, seed) if case["kind"] == "resolve" else [pb.s0 for pb in pbs]
    target = _targets(pbs, seed) if case["kind"] == "grad" else None
    sol = [None] * len(pbs)
    adj = [None] * len(pbs)
    for nm in sorted({(pb.n, pb.m) for pb in pbs}):
        ids = [j for j, pb in enumerate(pbs) if (pb.n, pb.m) == nm]
        K = _Kkt([pbs[j] for j in ids], [s0[j] for j in ids], not unique)
        w = K.solve(K.rhs)
        for j, v in zip(ids, K.split(w)):
            sol[j] = v
        if target is not None:
            gx, gu = [2 * (sol[j]["x"] - target[j]) for j in ids], [2 * sol[j]["u"] for j in ids]
            for j, v in zip(ids, K.split(K.solve(K.linear(gx, gu)), gx)):
                adj[j] = v
    cat = lambda vs: np.concatenate([np.asarray(v).ravel() for v in vs])  # noqa: E731
    if target is not None:
        return {"x": cat(s["x"] for s in sol), "u": cat(s["u"] for s in sol),
                **{"d" + k: cat(_gradient(k, pb, s, a) for pb, s, a in zip(pbs, sol, adj)) for k in autograd.PARAM_KEYS}}
    if case["kind"] == "resolve":
        return {"x": cat(s["x"] for s in sol), "u": cat(s["u"] for s in sol), "status": None}
    out = {k: cat(s[k] for s in sol) for k in OUTPUTS}
    if not unique:
        out.update(dict.fromkeys(("lam", "mu", "eta", "alpha")))
    return {**{k: v if v is None or v.size else np.zeros(1) for k, v in out.items()}, "status": None}


def _gradient(key, pb, w, a):
    """-a' dF/dtheta of the KKT map F (bilinear in matrices and variables) at the solution w, adjoint a."""
    x, u, l1 = w["x"], w["u"], w["lam"][1:]
    xb, ub, lb = a["x"], a["u"], a["lam"][1:]
    mu, mub, eta, etab = w["mu"], a["mu"], w["eta"], a["eta"]
    ip, iq = np.repeat(np.arange(pb.N), pb.p), np.repeat(np.arange(pb.N + 1), pb.q)
    o = lambda f, g: f[:, :, None] * g[:, None, :]  # noqa: E731
    col = lambda f: f[:, None]  # noqa: E731
    return {"A": lambda: -(o(l1, xb[:-1]) + o(lb, x[:-1])), "B": lambda: -(o(l1, ub) + o(lb, u)),
            "C": lambda: -(col(mu) * xb[ip] + col(mub) * x[ip]), "D": lambda: -(col(mu) * ub[ip] + col(mub) * u[ip]),
            "E": lambda: -(col(eta) * xb[iq] + col(etab) * x[iq]), "M": lambda: -(o(xb[:-1], u) + o(x[:-1], ub)),
            "Q": lambda: -0.5 * (o(xb, x) + o(x, xb)), "R": lambda: -0.5 * (o(ub, u) + o(u, ub)), "c": lambda: -lb,
            "d": lambda: -mub, "e": lambda: -etab, "qv": lambda: -xb, "rv": lambda: -ub, "s0": lambda: a["alpha"]}[key]()


class _Kkt:
    """The KKT systems of problems of equal (n, m), padded to the same horizon and row counts.

    Block i holds x_i (n), u_i (m), the multipliers of the stage's rows (r, padded) and lambda_{i+1} (n).
    Block 0 has x_0 = s_0 in the place of its state stationarity, which gives lambda_0 afterwards, and
    drops the rows that x_0 settles.  Padding is identity."""

    def __init__(self, pbs, s0, deficient):
        self.pbs, n, m = pbs, pbs[0].n, pbs[0].m
        self.n, self.m, N, P = n, m, max(pb.N for pb in pbs), len(pbs)
        self.deficient = deficient
        self.rows = [self._rows(pb) for pb in pbs]
        r = self.r = max([0] + [int(t.max()) + 1 for pair in self.rows for _, _, t in pair if len(t)])
        b = self.b = 2 * n + m + r
        D = np.zeros((N + 1, P, b, b))
        U = np.zeros((N + 1, P, b))
        x, u, y, l = slice(0, n), slice(n, n + m), n + m, slice(n + m + r, b)
        self.first = []
        for j, pb in enumerate(pbs):
            k = pb.N
            mixed, only = self.rows[j]
            D[:k + 1, j, x, x] = pb.Q
            D[:k, j, u, u] = pb.R
            D[:k, j, x, u] = pb.M
            D[:k, j, u, x] = pb.M.transpose(0, 2, 1)
            D[:k, j, l, x] = pb.A
            D[:k, j, x, l] = pb.A.transpose(0, 2, 1)
            D[:k, j, l, u] = pb.B
            D[:k, j, u, l] = pb.B.transpose(0, 2, 1)
            U[:k + 1, j, x], U[:k, j, u], U[:k, j, l] = -pb.qv, -pb.rv, -pb.c
            for F, G, o, (row, at, t) in ((pb.C, pb.D, pb.d, mixed), (pb.E, None, pb.e, only)):
                D[at, j, y + t, x] = F[row]
                D[at, j, x, y + t] = F[row]
                if G is not None:
                    D[at, j, y + t, u] = G[row]
                    D[at, j, u, y + t] = G[row]
                U[at, j, y + t] = -o[row]
            used = np.zeros((k + 1, r), bool)
            for _, at, t in (mixed, only):
                used[at, t] = True
            at, t = np.nonzero(~used)
            D[at, j, y + t, y + t] = 1.0
            pad = np.concatenate([np.arange(n, n + m), np.arange(b - n, b)])
            D[k, j, pad, pad] = 1.0
            D[k + 1:, j] = np.eye(b)
            self.first.append((D[0, j, x].copy(), pb.qv[0]))
            D[0, j, x], U[0, j, x] = np.eye(n, b), s0[j]
        dev = self.dev = "cuda" if P > 4 and torch.cuda.is_available() else "cpu"
        self.N, self.D, self.rhs = N, torch.from_numpy(D).to(dev), torch.from_numpy(U).to(dev)
        # lambda_{i+1} of block i meets x_{i+1} of block i + 1 with -1, inside each horizon
        self.on = torch.tensor([[float(i < pb.N) for pb in pbs] for i in range(N + 1)], dtype=torch.float64, device=dev)
        self._factor()

    def _rows(self, pb):
        """(row, stage, slot of its multiplier) of the mixed rows, and of the state-only ones after them."""
        def numbered(stage, keep):
            row = np.nonzero(keep)[0]
            start = np.searchsorted(stage[row], stage[row])
            return row, stage[row], np.arange(len(row)) - start

        sp, sq = np.repeat(np.arange(pb.N), pb.p), np.repeat(np.arange(pb.N + 1), pb.q)
        keep = (sp > 0) | np.any(pb.D != 0, axis=1)
        if self.deficient:  # repeated rows stand once
            for k in range(1, len(sp)):
                keep[k] &= not (sp[k] == sp[k - 1] and np.array_equal(pb.C[k], pb.C[k - 1]) and np.array_equal(pb.D[k], pb.D[k - 1]))
        mixed, only = numbered(sp, keep), numbered(sq, sq > 0)
        count = np.bincount(mixed[1], minlength=pb.N + 1)
        return mixed, (only[0], only[1], only[2] + count[only[1]])

    def _factor(self):
        n, b = self.n, self.b
        self.inv = torch.empty_like(self.D)
        for i in range(self.N, -1, -1):
            Di = self.D[i].clone()
            if i < self.N:
                Di[:, b - n:, b - n:] -= self.on[i][:, None, None] * self.inv[i + 1][:, :n, :n]
            self.inv[i] = torch.linalg.pinv(Di, rtol=1e-11) if self.deficient else torch.linalg.inv(Di)

    def _sweep(self, f):
        n, b = self.n, self.b
        f = f.clone()
        for i in range(self.N - 1, -1, -1):
            f[i][:, b - n:] += self.on[i][:, None] * (self.inv[i + 1][:, :n] @ f[i + 1][:, :, None])[:, :, 0]
        w = torch.empty_like(f)
        for i in range(self.N + 1):
            if i > 0:
                f[i][:, :n] += self.on[i - 1][:, None] * w[i - 1][:, b - n:]
            w[i] = (self.inv[i] @ f[i][:, :, None])[:, :, 0]
        return w

    def _apply(self, w):
        n, b = self.n, self.b
        f = (self.D @ w[..., None])[..., 0]
        f[:-1, :, b - n:] -= self.on[:-1, :, None] * w[1:, :, :n]
        f[1:, :, :n] -= self.on[:-1, :, None] * w[:-1, :, b - n:]
        return f

    def solve(self, rhs):
        w = self._sweep(rhs)
        for _ in range(2):
            w = w + self._sweep(rhs - self._apply(w))
        return w

    def linear(self, gx, gu):
        """The adjoint's right-hand side: dl/dx and dl/du, no offsets, s_0 = 0."""
        f = torch.zeros_like(self.rhs)
        for j, (a, c) in enumerate(zip(gx, gu)):
            f[:len(a), j, :self.n] = torch.as_tensor(a).to(self.dev)
            f[:len(c), j, self.n:self.n + self.m] = torch.as_tensor(c).to(self.dev)
        f[0, :, :self.n] = 0.0
        return f

    def split(self, w, gx=None):
        """Per problem x, u, lam, mu, eta, alpha = -lam_0; of the pairs (lam_0, eta_0) the one with the
        smallest lam_0.  gx: dl/dx of an adjoint, whose linear cost of x is -dl/dx."""
        n, m, b = self.n, self.m, self.b
        w = w.cpu().numpy()
        got = []
        for j, pb in enumerate(self.pbs):
            mixed, only = self.rows[j]
            mu, eta = np.zeros(len(pb.d)), np.zeros(len(pb.e))
            mu[mixed[0]] = w[mixed[1], j, n + m + mixed[2]]
            eta[only[0]] = w[only[1], j, n + m + only[2]]
            F, q = self.first[j]
            l0 = F @ w[0, j] + (q if gx is None else -gx[j][0])
            if pb.q[0]:
                E0 = pb.E[:pb.q[0]].T
                eta[:pb.q[0]] = -np.linalg.lstsq(E0, l0, rcond=None)[0]
                l0 = l0 + E0 @ eta[:pb.q[0]]
            lam = np.concatenate([l0[None], w[:pb.N, j, b - n:]])
            got.append({"x": w[:pb.N + 1, j, :n], "u": w[:pb.N, j, n:n + m], "lam": lam, "mu": mu, "eta": eta, "alpha": -lam[0]})
        return got
