"""The work this library is used for, as measured cases.

One case is one pass through the Python binding (paper_2112_03985_gb300.api) on
a handle that a user's program keeps: fits of all jackknife submodels from a
start, single concurrent MTTKRPs, the loss and its gradient, a run to
convergence, a batch of uneven problems, and one whole job from the tensor to
the standard errors.  Tensors, ranks and block layouts are those of the
package's own workloads (workloads.py) and generic ones between them.

Keys of a case:
  op      "mttkrp"    the concurrent MTTKRP of every mode for the current factors
          "fit"       set_factors(start), `sweeps` sweeps, factors and losses read back
          "converge"  set_factors(start), run(sweeps, tol), factors read back
          "loss"      JKCALS.loss(U) and its backward (torch autograd)
          "batch"     `problems` uneven problems advanced `sweeps` sweeps by one Batch
          "job"       create, `sweeps` sweeps, factors, jackknife standard errors, destroy
  dims    mode sizes; mode 0 is the sampled one
  blocks  "loo" (one submodel per sample), "loo+full" (and the full model),
          "groups" (contiguous groups of `d` samples), "models" (`models`
          concurrent fits of the full tensor, nothing left out)
  ranks   components per submodel; several: one submodel per sample and rank
  form    precision of the MTTKRP (api.JKCALS(precision=...))
  data    planted factors: "uniform", "normal", "bumps" (lognormal scores in
          mode 0, Gaussian bumps in the others); noise 1% (bumps: 2%)
  dtype   dtype of the tensor
"""
import itertools
import math

import numpy as np
import torch

from paper_2112_03985_gb300 import api

DEV = "cuda"


# -- the cases -----------------------------------------------------------------
def listed():
    return [
        # the smallest calls: a chemometrics-sized tensor (workload 1), one MTTKRP per
        # mode as a caller's own solver takes them, and a fit of its 21 submodels, all
        # launches and latency
        dict(name="mttkrp 20x30x40 fp64", op="mttkrp", dims="20x30x40", blocks="loo+full", ranks="3",
             form="fp64", data="uniform", dtype="f64"),
        dict(name="fit 20x30x40 exact", op="fit", dims="20x30x40", blocks="loo+full", ranks="3",
             form="exact_bf16", data="uniform", dtype="f64", sweeps=50),
        # model selection: every sample left out at ranks 3, 5, 7 and 9 in one handle of
        # odd sizes, until each submodel has converged (converged ones are compacted away)
        dict(name="converge 41x61x35 all fp64", op="converge", dims="41x61x35", blocks="loo", ranks="3,5,7,9",
             form="fp64", data="uniform", dtype="f64", sweeps=60, tol=1e-6),
        # the fluorescence workload (300 samples x 100 emission x 50 excitation): the
        # default form and the tensor-core form of the benchmark, a few sweeps from a start
        dict(name="fit 300x100x50 fp64", op="fit", dims="300x100x50", blocks="loo", ranks="5",
             form="fp64", data="bumps", dtype="f32", sweeps=5),
        dict(name="fit 300x100x50 exact", op="fit", dims="300x100x50", blocks="loo", ranks="5",
             form="exact_bf16", data="bumps", dtype="f32", sweeps=10),
        # the same as one job with nothing kept: tensor and start in, standard errors out
        dict(name="job 300x100x50 exact", op="job", dims="300x100x50", blocks="loo+full", ranks="5",
             form="exact_bf16", data="bumps", dtype="f32", sweeps=20),
        # ragged sizes and a single-pass form: exploratory sweeps over odd shapes
        dict(name="mttkrp 157x83x211 bf16", op="mttkrp", dims="157x83x211", blocks="loo", ranks="6",
             form="bf16", data="uniform", dtype="f32"),
        # the large synthetic workload, delete-10 groups: the tensor-core forms' MTTKRPs
        # and one FP64 sweep
        dict(name="mttkrp 400x400x400 exact", op="mttkrp", dims="400x400x400", blocks="groups", d=10, ranks="10",
             form="exact_bf16", data="normal", dtype="f32"),
        dict(name="mttkrp 400x400x400 3xtf32", op="mttkrp", dims="400x400x400", blocks="groups", d=10, ranks="20",
             form="3xtf32", data="normal", dtype="f32"),
        dict(name="fit 400x400x400 fp64", op="fit", dims="400x400x400", blocks="groups", d=10, ranks="10",
             form="fp64", data="normal", dtype="f32", sweeps=1),
        # gradient-based fitting: the summed loss and its backward, 4-way, 100 submodels
        dict(name="loss 100x60x60x40 fp64", op="loss", dims="100x60x60x40", blocks="loo", ranks="8",
             form="fp64", data="normal", dtype="f32"),
        # many independent problems of uneven sizes and ranks in one graph per sweep
        dict(name="batch 20 uneven 3xtf32", op="batch", problems=20, blocks="loo", form="3xtf32",
             data="uniform", dtype="f32", sweeps=5),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """A case of the same ranges: 3- and 4-way tensors from 20x30x30 to 400x400x400,
    ranks 2 to 20, 12 to 400 submodels, at most the largest listed case's work."""
    op = rng.choice(["mttkrp", "mttkrp", "fit", "fit", "fit", "loss", "converge", "job", "batch"])
    form = rng.choice(["fp64", "fp64", "exact_bf16", "exact_bf16", "3xtf32", "bf16", "tf32", "split_bf16"])
    if op in ("fit", "converge", "job", "loss"):
        form = rng.choice(["fp64", "exact_bf16"])
    data = rng.choice(["uniform", "normal", "bumps"])
    if op == "batch":
        return dict(op=op, problems=rng.randint(6, 20), blocks="loo", form=rng.choice(["3xtf32", "exact_bf16"]),
                    data="uniform", dtype="f32", sweeps=rng.randint(2, 6))
    while True:
        four = rng.random() < 0.25
        dims = [_log(rng, 20, 400)] + [_log(rng, 12 if four else 30, 80 if four else 400) for _ in range(3 if four else 2)]
        rank = rng.randint(2, 12 if op != "mttkrp" else 20)
        c = dict(op=op, dims="x".join(map(str, dims)), ranks=str(rank), form=form, data=data,
                 dtype=rng.choice(["f32", "f64"]))
        kind = rng.choice(["loo", "loo+full", "groups", "models"])
        if op == "job":   # standard errors need submodels of one rank, small enough to enumerate
            kind, c["ranks"] = rng.choice(["loo", "loo+full"]), str(min(rank, 5))
        c["blocks"] = kind
        if kind == "groups":
            d = [x for x in range(2, 21) if dims[0] % x == 0 and dims[0] // x >= 4]
            if not d:
                continue
            c["d"] = rng.choice(d)
        elif kind == "models":
            c["models"] = _log(rng, 1, 100)
        if op in ("fit", "job"):
            c["sweeps"] = rng.randint(2, 8)
        elif op == "converge":
            c["sweeps"], c["tol"] = rng.randint(20, 60), 1e-5
        columns = sum(_layout(c)[1])
        effort = 2.0 * columns * math.prod(dims) * len(dims) * c.get("sweeps", 1)
        if columns <= 3200 and effort <= (1.5e11 if form == "fp64" else 1.2e12):
            return c


# -- inputs ----------------------------------------------------------------------
def _dims(c):
    return [int(x) for x in c["dims"].split("x")]


def _layout(c):
    """(left-out sets, ranks) of the blocks."""
    I, ranks = _dims(c)[0], [int(r) for r in c["ranks"].split(",")]
    if c["blocks"] == "groups":
        sets = [list(range(g, g + c["d"])) for g in range(0, I, c["d"])]
    elif c["blocks"] == "models":
        sets = [[] for _ in range(c["models"])]
    else:
        sets = [[p] for p in range(I)] + ([[]] if c["blocks"] == "loo+full" else [])
    return [s for s in sets for _ in ranks], [r for _ in sets for r in ranks]


def _factors(dims, R, data, gen):
    if data == "uniform":
        return [torch.rand(I, R, generator=gen, device=DEV, dtype=torch.float64) for I in dims]
    if data == "normal":
        # columns of congruence one half, as the large synthetic workload's
        S = 0.5 + 0.5 * torch.eye(R, dtype=torch.float64, device=DEV)
        L = torch.linalg.cholesky(S)
        return [torch.randn(I, R, generator=gen, device=DEV, dtype=torch.float64) @ L.T for I in dims]
    out = [torch.exp(0.5 * torch.randn(dims[0], R, generator=gen, device=DEV, dtype=torch.float64))]
    for I in dims[1:]:
        mu = I * torch.rand(1, R, generator=gen, device=DEV, dtype=torch.float64)
        sg = I * (0.05 + 0.10 * torch.rand(1, R, generator=gen, device=DEV, dtype=torch.float64))
        x = torch.arange(I, device=DEV, dtype=torch.float64)[:, None]
        out.append(torch.exp(-((x - mu) ** 2) / (2 * sg ** 2)))
    return out


def _tensor(dims, R, c, gen):
    letters = "abcdefg"[:len(dims)]
    F = _factors(dims, R, c["data"], gen)
    T = torch.einsum(",".join(l + "z" for l in letters) + "->" + letters, *F)
    E = torch.randn(T.shape, generator=gen, device=DEV, dtype=torch.float64)
    T = T + E * ((0.02 if c["data"] == "bumps" else 0.01) * T.norm() / E.norm())
    return T.float().contiguous() if c["dtype"] == "f32" else T.contiguous()


def _start(dims, ranks, c, gen):
    """Initial multi-matrices: one factor set per rank, shared by its blocks (concurrent
    models of the full tensor: one set each)."""
    out = []
    for I in dims:
        shared, cols = {}, []
        for g, r in enumerate(ranks):
            key = (r, g) if c["blocks"] == "models" else r
            if key not in shared:
                shared[key] = torch.rand(I, r, generator=gen, device=DEV, dtype=torch.float64)
            cols.append(shared[key])
        out.append(torch.cat(cols, dim=1).contiguous())
    return out


def _problem(c, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    dims = _dims(c)
    left, ranks = _layout(c)
    T = _tensor(dims, max(ranks), c, gen)
    return T, left, ranks, _start(dims, ranks, c, gen)


def _batch_problems(c, seed):
    """The uneven batch: I1 in 20..400, I2 and I3 in 30..150, rank 2..8 per problem.  The
    sizes belong to the case, the values to the seed."""
    sizes = np.random.default_rng(4003)
    out = []
    for b in range(c["problems"]):
        dims = [int(sizes.integers(20, 401)), int(sizes.integers(30, 151)), int(sizes.integers(30, 151))]
        p = dict(c, dims="x".join(map(str, dims)), ranks=str(int(sizes.integers(2, 9))))
        out.append((p, seed * 1000 + b))
    return out


def _handle(c, T, left, ranks, U):
    return api.JKCALS(T, 0, ranks, left, U, precision=c["form"])


def prepare(case, seed):
    if case["op"] == "batch":
        hs, starts = [], []
        for p, s in _batch_problems(case, seed):
            T, left, ranks, U = _problem(p, s)
            hs.append(_handle(p, T, left, ranks, U))
            starts.append(U)
        return {"case": case, "handles": hs, "starts": starts, "batch": api.Batch(hs, max_sweeps=case["sweeps"])}
    T, left, ranks, U = _problem(case, seed)
    if case["op"] == "job":
        return {"case": case, "T": T, "left": left, "ranks": ranks, "U": U}
    return {"case": case, "h": _handle(case, T, left, ranks, U), "U": U}


# -- one pass --------------------------------------------------------------------
def run(state):
    c = state["case"]
    op = c["op"]
    if op == "batch":
        for h, U in zip(state["handles"], state["starts"]):
            h.set_factors(U)
        state["batch"].sweep(c["sweeps"])
        state["batch"].sync()
        return [torch.cat([u.reshape(-1) for u in h.get_factors(device=DEV)]) for h in state["handles"]]
    if op == "job":
        with _handle(c, state["T"], state["left"], state["ranks"], state["U"]) as h:
            losses = h.als_sweep(c["sweeps"])
            U = h.get_factors()
            S, perm, aligned = h.jackknife_se(ref_block=h.K - 1)
        return {"losses": losses, "U": U, "S": S, "perm": perm, "aligned": aligned}
    h = state["h"]
    if op == "mttkrp":
        return [h.mttkrp(n, device=DEV) for n in range(h.N)]
    if op == "loss":
        U = [u.detach().requires_grad_() for u in state["U"]]
        f = h.loss(U)
        f.backward()
        return {"loss": f.detach(), "grad": [u.grad for u in U]}
    h.set_factors(state["U"])
    if op == "fit":
        losses = h.als_sweep(c["sweeps"], device=DEV)
        return {"losses": losses, "U": h.get_factors(device=DEV)}
    done, loss = h.run(c["sweeps"], c["tol"])
    return {"sweeps": done, "loss": loss, "U": h.get_factors(device=DEV)}


# -- what it cannot do without ------------------------------------------------------
def work(case):
    if case["op"] == "batch":
        parts = [work(dict(p, op="fit")) for p, _ in _batch_problems(case, 0)]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    dims, (left, ranks) = _dims(case), _layout(case)
    C, size = sum(ranks), math.prod(dims)
    factors = 8 * C * sum(dims)
    # the tensor read once, the factors in and the result (as large) out; a run to
    # convergence needs about a third of the sweeps it may take
    sweeps = case.get("sweeps", 1) if case["op"] != "converge" else max(1, case["sweeps"] // 3)
    grams = sum(r * r for r in ranks) * sum(dims) * 4.0   # Grams and row solves of a sweep
    return {"bytes": size * (4 if case["dtype"] == "f32" else 8) + 2 * factors,
            "flops": sweeps * (2.0 * C * size * len(dims) + (0 if case["op"] == "mttkrp" else grams))}


# -- the same in 64 bits ------------------------------------------------------------
class _Plain:
    """Concurrent fits of every block in plain FP64 torch."""

    def __init__(self, T, left, ranks, U):
        self.T, self.N, self.ranks = T.double(), T.dim(), ranks
        self.U = [u.clone() for u in U]
        self.offs = np.concatenate([[0], np.cumsum(ranks)]).astype(int)
        self.keep = torch.ones(self.U[0].shape, dtype=torch.float64, device=DEV)
        slices = self.T.reshape(T.shape[0], -1).square().sum(1)
        norms = []
        for g, D in enumerate(left):
            self.keep[D, self.offs[g]:self.offs[g + 1]] = 0
            norms.append(slices.sum() - slices[D].sum())
        self.norms = torch.stack(norms)
        self.U[0] *= self.keep
        # blocks of one rank together: their columns as a (blocks x rank) table
        self.groups = []
        for r in sorted(set(ranks)):
            blocks = [g for g, x in enumerate(ranks) if x == r]
            cols = torch.tensor([[self.offs[g] + j for j in range(r)] for g in blocks], device=DEV)
            self.groups.append((torch.tensor(blocks, device=DEV), cols))

    def mttkrp(self, n):
        Tn = self.T.movedim(n, 0).reshape(self.T.shape[n], -1)
        others = [self.U[k] for k in range(self.N) if k != n]
        C, J = self.U[0].shape[1], Tn.shape[1]
        out = torch.empty(Tn.shape[0], C, dtype=torch.float64, device=DEV)
        step = max(1, int(1.5e8 // J))
        for c in range(0, C, step):
            K = others[0][:, c:c + step]
            for u in others[1:]:
                K = (K[:, None, :] * u[None, :, c:c + step]).reshape(-1, K.shape[1])
            out[:, c:c + step] = Tn @ K
        return out

    def of(self, M, cols):   # blocks x rows x rank
        return M[:, cols].permute(1, 0, 2)

    def gram(self, n, cols):
        X = self.of(self.U[n], cols)
        return X.transpose(1, 2) @ X

    def losses(self, M):
        e = torch.empty(len(self.ranks), dtype=torch.float64, device=DEV)
        for blocks, cols in self.groups:
            H = torch.ones_like(self.gram(0, cols))
            for n in range(self.N):
                H = H * self.gram(n, cols)
            cross = (self.of(self.U[-1], cols) * self.of(M, cols)).sum((1, 2))
            e[blocks] = self.norms[blocks] + H.sum((1, 2)) - 2 * cross
        return e

    def sweep(self, active=None):
        for n in range(self.N):
            M = self.mttkrp(n)
            for blocks, cols in self.groups:
                if active is not None:
                    cols = cols[active[blocks]]
                if not len(cols):
                    continue
                H = torch.ones(len(cols), cols.shape[1], cols.shape[1], dtype=torch.float64, device=DEV)
                for k in range(self.N):
                    if k != n:
                        H = H * self.gram(k, cols)
                X = torch.linalg.solve(H, self.of(M, cols).transpose(1, 2)).transpose(1, 2)
                if n == 0:
                    X = X * self.of(self.keep, cols)
                if n < self.N - 1:
                    s = X.norm(dim=1, keepdim=True)
                    X = X / torch.where(s > 0, s, torch.ones_like(s))
                self.U[n][:, cols] = X.permute(1, 0, 2)
        return self.losses(M)

    def grad(self):
        out = []
        for n in range(self.N):
            M, G = self.mttkrp(n), torch.empty_like(self.U[n])
            for _, cols in self.groups:
                H = torch.ones_like(self.gram(0, cols))
                for k in range(self.N):
                    if k != n:
                        H = H * self.gram(k, cols)
                G[:, cols] = 2 * (self.of(self.U[n], cols) @ H - self.of(M, cols)).permute(1, 0, 2)
            out.append(G * self.keep if n == 0 else G)
        return self.losses(M).sum(), out


def _standard_errors(U, left, ranks, ref_block):
    """Submodels adjusted to a reference (signs, then columns), and their standard errors."""
    R, N = ranks[0], len(U)
    F = [u.reshape(u.shape[0], -1, R).transpose(1, 0, 2) for u in U]
    ref = [f[ref_block] for f in F]
    sub = [g for g, D in enumerate(left) if len(D)]
    perms = list(itertools.permutations(range(R)))
    aligned = [np.empty((len(sub), u.shape[0], R)) for u in U]
    for i, g in enumerate(sub):
        X, score = [f[g].copy() for f in F], np.ones((R, R))
        for n in range(N - 1):
            top = np.abs(X[n]).argmax(0)
            s = np.where(X[n][top, range(R)] < 0, -1.0, 1.0)
            X[n] *= s
            X[-1] *= s
        for n in range(1, N):
            a, b = ref[n], X[n]
            score *= np.abs((a.T @ b) / (np.linalg.norm(a, axis=0)[:, None] * np.linalg.norm(b, axis=0)))
        best = max(perms, key=lambda p: sum(score[s, p[s]] for s in range(R)))
        for n in range(N):
            aligned[n][i] = X[n][:, best]
    G = len(sub)
    S = [None] + [np.sqrt((G - 1) / G * ((a - a.mean(0)) ** 2).sum(0)) for a in aligned[1:]]
    return S, aligned


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        out = []
        for p, s in _batch_problems(case, seed):
            plain = _Plain(*_problem(p, s))
            for _ in range(case["sweeps"]):
                plain.sweep()
            out.append(torch.cat([u.reshape(-1) for u in plain.U]))
        return out
    T, left, ranks, U = _problem(case, seed)
    p = _Plain(T, left, ranks, U)
    if op == "mttkrp":
        return [p.mttkrp(n) for n in range(p.N)]
    if op == "loss":
        loss, grad = p.grad()
        return {"loss": loss, "grad": grad}
    if op in ("fit", "job"):
        losses = torch.stack([p.sweep() for _ in range(case["sweeps"])])
        if op == "fit":
            return {"losses": losses, "U": p.U}
        F = [u.cpu().numpy() for u in p.U]
        S, aligned = _standard_errors(F, left, ranks, len(ranks) - 1)
        return {"losses": losses, "U": F, "S": S, "perm": None, "aligned": aligned}
    prev, last, active, done = None, None, torch.ones(len(ranks), dtype=torch.bool, device=DEV), 0
    while done < case["sweeps"] and bool(active.any()):
        e = p.sweep(active)
        done += 1
        last = e if last is None else torch.where(active, e, last)
        if prev is not None:
            active = active & ~((prev - e).abs() / p.norms < case["tol"])
        prev = e
    return {"sweeps": None, "loss": last, "U": p.U}
