"""The work that users of libls have it do, as cases for timing and comparison.

Every case goes through the public binding (paper_2212_11403_gb300.ls).  Inputs are founder-mosaic
haplotypes, log-uniform recombination probabilities and the mutation probabilities of the
repository's workloads, drawn on the GPU from the seed alone.

kinds
  dense    ls_run_all: forward, backward and distances of all haplotypes at D loci, with the uniform
           prior or a prior matrix (FP32 or BF16 format), scalar or per-locus mu
  walk     the table API one variant at a time: ls_forward / ls_backward by single steps, the tables
           read back, ls_distance where they meet
  ckpt     ls_checkpoints over all loci (FP32 or binary16), then ls_ckpt_replay to a locus between two
  grad     ls_pac_grad: PAC log-likelihood and its gradient in log mu and groups of log rho
  propose  ls_propose: donor sets of every window, by match counts alone or with the network
  sparse   ls_sparse_run_all over proposed donor sets
  train    ls_mlp_create, ls_mlp_train, ls_mlp_get: Adam steps of the proposal network
  score    ls_mlp_forward: the network's scores of many candidate rows
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2212_11403_gb300 import ls

EPS = 2.0 ** -52          # the distance clamp (DBL_EPSILON)
WINDOW = 256              # loci per proposal window
PARAMS = 8 * 256 + 256 + 256 * 256 + 256 + 256 + 1


def listed():
    return [
        # the smallest data set of the repository's workloads: a thousand dependent steps, each tiny
        dict(name="dense_small", kind="dense", N=200, L=1000, D=10, founders=20, switch=1e-2, flip=1e-3, mu=1e-4,
             prior="uniform", mu_kind="scalar"),
        # a cohort of ragged size: too small to fill the GPU by targets alone
        dict(name="dense_ragged", kind="dense", N=1003, L=4000, D=4, founders=200, switch=5e-3, flip=5e-4, mu=1e-5,
             prior="uniform", mu_kind="scalar"),
        # the benchmark's workload: the dense all-vs-all pipeline at the size users report
        dict(name="dense_bench", kind="dense", N=5000, L=20000, D=16, founders=200, switch=5e-3, flip=5e-4, mu=1e-5,
             prior="uniform", mu_kind="scalar"),
        # more haplotypes than the register tiles hold (one target per CTA, state in registers and shared memory)
        dict(name="dense_large", kind="dense", N=26000, L=400, D=1, founders=1040, switch=1e-3, flip=1e-4, mu=1e-5,
             prior="uniform", mu_kind="scalar"),
        # a copying-prior matrix with mu per locus, at the size of the prior workload
        dict(name="dense_prior", kind="dense", N=20000, L=200, D=1, founders=1000, switch=2e-3, flip=5e-4, mu=1e-6,
             prior="fp32", mu_kind="locus"),
        # tables moved one variant at a time, as an interactive scan of a region does
        dict(name="walk_tables", kind="walk", N=10000, L=9, steps=4, founders=200, switch=5e-3, flip=5e-4, mu=1e-5),
        # checkpoints for a long region and one replay between them
        dict(name="checkpoint_replay", kind="ckpt", N=4999, L=2001, f16=True, founders=200, switch=5e-3, flip=5e-4,
             mu=1e-5),
        # one evaluation of the log-likelihood and its gradient inside a parameter fit
        dict(name="pac_gradient", kind="grad", N=2003, L=1999, K=50, founders=200, switch=5e-3, flip=5e-4, mu=1e-5),
        # donor sets with the trained network, the first half of the sparse path; the last window is partial
        dict(name="propose_network", kind="propose", N=12345, L=2000, C=1024, K=512, network=True, founders=493,
             switch=1e-3, flip=1e-4),
        # the sparse recursions over proposed sets, the second half
        dict(name="sparse_sets", kind="sparse", N=20003, L=2000, K=512, D=2, founders=800, switch=1e-3, flip=1e-4,
             mu=1e-5),
        # training the proposal network
        dict(name="train_network", kind="train", rows=400000, batch=16384, steps=20),
        # scoring candidate rows with the trained network
        dict(name="score_rows", kind="score", rows=2000003),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "prior", "walk", "ckpt", "grad", "propose", "sparse", "train", "score"])
    pop = dict(switch=10.0 ** rng.uniform(-3.0, -2.0), flip=10.0 ** rng.uniform(-4.0, -3.0))
    if kind == "dense":
        N = _logint(rng, 50, 26000)
        L = _logint(rng, 64, max(65, min(20000, int(2.5e11 / (float(N) * N)))))
        D = rng.randint(1, max(1, min(16, L, int(4e8 / (float(N) * N)))))
        return dict(kind="dense", N=N, L=L, D=D, founders=max(8, min(1000, N // 25)), mu=10.0 ** rng.uniform(-6.0, -4.0),
                    prior="uniform", mu_kind=rng.choice(["scalar", "scalar", "locus"]), **pop)
    if kind == "prior":
        N = _logint(rng, 100, 20000)
        L = _logint(rng, 64, max(65, min(4000, int(8e10 / (float(N) * N)))))
        D = rng.randint(1, max(1, min(8, L, int(4e8 / (float(N) * N)))))
        return dict(kind="dense", N=N, L=L, D=D, founders=max(8, min(1000, N // 25)), mu=10.0 ** rng.uniform(-6.0, -4.0),
                    prior=rng.choice(["fp32", "bf16"]), mu_kind=rng.choice(["scalar", "locus"]), **pop)
    if kind == "walk":
        N = _logint(rng, 200, 10000)
        steps = rng.randint(1, 6)
        return dict(kind="walk", N=N, L=2 * steps + 1, steps=steps, founders=max(8, min(400, N // 25)), mu=1e-5, **pop)
    if kind == "ckpt":
        N = _logint(rng, 200, 6000)
        L = _logint(rng, 64, max(65, min(8000, int(5e10 / (float(N) * N)))))
        return dict(kind="ckpt", N=N, L=L, f16=rng.choice([False, True]), founders=max(8, min(400, N // 25)), mu=1e-5,
                    **pop)
    if kind == "grad":
        N = _logint(rng, 100, 2500)
        L = _logint(rng, 64, max(65, min(4000, int(8e9 / (float(N) * N)))))
        return dict(kind="grad", N=N, L=L, K=rng.randint(1, min(100, L - 1)), founders=max(8, min(400, N // 10)),
                    mu=10.0 ** rng.uniform(-6.0, -4.0), **pop)
    if kind == "propose":
        N = _logint(rng, 600, 16000)
        L = _logint(rng, 300, max(301, min(4000, int(3e11 / (float(N) * N)))))
        K = rng.choice([64, 100, 256, 512])
        return dict(kind="propose", N=N, L=L, C=min(2048, K * rng.choice([1, 2, 3, 4])), K=K,
                    network=rng.choice([False, True]), founders=max(8, N // 25), **pop)
    if kind == "sparse":
        N = _logint(rng, 1500, 20000)
        return dict(kind="sparse", N=N, L=_logint(rng, 300, 2000), K=rng.choice([32, 100, 256, 500, 512]),
                    D=rng.randint(1, 2), founders=max(8, N // 25), mu=1e-5, **pop)
    if kind == "train":
        return dict(kind="train", rows=_logint(rng, 20000, 400000), batch=_logint(rng, 512, 16384),
                    steps=rng.randint(3, 20))
    return dict(kind="score", rows=_logint(rng, 1000, 4000000))


# ---- inputs ------------------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _haplotypes(case, g):
    """uint8 [L, N] on the GPU: founder mosaics with allele frequencies U(0.01, 0.5), a switch of
    founder with probability `switch` per variant and allele flips with probability `flip`."""
    N, L, F = case["N"], case["L"], min(case["founders"], case["N"])
    af = torch.empty(L, 1, device="cuda").uniform_(0.01, 0.5, generator=g)
    founders = (torch.rand(L, F, device="cuda", generator=g) < af).to(torch.uint8)
    h = torch.empty(L, N, dtype=torch.uint8, device="cuda")
    copied = torch.randint(F, (1, N), device="cuda", generator=g)
    for l0 in range(0, L, 1000):
        n = min(1000, L - l0)
        moved = torch.rand(n, N, device="cuda", generator=g) < case["switch"]
        chosen = torch.cat([copied, torch.randint(F, (n, N), device="cuda", generator=g)])
        at = torch.arange(1, n + 1, device="cuda").unsqueeze(1) * moved  # row of `chosen` since the last switch
        here = chosen.gather(0, at.cummax(0).values)
        flipped = (torch.rand(n, N, device="cuda", generator=g) < case["flip"]).to(torch.uint8)
        h[l0:l0 + n] = founders[l0:l0 + n].gather(1, here) ^ flipped
        copied = here[-1:]
    return h


def _parameters(case, seed):
    """rho [L-1] log-uniform in (1e-5, 1e-2); mu a number, or [L] within a factor of ten around it."""
    r = np.random.default_rng([int(seed) % (1 << 62), 7])
    rho = np.exp(r.uniform(math.log(1e-5), math.log(1e-2), size=case["L"] - 1))
    mu = case["mu"]
    if case.get("mu_kind") == "locus":
        mu = mu * 10.0 ** r.uniform(-0.5, 0.5, size=case["L"])
    return rho, mu


def _prior(N, g):
    """float32 [N, N], entries Gamma(2, 1) off the diagonal, rows (recipients) normalised."""
    out = torch.empty(N, N, device="cuda")
    for r0 in range(0, N, 2048):
        n = min(2048, N - r0)
        x = torch.empty(n, N, dtype=torch.float64, device="cuda").exponential_(generator=g)
        x += torch.empty(n, N, dtype=torch.float64, device="cuda").exponential_(generator=g)
        x[torch.arange(n, device="cuda"), torch.arange(r0, r0 + n, device="cuda")] = 0.0
        out[r0:r0 + n] = x / x.sum(1, keepdim=True)
    return out


def _decode_loci(L, D):
    return np.array([(k * (L - 1)) // (D - 1) for k in range(D)] if D > 1 else [L // 2], dtype=np.int32)


def _groups(L, K):
    return np.minimum(np.arange(L - 1, dtype=np.int64) * K // (L - 1), K - 1).astype(np.int32)


def _network(seed):
    """float32 [PARAMS]: He-uniform weights (the eighth input unused), small biases."""
    r = np.random.default_rng([int(seed) % (1 << 62), 11])
    W1 = r.uniform(-1, 1, (8, 256)) * math.sqrt(6.0 / 7.0)
    W1[7] = 0.0
    parts = [W1, r.uniform(-0.1, 0.1, 256), r.uniform(-1, 1, (256, 256)) * math.sqrt(6.0 / 256.0),
             r.uniform(-0.1, 0.1, 256), r.uniform(-1, 1, 256) * math.sqrt(3.0 / 256.0), r.uniform(-0.1, 0.1, 1)]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _features(rows, g):
    """float32 [rows, 8] match fractions of seven windows (the eighth column 0) and labels [rows]."""
    level = torch.rand(rows, 1, device="cuda", generator=g)
    X = 1.0 - level * torch.rand(rows, 8, device="cuda", generator=g) * 0.5
    X = torch.round(X * 256.0) / 256.0
    X[:, 7] = 0.0
    y = (1.0 - 6.0 * (1.0 - X[:, 2:5].mean(1)) + 0.05 * torch.randn(rows, device="cuda", generator=g)).clamp(0.0, 1.0)
    return X.contiguous(), y.contiguous()


class State:
    """What a program keeps between calls: the library's handles, freed with the object."""

    def __init__(self, case):
        self.case = case
        self.ctx = None
        self.tables = []
        self.net = None

    def __del__(self):
        for t in self.tables:
            ls.ls_table_destroy(t)
        if self.net is not None:
            ls.ls_mlp_destroy(self.net)
        if self.ctx is not None:
            ls.ls_destroy(self.ctx)


def prepare(case, seed):
    s = State(case)
    kind, g = case["kind"], _generator(seed)
    if kind == "train":
        s.X, s.y = _features(case["rows"], g)
        s.weights = _network(seed)
        s.stream_seed = int(seed) % (1 << 31)
        return s
    if kind == "score":
        s.X, _ = _features(case["rows"], g)
        s.net = ls.ls_mlp_create(_network(seed))
        s.scores = torch.empty(case["rows"], device="cuda")
        return s
    N, L = case["N"], case["L"]
    s.ctx = ls.ls_create(_haplotypes(case, g).cpu().numpy())
    if kind == "propose":
        s.net = ls.ls_mlp_create(_network(seed)) if case["network"] else None
        s.idx = torch.empty(N, (L + WINDOW - 1) // WINDOW, case["K"], dtype=torch.int32, device="cuda")
        return s
    rho, mu = _parameters(case, seed)
    if case.get("prior", "uniform") != "uniform":
        ls.ls_set_prior_format(s.ctx, ls.LS_PRIOR_BF16 if case["prior"] == "bf16" else ls.LS_PRIOR_FP32)
        ls.ls_set_params(s.ctx, rho, mu, _prior(N, g))
    else:
        ls.ls_set_params(s.ctx, rho, mu)
    if kind == "dense":
        s.loci = _decode_loci(L, case["D"])
        s.d = torch.empty(len(s.loci), N, N, device="cuda")
    elif kind == "walk":
        s.fwd, s.bck = ls.ls_table_create(s.ctx, ls.LS_FWD, 0, N), ls.ls_table_create(s.ctx, ls.LS_BWD, 0, N)
        s.tables = [s.fwd, s.bck]
        s.alpha, s.beta, s.d = (torch.empty(N, N, device="cuda") for _ in range(3))
        s.logf, s.logg = (torch.empty(N, dtype=torch.float64, device="cuda") for _ in range(2))
    elif kind == "ckpt":
        s.fwd = ls.ls_table_create(s.ctx, ls.LS_FWD, 0, N)
        s.tables = [s.fwd]
        s.alpha = torch.empty(N, N, device="cuda")
        s.logf = torch.empty(N, dtype=torch.float64, device="cuda")
    elif kind == "grad":
        s.groups = _groups(L, case["K"])
    elif kind == "sparse":
        s.loci = _decode_loci(L, case["D"])
        s.idx = torch.empty(N, (L + WINDOW - 1) // WINDOW, case["K"], dtype=torch.int32, device="cuda")
        ls.ls_propose(s.ctx, case["K"], case["K"], None, s.idx)
        s.d = torch.empty(len(s.loci), N, N, device="cuda")
        s.trust = torch.empty(len(s.loci), N, (N + 31) // 32, dtype=torch.int32, device="cuda")
    return s


def _replay_locus(L):
    return (5 * (L - 1)) // 8  # between the snapshots at 1/2 and 3/4 of the region


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "dense":
        rc, pac = ls.ls_run_all(s.ctx, s.loci, s.d)
        return s.d, pac
    if kind == "walk":
        ls.ls_table_reset(s.fwd)
        ls.ls_table_reset(s.bck)
        for k in range(case["steps"] + 1):
            ls.ls_forward(s.ctx, s.fwd, k)
            ls.ls_backward(s.ctx, s.bck, case["L"] - 1 - k)
        ls.ls_table_read(s.fwd, s.alpha, s.logf)
        ls.ls_table_read(s.bck, s.beta, s.logg)
        ls.ls_distance(s.ctx, s.fwd, s.bck, s.d)
        return s.alpha, s.logf.float(), s.beta, s.logg.float(), s.d  # log scales: sums of FP32 logarithms
    if kind == "ckpt":
        ls.ls_table_reset(s.fwd)
        ck = ls.ls_checkpoints(s.ctx, s.fwd, 0, case["L"] - 1, ls.LS_CKPT_F16 if case["f16"] else ls.LS_CKPT_F32)
        ls.ls_ckpt_replay(s.ctx, ck, s.fwd, _replay_locus(case["L"]))
        ls.ls_table_read(s.fwd, s.alpha, s.logf)
        ls.ls_ckpt_destroy(ck)
        return s.alpha, s.logf.float()
    if kind == "grad":
        rc, pac, dmu, drho = ls.ls_pac_grad(s.ctx, s.groups, case["K"])
        return pac, dmu, drho.astype(np.float32)  # expectations under the FP32 recursions
    if kind == "propose":
        ls.ls_propose(s.ctx, case["C"], case["K"], s.net, s.idx)
        return s.idx
    if kind == "sparse":
        rc, pac, fallback = ls.ls_sparse_run_all(s.ctx, s.idx, case["K"], WINDOW, s.loci, s.d, trust_out=s.trust)
        return s.d, s.trust, pac, fallback
    if kind == "train":
        net = ls.ls_mlp_create(s.weights)
        loss = ls.ls_mlp_train(net, s.X, s.y, case["steps"], case["batch"], 1e-3, s.stream_seed)
        weights = ls.ls_mlp_get(net)
        ls.ls_mlp_destroy(net)
        return weights, loss
    ls.ls_mlp_forward(s.net, s.X, s.scores)
    return s.scores


def work(case):
    kind = case["kind"]
    if kind == "train":
        # per row: 7 x 256 + 256 x 256 + 256 products forward, twice that backward (no input gradient)
        f = 2.0 * (3 * 256 * 256 + 2 * 7 * 256 + 3 * 256) * case["batch"] * case["steps"]
        return dict(bytes=36.0 * case["batch"] * case["steps"] + 8.0 * PARAMS, flops=f)
    if kind == "score":
        return dict(bytes=36.0 * case["rows"] + 4.0 * PARAMS, flops=2.0 * (7 * 256 + 256 * 256 + 256) * case["rows"])
    N, L = float(case["N"]), float(case["L"])
    if kind == "dense":
        prior = case["prior"] != "uniform"
        return dict(bytes=N * L / 8 + 4.0 * case["D"] * N * N + (4.0 * N * N if prior else 0.0),
                    flops=(10.0 if prior else 8.0) * N * N * L)
    if kind == "walk":  # every call leaves its table in memory: written by the first, read and written by the others
        n = case["steps"]
        return dict(bytes=N * N * 4 * (2 * (1 + 2 * n) + 4 + 3), flops=8.0 * N * N * (n + 1))
    if kind == "ckpt":
        snaps = max(1, math.ceil(math.log2(L)))
        return dict(bytes=N * N * ((2 if case["f16"] else 4) * snaps + 8), flops=4.0 * N * N * L)
    if kind == "grad":
        return dict(bytes=N * L / 8, flops=16.0 * N * N * L)
    windows = math.ceil(L / WINDOW)
    if kind == "propose":  # 256 bit comparisons a pair (symmetric), the network's products a candidate
        f = N * N * windows * WINDOW
        if case["network"]:
            f += 2.0 * (7 * 256 + 256 * 256 + 256) * N * min(case["C"], N - 1) * windows
        return dict(bytes=N * L / 8 + 4.0 * N * windows * case["K"], flops=f)
    return dict(bytes=N * L / 8 + 4.0 * N * windows * case["K"] + case["D"] * N * N * 4.125,
                flops=8.0 * N * L * min(3.0 * case["K"], N - 1))


# ---- the same results in 64 bits ---------------------------------------------------------------
class _Dense:
    """The rescaled recursions over all recipients (rows) and donors (columns), in float64."""

    def __init__(self, case, seed):
        g = _generator(seed)
        self.N, self.L = case["N"], case["L"]
        self.h = _haplotypes(case, g).bool()
        self.rho, mu = _parameters(case, seed)
        self.mu = np.broadcast_to(np.asarray(mu, dtype=np.float64), (self.L,))
        self.pi = 1.0 / (self.N - 1)
        self.prior = None
        if case.get("prior", "uniform") != "uniform":
            p = _prior(self.N, g)
            self.prior = (p.to(torch.bfloat16) if case["prior"] == "bf16" else p).double()

    def theta(self, l, rows=slice(None)):
        same = self.h[l, rows, None] == self.h[l, None, :]
        return torch.where(same, 1.0 - self.mu[l], self.mu[l]).double()

    def forward(self, to, keep=(), rows=slice(None)):
        """(alpha at `to`, log F at `to`, {l: alpha} for l in keep)."""
        ids = torch.arange(self.N, device="cuda")[rows]
        mine = torch.arange(len(ids), device="cuda"), ids
        pi = self.prior[rows] if self.prior is not None else self.pi
        kept, a, logf = {}, None, 0.0
        for l in range(to + 1):
            t = self.theta(l, rows)
            if a is None:
                a = t * pi
            else:
                a.mul_((1.0 - self.rho[l - 1]) / a.sum(1, keepdim=True)).add_(self.rho[l - 1] * pi).mul_(t)
            a[mine] = 0.0
            logf = logf + a.sum(1).log()
            if l in keep:
                kept[l] = a.clone()
        return a, logf, kept

    def backward(self, to, rows=slice(None)):
        """yields (l, beta at l, log G at l) for l = L-1 .. to."""
        ids = torch.arange(self.N, device="cuda")[rows]
        mine = torch.arange(len(ids), device="cuda"), ids
        pi = self.prior[rows] if self.prior is not None else self.pi
        b, logg = None, torch.zeros(len(ids), dtype=torch.float64, device="cuda")
        for l in range(self.L - 1, to - 1, -1):
            if b is None:
                b = torch.ones(len(ids), self.N, dtype=torch.float64, device="cuda")
            else:
                b.mul_(self.theta(l + 1, rows))
                s = (b * pi).sum(1, keepdim=True)
                logg = logg + s[:, 0].log()
                b.mul_((1.0 - self.rho[l]) / s).add_(self.rho[l])
            b[mine] = 0.0
            yield l, b, logg

    @staticmethod
    def distance(p):
        h = -0.5 * torch.log(torch.clamp(p, min=EPS))
        d = h + h.T
        d.fill_diagonal_(0.0)
        return d


def _exact_dense(case, seed):
    if float(case["N"]) ** 2 * case["L"] > 1.2e11:
        return None
    m = _Dense(case, seed)
    loci = [int(l) for l in _decode_loci(case["L"], case["D"])]
    d = torch.empty(len(loci), m.N, m.N, dtype=torch.float64)
    _, logf, alpha = m.forward(m.L - 1, set(loci))
    for l, b, _ in m.backward(loci[0]):
        if l in alpha:
            p = alpha.pop(l).mul_(b)
            d[loci.index(l)] = m.distance(p.div_(p.sum(1, keepdim=True))).cpu()
    return d, float(logf.sum())


def _exact_walk(case, seed):
    m, l = _Dense(case, seed), case["steps"]
    a, logf, _ = m.forward(l)
    for _, b, logg in m.backward(l):
        pass
    p = a * b
    return a, logf, b, logg, m.distance(p / p.sum(1, keepdim=True))


def _exact_ckpt(case, seed):
    if float(case["N"]) ** 2 * case["L"] > 6e10:
        return None
    a, logf, _ = _Dense(case, seed).forward(_replay_locus(case["L"]))
    return a, logf


def _exact_grad(case, seed):
    m, K = _Dense(case, seed), case["K"]
    N, L = m.N, m.L
    groups = _groups(L, K)
    block = max(1, min(N, int(1.2e9 / (float(N) * L))))
    pac = torch.zeros((), dtype=torch.float64, device="cuda")
    dmu = torch.zeros_like(pac)
    drho = torch.zeros(L - 1, dtype=torch.float64, device="cuda")
    for r0 in range(0, N, block):
        rows = slice(r0, min(N, r0 + block))
        ids = torch.arange(N, device="cuda")[rows]
        mine = torch.arange(len(ids), device="cuda"), ids
        _, logf, alpha = m.forward(L - 1, range(L), rows)
        pac += logf.sum()
        after = None  # theta beta at the locus after l
        for l, b, _ in m.backward(0, rows):
            a = alpha.pop(l)
            if after is not None:
                # d log P / d log rho of the interval (l, l + 1): the change of the transition's mass
                x = a / a.sum(1, keepdim=True)
                pi = torch.full_like(x, m.pi)
                pi[mine] = 0.0
                mass = (after * ((1.0 - m.rho[l]) * x + m.rho[l] * pi)).sum(1)
                drho[l] += m.rho[l] * ((after * (pi - x)).sum(1) / mass).sum()
            p = a * b
            differ = m.h[l, rows, None] != m.h[l, None, :]
            wrong = (p * differ).sum(1) / p.sum(1)
            dmu += (wrong - (1.0 - wrong) * m.mu[l] / (1.0 - m.mu[l])).sum()
            after = b * m.theta(l, rows)
            after[mine] = 0.0
    out = np.zeros(K)
    np.add.at(out, groups, drho.cpu().numpy())
    return float(pac), float(dmu), out


def _exact_sparse(case, seed):
    """The pooled chain over the unions of each window's set with its neighbours' sets."""
    s = prepare(case, seed)
    sets = s.idx.long()  # the proposed sets are inputs of the call
    m = _Dense(case, seed)
    N, L, K = m.N, m.L, case["K"]
    W = sets.shape[1]
    h8 = torch.cat([m.h, torch.zeros(L, 1, dtype=torch.bool, device="cuda")], 1)  # a dummy donor N
    ones = m.h.sum(1)
    loci = [int(l) for l in _decode_loci(L, case["D"])]

    def union(w):
        """(donor ids [N, 3K] ascending with N for padding, valid as float64)."""
        u = torch.cat([sets[:, v] for v in range(max(0, w - 1), min(W, w + 2))], 1)
        u = torch.where(u < 0, N, u).sort(1).values
        u[:, 1:][u[:, 1:] == u[:, :-1]] = N
        u = u.sort(1).values
        return u, (u < N).double()

    def sweep(order, forward, alpha, pool_at):
        """one direction; calls back at the decode loci with the quantities that the posterior needs"""
        x = o = tot = w = None
        logf, out = 0.0, {}
        for l in order:
            if w is None:
                w = l // WINDOW
                u, v = union(w)
                nout = N - 1 - v.sum(1)
                x, o = torch.zeros_like(v), torch.zeros(N, dtype=torch.float64, device="cuda")
                c, r = torch.zeros(N, dtype=torch.float64, device="cuda"), (m.pi if forward else 1.0)
            else:
                if l // WINDOW != w:
                    w = l // WINDOW
                    had = (x * v).sum(1)
                    fill = torch.where(nout > 0, o / nout.clamp(min=1), 0.0)
                    dense = torch.full((N, N + 1), -1.0, dtype=torch.float64, device="cuda")
                    dense.scatter_(1, u, torch.where(v > 0, x, -1.0))
                    u, v = union(w)
                    old = dense.gather(1, u)
                    del dense
                    old[u == N] = -1.0
                    stayed = old >= 0
                    mapped = torch.where(stayed, old, 0.0).sum(1)
                    entered = v.sum(1) - stayed.sum(1)
                    x = torch.where(stayed, old, fill[:, None]) * v
                    o = (o + (had - mapped) - entered * fill).clamp(min=0.0)
                    nout = N - 1 - v.sum(1)
                i = l - 1 if forward else l
                c = (1.0 - m.rho[i]) / (tot if forward else m.pi * tot)
                r = m.rho[i] * m.pi if forward else m.rho[i]
            before = x * c[:, None] + r
            if l in loci and not forward:
                z = (alpha[l] * before * v).sum(1)
                zp = torch.where(nout > 0, pool_at[l] * (c * o / nout.clamp(min=1) + r), 0.0)
                z = z + zp
                out[l] = (u, v, alpha[l] * before / z[:, None], zp / z / nout.clamp(min=1))
            same = h8[l][u] == m.h[l][:, None]
            x = torch.where(same, 1.0 - m.mu[l], m.mu[l]) * before * v
            match = (same * v).sum(1)
            mout = (torch.where(m.h[l], ones[l], N - ones[l]) - 1 - match).clamp(min=0)
            mout = torch.minimum(mout, nout)
            th = (1.0 - m.mu[l]) * mout + m.mu[l] * (nout - mout)
            o = torch.where(nout > 0, th / nout.clamp(min=1), 0.0) * (c * o) + r * th
            tot = x.sum(1) + o
            if forward:
                logf = logf + tot.log()
                if l in loci:
                    out[l] = (x.clone(), o.clone())
        return logf, out

    logf, fw = sweep(range(L), True, None, None)
    _, bw = sweep(range(L - 1, -1, -1), False, {l: fw[l][0] for l in loci}, {l: fw[l][1] for l in loci})
    d = torch.empty(len(loci), N, N, dtype=torch.float64)
    trust = torch.zeros(len(loci), N, (N + 31) // 32, dtype=torch.int32)
    for k, l in enumerate(loci):
        u, v, p, share = bw.pop(l)
        full = share[:, None].expand(N, N + 1).contiguous()
        full.scatter_(1, u, torch.where(v > 0, p, share[:, None]))
        d[k] = _Dense.distance(full[:, :N].clamp(max=1.0)).cpu()
        inside = torch.zeros(N, N + 1, dtype=torch.bool, device="cuda")
        inside.scatter_(1, u, v > 0)
        both = inside[:, :N] & inside[:, :N].T
        both.fill_diagonal_(False)
        words = torch.zeros(N, 32 * trust.shape[2], dtype=torch.int64, device="cuda")
        words[:, :N] = both
        words = (words.view(N, -1, 32) << torch.arange(32, device="cuda")).sum(2)
        trust[k] = (words - (words >> 31 << 32)).to(torch.int32).cpu()
    return d, trust, float(logf.sum()), 0


def _unpack(p):
    sizes, out, at = [(8, 256), (256,), (256, 256), (256,), (256,), (1,)], [], 0
    for z in sizes:
        n = int(np.prod(z))
        out.append(p[at:at + n].view(z))
        at += n
    return out


def _exact_train(case, seed):
    X, y = _features(case["rows"], _generator(seed))
    X, y = X.double(), y.double()
    p = torch.from_numpy(_network(seed)).double().cuda()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    state, tail = np.uint64(int(seed) % (1 << 31)), []
    steps, B = case["steps"], case["batch"]
    for it in range(steps):
        # the minibatch: a splitmix64 stream modulo the number of rows
        with np.errstate(over="ignore"):
            z = state + np.arange(1, B + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
            state = z[-1]
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = z ^ (z >> np.uint64(31))
        sel = torch.from_numpy((z % np.uint64(case["rows"])).astype(np.int64)).cuda()
        q = p.clone().requires_grad_(True)
        W1, b1, W2, b2, w3, b3 = _unpack(q)
        s = torch.relu(torch.relu(X[sel] @ W1 + b1) @ W2 + b2) @ w3 + b3
        loss = 0.5 * ((s - y[sel]) ** 2).sum() / B
        (grad,) = torch.autograd.grad(loss, q)
        if it >= steps - max(1, steps // 10):
            tail.append(float(loss))
        m = 0.9 * m + 0.1 * grad
        v = 0.999 * v + 0.001 * grad * grad
        mhat, vhat = m / (1.0 - 0.9 ** (it + 1)), v / (1.0 - 0.999 ** (it + 1))
        p = p - 1e-3 * mhat / (vhat.sqrt() + 1e-8)
    return p, float(np.mean(tail))


def _exact_score(case, seed):
    X, _ = _features(case["rows"], _generator(seed))
    W1, b1, W2, b2, w3, b3 = _unpack(torch.from_numpy(_network(seed)).double().cuda())
    out = torch.empty(case["rows"], dtype=torch.float64, device="cuda")
    for r0 in range(0, case["rows"], 1 << 18):
        x = X[r0:r0 + (1 << 18)].double()
        out[r0:r0 + (1 << 18)] = torch.relu(torch.relu(x @ W1 + b1) @ W2 + b2) @ w3 + b3
    return out


def exact(case, seed):
    """Results in 64 bits; None where the outputs are whole numbers or the case is too large."""
    f = dict(dense=_exact_dense, walk=_exact_walk, ckpt=_exact_ckpt, grad=_exact_grad, sparse=_exact_sparse,
             train=_exact_train, score=_exact_score).get(case["kind"])
    with torch.no_grad() if case["kind"] != "train" else torch.enable_grad():
        return f(case, seed) if f else None
