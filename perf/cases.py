"""The performance cases of the cloning library: what a user's programs ask of it, over
the range of sizes it is used at.

Four kinds of call, each through the package's public entry points:

  run     a batch of populations advances by a number of intervals (``run``), then its
          estimates are read (``estimate_psi``, ``events``, for some ``density_mode``);
          batches of at most STATE_CLONES clones are copied out whole as well
  steps   the per-step calls with the ancestry composed across every cloning stage
          (``evolve``, ``resample``, ``lineage``), as the ancestral samples are gathered
  select  the allocation-free cloning-stage selection of one population
  grad    loss and gradient of the window network on a batch of configurations

A batch's configurations continue from one pass to the next, as in a long run that is
read at intervals.
"""
import math

import numpy as np
import torch

import paper_1711_05095_gb300 as pg
from paper_1711_05095_gb300 import potential

STATE_CLONES = 1 << 18


def _run(name, **kw):
    case = dict(name=name, kind="run", L=50, n_pops=1, n_clones=1000, dt=0.1, intervals=10, lam_lo=20.0,
                lam_hi=20.0, weights="plain", selection="eq", density=False, uneven=0)
    case.update(kw)
    return case


def listed():
    return [
        # one small population, the first thing a new user runs: L = 20, s = 0.05,
        # N_c = 1000; a tenth of its 2000 intervals, then everything read back.  One
        # interval is a few microseconds of work: launches and latencies count.
        _run("ring", L=20, n_clones=1000, intervals=200),
        # psi(s) at 64 biases in one batch: L = 50, N_c = 16384, lambda in [-20, 40]
        _run("s_sweep", L=50, n_pops=64, n_clones=16384, intervals=200, lam_lo=-20.0, lam_hi=40.0),
        # large populations near the transition: L = 128, N_c = 2^20, lambda in
        # {5, 10, 15, 20} x 2 seeds, dt = 0.05, with the density mode that follows the
        # clustering
        _run("large_population", L=128, n_pops=8, n_clones=1 << 20, dt=0.05, intervals=100, lam_lo=5.0, lam_hi=20.0,
             density=True),
        # 256 populations of mixed ring lengths and of 2^10 to 2^18 clones in one batch
        _run("uneven_batch", L=128, n_pops=256, n_clones=1 << 18, intervals=40, lam_lo=-10.0, lam_hi=30.0,
             uneven=12345),
        # the study of the cloning interval at lambda = 28, plain and MODIFIED weights
        # side by side: the longest interval ([eq]), some 250 hops per clone, ...
        _run("study_long_dt", L=50, n_pops=32, n_clones=1 << 16, dt=10.0, intervals=6, lam_lo=28.0, lam_hi=28.0,
             weights="both"),
        # ... and [iid] selection at a middle one
        _run("study_iid", L=50, n_pops=32, n_clones=1 << 16, dt=1.0, intervals=20, lam_lo=28.0, lam_hi=28.0,
             weights="both", selection="iid"),
        # guided cloning at L = 128 under a window potential, 32 seeds
        _run("guided", L=128, n_pops=32, n_clones=1 << 14, dt=0.05, intervals=20, lam_lo=15.0, lam_hi=15.0,
             weights="guided"),
        # rings beyond 128 sites
        _run("wide_ring", L=256, n_pops=8, n_clones=8192, dt=0.05, intervals=50, lam_lo=10.0, lam_hi=10.0),
        # gathering ancestral configurations: per-step calls on large populations
        dict(name="ancestry", kind="steps", L=128, n_pops=4, n_clones=1 << 20, dt=0.05, intervals=10, lam=15.0),
        # selection for a caller that may not allocate, at its clone limit
        dict(name="select", kind="select", n_clones=1 << 20, mean=3.2, s=0.0012),
        # one minibatch of the window network's training
        dict(name="train_batch", kind="grad", L=128, n=16384),
        # the loss on held-out configurations (and a full-batch gradient)
        dict(name="held_out", kind="grad", L=128, n=1 << 20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "modified", "iid", "guided", "wide", "uneven", "steps", "select", "grad"])
    lam_lo = rng.uniform(-10.0, 15.0)
    lam = dict(lam_lo=lam_lo, lam_hi=lam_lo + rng.uniform(0.0, 20.0))
    if kind == "run":
        total = _log_int(rng, 500, 1 << 21)
        n_pops = min(_log_int(rng, 1, 128), max(1, total // 300))
        case = _run("", L=rng.randint(10, 128), n_pops=n_pops, n_clones=total // n_pops + 1,
                    dt=rng.choice([0.05, 0.1, 0.2, 0.3]), intervals=rng.randint(20, 60), density=rng.random() < 0.3,
                    **lam)
    elif kind == "modified":
        n_pops = 2 * rng.randint(1, 16)
        case = _run("", L=rng.randint(16, 100), n_pops=n_pops, n_clones=_log_int(rng, 500, 1 << 15),
                    dt=rng.choice([0.1, 0.3, 1.0, 3.0]), intervals=rng.randint(5, 20), weights="both", **lam)
    elif kind == "iid":
        n_pops = 2 * rng.randint(1, 16)
        case = _run("", L=rng.randint(16, 100), n_pops=n_pops, n_clones=_log_int(rng, 500, 1 << 16),
                    dt=rng.choice([0.1, 0.3, 1.0]), intervals=rng.randint(5, 20), weights="both", selection="iid",
                    **lam)
    elif kind == "guided":
        case = _run("", L=rng.randint(20, 128), n_pops=rng.randint(1, 32), n_clones=_log_int(rng, 500, 1 << 14),
                    dt=0.05, intervals=rng.randint(5, 20), weights="guided", **lam)
    elif kind == "wide":
        case = _run("", L=_log_int(rng, 129, 1024), n_pops=rng.randint(1, 8), n_clones=_log_int(rng, 300, 4096),
                    dt=0.05, intervals=rng.randint(5, 20), **lam)
    elif kind == "uneven":
        case = _run("", L=128, n_pops=rng.randint(8, 96), n_clones=_log_int(rng, 1 << 13, 1 << 17),
                    intervals=rng.randint(10, 30), uneven=rng.randint(1, 1 << 20), **lam)
    elif kind == "steps":
        case = dict(kind="steps", L=rng.randint(20, 128), n_pops=rng.randint(1, 4), n_clones=_log_int(rng, 1000, 1 << 19),
                    dt=rng.choice([0.05, 0.1]), intervals=rng.randint(3, 10), lam=rng.uniform(-10.0, 20.0))
    elif kind == "select":
        mean = rng.uniform(2.0, 60.0)
        case = dict(kind="select", n_clones=_log_int(rng, 1000, 1 << 20), mean=mean,
                    s=rng.choice([-1.0, 1.0]) * rng.uniform(0.0005, 0.3))
    else:
        case = dict(kind="grad", L=rng.randint(16, 128), n=_log_int(rng, 1000, 1 << 19))
    case.pop("name", None)
    return case


def _batch_of(case, seed):
    """The populations and biases of a run case: sizes from the case, streams from the seed."""
    n = case["n_pops"]
    seeds = [1000003 * int(seed) + i for i in range(n)]
    sel = pg.POP_IID if case["selection"] == "iid" else pg.POP_EQ
    if case["uneven"]:
        g = np.random.Generator(np.random.Philox(case["uneven"]))
        Ls = [int(v) for v in g.choice([32, 64, 100, 128], size=n)]
        ncs = [int(v) for v in np.floor(2.0 ** g.uniform(10, math.log2(case["n_clones"]), size=n))]
        lams = list(g.uniform(case["lam_lo"], case["lam_hi"], size=n))
    else:
        Ls, ncs = [case["L"]] * n, [case["n_clones"]] * n
        lams = list(np.linspace(case["lam_lo"], case["lam_hi"], n)) if n > 1 else [case["lam_lo"]]
    modes = {"plain": [pg.POP_PLAIN], "both": [pg.POP_PLAIN, pg.POP_MODIFIED], "guided": [pg.POP_GUIDED]}[case["weights"]]
    pops = [dict(L=Ls[i], N=Ls[i] // 2, n_clones=ncs[i], seed=seeds[i], weight_mode=modes[i * len(modes) // n],
                 selection=sel) for i in range(n)]
    return pops, [float(lam) / L ** 2 for lam, L in zip(lams, Ls)]


def _configurations(n, L, seed):
    """Uniform half-filled configurations as the words pop_copy_state gives, and labels."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    W = (L + 63) // 64
    words = torch.zeros((n, W), dtype=torch.int64, device="cuda")
    for at in range(0, n, 1 << 18):
        m = min(1 << 18, n - at)
        rank = torch.rand((m, L), generator=g, device="cuda").argsort(dim=1)
        sites = torch.zeros((m, 64 * W), dtype=torch.int64, device="cuda")
        sites.scatter_(1, rank[:, : L // 2], 1)
        bits = torch.arange(64, device="cuda")
        words[at:at + m] = (sites.view(m, W, 64) << bits).sum(dim=2)
    labels = torch.randint(0, 2, (n,), generator=g, device="cuda", dtype=torch.uint8)
    return words, labels


def prepare(case, seed):
    kind = case["kind"]
    if kind == "run":
        pops, s = _batch_of(case, seed)
        batch = pg.PopulationBatch(pops)
        if case["weights"] == "guided":
            phi = np.random.default_rng(seed).normal(0.0, 0.05, 512).astype(np.float32)
            for p in range(len(pops)):
                batch.set_potential(p, phi)
        return dict(case=case, batch=batch, s=s)
    if kind == "steps":
        n = case["n_pops"]
        pops = [dict(L=case["L"], N=case["L"] // 2, n_clones=case["n_clones"], seed=1000003 * int(seed) + i)
                for i in range(n)]
        batch = pg.PopulationBatch(pops)
        identity = torch.zeros(batch.slots, dtype=torch.int32, device="cuda")
        for p, q in enumerate(pops):
            off = batch.first_slot(p)
            identity[off:off + q["n_clones"]] = torch.arange(q["n_clones"], dtype=torch.int32, device="cuda")
        return dict(case=case, batch=batch, s=[case["lam"] / case["L"] ** 2] * n, identity=identity,
                    a=torch.zeros_like(identity), b=torch.zeros_like(identity))
    if kind == "select":
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed))
        mean = torch.full((case["n_clones"],), case["mean"], device="cuda")
        dk = torch.poisson(mean, generator=g).to(torch.int32)
        return dict(case=case, dk=dk, anc=torch.empty_like(dk), seed=int(seed))
    words, labels = _configurations(case["n"], case["L"], seed)
    return dict(case=case, words=words, labels=labels, trainer=potential.Trainer(seed=seed % (1 << 31)))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "run":
        batch = state["batch"]
        batch.run(case["dt"], state["s"], case["intervals"])
        psi, k_hat, t_obs = batch.estimate_psi()
        out = dict(psi=psi, k_hat=k_hat, t_obs=t_obs, events=batch.events().view(np.int64))
        if case["density"]:
            out["density"] = batch.density_mode(1)
        if sum(q["n_clones"] for q in batch.pops) <= STATE_CLONES:
            states = [batch.copy_state(p) for p in range(batch.n_pops)]
            out["lattice"] = np.concatenate([st["lattice"] for st in states]).view(np.int64)
            for name in ("K", "anc", "dK"):
                out[name] = np.concatenate([st[name] for st in states])
        return out
    if kind == "steps":
        batch, lin, other = state["batch"], state["a"], state["b"]
        lin.copy_(state["identity"])
        for _ in range(case["intervals"]):
            batch.evolve(case["dt"], state["s"])
            batch.resample()
            batch.lineage(lin, other)
            lin, other = other, lin
        psi, k_hat, t_obs = batch.estimate_psi()
        return dict(lineage=lin, psi=psi, k_hat=k_hat, t_obs=t_obs)
    if kind == "select":
        term = pg.select_noalloc(state["dk"], case["s"], state["seed"], 1, state["anc"])
        return dict(anc=state["anc"], psi_term=np.float64(term))
    loss, grad = state["trainer"].grad(state["words"], state["labels"], case["L"])
    return dict(loss=loss, grad=grad)


def work(case):
    """Bytes: the state (configurations, K, activities) in and out once per pass, or a
    batch's configurations and labels and the gradient.  flops: 32-bit operations, as
    integer work: per hop the active bonds, their count, the draw, the waiting time, the
    bond and the flip (140 for two lattice words, 115 for one), 24 per clone for a cloning
    stage."""
    kind = case["kind"]
    if kind in ("run", "steps"):
        if kind == "run":
            pops, _ = _batch_of(case, 0)
        else:
            pops = [dict(L=case["L"], N=case["L"] // 2, n_clones=case["n_clones"])] * case["n_pops"]
        W = (max(q["L"] for q in pops) + 63) // 64
        nbytes = ops = 0.0
        for q in pops:
            L, N, n = q["L"], q["N"], q["n_clones"]
            hops = case["dt"] * 2.0 * N * (L - N) / max(1, L - 1)
            nbytes += n * 2.0 * (8 * W + 8)
            ops += n * case["intervals"] * ((hops + 1.0) * (115 if W == 1 else 140) + 24)
        return dict(bytes=nbytes, flops=ops)
    if kind == "select":
        return dict(bytes=8.0 * case["n_clones"], flops=24.0 * case["n_clones"])
    W = (case["L"] + 63) // 64
    n = case["n"]
    return dict(bytes=n * (8.0 * W + 1) + 2 * 4.0 * potential.N_PARAMS,
                flops=2.0 * 512 * 128 * 128 * 3 + 3.0 * n * case["L"])


def exact(case, seed):
    """64-bit values where there are any: the psi term of one selection, and the loss
    and gradient of the window network without BF16 rounding.  The estimates of a run are
    those of its own random numbers: no plain evaluation gives them."""
    if case["kind"] == "select":
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed))
        mean = torch.full((case["n_clones"],), case["mean"], device="cuda")
        dk = torch.poisson(mean, generator=g).to(torch.int32).cpu().numpy().astype(np.float64)
        ref = dk.min() if case["s"] >= 0 else dk.max()
        term = -case["s"] * ref + math.log1p(math.fsum(np.expm1(-case["s"] * (dk - ref))) / dk.size)
        return dict(anc=None, psi_term=np.float64(term))
    if case["kind"] != "grad":
        return None
    L, n = case["L"], case["n"]
    words, labels = _configurations(n, L, seed)
    theta = torch.from_numpy(potential.init_params(seed % (1 << 31)).astype(np.float64)).cuda().requires_grad_(True)
    H = potential.HIDDEN
    cut = np.cumsum([0, H * 9, H, H * H, H, H, 1, 1])
    W1, b1, W2, b2, W3, b3, c = (theta[cut[i]:cut[i + 1]] for i in range(7))
    bits = (torch.arange(512, device="cuda")[:, None] >> torch.arange(9, device="cuda")) & 1
    h1 = torch.nn.functional.gelu(bits.double() @ W1.view(H, 9).T + b1)
    h2 = torch.nn.functional.gelu(h1 @ W2.view(H, H).T + b2)
    phi = h2 @ W3 + b3
    total = torch.zeros((), dtype=torch.float64, device="cuda")
    table = phi.detach()
    d_phi = torch.zeros(512, dtype=torch.float64, device="cuda")
    d_c = torch.zeros((), dtype=torch.float64, device="cuda")
    site = torch.arange(L, device="cuda")
    for at in range(0, n, 1 << 17):
        w, y = words[at:at + (1 << 17)], labels[at:at + (1 << 17)].double()
        x = (w[:, site // 64] >> (site % 64)) & 1
        pat = sum(torch.roll(x, 4 - k, dims=1) << k for k in range(9))
        z = 0.5 * table[pat].sum(dim=1) + c.detach()
        total += (torch.nn.functional.softplus(z, threshold=700.0) - y * z).sum()
        dz = (torch.sigmoid(z) - y) / n
        d_c += dz.sum()
        d_phi += torch.bincount(pat.reshape(-1), weights=(0.5 * dz)[:, None].expand(-1, L).reshape(-1), minlength=512)
    (grad,) = torch.autograd.grad((phi * d_phi).sum() + (c * d_c).sum(), theta)
    return dict(loss=np.float64(float(total) / n), grad=grad.cpu().numpy())
