"""Performance cases: the work a user of this library has it do, through its
public entry points, with inputs drawn from a seed.

  travel_time   the travel-time networks alone: torch autograd over a list of
                (source, station) pairs, or the raw device-pointer call
  gradient      one full-batch gradient of the log posterior
  chain         a stretch of sampler steps, then the state read back
  batch         the same for several catalogs x chains in one context
  stage1        Adam steps on the L1 objective, then the two observation filters
  summary       posterior summaries of the stored samples

`exact` restates each of them in 64-bit torch (the summaries excepted: their
input is the chain itself)."""
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_2508_12117_gb300 import binding, synth
from paper_2508_12117_gb300.autograd import travel_time

PRECISION = {"fp32": binding.FP32, "bf16": binding.BF16, "fp8": binding.FP8}
UPDATE = {"sgld": binding.UPDATE_SGLD, "psgld": binding.UPDATE_PSGLD, "adam": binding.UPDATE_ADAM}
# step sizes: plain SGLD takes the workload's own; km per step for the others
EPS = {"psgld": 2e-5, "adam": 1e-3}
ALL = 0                                    # batch of 0: every observation in every step


def listed():
    return [
        # locating one event interactively: its travel times and their gradient at the network's stations
        dict(name="travel-time-one-event", kind="travel_time", route="autograd", precision="fp32", hidden=64, pairs=47),
        # a misfit over a small catalog in a user's own torch loop, in the default precision
        dict(name="travel-time-fp32", kind="travel_time", route="autograd", precision="fp32", hidden=128, pairs=250_007),
        # the travel times of one minibatch of the million-event catalog
        dict(name="travel-time-bf16", kind="travel_time", route="pairs", precision="bf16", hidden=256, pairs=1_570_001),
        # the same network for a smaller catalog in the narrowest arithmetic
        dict(name="travel-time-fp8", kind="travel_time", route="pairs", precision="fp8", hidden=256, pairs=400_003),
        # the smallest catalog: a cluster of 200 events in a homogeneous medium, one gradient
        dict(name="gradient-small", kind="gradient", recipe=1, events=200, precision="fp32", hidden=0),
        # a regional catalog at full batch: 10,000 events, 2 million differential times
        dict(name="gradient-regional", kind="gradient", recipe=2, events=10_000, precision="fp32", hidden=128),
        # sampling the small cluster at full batch
        dict(name="chain-small", kind="chain", recipe=1, events=200, precision="fp32", hidden=0, update="sgld",
             minibatch=ALL, steps=16),
        # minibatch SGLD with the tensor-core network, density of the million-event catalog
        dict(name="chain-bf16", kind="chain", recipe=4, events=20_000, precision="bf16", hidden=256, update="sgld",
             minibatch=1 << 18, steps=8),
        # stage-2 warm-up (pSGLD with the noise off) in the default precision on a dense catalog
        dict(name="chain-fp32-psgld", kind="chain", recipe=3, events=4_000, precision="fp32", hidden=128,
             update="psgld", minibatch=1 << 16, steps=4),
        # several uneven catalogs, some smaller than the minibatch, with two chains each
        dict(name="batch-chains", kind="batch", catalogs=4, chains=2, events=5_000, precision="bf16", hidden=128,
             minibatch=1 << 16, steps=2),
        # stage 1 of the workflow: a few L1 + Adam steps, outlier and linearisation filters
        dict(name="stage1-filters", kind="stage1", recipe=3, events=2_000, precision="fp32", hidden=64,
             minibatch=1 << 17, steps=4),
        # medians, credible intervals and effective sample sizes of a finished chain
        dict(name="posterior-summary", kind="summary", recipe=4, events=5_000, samples=400),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["travel_time", "travel_time", "travel_time", "gradient", "chain", "chain", "batch",
                       "stage1", "summary"])
    if kind == "travel_time":
        precision = rng.choice(["fp32", "bf16", "fp8"])
        hidden = rng.choice({"fp32": [32, 64, 128, 256], "bf16": [64, 128, 256], "fp8": [128, 256]}[precision])
        most = 250_000 * 128 * 128 // (hidden * hidden) if precision == "fp32" else 1_500_000
        return dict(kind=kind, route=rng.choice(["autograd", "pairs"]), precision=precision, hidden=hidden,
                    pairs=_spread(rng, 30, min(most, 1_500_000)))
    if kind == "gradient":
        if rng.random() < 0.3:
            return dict(kind=kind, recipe=1, events=_spread(rng, 60, 600), precision="fp32", hidden=0)
        return dict(kind=kind, recipe=2, events=_spread(rng, 300, 9_000), precision=rng.choice(["fp32", "bf16"]),
                    hidden=rng.choice([64, 128]))
    if kind == "chain":
        if rng.random() < 0.2:
            return dict(kind=kind, recipe=1, events=_spread(rng, 60, 400), precision="fp32", hidden=0,
                        update=rng.choice(["sgld", "psgld"]), minibatch=ALL, steps=rng.randint(4, 16))
        recipe = rng.choice([3, 4])
        precision = rng.choice(["fp32", "bf16", "bf16"])
        events = _spread(rng, 1_000, 20_000 if recipe == 4 else 5_000)
        blocks = events * (200 if recipe == 4 else 500) // 4096
        # a minibatch is a small part of its catalog
        part = max(2, int(round(blocks * math.exp(rng.uniform(math.log(0.01), math.log(0.1))))))
        return dict(kind=kind, recipe=recipe, events=events, precision=precision,
                    hidden=128 if precision == "fp32" else rng.choice([128, 256]),
                    update=rng.choice(["sgld", "psgld"]), minibatch=4096 * part, steps=rng.randint(1, 6))
    if kind == "batch":
        return dict(kind=kind, catalogs=rng.randint(2, 4), chains=rng.randint(1, 2), events=_spread(rng, 800, 4_500),
                    precision=rng.choice(["fp32", "bf16"]), hidden=rng.choice([64, 128]),
                    minibatch=4096 * _spread(rng, 4, 16), steps=rng.randint(1, 2))
    if kind == "stage1":
        return dict(kind=kind, recipe=3, events=_spread(rng, 300, 2_000), precision="fp32",
                    hidden=rng.choice([32, 64]), minibatch=4096 * _spread(rng, 4, 48), steps=rng.randint(1, 6))
    return dict(kind=kind, recipe=4, events=_spread(rng, 300, 5_000), samples=rng.randint(50, 400))


# ------------------------------------------------------------------ inputs
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _network(case, seed):
    """A network whose learned part is a good share of the travel time."""
    return synth.strong_mlp_weights(case["hidden"], seed)


def _pairs(case, seed):
    """Events of a 60 x 60 km region at 2 to 16 km depth, surface stations, and
    the incoming gradient of a misfit."""
    g = torch.Generator(device=_device()).manual_seed(seed)
    u = torch.rand(case["pairs"], 7, device=_device(), generator=g)
    src = torch.stack([60 * u[:, 0], 60 * u[:, 1], 2 + 14 * u[:, 2]], 1)
    rcv = torch.stack([80 * u[:, 3] - 10, 80 * u[:, 4] - 10, 0 * u[:, 5]], 1)
    return src, rcv, u[:, 6] - 0.5


@functools.lru_cache(maxsize=8)
def _layout(recipe, events, forward, hidden):
    """Events, stations and pairs of one of the repository's recipes at another size."""
    s = synth.scaled_spec(recipe, events)
    s.forward, s.hidden = forward, hidden
    return synth.make_catalog(s)


def _catalog(case, seed, events=None):
    """A catalog whose observed times and network come from the seed, and the
    state to start from: a little off the catalog, as in a chain that is resumed."""
    H = case.get("hidden", 0)
    cat = _layout(case.get("recipe", 4), events or case["events"], "mlp" if H else "homogeneous", H)
    rng = np.random.default_rng(seed)
    theta = cat.init_xyzt + rng.normal(0.0, 1.0, (cat.M, 4)) * [0.05, 0.05, 0.05, 0.01]
    theta[:, 2] = np.maximum(theta[:, 2], 0.1)
    return dataclasses.replace(cat, dt=cat.dt + rng.normal(0.0, 0.002, cat.N),
                               net=synth.mlp_weights(H, seed) if H else None), theta


def _batch_events(case):
    """Catalogs of a batch: the largest first, each a half of the one before."""
    return [max(200, case["events"] >> c) for c in range(case["catalogs"])]


def _eps(case, cat):
    return EPS.get(case.get("update", "adam" if case["kind"] == "stage1" else "sgld"), cat.spec.hyper.eps)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "next": 1000 * seed + 1}
    if kind == "travel_time":
        n = case["pairs"]
        s["net"] = binding.NetDevice(binding.Net(binding.TT_MLP, mlp=_network(case, seed)),
                                     PRECISION[case["precision"]])
        src, rcv, s["gT"] = _pairs(case, seed)
        if case["route"] == "autograd":
            s["src"], s["rcv"] = src.requires_grad_(True), rcv
        else:
            pad = torch.zeros(n, 1, device=src.device)
            s["src"], s["rcv"] = torch.cat([src, pad], 1).contiguous(), torch.cat([rcv, pad], 1).contiguous()
            s["T"] = torch.empty(n, device=src.device)
            s["J"] = torch.empty(n, 4, device=src.device)
        return s
    precision = PRECISION[case.get("precision", "fp32")]
    if kind == "batch":
        cats, thetas = zip(*(_catalog(case, 10 * seed + c, m) for c, m in enumerate(_batch_events(case))))
        s["eps"] = _eps(case, cats[0])
        s["ctx"] = binding.Context.batch(
            cats, case["chains"], binding.Net(binding.TT_MLP, mlp=cats[0].net),
            binding.config_for_catalog(cats[0], batch_n=case["minibatch"], precision=precision))
        s["ctx"].spider_set_state(np.concatenate([t for t in thetas for _ in range(case["chains"])]), 0)
        return s
    cat, theta = _catalog(case, seed)
    s["eps"] = _eps(case, cat)
    over = dict(precision=precision, batch_n=case.get("minibatch", ALL))
    if kind == "chain":
        over["update"] = UPDATE[case["update"]]
        if case["update"] == "psgld":
            over["noise_scale"] = 0.0      # as in the warm-up, where this update is used
    elif kind == "stage1":
        over.update(update=binding.UPDATE_ADAM, loss=binding.LOSS_L1)
    elif kind == "summary":
        over.update(batch_n=1 << 14, sample_cap=case["samples"])
    s["ctx"] = binding.Context.from_catalog(cat, **over)
    s["ctx"].spider_set_state(theta, 0)
    if kind == "summary":
        s["truth"] = cat.true_xyzt
        for t in range(case["samples"]):
            s["ctx"].spider_sgld_step(s["eps"], s["next"] + t)
        s["ctx"].spider_sync()
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "travel_time":
        if case["route"] == "autograd":
            T = travel_time(s["src"], s["rcv"], s["net"])
            (g,) = torch.autograd.grad(T, s["src"], s["gT"])
            return {"T": T.detach(), "grad": g}
        # a caller that needs T to single precision leaves out its low part
        s["net"].spider_tt_pairs(case["pairs"], s["src"].data_ptr(), s["rcv"].data_ptr(), s["T"].data_ptr(), 0,
                                 s["J"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"T": s["T"], "J": s["J"]}
    ctx = s["ctx"]
    if kind == "gradient":
        g, logpost = ctx.spider_grad_logpost(0)
        # a sum over single-precision observations: reported as one
        return {"grad": g, "logpost": np.float32(logpost)}
    if kind == "summary":
        return ctx.spider_uq(s["truth"])
    for _ in range(case["steps"]):
        ctx.spider_sgld_step(s["eps"], s["next"])
        s["next"] += 1
    theta, _ = ctx.spider_get_state()
    if kind == "stage1":
        keep, median, mad = ctx.spider_outlier_mask(4.0)
        return {"theta": theta, "keep": keep, "median": median, "mad": mad,
                "linear": ctx.spider_linearisation_mask(0.05)}
    return {"theta": theta}


# ------------------------------------------------------------------ what a pass cannot do without
def _network_flops(H):
    """Forward and reverse products of one pair (the closed form in a homogeneous medium)."""
    return 12.0 * H * H + 20.0 * H if H else 60.0


def work(case):
    kind, H = case["kind"], case.get("hidden", 0)
    if kind == "travel_time":
        n = case["pairs"]
        return {"bytes": 44.0 * n if case["route"] == "autograd" else 52.0 * n, "flops": n * _network_flops(H)}
    if kind == "summary":
        n = 4.0 * case["events"] * case["samples"]
        return {"bytes": 4.0 * n + 5 * 32.0 * case["events"], "flops": n * (math.log2(case["samples"]) ** 2 + 8)}
    if kind == "batch":
        sizes = [(m, 200 * m) for m in _batch_events(case) for _ in range(case["chains"])]
    else:
        per = {1: 46, 2: 200, 3: 500, 4: 200}[case["recipe"]]
        sizes = [(case["events"], per * case["events"])]
    total = {"bytes": 0.0, "flops": 0.0}

    def evaluation(events, obs, pairs):
        # observation: two local pair indices, time, weight; pair: event, station; event: state in, result out
        total["bytes"] += 12.0 * obs + 8.0 * pairs + 48.0 * events
        total["flops"] += pairs * _network_flops(H) + 20.0 * obs

    for m, n in sizes:
        stations = {1: 10, 2: 10, 3: 20}.get(case.get("recipe"), 20)
        mb = case.get("minibatch", ALL)
        part = n if not mb else min(n, mb)
        pairs = min(1.1 * m * stations, 0.37 * part if part < n else 1.1 * m * stations)
        for _ in range(case.get("steps", 1)):
            evaluation(m, part, pairs)
        if kind == "stage1":
            evaluation(m, n, 1.1 * m * stations)
            total["bytes"] += 14.0 * n
        total["bytes"] += 32.0 * m
    return total


# ------------------------------------------------------------------ the same in 64 bits
def _mlp(x, net):
    """T, dT/dx of T = |x - s| tau(x, s) for rows [source, station]."""
    W = [torch.as_tensor(w, device=x.device).double() for w in net["W"]]
    b = [torch.as_tensor(v, device=x.device).double() for v in net["b"]]
    T, J = [], []
    for rows in x.split(1 << 18):
        h, ds = rows, []
        for l in range(4):
            z = h @ W[l].T + b[l]
            sg = torch.sigmoid(z)
            h = z * sg
            ds.append(sg * (1 + z * (1 - sg)))
        tau = (h @ W[4].T + b[4])[:, 0]
        d = W[4] * ds[3]
        for l in (3, 2, 1):
            d = (d @ W[l]) * ds[l - 1]
        diff = rows[:, :3] - rows[:, 3:]
        r = diff.norm(dim=1)
        T.append(r * tau)
        J.append((tau / r)[:, None] * diff + r[:, None] * (d @ W[0])[:, :3])
    return torch.cat(T), torch.cat(J)


def _philox(counter, seed):
    """Philox4x32-10 (Salmon et al. 2011) of the rows of counter, 64-bit key."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.array(a, dtype=np.uint64) for a in counter]
    k = [np.uint64(seed & 0xFFFFFFFF), np.uint64((seed >> 32) & 0xFFFFFFFF)]
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        s = np.uint64(32)
        c = [(p1 >> s) ^ c[1] ^ k[0], p1 & m32, (p0 >> s) ^ c[3] ^ k[1], p0 & m32]
        k = [(k[0] + np.uint64(0x9E3779B9)) & m32, (k[1] + np.uint64(0xBB67AE85)) & m32]
    return c


def _noise(m, seed, chain, catalog):
    one = np.ones(m, np.uint64)
    w = _philox([np.arange(m), one * np.uint64(chain), one * np.uint64(catalog), one * np.uint64(0x4E4F4953)], seed)
    u = [((a >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0 ** -23 for a in w]
    out = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        rad = np.sqrt(-2 * np.log(a))
        out += [rad * np.cos(2 * math.pi * b), rad * np.sin(2 * math.pi * b)]
    return np.stack(out, 1)


def _selected(n_obs, block, batch, seed):
    """Observations of a minibatch: whole blocks, drawn by a keyed Feistel permutation."""
    nb = -(-n_obs // block)
    want = min(nb, -(-batch // block)) if batch else nb
    if want == nb:
        return np.arange(n_obs)
    bits = max(2, (nb - 1).bit_length())
    h = (bits + 1) // 2
    parts = []
    for x in range(want):
        while True:
            left, right = x >> h, x & ((1 << h) - 1)
            for rnd in range(4):
                f = int(_philox([[right], [rnd], [0], [0x46454953]], seed)[0][0]) & ((1 << h) - 1)
                left, right = right, left ^ f
            x = (left << h) | right
            if x < nb:
                break
        parts.append(np.arange(x * block, min(n_obs, (x + 1) * block)))
    return np.sort(np.concatenate(parts))


class _Posterior:
    def __init__(self, cat, net):
        dev = _device()

        def put(a):
            return torch.as_tensor(np.asarray(a), device=dev)

        self.h, self.net = cat.spec.hyper, net
        self.th0, self.sta, self.dt = put(cat.init_xyzt), put(cat.stations), put(cat.dt)
        self.i, self.j, self.k = put(cat.i).long(), put(cat.j).long(), put(cat.k).long()
        d = (self.th0[self.i, :3] - self.th0[self.j, :3]).norm(dim=1)
        w = (d / self.h.ell) ** self.h.p + self.h.eps_w
        S = len(self.sta)
        mean = torch.bincount(self.k, w, S) / torch.bincount(self.k, minlength=S).clamp(min=1)
        self.w = w / mean[self.k]

    def times(self, theta, sel):
        i, j, k = self.i[sel], self.j[sel], self.k[sel]
        S = len(self.sta)
        node, where = torch.unique(torch.cat([i * S + k, j * S + k]), return_inverse=True)
        x = torch.cat([theta[node // S, :3], self.sta[node % S]], 1)
        if self.net is not None:
            T, J = _mlp(x, self.net)
        else:
            d = x[:, :3] - x[:, 3:]
            r = d.norm(dim=1)
            T, J = r / 6.0, d / (6.0 * r)[:, None]
        return i, j, where[:len(i)], where[len(i):], node // S, T, J

    def gradient(self, theta, sel=None, l1=False):
        """Gradient and value of the log posterior on the observations sel."""
        h, n = self.h, len(self.dt)
        sel = torch.arange(n, device=theta.device) if sel is None else sel
        i, j, a, b, ev, T, J = self.times(theta, sel)
        r = self.dt[sel] - ((T[a] + theta[i, 3]) - (T[b] + theta[j, 3]))
        if l1:
            q, quad = r.sign(), 2 * r.abs().sum()
        else:
            q = (r - self._shared(r, a, b, self.w[sel], len(T))) / h.sigma ** 2
            quad = (r * q).sum()
        node = torch.zeros_like(T).index_add_(0, a, q).index_add_(0, b, -q) * (n / len(sel))
        g = torch.zeros_like(theta)
        g.index_add_(0, ev, torch.cat([node[:, None] * J, node[:, None]], 1))
        se, sc = (torch.tensor(v, device=theta.device, dtype=torch.float64) for v in (h.sig_e, h.sig_c))
        dev = theta - self.th0
        c = dev.mean(0)
        g -= dev / se ** 2 + c / (len(theta) * sc ** 2)
        return g, -0.5 * (quad * (n / len(sel)) + ((dev / se) ** 2).sum() + ((c / sc) ** 2).sum())

    def _shared(self, r, a, b, w, nodes):
        """The part of r the shared-event term explains: B z with
        (sigma^2 / kappa^2 I + B^T B) z = B^T r, by conjugate gradients."""
        lam, sw = (self.h.sigma / self.h.kappa) ** 2, w.sqrt()

        def down(e):
            return torch.zeros(nodes, device=r.device, dtype=torch.float64).index_add_(0, a, e).index_add_(0, b, -e)

        diag = lam + torch.bincount(a, w, nodes) + torch.bincount(b, w, nodes)
        rhs = down(sw * r)
        z, res = torch.zeros_like(rhs), rhs.clone()
        y = res / diag
        p, rz = y.clone(), (res * y).sum()
        for it in range(6000):
            Ap = lam * p + down(w * (p[a] - p[b]))
            alpha = rz / (p * Ap).sum()
            z += alpha * p
            res -= alpha * Ap
            if it % 25 == 0 and float(res.norm()) <= 1e-13 * float(rhs.norm()):
                break
            y = res / diag
            new = (res * y).sum()
            p, rz = y + (new / rz) * p, new
        return sw * (z[a] - z[b])


def _walk(case, post, theta, seed, eps, sub=0, chain=0, catalog=0, update="sgld", l1=False):
    """The state after the steps of one pass."""
    theta, h = torch.as_tensor(theta, device=post.dt.device), post.h
    m, v = torch.zeros_like(theta), torch.zeros_like(theta)
    for t in range(case["steps"]):
        key = 1000 * seed + 1 + t
        sel = _selected(len(post.dt), h.block_obs, case["minibatch"],
                        key ^ ((0x9E3779B97F4A7C15 * sub) & 0xFFFFFFFFFFFFFFFF))
        g, _ = post.gradient(theta, torch.as_tensor(sel, device=theta.device), l1)
        v = 0.99 * v + 0.01 * g * g
        if update == "adam":
            m = 0.9 * m + 0.1 * g
            theta = theta + eps * (m / (1 - 0.9 ** (t + 1))) / ((v / (1 - 0.99 ** (t + 1))).sqrt() + 1e-5)
            continue
        if update == "psgld":              # noise off
            theta = theta + eps * g / (v.sqrt() + 1e-5)
            continue
        eta = torch.as_tensor(_noise(len(theta), key, chain, catalog), device=theta.device)
        theta = theta + eps * g + math.sqrt(2 * eps) * eta
    return theta


def exact(case, seed):
    kind = case["kind"]
    if kind == "summary":
        return None                        # computed from the chain, which only the library has
    if kind == "travel_time":
        src, rcv, gT = _pairs(case, seed)
        T, J = _mlp(torch.cat([src, rcv], 1).double(), _network(case, seed))
        if case["route"] == "autograd":
            return {"T": T, "grad": gT.double()[:, None] * J}
        return {"T": T, "J": torch.cat([J, torch.zeros_like(T)[:, None]], 1)}
    if kind == "batch":
        out, first = [], None
        for c, m in enumerate(_batch_events(case)):
            cat, theta = _catalog(case, 10 * seed + c, m)
            first = first or cat
            post = _Posterior(cat, first.net)
            out += [_walk(case, post, theta, seed, _eps(case, first), len(out) + h, h, c) for h in range(case["chains"])]
        return {"theta": torch.cat(out)}
    cat, theta = _catalog(case, seed)
    post = _Posterior(cat, cat.net)
    if kind == "gradient":
        g, logpost = post.gradient(torch.as_tensor(theta, device=post.dt.device))
        return {"grad": g, "logpost": float(logpost)}
    if kind == "chain":
        return {"theta": _walk(case, post, theta, seed, _eps(case, cat), update=case["update"])}
    theta = _walk(case, post, theta, seed, _eps(case, cat), update="adam", l1=True)
    every = torch.arange(len(post.dt), device=theta.device)
    i, j, a, b, _, T, _ = post.times(theta, every)
    r = (post.dt - ((T[a] + theta[i, 3]) - (T[b] + theta[j, 3]))).cpu().numpy()
    median = np.median(r)
    return {"theta": theta, "keep": None, "median": np.array([median]), "mad": np.array([np.median(abs(r - median))]),
            "linear": None}
