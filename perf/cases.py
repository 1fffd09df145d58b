"""The calls whose speed is measured: what they stand for, their inputs and their exact values.

A tremor catalogue is a chain of hourly observations (none, or a location in
km). Fitting it evaluates the forward log likelihood, once per proposal of a
sampler; analysing the fit asks for posterior state probabilities, EM steps
and the most probable path. The inputs come from the package's own generator
(``synth``), seeded, with the value ranges of its docstring.

log L is a sum over up to 10^6 steps computed in FP32 or narrower arithmetic
and carried in a double; it is handed on as the float32 number a user keeps.
"""
import math

import numpy as np
import torch

from paper_2003_03508_gb300 import api, synth

# what a drawn case may cost: proposals x steps x K^3 of the largest listed
# case on the tensor cores, and a sixteenth of it on the CUDA cores
MOST_TC = 256 * (1 << 20) * 32 ** 3
MOST_FP32 = MOST_TC // 16


def listed():
    return [
        # the smallest real call: one parameter set on a short chain (K=4, T=10^4), as an optimiser loop makes it
        dict(name="loglik_k4_t1e4", kind="loglik", K=4, T=10_000, prec="fp32", quiet=False),
        # one parameter set at catalogue scale: 24 spatial states and a quiescent one, T=2^20
        dict(name="loglik_k25_t2p20", kind="loglik", K=25, T=1 << 20, prec="fp32", quiet=True),
        # the benchmark's workload: 256 proposals of a batched sampler on one long chain, TF32
        dict(name="batched_k32_t2p20_p256_tf32", kind="batched", K=32, T=1 << 20, props=256, segs=1, prec="tf32"),
        # a batch from host buffers on 64 uneven segments (a catalogue with gaps), FP32
        dict(name="host_k32_seg64_p64_fp32", kind="host", K=32, T=300_007, props=64, segs=64, prec="fp32"),
        # wide state spaces, for model-order sweeps
        dict(name="batched_k64_p64_tf32", kind="batched", K=64, T=300_001, props=64, segs=1, prec="tf32"),
        dict(name="batched_k80_p32_bf16", kind="batched", K=80, T=131_072, props=32, segs=3, prec="bf16"),
        # one iteration's work of 512 chains: states to parameters and prior, then their likelihood
        dict(name="chains_k16_c512_split", kind="chains", K=16, T=16_384, props=512, segs=1, prec="tf32_split"),
        # hours with a tremor are rare: the run-length option
        dict(name="runlen_k32_p64", kind="runlen", K=32, T=262_144, props=64, segs=1, prec="fp32"),
        # classifying a catalogue's hours by state (105,000 hourly points)
        dict(name="posterior_k25_t105000", kind="posterior", K=25, T=105_000, prec="fp32", quiet=True),
        # one EM iteration of a point estimate
        dict(name="em_k12_t200003", kind="em", K=12, T=200_003, prec="fp32", quiet=False),
        # the most probable path of a catalogue
        dict(name="viterbi_k25_t105000", kind="viterbi", K=25, T=105_000, prec="fp32", quiet=True),
        # gradient of the learned proposal's loss on a minibatch (K=16 chains: d=351)
        dict(name="mlp_d351_b512", kind="mlp", K=16, T=512, hidden=256),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["loglik", "loglik", "batched", "batched", "batched", "host", "chains", "runlen", "posterior",
                       "em", "viterbi", "mlp"])
    if kind == "mlp":
        return dict(kind=kind, K=rng.randint(4, 20), T=_log_int(rng, 32, 2048), hidden=rng.choice([64, 100, 256]))
    if kind in ("loglik", "posterior", "em", "viterbi"):
        T = _log_int(rng, 1000, {"loglik": 1 << 20, "posterior": 1 << 18, "em": 1 << 18, "viterbi": 1 << 17}[kind])
        return dict(kind=kind, K=_log_int(rng, 3, 48 if kind == "loglik" else 40), T=T, prec="fp32",
                    quiet=rng.random() < 0.5)
    if kind == "runlen":
        K, prec = _log_int(rng, 4, 48), "fp32"
    elif kind == "chains":
        K, prec = _log_int(rng, 3, 24), rng.choice(["fp32", "tf32_split"])
    elif kind == "host":
        K, prec = _log_int(rng, 4, 40), rng.choice(["fp32", "tf32_split"])
    else:
        prec = rng.choice(["fp32", "tf32", "tf32", "tf32_split", "bf16"])
        K = _log_int(rng, 24, 80) if prec in ("tf32", "bf16") else _log_int(rng, 3, 80)
    props = _log_int(rng, 4, 512)
    T = _log_int(rng, 2000, 1 << 20)
    most = MOST_FP32 if prec == "fp32" else MOST_TC
    cost = max(K, 16) ** 3
    T = max(2000, min(T, most // (props * cost)))
    props = max(1, min(props, most // (T * cost)))
    segs = rng.randint(2, 64) if rng.random() < 0.4 else 1
    return dict(kind=kind, K=K, T=T, props=props, segs=segs, prec=prec)


# ---------------------------------------------------------------- inputs

def _inputs(case, seed):
    """The case's inputs as numpy arrays."""
    K, T, kind = case["K"], case["T"], case["kind"]
    rng = np.random.default_rng(seed)
    if kind == "mlp":
        d, H = K * K + 6 * K - 1, case["hidden"]
        n = H * d + H + H * H + H + 2 * d * H + 2 * d
        w = np.concatenate([
            rng.uniform(-1, 1, H * d) * math.sqrt(6.0 / d), rng.normal(0, 0.01, H),
            rng.uniform(-1, 1, H * H) * math.sqrt(6.0 / H), rng.normal(0, 0.01, H),
            rng.uniform(-1, 1, 2 * d * H) * 0.3 * math.sqrt(6.0 / H), rng.normal(0, 0.01, 2 * d)]).astype(np.float32)
        assert w.size == n
        mean = rng.normal(0, 3.0, d).astype(np.float32)
        sd = np.exp(rng.normal(-2.0, 0.5, d)).astype(np.float32)
        theta = (mean + sd * rng.standard_normal((T, d))).astype(np.float32)
        y = (theta + 1.4 * sd * rng.standard_normal((T, d))).astype(np.float32)
        return dict(w=w, mean=mean, sd=sd, scale=(1.4 * sd).astype(np.float32), theta=theta, y=y)
    if kind in ("loglik", "posterior", "em", "viterbi"):
        gen = synth.quiescent_params(K, rng) if case["quiet"] else synth.random_params(K, rng)
        o = synth.sample_observations(gen, T, rng)
        prm = synth.perturb_params(gen, rng)
        return dict(params=prm, xy=o.xy, tremor=o.tremor, offsets=np.array([0, T], np.int64))
    d = synth.batched_inputs(K=K, T=T, n_prop=case["props"], seed=seed, n_seg=case["segs"], sparse=kind == "runlen")
    if kind == "chains":
        d["theta"] = np.stack([_theta(*(a[q].astype(np.float64) for a in d["params"].as_tuple()))
                               for q in range(case["props"])]).astype(np.float32)
    return d


def _theta(pi, P, p, mu, cov):
    """The sampler's coordinates of one parameter set (header: hmm_theta_dim)."""
    K = len(pi)
    off = ~np.eye(K, dtype=bool)
    sx, sy = np.sqrt(cov[:, 0]), np.sqrt(cov[:, 2])
    return np.concatenate([np.log(P / np.diag(P)[:, None])[off], np.log(pi[1:] / pi[0]), np.log(p / (1 - p)),
                           mu.reshape(-1), np.stack([np.log(sx), np.log(sy)], 1).reshape(-1),
                           np.arctanh(cov[:, 1] / (sx * sy))])


def _opts(case):
    return api.make_opts(precision=case["prec"], runlen_min=4 if case["kind"] == "runlen" else 0)


def prepare(case, seed):
    d = _inputs(case, seed)
    if case["kind"] == "mlp":
        t = {k: torch.from_numpy(v).cuda() for k, v in d.items()}
        net = api.MLP(t["theta"].shape[1], case["hidden"], seed=1)
        net.set_params(t["w"])
        net.set_scaling(t["mean"], t["sd"], t["scale"], 1.0)
        return dict(kind="mlp", net=net, theta=t["theta"], y=t["y"])
    s = dict(kind=case["kind"], ctx=api.Context(), opts=_opts(case), offsets=d["offsets"])
    if case["kind"] == "host":
        pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()  # noqa: E731
        s.update(params=[pin(a) for a in d["params"].as_tuple()], xy=pin(d["xy"]), tremor=pin(d["tremor"]))
        return s
    s.update(xy=torch.from_numpy(d["xy"]).cuda(), tremor=torch.from_numpy(d["tremor"]).cuda())
    if case["kind"] == "chains":
        s.update(K=case["K"], theta=torch.from_numpy(d["theta"]).cuda(), prior=api.make_prior(case["K"], alpha_P=0.5))
    else:
        s.update(params=api.to_device(d["params"]))
    return s


def run(s):
    kind = s["kind"]
    if kind == "mlp":
        loss, grads = s["net"].loss_grad(s["theta"], s["y"])
        return loss.float(), grads
    ctx, xy, tr, o = s["ctx"], s["xy"], s["tremor"], s["opts"]
    if kind == "loglik":
        return ctx.hmm_loglik(*s["params"], xy, tr, opts=o).float()
    if kind == "host":
        return ctx.hmm_loglik_batched_host(*s["params"], s["offsets"], xy, tr, opts=o).astype(np.float32)
    if kind == "chains":
        params, logprior = api.theta_to_params(s["theta"], s["K"], s["prior"])
        ll = ctx.hmm_loglik_batched(*params, s["offsets"], xy, tr, opts=o)
        return params, logprior, (ll + logprior).float()
    if kind == "posterior":
        gamma, ll = ctx.hmm_posterior(*s["params"], xy, tr, opts=o)
        return gamma, ll.float()
    if kind == "em":
        new, ll = ctx.hmm_em_step(*s["params"], xy, tr, opts=o)
        return new, ll.float()
    if kind == "viterbi":
        path, score, ll = ctx.hmm_viterbi(*s["params"], xy, tr, opts=o)
        return path, score.float(), ll.float()
    return ctx.hmm_loglik_batched(*s["params"], s["offsets"], xy, tr, opts=o).float()


def work(case):
    """The forward recursion needs 2 K^2 flops per proposal and step (and the emissions); smoothing three such
    recursions, Viterbi one. Bytes: parameters, observations and results once."""
    K, T, kind = case["K"], case["T"], case["kind"]
    if kind == "mlp":
        d, H = K * K + 6 * K - 1, case["hidden"]
        n = H * d + H * H + 2 * d * H
        return dict(bytes=4.0 * (2 * n + 2 * T * d), flops=2.0 * T * (3 * n - H * d))
    props = case.get("props", 1)
    passes = {"posterior": 2, "em": 3}.get(kind, 1)
    out = {"posterior": 4 * T * K, "em": 4 * K * K, "viterbi": 4 * T}.get(kind, 8 * props)
    return dict(bytes=9.0 * T + 4.0 * props * (K * K + 7 * K) + out,
                flops=float(props) * T * (2 * K * K * passes + 12 * K))


# ---------------------------------------------------------------- exact values, 64 bits

def _emissions(prm, x, y, tr):
    """log emission densities [props, n, K] of n observations."""
    _, _, p, mu, cov = prm
    sxx, sxy, syy = (cov[:, None, :, i] for i in range(3))
    det = sxx * syy - sxy * sxy
    dx, dy = x[None, :, None] - mu[:, None, :, 0], y[None, :, None] - mu[:, None, :, 1]
    q = (syy * dx * dx - 2 * sxy * dx * dy + sxx * dy * dy) / det
    hit = torch.log(p)[:, None] - math.log(2 * math.pi) - 0.5 * torch.log(det) - 0.5 * q
    return torch.where(tr[None, :, None], hit, torch.log1p(-p)[:, None])


class _Chain:
    """The scaled recursions in 64 bits over all pieces of the segments at once. A piece starts `warm` steps
    early from a flat vector (or at its segment's start from pi); where the vector it reaches at its own start
    differs from the one the piece before ends with, `warm` was too short and the pass is made again."""

    def __init__(self, d, dev):
        t64 = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev).double()  # noqa: E731
        prm = [t64(a) for a in d["params"].as_tuple()]
        self.prm = [a if a.dim() == n else a[None] for a, n in zip(prm, (2, 3, 2, 3, 3))]
        xy = t64(d["xy"])
        self.x, self.y = xy[:, 0].contiguous(), xy[:, 1].contiguous()
        self.tr = torch.from_numpy(d["tremor"]).to(dev) > 0
        self.offs, self.dev = [int(v) for v in d["offsets"]], dev
        self.K = self.prm[0].shape[1]

    def pieces(self, length):
        got = []
        for lo, hi in zip(self.offs[:-1], self.offs[1:]):
            n = max(1, -(-(hi - lo) // length))
            cut = [lo + (hi - lo) * i // n for i in range(n + 1)]
            got += [(lo, hi, a, b) for a, b in zip(cut[:-1], cut[1:]) if b > a]
        return got

    def sweep(self, length, warm, back=False, keep=None):
        """One pass: (log scale [props, pieces], largest mismatch at a piece's start). keep: [T, K] gets the
        normalised vectors of proposal 0."""
        pi, P = self.prm[0], self.prm[1]
        pc = torch.tensor(self.pieces(length), device=self.dev)
        lo, hi, a, b = pc.unbind(1)
        n = len(pc)
        first = torch.minimum(b + warm, hi) - 1 if back else torch.maximum(a - warm, lo)
        steps = int(((first - a) if back else (b - 1 - first)).max()) + 1
        M = P.transpose(1, 2).contiguous() if back else P
        v = torch.ones(pi.shape[0], n, self.K, device=self.dev, dtype=torch.float64)
        scale = torch.zeros(pi.shape[0], n, device=self.dev, dtype=torch.float64)
        start = v.clone()
        prev = torch.zeros_like(first)
        for k in range(steps):
            t = first - k if back else first + k
            live = (t >= a) if back else (t < b)
            tt = torch.where(live, t, a)
            if back:
                # v is b_t; entering the piece it is compared with what the piece after it ends with
                at = t == b - 1
                if k:
                    le = _emissions(self.prm, self.x[prev], self.y[prev], self.tr[prev])
                    w = torch.bmm(torch.exp(le - le.amax(2, keepdim=True)) * v, M)
                else:
                    w = v
                c = w.amax(2)
                w = w / c[..., None]
            else:
                at = t == a
                le = _emissions(self.prm, self.x[tt], self.y[tt], self.tr[tt])
                m = le.amax(2)
                head = (t == lo)[None, :, None]
                if k:
                    w = torch.bmm(v, M)
                else:
                    w = torch.full_like(v, 1.0 / self.K)
                w = torch.where(head, pi[:, None, :], w) * torch.exp(le - m[..., None])
                c = w.sum(2)
                w = w / c[..., None]
                scale += torch.where((live & (t >= a))[None], m + torch.log(c), torch.zeros_like(m))
            v = torch.where(live[None, :, None], w, v)
            prev = tt
            start = torch.where(at[None, :, None], v, start)
            if keep is not None:
                own = live & ((t < b) if back else (t >= a))
                keep[t[own]] = v[0][own]
        off = 0.0
        if n > 1:
            if back:  # the piece after ends one step later than this one starts: step its vector once
                t = a[1:]
                le = _emissions(self.prm, self.x[t], self.y[t], self.tr[t])
                nxt = torch.bmm(torch.exp(le - le.amax(2, keepdim=True)) * v[:, 1:], M)
                nxt, mine, same = nxt / nxt.amax(2, keepdim=True), start[:, :-1], hi[1:] == hi[:-1]
            else:
                t = a[1:]
                le = _emissions(self.prm, self.x[t], self.y[t], self.tr[t])
                nxt = torch.bmm(v[:, :-1], M) * torch.exp(le - le.amax(2, keepdim=True))
                nxt, mine, same = nxt / nxt.sum(2, keepdim=True), start[:, 1:], lo[1:] == lo[:-1]
            if bool(same.any()):
                off = float((nxt - mine)[:, same].abs().max())
        return scale, off

    def passes(self, back=False, keep=None):
        length, warm = max(512, self.offs[-1] // 256), 768
        while True:
            scale, off = self.sweep(length, warm, back, keep)
            if off < 1e-12 or warm > self.offs[-1]:
                return scale
            warm *= 3

    def loglik(self):
        return self.passes().sum(1)


def _prior64(theta, K, pr):
    """Parameters and log prior + log Jacobian of the sampler's coordinates."""
    n = theta.shape[0]
    at = [0, K * (K - 1), K - 1, K, 2 * K, 2 * K, K]
    c = np.cumsum(at)
    z, zp, w, mu, ls, r = (theta[:, c[i]:c[i + 1]] for i in range(6))
    full = torch.zeros(n, K, K, device=theta.device, dtype=torch.float64)
    full[:, ~torch.eye(K, dtype=torch.bool, device=theta.device)] = z
    lP = torch.log_softmax(full, 2)
    lpi = torch.log_softmax(torch.cat([torch.zeros_like(zp[:, :1]), zp], 1), 1)
    lp = pr.alpha_P * lP.sum((1, 2)) + pr.alpha_pi * lpi.sum(1)
    m = torch.where(torch.arange(K, device=theta.device) < K // 2, float(pr.p_mean_lo), float(pr.p_mean_hi)).double()
    p = torch.sigmoid(w)
    lp = lp + (m * m / pr.p_var * torch.nn.functional.logsigmoid(w) - m / pr.p_var * p
               + torch.nn.functional.logsigmoid(-w)).sum(1)
    xy = mu.reshape(n, K, 2)
    inside = ((xy[..., 0] >= pr.box[0]) & (xy[..., 0] <= pr.box[1]) & (xy[..., 1] >= pr.box[2])
              & (xy[..., 1] <= pr.box[3])).all(1)
    u, v = ls.reshape(n, K, 2).unbind(2)
    sx, sy, rho = torch.exp(u), torch.exp(v), torch.tanh(r)
    cov = torch.stack([sx * sx, rho * sx * sy, sy * sy], 2)
    det = cov[..., 0] * cov[..., 2] - cov[..., 1] ** 2
    lp = lp + (-0.5 * (pr.iw_df + 3.0) * torch.log(det) - 0.5 * (cov[..., 0] + cov[..., 2]) / det + math.log(4.0)
               + torch.log1p(-rho * rho) + 3.0 * u + 3.0 * v).sum(1)
    lp = torch.where(inside, lp, torch.full_like(lp, -math.inf))
    return (torch.exp(lpi), torch.exp(lP), p, xy, cov), lp


def _mlp64(d, H, dev):
    t = {k: torch.from_numpy(v).to(dev).double() for k, v in d.items()}
    n = t["theta"].shape[1]
    w = t["w"].requires_grad_(True)
    cut = np.cumsum([0, H * n, H, H * H, H, 2 * n * H, 2 * n])
    W1, b1, W2, b2, W3, b3 = (w[cut[i]:cut[i + 1]] for i in range(6))
    h = torch.relu((t["theta"] - t["mean"]) / t["sd"] @ W1.view(H, n).T + b1)
    out = torch.relu(h @ W2.view(H, H).T + b2) @ W3.view(2 * n, H).T + b3
    fs = out[:, n:].clamp(-6.0, 3.0)
    res = (t["y"] - t["theta"]) / t["scale"] - out[:, :n]
    loss = (0.5 * res * res * torch.exp(-2 * fs) + fs).sum(1).mean()
    loss.backward()
    return loss.detach().reshape(1), w.grad


def _viterbi64(d):
    """The best path's log joint probability (numpy, one step after another)."""
    ch = _Chain(d, "cpu")
    lP = torch.log(ch.prm[1][0]).numpy()
    T = len(d["tremor"])
    le = torch.cat([_emissions(ch.prm, ch.x[i:i + 65536], ch.y[i:i + 65536], ch.tr[i:i + 65536])[0]
                    for i in range(0, T, 65536)]).numpy()
    v = torch.log(ch.prm[0][0]).numpy() + le[0]
    lPT = np.ascontiguousarray(lP.T)
    for t in range(1, T):
        v = (lPT + v).max(1) + le[t]
    return np.array([v.max()])


def exact(case, seed):
    kind, d = case["kind"], _inputs(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "mlp":
        return _mlp64(d, case["hidden"], dev)
    if kind == "chains":
        theta = torch.from_numpy(d["theta"]).to(dev).double()
        params, lp = _prior64(theta, case["K"], api.make_prior(case["K"], alpha_P=0.5))
        # the likelihood is evaluated at the parameters rounded to float32, as the call takes them
        ch = _Chain(d, dev)
        ch.prm = [a.float().double() for a in params]
        return params, lp, lp + ch.loglik()
    ch = _Chain(d, dev)
    if kind == "posterior" or kind == "em":
        T, K = len(d["tremor"]), case["K"]
        f = torch.zeros(T, K, device=dev, dtype=torch.float64)
        b = torch.zeros_like(f)
        ll = ch.passes(keep=f).sum(1)
        ch.passes(back=True, keep=b)
        g = f * b
        g = g / g.sum(1, keepdim=True)
        if kind == "posterior":
            return g, ll
        le = _emissions(ch.prm, ch.x, ch.y, ch.tr)[0]
        P = ch.prm[1][0]
        u = torch.exp(le[1:] - le[1:].amax(1, keepdim=True)) * b[1:]
        Z = ((f[:-1] @ P) * u).sum(1, keepdim=True)
        N = P * (f[:-1].T @ (u / Z))
        gr = g * ch.tr[:, None]
        r = gr.sum(0)
        mu = torch.stack([(gr * ch.x[:, None]).sum(0), (gr * ch.y[:, None]).sum(0)], 1) / r[:, None]
        dx, dy = ch.x[:, None] - mu[:, 0], ch.y[:, None] - mu[:, 1]
        cov = torch.stack([(gr * dx * dx).sum(0), (gr * dx * dy).sum(0), (gr * dy * dy).sum(0)], 1) / r[:, None]
        return (g[0], N / N.sum(1, keepdim=True), r / g.sum(0), mu, cov), ll
    if kind == "viterbi":
        return None, _viterbi64(d), ch.loglik()
    return ch.loglik()
