"""The work this library is measured on: one training iteration of each of its
workloads, and the calls that programs make around it (evaluation batches, log
pi with its gradient, the gradient for an optimiser of one's own).

A case is a dict:
  call       step      one VQMC.step: samples, energies, gradient, Adam
             sr        one VQMC.sr_step: the same with stochastic reconfiguration
             batch     one graph launch of a VQMCBatch: a step of many instances
             evaluate  an evaluation batch: VQMC.sample and VQMC.local_energy
             logprob   LogProb forward and backward, as torch.autograd runs it
             grad      sample, local_energy and grad: the score-function gradient
  graph      the Hamiltonian: "regular" (3-regular graph, weights +-1), "er"
             (random graph of average degree 8, weights 1..10), "unit" (random
             graph of density 1/2, unit weights), "sk" (dense spin glass), "tim"
             (dense couplings, fields and a transverse field)
  n, h, B    spins, hidden units, samples (batch: the largest n, the number of
             instances in place of h, samples of each)
  act, prec  "relu" / "sigmoid", "fp32" / "bf16"

The outputs are the tensors a program reads: samples, log pi, energies and
gradients, and for a training step the updated parameters.
"""
import math

import numpy as np
import torch

from paper_2106_13308_gb300 import inputs
from paper_2106_13308_gb300.vqmc import LogProb, VQMC, VQMCBatch

LR, BETA1, BETA2, EPS = 1e-2, 0.9, 0.999, 1e-8
SR_LR, SR_LAMBDA = 0.1, 1e-3
DEGREE = 6.0  # average degree of a batch's graphs
EVAL_COUNTER = 1 << 62  # evaluation batches draw from Philox counters above it


def _case(name, call, graph, n, h, B, act="relu", prec="bf16"):
    return {"name": name, "call": call, "graph": graph, "n": n, "h": h, "B": B, "act": act, "prec": prec}


def listed():
    return [
        # a toy problem at full precision, with sigmoid units: launches and latency
        _case("step_er20_fp32", "step", "unit", 20, 40, 1024, act="sigmoid", prec="fp32"),
        # the ordinary Max-Cut problem: sparse graph, as many hidden units as spins
        _case("step_regular1000", "step", "regular", 1000, 1000, 4096),
        # the benchmark: the large Max-Cut problem
        _case("step_er10000", "step", "er", 10000, 2000, 2048),
        # the benchmark's plain full-precision arm
        _case("step_er10000_fp32", "step", "er", 10000, 2000, 2048, prec="fp32"),
        # dense couplings with a large batch
        _case("step_sk2000", "step", "sk", 2000, 2000, 8192),
        # transverse field: n + 1 rows of log pi for each sample's energy
        _case("step_tim500", "step", "tim", 500, 193, 1024),
        # the paper's second optimiser, on the same problem; full precision only
        _case("sr_tim500", "sr", "tim", 500, 193, 1024, prec="fp32"),
        # uneven instances trained together, hidden units = spins, 512 samples each
        _case("batch_16", "batch", "er", 5000, 16, 512),
        # the evaluation batch between training steps, on both kinds of model
        _case("evaluate_er10000", "evaluate", "er", 10000, 2000, 1024),
        _case("evaluate_regular1000", "evaluate", "regular", 1000, 1000, 1024),
        # log pi of given configurations in an autograd program, odd sizes
        _case("logprob_1537", "logprob", "er", 1537, 771, 1023),
        # the gradient for an optimiser of one's own, full precision, odd sizes
        _case("grad_301_fp32", "grad", "er", 301, 203, 777, prec="fp32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "step", "tim", "sr", "batch", "evaluate", "evaluate", "logprob", "grad"])
    if call == "batch":
        return {"call": "batch", "graph": "er", "n": _log(rng, 300, 3000), "h": rng.randint(2, 12),
                "B": _log(rng, 64, 512), "act": "relu", "prec": "bf16"}
    act = rng.choice(["relu", "relu", "relu", "sigmoid"])
    if call in ("tim", "sr"):
        n = _log(rng, 20, 500)
        return {"call": "step" if call == "tim" else "sr", "graph": "tim", "n": n,
                "h": max(2, int(5 * math.log(n) ** 2)), "B": _log(rng, 64, 1024), "act": act,
                "prec": "bf16" if call == "tim" else "fp32"}
    prec = rng.choice(["bf16", "bf16", "fp32"])
    n = _log(rng, 20, 10000)
    h = min(2000, max(8, int(n * rng.choice([rng.uniform(0.15, 0.5), rng.uniform(0.5, 1.2), 1.0, 2.0]))))
    top = 1.5e10 if prec == "bf16" else 8e9
    B = max(16, min(_log(rng, 64, 8192), int(top / (float(n) * h))))
    graph = rng.choice(["er", "regular"] if n > 3000 else ["er", "regular", "sk"])
    if graph == "regular":
        n += n % 2  # a 3-regular graph has an even number of vertices
    if graph == "er" and n < 64:
        graph = "unit"
    return {"call": call, "graph": graph, "n": n, "h": h, "B": B, "act": act, "prec": prec}


# ------------------------------------------------------------------ inputs

def _instance(graph, n, seed):
    if graph == "sk":
        return inputs.sk(n, seed)
    if graph == "tim":
        return inputs.tim(n, seed)
    if graph == "regular":
        e = inputs.random_regular(n, 3, seed)
        return inputs.to_csr(n, e, inputs.pm1_weights(len(e), seed + 1))
    if graph == "unit":
        e = inputs.erdos_renyi(n, 0.5, seed)
        return inputs.to_csr(n, e, np.ones(len(e), dtype=np.int32))
    e = inputs.erdos_renyi(n, 8.0 / (n - 1), seed)
    return inputs.to_csr(n, e, inputs.int_weights(len(e), 1, 10, seed + 1))


def _theta(case, n, h, seed):
    """Parameters on the GPU: where training starts (N(0, 0.01), no biases) for
    a training step, else conditionals spread over (0, 1) as in a trained model."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    t = torch.randn(2 * n * h + h + n, generator=g, device="cuda")
    nh = n * h
    if case["call"] in ("step", "sr", "batch"):
        t *= 0.01
        t[nh: nh + h] = 0.0
        t[2 * nh + h:] = 0.0
    else:
        t[:nh] *= 1.5 / math.sqrt(n)
        t[nh: nh + h] *= 0.5
        t[nh + h: 2 * nh + h] *= 3.0 / math.sqrt(h)
        t[2 * nh + h:] *= 0.5
    return t


def _past_gradient(d, seed):
    """The gradient of an earlier iteration: gives Adam its moments."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    x = torch.rand(d, generator=g, device="cuda") * 2.0 - 1.0
    return x + torch.sign(x)


def _model(case, n, h, B, inst, seed):
    m = VQMC(n, h, B, inst, act=case["act"], precision=case["prec"], lr=LR, beta1=BETA1, beta2=BETA2, eps=EPS,
             seed=seed)
    m.set_params(_theta(case, n, h, seed))
    return m


def _parameters(model, owner):
    """The model's parameters as a tensor that keeps their owner alive."""
    t = model.params_view()
    t.owner = owner
    return t


def _members(case):
    """The sizes of a batch's instances: they belong to the case."""
    return inputs.batched_configs(case["h"], n_lo=100, n_hi=case["n"], avg_deg=DEGREE)


def prepare(case, seed):
    n, h, B = case["n"], case["h"], case["B"]
    if case["call"] == "batch":
        problems = []
        for q, c in enumerate(_members(case)):
            e = inputs.erdos_renyi(c["n"], c["p"], seed + 1000 * q)
            problems.append(dict(n=c["n"], h=c["h"], max_batch=B, act=case["act"], precision=case["prec"], lr=LR,
                                 instance=inputs.to_csr(c["n"], e, inputs.pm1_weights(len(e), seed + 1000 * q + 1)),
                                 seed=seed + q))
        batch = VQMCBatch(problems)
        for q, m in enumerate(batch.members):
            m.set_params(_theta(case, m.n, m.h, seed + 1000 * q))
            m.adam(_past_gradient(m.d, seed + 1000 * q))
        batch.graph_capture(B, stream=torch.cuda.Stream())
        return {"call": "batch", "batch": batch, "theta": [_parameters(m, batch) for m in batch.members]}
    m = _model(case, n, h, B, _instance(case["graph"], n, seed), seed)
    state = {"call": case["call"], "model": m, "B": B, "iteration": EVAL_COUNTER + seed}
    if case["call"] in ("step", "sr"):
        if case["call"] == "step":
            m.adam(_past_gradient(m.d, seed))
        state["theta"] = _parameters(m, m)
    if case["call"] == "logprob":
        g = torch.Generator(device="cuda").manual_seed(seed + 2)
        state["theta"] = _parameters(m, m).requires_grad_()
        state["spins"] = torch.randint(0, 2, (B, n), generator=g, device="cuda", dtype=torch.int8) * 2 - 1
        state["weight"] = torch.randn(B, generator=g, device="cuda") / B
    return state


def run(state):
    call = state["call"]
    if call == "batch":
        state["batch"].graph_launch()
        return state["theta"]
    m, B = state["model"], state["B"]
    if call == "step":
        m.step(B)
        return state["theta"]
    if call == "sr":
        m.sr_step(B, lr=SR_LR, lam=SR_LAMBDA)
        return state["theta"]
    if call == "logprob":
        state["theta"].grad = None
        lp = LogProb.apply(state["theta"], state["spins"], m)
        lp.backward(state["weight"])
        return {"logp": lp, "grad": state["theta"].grad}
    s, lp = m.sample(B, None, iteration=state["iteration"])
    e = m.local_energy(s)
    if call == "evaluate":
        return {"s": s, "logp": lp, "e": e}
    g, stats = m.grad(s, e)
    return {"s": s, "logp": lp, "e": e, "grad": g, "stats": stats}


# -------------------------------------------------------------------- work

def _work(call, graph, n, h, B, prec, sparse_edges):
    w = 2 if prec == "bf16" else 4  # bytes of a weight as the kernels read it
    hn = float(h) * n               # weights inside the masks (half of W1, half of W2)
    flops = bytes_ = 0.0
    if call != "logprob":
        flops += 2.0 * hn * B       # sampling: half the weights in updates, half in logits
        bytes_ += hn * w + float(B) * n
        flops += 2.0 * B * (sparse_edges if sparse_edges else 0.5 * n * n)
        bytes_ += sparse_edges * 12 if sparse_edges else 2.0 * n * n
        if graph == "tim":          # each sample's n flips: the outputs after the flipped spin
            flops += hn * n * B * 2.0 / 3.0
    else:
        flops += 2.0 * hn * B       # the forward pass
        bytes_ += hn * w + float(B) * n
    if call != "evaluate":
        flops += 3.0 * hn * B       # the hidden adjoint and the two weight gradients
    if call in ("step", "batch"):
        bytes_ += 24.0 * hn         # theta and both moments, read and written
    elif call == "sr":
        flops += 2.5 * (n + h) * B * B + B ** 3 / 3.0
        bytes_ += 8.0 * hn
    elif call in ("logprob", "grad"):
        bytes_ += 8.0 * hn          # the gradient, masked entries included
    return flops, bytes_


def work(case):
    n, h, B = case["n"], case["h"], case["B"]
    if case["call"] == "batch":
        each = [_work("batch", "er", c["n"], c["n"], B, case["prec"], DEGREE / 2.0 * c["n"]) for c in _members(case)]
        return {"flops": sum(f for f, _ in each), "bytes": sum(b for _, b in each)}
    edges = {"regular": 1.5 * n, "er": 4.0 * n, "unit": 0.25 * n * (n - 1)}.get(case["graph"], 0.0)
    f, b = _work(case["call"], case["graph"], n, h, B, case["prec"], edges)
    return {"flops": f, "bytes": b}


# ------------------------------------------------------- the same in 64 bits

class _Made:
    """The masked model in FP64, weights and hidden activations rounded to
    bfloat16 for the bf16 model, on the GPU."""

    def __init__(self, theta, case):
        n, h = case["n"], case["h"]
        self.n, self.h, self.act, self.bf16 = n, h, case["act"], case["prec"] == "bf16"
        self.deg = 1 + torch.arange(h, device="cuda", dtype=torch.int64) * (n - 1) // h
        row = torch.arange(n, device="cuda", dtype=torch.int64)[:, None]
        self.m1 = row < self.deg[None, :]     # W1^T (n, h)
        self.m2 = self.deg[None, :] <= row    # W2 (n, h)
        nh = n * h
        self.W1t = self._weight(theta[:nh].view(n, h)) * self.m1
        self.b1 = theta[nh: nh + h].double()
        self.W2 = self._weight(theta[nh + h: 2 * nh + h].view(n, h)) * self.m2
        self.b2 = theta[2 * nh + h:].double()

    def _weight(self, w):
        return w.float().bfloat16().double() if self.bf16 else w.double()

    def hidden(self, a):
        g = torch.relu(a) if self.act == "relu" else torch.sigmoid(a)
        return g.float().bfloat16().double() if self.bf16 else g

    def logp(self, S):
        H = self.hidden(S @ self.W1t + self.b1)
        return torch.nn.functional.logsigmoid(S * (H @ self.W2.T + self.b2)).sum(1)

    def sample(self, U):
        """Exact samples (B, n) from uniforms (B, n), spin by spin."""
        B = U.shape[0]
        A = self.b1[:, None].expand(self.h, B).contiguous()
        G = torch.empty_like(A)
        S = torch.empty(self.n, B, device="cuda", dtype=torch.float64)
        done = torch.searchsorted(self.deg, torch.arange(self.n + 1, device="cuda"), right=True).tolist()
        W1 = self.W1t.T.contiguous()
        for i in range(self.n):
            z = self.W2[i, : done[i]] @ G[: done[i]] + self.b2[i]
            S[i] = torch.where(U[:, i] < torch.sigmoid(z), 1.0, -1.0)
            A[done[i]:] += W1[done[i]:, i, None] * S[i]
            G[done[i]: done[i + 1]] = self.hidden(A[done[i]: done[i + 1]])
        return S.T.contiguous()

    def scores(self, S):
        """(delta, H, GA): the factors of each sample's gradient of log pi."""
        H = self.hidden(S @ self.W1t + self.b1)
        D = S * torch.sigmoid(-S * (H @ self.W2.T + self.b2))
        GA = (D @ self.W2) * ((H > 0).double() if self.act == "relu" else H * (1.0 - H))
        return D, H, GA

    def gradient(self, S, c):
        """sum_b c_b grad log pi(s_b), in theta's layout."""
        D, H, GA = self.scores(S)
        D, GA = D * c[:, None], GA * c[:, None]
        return torch.cat([((S.T @ GA) * self.m1).view(-1), GA.sum(0), ((D.T @ H) * self.m2).view(-1), D.sum(0)])

    def natural(self, S, c, lam):
        """(O^T O / B + lam)^-1 O^T c from the B x B Gram matrix of the score vectors O."""
        D, H, GA = self.scores(S)
        B = S.shape[0]
        O = torch.cat([((S[:, :, None] * GA[:, None, :]) * self.m1).view(B, -1), GA,
                       ((D[:, :, None] * H[:, None, :]) * self.m2).view(B, -1), D], 1)
        x = torch.linalg.solve(O @ O.T / B + lam * torch.eye(B, device="cuda", dtype=torch.float64), c)
        return O.T @ x


def _uniforms(B, n, seed, iteration):
    """Philox4x32-10 uniforms of (sample b, spin i): word i % 4 of counter
    (i // 4, b, iteration), the high 24 bits."""
    low = 0xFFFFFFFF

    def mul(k, x):  # 32 x 32 -> (high, low) words
        p0, p1 = k * (x & 0xFFFF), k * (x >> 16)
        mid = p0 + ((p1 & 0xFFFF) << 16)
        return (p1 >> 16) + (mid >> 32), mid & low

    groups = (n + 3) // 4
    c0 = torch.arange(groups, device="cuda", dtype=torch.int64).expand(B, groups)
    c1 = torch.arange(B, device="cuda", dtype=torch.int64)[:, None].expand(B, groups)
    c2, c3 = torch.full_like(c0, iteration & low), torch.full_like(c0, iteration >> 32)
    k0, k1 = seed & low, seed >> 32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    words = torch.stack([c0, c1, c2, c3], 2).reshape(B, 4 * groups)[:, :n]
    return (words >> 8).double() / float(1 << 24)


def _energy(inst, S, made):
    """Local energies of the configurations S."""
    if inst["kind"] == "dense":
        J = torch.from_numpy(inst["J"]).cuda().double()
        e = 0.5 * ((S @ J) * S).sum(1)
    else:
        rows = np.repeat(np.arange(inst["n"]), np.diff(inst["row_ptr"]))
        i, j = torch.from_numpy(rows).cuda(), torch.from_numpy(inst["col"].astype(np.int64)).cuda()
        w = torch.from_numpy(inst["w"]).cuda().double()
        e = torch.zeros(S.shape[0], device="cuda", dtype=torch.float64)
        for p in range(0, len(w), 4096):
            e += (S[:, i[p: p + 4096]] * S[:, j[p: p + 4096]]) @ w[p: p + 4096]
    if inst.get("field") is not None:
        e = e + S @ torch.from_numpy(inst["field"]).cuda().double()
    if inst.get("alpha") is not None:
        alpha = torch.from_numpy(inst["alpha"]).cuda().double()
        n = made.n
        flips = 1.0 - 2.0 * torch.eye(n, device="cuda", dtype=torch.float64)
        lp = made.logp(S)
        for b in range(0, S.shape[0], 32):
            x = (S[b: b + 32, None, :] * flips).reshape(-1, n)
            e[b: b + 32] -= torch.exp(0.5 * (made.logp(x).view(-1, n) - lp[b: b + 32, None])) @ alpha
    return e


def exact(case, seed):
    if case["call"] == "batch":
        return None
    n, h, B = case["n"], case["h"], case["B"]
    theta = _theta(case, n, h, seed)
    made = _Made(theta, case)
    if case["call"] == "logprob":
        g = torch.Generator(device="cuda").manual_seed(seed + 2)
        S = (torch.randint(0, 2, (B, n), generator=g, device="cuda", dtype=torch.int8) * 2 - 1).double()
        c = (torch.randn(B, generator=g, device="cuda") / B).double()
        return {"logp": made.logp(S), "grad": made.gradient(S, c)}
    inst = _instance(case["graph"], n, seed)
    if case["call"] in ("evaluate", "grad"):
        S = made.sample(_uniforms(B, n, seed, EVAL_COUNTER + seed))
        e = _energy(inst, S, made)
        out = {"s": None, "logp": made.logp(S), "e": None if inst["kind"] == "sparse_i32" else e}
        if case["call"] == "grad":
            mean, var = e.mean(), e.var(unbiased=False)
            out["grad"] = made.gradient(S, (e - mean) / B)
            out["stats"] = torch.stack([mean, var, e.min(), e.max()])
        return out
    t = torch.cat([(theta[: n * h].view(n, h) * made.m1).view(-1), theta[n * h: n * h + h],
                   (theta[n * h + h: 2 * n * h + h].view(n, h) * made.m2).view(-1), theta[2 * n * h + h:]]).double()
    if case["call"] == "sr":
        S = made.sample(_uniforms(B, n, seed, 0))
        e = _energy(inst, S, made)
        return t - SR_LR * made.natural(S, (e - e.mean()) / B, SR_LAMBDA)
    # Adam's second step, after one with the past gradient
    one = torch.ones(1, device="cuda", dtype=torch.bool)
    kept = torch.cat([made.m1.view(-1), one.expand(h), made.m2.view(-1), one.expand(n)]).double()
    g0 = _past_gradient(t.numel(), seed).double() * kept
    m, v = (1 - BETA1) * g0, (1 - BETA2) * g0 * g0
    t -= LR * (m / (1 - BETA1)) / ((v / (1 - BETA2)).sqrt() + EPS)
    made = _Made(t.float(), case)
    S = made.sample(_uniforms(B, n, seed, 0))
    e = _energy(inst, S, made)
    g = made.gradient(S, (e - e.mean()) / B)
    m, v = BETA1 * m + (1 - BETA1) * g, BETA2 * v + (1 - BETA2) * g * g
    return t - LR * (m / (1 - BETA1 ** 2)) / ((v / (1 - BETA2 ** 2)).sqrt() + EPS)
