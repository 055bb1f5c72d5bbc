"""The work that this library is measured on: expert-choice and token-choice MoE layers, from a
256-token fp32 layer to full training steps, through the public Python entry points.

Sizes are those of the benchmark and the tests (d 2048 with 64 experts, 128 small experts, wide
d 4096 layers, the tiny fp32 layer) and generic smaller, ragged and odd ones between them. Inputs
follow the workloads' recipes: unit-norm token rows and N(0, 0.02^2) weights in bf16, N(0, 1)
tokens and fan-in weights in fp32; with timestep capacity a drawn fraction of each sequence holds
one mask vector, so that scores tie exactly.

A case is a dict of
  kind      "train" (forward + backward), "infer" (forward), "tc" (token choice, forward +
            backward), "route" (router and selection), "select" (selection from given scores)
  dtype     "bf16" or "f32"
  G, N      sequences (selection groups) and tokens in all; ragged: unequal sequence lengths
  d, E, F   model width, experts, hidden width of an expert
  k         experts per token on average: a sequence of L tokens has capacity round(k L / E)
  timestep  per-sequence capacities from masking ratios, given on the device before each step
  bias, residual, shared (hidden width of the shared experts), cf (token-choice capacity
  factor, 0: dropless), outputs (also return the selection and the scores)
"""
import math

import numpy as np
import torch

from paper_2604_01622_gb300.inputs import timestep_capacity
from paper_2604_01622_gb300.layer import ECMoELayer, TCMoELayer, tc_capacity


def _case(kind, G, N, E, k, d=64, F=64, dtype="bf16", ragged=False, timestep=False, bias=False,
          residual=False, shared=0, cf=0.0, outputs=True, name=None):
    c = dict(kind=kind, dtype=dtype, G=G, N=N, d=d, E=E, F=F, k=k, ragged=ragged,
             timestep=timestep, bias=bias, residual=residual, shared=shared, cf=cf,
             outputs=outputs)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest layer of the benchmark: a unit-test-sized model in fp32, all latency
        _case("train", 2, 256, 8, 1, 64, 128, "f32", name="tiny_f32"),
        # a small model trained in fp32 (debugging, reference runs); no size a multiple of a tile
        _case("train", 4, 4000, 16, 4, 500, 364, "f32", ragged=True, bias=True,
              name="f32_ragged"),
        # one denoising step of one 256-token block at the d 2048 layer: weights dominate
        _case("infer", 1, 256, 64, 8, 2048, 1024, outputs=False, name="infer_block"),
        # a served batch of requests of unequal lengths on the 128-expert layer
        _case("infer", 6, 5000, 128, 8, 1024, 512, ragged=True, bias=True, name="infer_ragged"),
        # a small research model on a few ragged documents; odd widths, 12 experts
        _case("train", 3, 777, 12, 2, 192, 320, ragged=True, name="train_small"),
        # an ordinary micro-batch of a mid-sized model
        _case("train", 4, 4096, 32, 4, 1024, 512, outputs=False, name="train_mid"),
        # a micro-batch of the d 2048 layer with two shared experts
        _case("train", 2, 8192, 64, 8, 2048, 1024, shared=2048, outputs=False,
              name="train_shared"),
        # the token-choice comparison at the same layer, capacity factor 1.25
        _case("tc", 1, 8192, 64, 8, 2048, 1024, cf=1.25, outputs=False, name="tc_train"),
        # full training step of the 128-small-experts layer, skewed router bias
        _case("train", 16, 32768, 128, 8, 1024, 512, bias=True, outputs=False,
              name="train_e128"),
        # full training step of the headline layer with capacities that follow the masking ratio
        _case("train", 8, 32768, 64, 8, 2048, 1024, timestep=True, outputs=False,
              name="train_timestep"),
        # one layer of the wide residual stack, 8192-token sequences
        _case("train", 4, 32768, 32, 2, 4096, 2048, timestep=True, residual=True, outputs=False,
              name="train_wide"),
        # selection from given scores over long sequences (retrofit and analysis runs)
        _case("select", 4, 131072, 64, 8, name="select_long"),
    ]


_MAX_FLOPS = 9.0e12       # of the largest listed case, rounded down
_MAX_WEIGHTS = 64 * 2048 * 1024


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["train"] * 5 + ["infer"] * 3 + ["tc"] * 2 + ["route", "select"])
        if kind in ("route", "select"):
            G = log(1, 16)
            N = max(G, log(512, 131072 if kind == "select" else 32768))
            E = rng.choice([8, 16, 24, 40, 64, 96, 128])
            return _case(kind, G, N, E, rng.randint(1, min(8, E)),
                         d=64 * log(1, 64) if kind == "route" else 64,
                         ragged=rng.random() < 0.5, bias=kind == "route" and rng.random() < 0.5)
        f32 = kind != "tc" and rng.random() < 0.25
        unit = 4 if f32 else 64
        N = log(64, 4096 if f32 else 32768)
        G = min(log(1, 16), max(1, N // 16))
        d = unit * max(1, log(64, 1024 if f32 else 4096) // unit)
        F = unit * max(1, log(64, 512 if f32 else 2048) // unit)
        E = rng.choice([4, 8, 12, 16, 32, 48, 64, 100, 128])
        k = rng.randint(1, min(8, E))
        timestep = kind != "tc" and not f32 and rng.random() < 0.3
        if timestep:
            N -= N % G
        c = _case(kind, G, N, E, k, d, F, "f32" if f32 else "bf16",
                  ragged=not timestep and rng.random() < 0.5, timestep=timestep,
                  bias=rng.random() < 0.3, residual=kind != "tc" and rng.random() < 0.3,
                  shared=64 * log(1, 32) if kind == "train" and not f32 and rng.random() < 0.2
                  else 0,
                  cf=rng.choice([0.0, 1.0, 1.25]) if kind == "tc" else 0.0,
                  outputs=rng.random() < 0.5)
        if (work(c)["flops"] <= _MAX_FLOPS / (16 if f32 else 1) and E * d * F <= _MAX_WEIGHTS
                and (not timestep or G * _uniform_k(N // G, c) <= N // G)):
            return c


# ------------------------------------------------------------------ shapes and inputs
def _group_off(c):
    """Sequence boundaries: equal, or lengths spread by a factor of about four."""
    G, N = c["G"], c["N"]
    if not c["ragged"]:
        base, extra = divmod(N, G)
        sizes = [base + (g < extra) for g in range(G)]
    else:
        w = np.random.RandomState(G * 1000003 + N).uniform(0.4, 1.6, G)
        sizes = np.maximum(1, np.floor(N * w / w.sum())).astype(int)
        sizes[-1] += N - sizes.sum()
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)


def _uniform_k(L, c):
    return int(min(L, max(1, math.floor(c["k"] * L / c["E"] + 0.5))))


def _uniform_k_g(c):
    return np.array([_uniform_k(int(L), c) for L in np.diff(_group_off(c))], np.int32)


def _rows(c):
    """Token-expert pairs that the experts process."""
    if c["kind"] == "tc":
        return c["N"] * c["k"]
    return c["E"] * int(_uniform_k_g(c).sum())


class _Inputs:
    pass


def _inputs(c, seed):
    f32 = c["dtype"] == "f32"
    dt = torch.float32 if f32 else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 1000 + 17)
    N, d, E, F = c["N"], c["d"], c["E"], c["F"]

    def normal(*shape, std=1.0, dtype=dt):
        x = torch.empty(shape, dtype=dtype, device="cuda")
        flat = x.view(-1)
        for i in range(0, flat.numel(), 1 << 28):      # fp32 draws, a part at a time
            part = flat[i:i + (1 << 28)]
            part.copy_(torch.randn(part.numel(), device="cuda", generator=gen).mul_(std))
        return x

    p = _Inputs()
    p.group_off, p.k_g = _group_off(c), _uniform_k_g(c)
    if c["kind"] == "select":
        # router scores of E experts: softmax of logits with a spread of a few percent
        p.S = torch.softmax(normal(E, N, std=0.03, dtype=torch.float32), dim=0).contiguous()
        return p
    x = normal(N, d, dtype=torch.float32)
    if not f32:
        x /= x.norm(dim=1, keepdim=True)
    if c["timestep"]:
        r = np.random.RandomState(seed % (1 << 31))
        t = r.uniform(0.0, 1.0, c["G"])
        L = N // c["G"]
        p.k_g = timestep_capacity(t, int(p.k_g[0]), L)
        mask = normal(d, dtype=torch.float32)
        mask = mask if f32 else mask / mask.norm()
        hit = torch.rand(c["G"], L, device="cuda", generator=gen) < torch.tensor(
            t, device="cuda").float()[:, None]
        x[hit.view(-1)] = mask
    p.X = x.to(dt)
    s_in, s_ff = (d ** -0.5, F ** -0.5) if f32 else (0.02, 0.02)
    p.Wr = normal(d, E, std=s_in)
    p.br = normal(E, std=1.0, dtype=torch.float32) if c["bias"] else None
    if c["kind"] == "route":
        return p
    p.Wg, p.Wu = normal(E, d, F, std=s_in), normal(E, d, F, std=s_in)
    p.Wd = normal(E, F, d, std=s_ff)
    p.shared = None
    if c["shared"]:
        fs = c["shared"]
        p.shared = (normal(d, fs, std=s_in), normal(d, fs, std=s_in), normal(fs, d, std=s_ff))
    if c["kind"] != "infer":
        p.dY = normal(N, d)
    return p


# ------------------------------------------------------------------ the measured pass
def prepare(case, seed):
    c = case
    p = _inputs(c, seed)
    p.case = c
    p.k_dev = None
    if c["kind"] == "tc":
        cap = tc_capacity(c["cf"] or None, c["k"], c["N"], c["E"])
        p.layer = TCMoELayer(c["N"], c["d"], c["E"], c["F"], c["k"], cap)
    else:
        p.layer = ECMoELayer(c["N"], c["d"], c["E"], c["F"], p.group_off, p.k_g,
                             dtype=c["dtype"] if c["kind"] != "select" else "f32",
                             d_ff_shared=c["shared"])
        if c["timestep"]:
            p.k_dev = torch.from_numpy(p.k_g.copy()).cuda()
    if c["residual"]:
        p.layer.set_residual(True)
    return p


def run(state):
    p = state
    c = p.case
    if c["kind"] == "select":
        idx, gate, S = p.layer.route(S_in=p.S)
        return {"idx": idx, "gate": gate, "S": S}
    if c["kind"] == "route":
        idx, gate, S = p.layer.route(p.X, p.Wr, p.br)
        return {"idx": idx, "gate": gate, "S": S}
    if p.k_dev is not None:
        p.layer.set_capacity_async(p.k_dev)
    out = p.layer.forward(p.X, p.Wr, p.br, p.Wg, p.Wu, p.Wd, outputs=c["outputs"],
                          shared=p.shared)
    names = (("Y", "choice", "gate", "kept", "load", "S") if c["kind"] == "tc"
             else ("Y", "idx", "gate", "S"))
    got = dict(zip(names, out))
    if c["kind"] != "infer":
        got.update(p.layer.backward(p.dY, with_bias=c["bias"]))
    return got


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    c = case
    N, d, E, F, Fs, P = c["N"], c["d"], c["E"], c["F"], c["shared"], _rows(c)
    b = 4 if c["dtype"] == "f32" else 2
    sel = 4 * N * E + 8 * P                               # scores, indices and gates
    if c["kind"] == "select":
        return {"bytes": 4 * N * E + sel, "flops": 0}
    router = 2 * N * d * E
    if c["kind"] == "route":
        return {"bytes": b * (N * d + d * E) + sel, "flops": router}
    weights = d * E + 3 * E * d * F + 3 * d * Fs
    flops = router + 6 * P * d * F + 6 * N * d * Fs
    nbytes = b * (2 * N * d + weights) + (sel if c["outputs"] else 0)
    if c["kind"] != "infer":
        flops *= 3
        nbytes += b * 2 * N * d + 4 * weights             # dY in, dX and the fp32 gradients out
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "select":
        return "exact"
    if case["dtype"] == "f32":
        # fp32 sums in another order: 2e-7 to 5e-7 against 64 bits
        return {"rel": 4e-6, "max": 4e-4, "differ": 2e-3}
    # bf16 activations between the GEMMs: 3e-3 to 5e-3 against 64 bits; scores a rounding apart
    # can swap two tokens at a capacity's edge, which moves the indices after them
    return {"rel": 1.5e-2, "max": 0.6, "differ": 0.01}


# ------------------------------------------------------------------ the same in 64 bits
def _select64(S, group_off, k_g):
    """S [N][E] in 64 bits -> idx [E][M]: per expert and group the k_g largest scores (ranked as
    32-bit values, so that equal inputs tie), ties to the lower token, in token order."""
    parts = []
    for g in range(len(k_g)):
        lo, hi, k = int(group_off[g]), int(group_off[g + 1]), int(k_g[g])
        order = torch.sort(S[lo:hi].float().t(), dim=1, descending=True, stable=True)[1][:, :k]
        parts.append(lo + order.sort(dim=1)[0])
    return torch.cat(parts, dim=1)


def exact(case, seed):
    c = case
    p = _inputs(c, seed)
    N, E = c["N"], c["E"]
    if c["kind"] == "select":
        idx = _select64(p.S.t().double(), p.group_off, p.k_g)
        return {"idx": idx.int(), "gate": p.S.gather(1, idx), "S": p.S}
    X, Wr = p.X.double(), p.Wr.double()
    logits = X @ Wr + (0 if p.br is None else p.br.double())
    S = torch.softmax(logits, dim=1)
    out = {}
    if c["kind"] == "tc":
        k = c["k"]
        choice = torch.sort(S.float(), dim=1, descending=True, stable=True)[1][:, :k]
        top = S.gather(1, choice)
        Z = top.sum(dim=1, keepdim=True)
        gates = top / Z
        cap = math.ceil(c["cf"] * k * N / E) if c["cf"] else N
        hit = torch.zeros(N, E, dtype=torch.int64, device="cuda").scatter_(1, choice, 1)
        kept = (hit.cumsum(0).gather(1, choice) <= cap)
        if c["outputs"]:
            out.update(choice=choice.int(), gate=gates, kept=kept.int(),
                       load=hit.sum(0).clamp(max=cap).int(), S=S)
        full_gate = torch.zeros(N, E, dtype=torch.float64, device="cuda").scatter_(
            1, choice, gates * kept)
        rows = [torch.nonzero((hit * 0).scatter_(1, choice, kept.long())[:, e])[:, 0]
                for e in range(E)]
    else:
        idx = _select64(S, p.group_off, p.k_g)
        rows = list(idx)
        full_gate = S
        if c["outputs"] or c["kind"] == "route":
            out.update(idx=idx.int(), gate=S.t().gather(1, idx), S=S.t().contiguous())
    if c["kind"] == "route":
        return out
    back = c["kind"] != "infer"
    Y = X.clone() if c["residual"] else torch.zeros_like(X)
    if back:
        dY = p.dY.double()
        dX = dY.clone() if c["residual"] else torch.zeros_like(X)
        dS = torch.zeros_like(S)
        grads = {n: torch.empty(w.shape, dtype=torch.float64, device="cuda")
                 for n, w in (("dWg", p.Wg), ("dWu", p.Wu), ("dWd", p.Wd))}

    def ffn(t, g, Wg, Wu, Wd, grad_out):
        """SwiGLU of the rows t scaled by g (None: 1); adds to Y and dX, fills grad_out;
        returns the gate gradients."""
        Wg, Wu, Wd = Wg.double(), Wu.double(), Wd.double()
        h = X[t]
        a, u = h @ Wg, h @ Wu
        sg = torch.sigmoid(a)
        v = a * sg * u
        o = v @ Wd
        Y.index_add_(0, t, o if g is None else g[:, None] * o)
        if not back:
            return None
        dy = dY[t]
        do = dy if g is None else g[:, None] * dy
        dv = do @ Wd.t()
        da, du = dv * u * sg * (1 + a * (1 - sg)), dv * a * sg
        dX.index_add_(0, t, da @ Wg.t() + du @ Wu.t())
        grad_out[0].copy_(h.t() @ da)
        grad_out[1].copy_(h.t() @ du)
        grad_out[2].copy_(v.t() @ do)
        return (dy * o).sum(dim=1)

    for e in range(E):
        t = rows[e]
        dg = ffn(t, full_gate[t, e], p.Wg[e], p.Wu[e], p.Wd[e],
                 [grads[n][e] for n in ("dWg", "dWu", "dWd")] if back else None)
        if back:
            dS[t, e] = dg
    if c["shared"]:
        if back:
            for n, w in zip(("dWg_s", "dWu_s", "dWd_s"), p.shared):
                grads[n] = torch.empty(w.shape, dtype=torch.float64, device="cuda")
        ffn(torch.arange(N, device="cuda"), None, *p.shared,
            [grads[n] for n in ("dWg_s", "dWu_s", "dWd_s")] if back else None)
    out["Y"] = Y
    if back:
        if c["kind"] == "tc":      # dS holds the gradients of the normalised gates of kept pairs
            common = (dS * full_gate).sum(dim=1, keepdim=True)
            dS = (dS - common) / Z * hit
        dZ = S * (dS - (dS * S).sum(dim=1, keepdim=True))
        out.update(grads, dX=dX + dZ @ Wr.t(), dWr=X.t() @ dZ)
        out["dbr"] = dZ.sum(dim=0) if c["bias"] else None
    return out
