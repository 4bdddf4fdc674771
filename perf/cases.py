"""What the MoE layer's users run, as cases that can be timed and compared.

A case is one pass through the public entry points of ``paper_2606_00395_gb300.binding``: a layer
in rollout mode (route predicted, recorded and applied), a layer in training mode (a recorded
route replayed), the multi-layer decode loop, the routing call by itself, the predictive loss with
its gradient, and the two bookkeeping calls around them.  Shapes are the repository's own: a
Qwen3-30B-A3B-shaped layer (d = 2048, 128 experts, top-8, expert width 768), a DeepSeek-V3-shaped
layer (d = 7168, 256 experts and a shared one, top-8, expert width 2048) and the small fp32 layer.

Inputs are seeded draws on the GPU: tokens N(0, 1), weights N(0, 0.02^2), router drift between
rollout and training N(0, 0.002^2), routes either spread evenly or Zipf(1.2)-skewed.
"""
import math

import torch

from paper_2606_00395_gb300 import binding as B

QWEN = dict(d=2048, N=128, k=8, m=768, shared=0, dtype="bf16")
DEEPSEEK = dict(d=7168, N=256, k=8, m=2048, shared=1, dtype="bf16")
TINY = dict(d=128, N=8, k=2, m=256, shared=0, dtype="fp32")

WEIGHT_STD = 0.02
DRIFT_STD = 0.002


def listed():
    return [
        # The tail of a rollout batch: a few sequences still decoding, one token each.  Latency.
        dict(name="decode_tail", kind="rollout", T=4, norm=False, **QWEN),
        # A rollout decode step of a full batch, one token per sequence.
        dict(name="decode_batch", kind="rollout", T=256, norm=False, **QWEN),
        # The same through the multi-layer loop, at a batch that is not a multiple of anything.
        dict(name="decode_layers", kind="layers", T=93, L=4, **QWEN),
        # A prompt chunk in rollout mode, the feature-cache logits and the expert loads recorded.
        dict(name="rollout_prefill", kind="rollout", T=4096, norm=False, **QWEN),
        # A ragged training micro-batch replayed on its recorded route; the probabilities are the
        # teacher of the predictive loss, the gates renormalised as this model family does.
        dict(name="replay_train", kind="replay", T=3001, zipf=False, norm=True, **QWEN),
        # Training on long sequences whose routes load the experts very unevenly.
        dict(name="replay_long", kind="replay", T=32768, zipf=True, norm=False, **QWEN),
        # A training micro-batch through the widest layer, with its shared expert.
        dict(name="replay_wide", kind="replay", T=8192, zipf=False, norm=False, **DEEPSEEK),
        # The route recorded without running the experts (they live elsewhere).
        dict(name="route_record", kind="route", T=4001, norm=False, **QWEN),
        # The predictor's training step: loss and gradient of one layer's cached tokens.
        dict(name="predictor_loss", kind="loss", T=2048, delta=False, d=2048, N=128, dtype="bf16"),
        # A layer's fixed-length feature cache, written after its rollout pass.
        dict(name="feature_cache", kind="cache", T=4096, Tc=2048, d=2048, N=128, dtype="bf16"),
        # Route-tracking metrics of a training step, summed over its layers.
        dict(name="route_tracking", kind="track", T=4096, L=6, N=128, k=8),
        # The exact-fp32 layer in both modes: a reference run or a small research model.
        dict(name="fp32_step", kind="step", T=256, norm=False, **TINY),
    ]


def _log_int(rng, lo, hi):
    """A whole number between lo and hi, even over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _shape(rng):
    """A bf16 layer: the Qwen3 shape half of the time, else one around it."""
    if rng.random() < 0.5:
        return dict(QWEN)
    return dict(d=64 * rng.randint(8, 48), N=16 * rng.randint(2, 16), k=rng.choice([2, 4, 6, 8]),
                m=64 * rng.randint(4, 24), shared=rng.choice([0, 0, 1]), dtype="bf16")


def draw(rng):
    kind = rng.choice(["rollout", "rollout", "rollout", "replay", "replay", "replay", "wide",
                       "layers", "route", "loss", "cache", "track", "step", "step"])
    if kind == "rollout":
        return dict(kind=kind, T=_log_int(rng, 1, 8192), norm=rng.random() < 0.3, **_shape(rng))
    if kind == "replay":
        return dict(kind=kind, T=_log_int(rng, 64, 32768), zipf=rng.random() < 0.5,
                    norm=rng.random() < 0.3, **_shape(rng))
    if kind == "wide":
        return dict(kind=rng.choice(["rollout", "replay"]), T=_log_int(rng, 64, 8000), zipf=False,
                    norm=False, **DEEPSEEK)
    if kind == "layers":
        return dict(kind=kind, T=_log_int(rng, 1, 512), L=rng.randint(2, 6), **QWEN)
    if kind == "route":
        return dict(kind=kind, T=_log_int(rng, 16, 32768), norm=rng.random() < 0.3, **_shape(rng))
    if kind == "loss":
        if rng.random() < 0.25:
            return dict(kind=kind, T=_log_int(rng, 32, 1024), delta=rng.random() < 0.5,
                        d=4 * rng.randint(16, 128), N=rng.randint(4, 64), dtype="fp32")
        return dict(kind=kind, T=_log_int(rng, 128, 8192), delta=rng.random() < 0.5,
                    d=64 * rng.randint(8, 64), N=16 * rng.randint(2, 16), dtype="bf16")
    if kind == "cache":
        T = _log_int(rng, 512, 32768)
        return dict(kind=kind, T=T, Tc=max(1, int(T * rng.uniform(0.05, 1.0))),
                    d=64 * rng.randint(8, 64), N=16 * rng.randint(2, 16), dtype="bf16")
    if kind == "track":
        return dict(kind=kind, T=_log_int(rng, 256, 32768), L=rng.randint(1, 8),
                    N=rng.randint(16, 256), k=rng.choice([2, 4, 6, 8]))
    N = rng.randint(4, 64)
    return dict(kind="step", T=_log_int(rng, 32, 2048), norm=rng.random() < 0.3,
                d=4 * rng.randint(16, 128), N=N, k=rng.randint(1, min(8, N)),
                m=4 * rng.randint(16, 128), shared=rng.choice([0, 0, 1]), dtype="fp32")


# ---- inputs ----------------------------------------------------------------------------------

def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


class _Draw:
    """Seeded draws on the GPU, in the order in which they are asked for."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed))

    def normal(self, *shape, std=1.0, dtype=torch.float32):
        return torch.empty(*shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=self.gen)

    def uniform(self, *shape):
        return torch.rand(*shape, device="cuda", generator=self.gen)


def _gumbel_topk(dr, weights, T, k):
    """k distinct experts per token, drawn without replacement in proportion to `weights`."""
    g = -torch.log(-torch.log(dr.uniform(T, weights.numel()).clamp_(1e-7, 1 - 1e-7)))
    return torch.topk(weights.log() + g, k, dim=1).indices.to(torch.int32).contiguous()


def _weights(dr, case, lead=()):
    dt = _dtype(case)
    d, N, m, s = case["d"], case["N"], case["m"], case["shared"]
    w = lambda *shape: dr.normal(*lead, *shape, std=WEIGHT_STD, dtype=dt)  # noqa: E731
    out = dict(W_router=w(N, d), W_pred=w(N, d), W_gate=w(N, m, d), W_up=w(N, m, d), W_down=w(N, d, m))
    out.update(Ws_gate=w(s, m, d) if s else None, Ws_up=w(s, m, d) if s else None,
               Ws_down=w(s, d, m) if s else None)
    return out


def _experts(st):
    return [st["w"][n] for n in ("W_gate", "W_up", "W_down", "Ws_gate", "Ws_up", "Ws_down")]


def _inputs(case, seed):
    """The input tensors of a case alone (what both run() and exact() start from)."""
    dr, kind = _Draw(seed), case["kind"]
    if kind == "loss":
        T, d, N = case["T"], case["d"], case["N"]
        p_old = dr.normal(T, N, std=0.9)
        T_rho = 2 * T + 1
        pos = torch.arange(T, device="cuda", dtype=torch.int64) * T_rho // T
        rho = dr.normal(T_rho, N, std=0.9)
        rho[pos] = p_old + dr.normal(T, N, std=0.1)  # the router has moved a little since
        return dict(p_old=p_old, rho=torch.softmax(rho, 1), pos=pos.to(torch.int32),
                    h_old=dr.normal(T, d, dtype=_dtype(case)),
                    W_pred=dr.normal(N, d, std=WEIGHT_STD, dtype=_dtype(case)))
    if kind == "cache":
        return dict(h=dr.normal(case["T"], case["d"], dtype=_dtype(case)),
                    logits=dr.normal(case["T"], case["N"], std=0.9))
    if kind == "track":
        z = dr.normal(case["L"], case["T"], case["N"], std=0.9)
        old = z + dr.normal(*z.shape, std=0.1)
        return dict(rho=[torch.softmax(layer, 1) for layer in z],
                    idx=[torch.topk(layer, case["k"], dim=1).indices.to(torch.int32) for layer in old])
    x = dr.normal(case["T"], case["d"], dtype=_dtype(case))
    if kind == "route":
        w = lambda: dr.normal(case["N"], case["d"], std=WEIGHT_STD, dtype=_dtype(case))  # noqa: E731
        return dict(x=x, w=dict(W_router=w(), W_pred=w()))
    st = dict(x=x, w=_weights(dr, case, (case["L"],) if kind == "layers" else ()))
    if kind in ("replay", "step"):  # the router as training has it now
        W = st["w"]["W_router"]
        st["W_now"] = (W.float() + dr.normal(*W.shape, std=DRIFT_STD)).to(W.dtype)
    if kind == "replay":
        e = torch.arange(1, case["N"] + 1, device="cuda", dtype=torch.float32)
        st["idx"] = _gumbel_topk(dr, e ** (-1.2 if case["zipf"] else 0.0), case["T"], case["k"])
    return st


def prepare(case, seed):
    """Inputs plus what a program keeps between calls: dimensions, workspaces, output buffers."""
    st = _inputs(case, seed)
    kind, T, N = case["kind"], case["T"], case["N"]
    st["kind"] = kind
    st["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    f32 = lambda *shape: torch.empty(*shape, device="cuda")  # noqa: E731
    i32 = lambda *shape: torch.empty(*shape, dtype=torch.int32, device="cuda")  # noqa: E731
    if kind == "loss":
        dm = B.dims(T, case["d"], N, 1, 64, 0, case["dtype"], B.PR2_F_DELTA_LOSS if case["delta"] else 0)
        st.update(dm=dm, ws=B.alloc_loss_workspace(dm), loss=f32(1), kl=f32(T), grad=f32(N, case["d"]))
        return st
    if kind == "cache":
        Tc = case["Tc"]
        st.update(dm=B.dims(T, case["d"], N, 1, 64, 0, case["dtype"]), Tc=Tc, pos=i32(Tc), cache_p=f32(Tc, N),
                  cache_h=torch.empty(Tc, case["d"], dtype=_dtype(case), device="cuda"))
        return st
    if kind == "track":
        st.update(dm=B.dims(T, 64, N, case["k"], 64, 0, "fp32"),
                  counters=torch.zeros(case["k"] + 2, dtype=torch.int64, device="cuda"))
        return st
    k = case["k"]
    flags = B.PR2_F_NORMALIZE_TOPK if case.get("norm") else 0
    dm = B.dims(T, case["d"], N, k, case["m"], case["shared"], case["dtype"], flags)
    lead = (case["L"],) if kind == "layers" else ()
    st.update(dm=dm, gates=f32(*lead, T, k), aux=f32(*lead, T, N))
    if kind != "replay":
        st["idx"] = i32(*lead, T, k)
    if kind != "route":
        st.update(ws=B.alloc_workspace(dm), out=torch.empty_like(st["x"]), counts=i32(N))
    if kind == "layers":
        st["L"] = case["L"]
    if kind == "step":
        st.update(gates2=f32(T, k), probs=f32(T, N), out2=torch.empty_like(st["x"]))
    return st


# ---- one pass --------------------------------------------------------------------------------

def _rollout(st):
    B.check(B.pr2_moe_rollout_forward(
        st["dm"], st["x"], st["w"]["W_router"], st["w"]["W_pred"], st["idx"], st["gates"], st["aux"], None,
        *_experts(st), st["out"], counts=st["counts"], workspace=st["ws"], status=st["status"]))
    return dict(idx=st["idx"], gates=st["gates"], logits=st["aux"], out=st["out"], counts=st["counts"])


def _replay(st, gates, probs, out):
    B.check(B.pr2_moe_replay_forward(
        st["dm"], st["x"], st["W_now"], st["idx"], gates, probs, *_experts(st), out,
        workspace=st["ws"], status=st["status"]))
    return dict(gates=gates, probs=probs, out=out)


def run(st):
    kind = st["kind"]
    if kind == "rollout":
        return _rollout(st)
    if kind == "replay":
        return _replay(st, st["gates"], st["aux"], st["out"])
    if kind == "step":
        return dict(rollout=_rollout(st), replay=_replay(st, st["gates2"], st["probs"], st["out2"]))
    if kind == "layers":
        w = st["w"]
        h = st["out"].copy_(st["x"])  # the loop updates its residual stream in place
        B.check(B.pr2_rollout_layers(
            st["dm"], st["L"], h, w["W_router"], w["W_pred"], w["W_gate"], w["W_up"], w["W_down"], st["idx"],
            st["gates"], logits_old=st["aux"], workspace=st["ws"], status=st["status"]))
        # The routes of later layers are not compared: they turn on the rounding of the layers before.
        return dict(h=h, gates=st["gates"], logits=st["aux"])
    if kind == "route":
        B.check(B.pr2_route_predict(st["dm"], st["x"], st["w"]["W_router"], st["w"]["W_pred"], st["idx"],
                                    st["gates"], st["aux"], status=st["status"]))
        return dict(idx=st["idx"], gates=st["gates"], logits=st["aux"])
    if kind == "loss":
        B.check(B.pr2_predictor_loss(
            st["dm"], st["h_old"], st["p_old"], st["W_pred"], st["rho"], st["loss"], st["grad"], pos=st["pos"],
            kl_tok=st["kl"], workspace=st["ws"], status=st["status"]))
        return dict(loss=st["loss"], kl=st["kl"], grad=st["grad"])
    if kind == "cache":
        B.check(B.pr2_feature_cache_write(st["dm"], st["Tc"], st["h"], st["logits"], st["pos"], st["cache_h"],
                                          st["cache_p"]))
        return dict(pos=st["pos"], h=st["cache_h"], p=st["cache_p"])
    hist, overlap = st["counters"][:-1], st["counters"][-1:]
    st["counters"].zero_()
    for rho, idx in zip(st["rho"], st["idx"]):
        B.check(B.pr2_route_diagnostics(st["dm"], rho, idx, hist, overlap))
    return dict(hist=hist, overlap=overlap)


# ---- work and accuracy -----------------------------------------------------------------------

def work(case):
    """Each input read once, each output written once; multiplies and adds of the contractions."""
    kind, T, N = case["kind"], case["T"], case["N"]
    if kind == "track":
        return dict(bytes=case["L"] * T * 4 * (N + case["k"]), flops=0)
    d, es = case["d"], 2 if case["dtype"] == "bf16" else 4
    if kind == "loss":
        return dict(bytes=T * (es * d + 8 * N + 8) + N * d * (es + 4), flops=4 * T * N * d)
    if kind == "cache":
        return dict(bytes=case["Tc"] * (2 * (es * d + 4 * N) + 4), flops=0)
    k, m, s = case["k"], case["m"], case["shared"]
    tokens, route = T * es * d, T * (8 * k + 4 * N)
    if kind == "route":
        return dict(bytes=tokens + 2 * N * d * es + route, flops=4 * T * N * d)
    hit = sum(1 - (1 - p) ** T for p in _expert_share(case))
    experts, mlp = (hit + s) * 3 * m * d * es, 6 * T * (k + s) * m * d
    if kind == "replay":
        return dict(bytes=2 * tokens + N * d * es + route + experts, flops=mlp + 2 * T * N * d)
    rollout = dict(bytes=2 * tokens + 2 * N * d * es + route + experts, flops=mlp + 4 * T * N * d)
    if kind == "step":
        return dict(bytes=2 * rollout["bytes"] - N * d * es, flops=2 * rollout["flops"] - 2 * T * N * d)
    return {n: v * case.get("L", 1) for n, v in rollout.items()}


def _expert_share(case):
    """About the share of tokens that each expert serves."""
    w = [(e + 1) ** (-1.2 if case.get("zipf") else 0.0) for e in range(case["N"])]
    return [min(1.0, case["k"] * x / sum(w)) for x in w]


def tolerance(case):
    kind = case["kind"]
    if kind in ("cache", "track"):
        return "exact"  # copies and counts
    if case["dtype"] == "fp32":
        return {"rel": 2e-5, "max": 1e-3, "differ": 1e-3}
    if kind == "route":  # fp32 sums of exact products; `differ`: ties between experts
        return {"rel": 2e-5, "max": 1e-3, "differ": 1e-3}
    # bf16 hidden activations and outputs (layers), bf16 dKL/dz in the gradient (loss)
    return {"rel": 1e-2, "max": 0.3, "differ": 1e-3}


def _topk(z, k):
    """Indices of the k largest per row, ties to the lower index."""
    return torch.sort(z, dim=1, descending=True, stable=True).indices[:, :k]


def _layer64(x, w, idx, gates):
    """sum_s gates[t, s] E_idx[t, s](x_t) + shared experts, and the tokens per expert."""
    def expert(v, wg, wu, wd):
        return (torch.nn.functional.silu(v @ wg.double().T) * (v @ wu.double().T)) @ wd.double().T

    N = w["W_gate"].shape[0]
    out = torch.zeros_like(x)
    counts = torch.bincount(idx.reshape(-1), minlength=N)
    for e in range(N):
        t, slot = (idx == e).nonzero(as_tuple=True)
        if t.numel():
            y = expert(x[t], w["W_gate"][e], w["W_up"][e], w["W_down"][e])
            out.index_add_(0, t, y * gates[t, slot].unsqueeze(1))
    if w["Ws_gate"] is not None:
        for e in range(w["Ws_gate"].shape[0]):
            out += expert(x, w["Ws_gate"][e], w["Ws_up"][e], w["Ws_down"][e])
    return out, counts.to(torch.int32)


def _predict64(x, w, k, norm):
    p = x @ w["W_router"].double().T
    rho = torch.softmax(p + x @ w["W_pred"].double().T, 1)
    idx = _topk(rho, k)
    gates = rho.gather(1, idx)
    return p, idx, gates / gates.sum(1, keepdim=True) if norm else gates


def _replay64(x, st, idx, norm):
    rho = torch.softmax(x @ st["W_now"].double().T, 1)
    gates = rho.gather(1, idx.long())
    if norm:
        gates = gates / gates.sum(1, keepdim=True)
    return dict(gates=gates, probs=rho, out=_layer64(x, st["w"], idx.long(), gates)[0])


def exact(case, seed):
    kind = case["kind"]
    st = _inputs(case, seed)
    if kind == "loss":
        h, p_old, rho = st["h_old"].double(), st["p_old"].double(), st["rho"][st["pos"].long()].double()
        b = h @ st["W_pred"].double().T
        target = torch.softmax(rho.log() - p_old, 1) if case["delta"] else rho
        log_pred = torch.log_softmax(b if case["delta"] else p_old + b, 1)
        kl = (target * (target.log() - log_pred)).sum(1)
        return dict(loss=kl.mean().reshape(1), kl=kl, grad=(log_pred.exp() - target).T @ h / case["T"])
    if kind == "cache":
        pos = torch.arange(case["Tc"], device="cuda") * case["T"] // case["Tc"]
        return dict(pos=pos.to(torch.int32), h=st["h"][pos].double(), p=st["logits"][pos].double())
    if kind == "track":
        k, over = case["k"], []
        for rho, idx in zip(st["rho"], st["idx"]):
            now = _topk(rho, k)
            over.append((now.unsqueeze(2) == idx.long().unsqueeze(1)).sum((1, 2)))
        over = torch.cat(over)
        return dict(hist=torch.bincount(k - over, minlength=k + 1), overlap=over.sum().reshape(1))
    x, k, norm = st["x"].double(), case["k"], bool(case.get("norm"))
    if kind == "replay":
        return _replay64(x, st, st["idx"], norm)
    if kind == "layers":
        gates, logits = [], []
        for l in range(case["L"]):
            w = {n: None if v is None else v[l] for n, v in st["w"].items()}
            p, idx, g = _predict64(x, w, k, False)
            x = (x + _layer64(x, w, idx, g)[0]).bfloat16().double()  # the stream is kept in bf16
            gates.append(g)
            logits.append(p)
        return dict(h=x, gates=torch.stack(gates), logits=torch.stack(logits))
    p, idx, gates = _predict64(x, st["w"], k, norm)
    rec = dict(idx=idx.to(torch.int32), gates=gates, logits=p)
    if kind == "route":
        return rec
    out, counts = _layer64(x, st["w"], idx, gates)
    rollout = dict(rec, out=out, counts=counts)
    if kind == "rollout":
        return rollout
    return dict(rollout=rollout, replay=_replay64(x, st, idx, norm))
