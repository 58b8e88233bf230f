"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one call (or one forward and backward pair) through the public Python entry points on a stated shape: training
steps, prompts (prefill) and decode steps, over the sizes, storage types and options that the repository's configurations
and tests use.  `listed()` names the fixed cases, `draw(rng)` gives further ones from the same ranges.
"""
import math

import torch

from paper_2606_08804_b200 import autograd as qa
from paper_2606_08804_b200 import binding as qd

# ---- the cases --------------------------------------------------------------------------------------------------------
# kind    "train"    forward that keeps what the backward needs, then backward
#         "autograd" the same pair through torch.autograd (qdelta_chunk), as a model's training step reaches it
#         "prefill"  forward only: a prompt
#         "decode"   S tokens per sequence through the recurrence, state updated in place
# gates   "config"   beta, alpha, lambda = sigmoid(N(0, 1)), the benchmark configurations' distribution
#         "trained"  slowly forgetting gates as a trained model has them (alpha near 0.98, small beta)
# raw     q, k un-normalised and the gates as logits: the kernels normalise and apply the sigmoids (norm_qk, logits)
# pool    keys from a pool of 512 vectors per head plus noise (long contexts with colliding keys)


def _chunk(kind, B, T, H, dk=128, dv=128, dtype="bf16", gates="config", raw=False, pool=False, h0=True):
    return {"kind": kind, "B": B, "T": T, "H": H, "dk": dk, "dv": dv, "dtype": dtype, "gates": gates, "raw": raw,
            "pool": pool, "h0": h0}


def _decode(B, S, H, dk=128, dv=128, dtype="bf16", gates="config", raw=False, state="f32", api="step"):
    return {"kind": "decode", "B": B, "S": S, "H": H, "dk": dk, "dv": dv, "dtype": dtype, "gates": gates, "raw": raw,
            "state": state, "api": api}


def listed():
    c = [
        # a language-model training step of one layer, 16384 tokens: the headline configuration
        ("train lm", _chunk("train", 8, 2048, 16)),
        # long-context training: one sequence of 32768 tokens, few heads, colliding keys (the largest case)
        ("train long", _chunk("train", 1, 32768, 32, pool=True)),
        # a model's training step through torch.autograd, raw q, k and gate logits, ragged length
        ("train autograd ragged raw", _chunk("autograd", 6, 1000, 12, gates="trained", raw=True, h0=False)),
        # training with head dimension 64
        ("train d64", _chunk("train", 4, 1024, 16, dk=64, dv=64)),
        # full-precision training of a small model (debugging, reference runs)
        ("train f32", _chunk("train", 2, 512, 8, dtype="f32")),
        # prompts of a batch, state handed on to decode: the forward configuration
        ("prefill lm", _chunk("prefill", 8, 2048, 16)),
        # one user's prompt of odd length, raw q, k and gate logits
        ("prefill one ragged raw", _chunk("prefill", 1, 777, 16, gates="trained", raw=True, h0=False)),
        # the tiny full-precision forward configuration
        ("prefill tiny f32", _chunk("prefill", 1, 256, 2, dk=64, dv=64, dtype="f32", h0=False)),
        # the decode configuration: 256 sequences, one token each
        ("decode 256", _decode(256, 1, 16)),
        # a few users, one token each: latency
        ("decode 3", _decode(3, 1, 16, gates="trained")),
        # verification of several draft tokens per call, raw inputs
        ("decode 48 x 4 raw", _decode(48, 4, 16, gates="trained", raw=True, api="steps")),
        # memory-lean decode: bf16 state, one token per call
        ("decode 256 state bf16", _decode(256, 1, 16, gates="trained", state="bf16", api="steps")),
    ]
    return [dict(d, name=n) for n, d in c]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["train", "train", "autograd", "prefill", "prefill", "small dims", "f32", "decode", "decode", "steps"])
    gates = rng.choice(["config", "trained"])
    if what in ("train", "autograd", "prefill"):
        # 128-dimensional heads in bf16: short prompts up to long contexts, at most 2^19 token-heads per call
        T = _log_int(rng, 64, 16384)
        if rng.random() < 0.4:
            T = max(64, T // 64 * 64)
        H = rng.choice([4, 8, 12, 16, 32])
        B = min(_log_int(rng, 1, 32), max(1, (1 << 19) // (T * H)))
        raw = what == "autograd" or rng.random() < 0.3
        return _chunk(what, B, T, H, gates=gates, raw=raw, pool=rng.random() < 0.2, h0=rng.random() < 0.5)
    if what in ("small dims", "f32"):
        # other head dimensions in bf16, and full precision: small models and checks, at most 2^16 token-heads per call
        f32 = what == "f32"
        dk, dv = rng.choice([(64, 64), (64, 64), (128, 64), (64, 128)] + ([(128, 128)] if f32 else []))
        T = _log_int(rng, 64, 4096)
        H = rng.choice([2, 4, 8, 16])
        B = min(_log_int(rng, 1, 8), max(1, (1 << (13 if f32 else 16)) // (T * H)))
        return _chunk(rng.choice(["train", "prefill"]), B, T, H, dk=dk, dv=dv, dtype="f32" if f32 else "bf16", gates=gates,
                      raw=rng.random() < 0.2, h0=rng.random() < 0.5)
    B, H = _log_int(rng, 1, 256), rng.choice([4, 8, 16])
    if what == "decode":
        d = rng.choice([128, 128, 128, 64])
        return _decode(B, 1, H, dk=d, dv=d, dtype=rng.choice(["bf16", "bf16", "bf16", "f32"]), gates=gates)
    return _decode(B, rng.randint(1, 8), H, gates=gates, raw=rng.random() < 0.5, state=rng.choice(["f32", "f32", "bf16"]),
                   api="steps")


# ---- inputs -----------------------------------------------------------------------------------------------------------
_DT = {"bf16": torch.bfloat16, "f32": torch.float32}


def _unit(x):
    return torch.nn.functional.normalize(x, dim=-1)


def _tokens(case, gen, shape):
    """q, k, v and the coefficients of `shape` = (batch, tokens, heads) or (batch, heads), in the storage type."""
    dt = _DT[case["dtype"]]

    def normal(*dims):
        return torch.randn(*dims, device="cuda", generator=gen)

    q, k = normal(*shape, case["dk"]), normal(*shape, case["dk"])
    if case.get("pool"):
        B, T, H = shape
        pool = _unit(normal(B * H, 512, case["dk"]))
        pick = torch.randint(0, 512, (B * H, T), device="cuda", generator=gen)
        rows = pool[torch.arange(B * H, device="cuda")[:, None], pick]
        k = k.mul_(0.1).add_(rows.view(B, H, T, case["dk"]).transpose(1, 2))
    if case["raw"]:          # rows of very different lengths
        q, k = q * normal(*shape, 1).exp(), k * normal(*shape, 1).exp()
    else:
        q, k = _unit(q), _unit(k)
    zb, za, zl = normal(*shape), normal(*shape), normal(*shape)
    if case["gates"] == "trained":
        zb, za, zl = -3.0 + 0.5 * zb, 4.0 + za, -0.8 + 0.5 * zl
    if not case["raw"]:
        zb, za, zl = torch.sigmoid(zb), torch.sigmoid(za), torch.sigmoid(zl)
    t = {"q": q, "k": k, "v": normal(*shape, case["dv"]), "beta": zb, "alpha": za, "lam": zl}
    return {n: x.to(dt).contiguous() for n, x in t.items()}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    s = {"case": case}
    if case["kind"] == "decode":
        B, S, H, dk, dv = (case[n] for n in ("B", "S", "H", "dk", "dv"))
        s["t"] = _tokens(case, gen, (B, H) if case["api"] == "step" else (B, S, H))
        s["state"] = (torch.randn(B, H, dk, dv, device="cuda", generator=gen) * 0.02).to(_DT[case["state"]])
        return s
    B, T, H, dk, dv = (case[n] for n in ("B", "T", "H", "dk", "dv"))
    t = s["t"] = _tokens(case, gen, (B, T, H))
    s["h0"] = torch.randn(B, H, dk, dv, device="cuda", generator=gen) * 0.02 if case["h0"] else None
    if case["kind"] != "prefill":
        s["dO"] = torch.randn(B, T, H, dv, device="cuda", generator=gen).to(t["q"].dtype)
        s["dhT"] = torch.randn(B, H, dk, dv, device="cuda", generator=gen) * 0.02
    if case["kind"] == "autograd":
        s["wanted"] = [x.requires_grad_() for x in t.values()]
        # other layers of the model have run backward before this one
        torch.nn.Linear(8, 8, device="cuda")(torch.ones(8, 8, device="cuda")).sum().backward()
    else:
        # a program that calls with one shape again and again keeps its workspace
        s["ws"] = qd.alloc_workspace(qd.make_shape(t["q"], t["v"], 64), case["kind"] == "train", t["q"].device)
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------------
def run(s):
    case, t = s["case"], s["t"]
    q, k, v, beta, alpha, lam, raw = t["q"], t["k"], t["v"], t["beta"], t["alpha"], t["lam"], case["raw"]
    if case["kind"] == "decode":
        if case["api"] == "step":
            return {"o": qd.recurrent_step(q, k, v, beta, alpha, lam, s["state"]), "state": s["state"]}
        o = qd.recurrent_steps(q, k, v, beta, alpha, lam, s["state"], logits=raw, norm_qk=raw)
        return {"o": o, "state": s["state"]}
    if case["kind"] == "autograd":
        o, hT = qa.qdelta_chunk(q, k, v, beta, alpha, lam, s["h0"], logits=raw, norm_qk=raw)
        grads = torch.autograd.grad((o, hT), s["wanted"], (s["dO"], s["dhT"]))
        return {"o": o.detach(), "hT": hT.detach(), "grads": list(grads)}
    train = case["kind"] == "train"
    o, hT, ws = qd.chunk_fwd(q, k, v, beta, alpha, lam, s["h0"], save_for_bwd=train, workspace=s["ws"], logits=raw,
                             norm_qk=raw)
    if not train:
        return {"o": o, "hT": hT}
    g = qd.chunk_bwd(q, k, v, beta, alpha, lam, s["h0"], s["dO"], s["dhT"], workspace=ws, reuse_fwd=True,
                     want_dh0=case["h0"], logits=raw, norm_qk=raw)
    return {"o": o, "hT": hT, "grads": {n: x for n, x in g.items() if x is not None}}


# ---- what a pass cannot do without, and how exact its results are --------------------------------------------------------
def work(case):
    B, H, dk, dv = (case[n] for n in ("B", "H", "dk", "dv"))
    io = 2 if case["dtype"] == "bf16" else 4
    state = dk * dv * B * H
    if case["kind"] == "decode":
        rows = B * H * case["S"]
        st = 2 if case["state"] == "bf16" else 4
        # read q, k, v and three coefficients, write o; the state is read and written once.  Per token: h^T x, h^T q, k delta^T
        return {"bytes": rows * io * (2 * dk + 2 * dv + 3) + 2 * st * state, "flops": 6.0 * rows * dk * dv}
    # the chunkwise form with 64-token chunks, dense tiles; S: a 64 x 64 x d product per token, M: a 64 x dk x dv product
    C, rows = 64, B * case["T"] * H
    nbytes = rows * io * (2 * dk + 2 * dv + 3) + 4 * state * (2 if case["h0"] else 1)
    flops = rows * (2.0 * C * (3 * dk + 2 * dv) + 6.0 * dk * dv)
    if case["kind"] != "prefill":
        # read q, k, v, dO, the coefficients and dhT (and h0), write dq, dk, dv, three gradients of gates (fp32) and dh0
        co = io if case["kind"] == "autograd" else 4
        nbytes += rows * (io * (2 * dk + 2 * dv + 3) + io * (2 * dk + dv) + 3 * co) + 4 * state * (3 if case["h0"] else 1)
        flops += rows * (2.0 * C * (7 * dk + 4 * dv) + 12.0 * dk * dv)
    return {"bytes": float(nbytes), "flops": flops}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5}                     # fp32 products and sums, another order of summation
    if case["kind"] == "decode":
        # fp32 arithmetic on the state; o (and a bf16 state) is rounded once, where a last bit may fall the other way
        return {"rel": 1e-3, "max": 1.6e-2}
    # bf16 operands of the products, fp32 accumulation: gradients of gates are up to 5e-3 off the exact ones, so two
    # correct implementations differ by up to 7e-3 on a typical tensor
    return {"rel": 1.2e-2, "max": 0.5}
