"""The fp32-accurate kernels at the edges of their dispatch: both slice widths of the state chains, every head-dimension
pair, ragged last chunks, against the oracle."""
from dataclasses import replace

import numpy as np
import pytest

import gpu_util as gu
from paper_2606_08804_b200 import inputs as gen
from test_gpu_chunk import _bwd_check, _fwd_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,B,H,T,dk,dv", [
    ("f32", 4, 15, 65, 64, 64),       # wide slices (32 columns), one token in the last chunk
    ("f32", 7, 17, 63, 64, 64),       # wide slices, one short chunk
    ("f32", 2, 15, 130, 128, 128),    # wide slices, both head dimensions 128
    ("f32", 1, 3, 129, 128, 128),     # narrow slices (16 columns)
    ("bf16", 4, 15, 100, 64, 64),
    ("bf16", 1, 2, 1, 64, 64),
    ("bf16", 5, 12, 70, 128, 64),
    ("bf16", 3, 10, 127, 64, 128),
    ("bf16", 2, 37, 65, 64, 64),      # 148 CTAs of the state chains: copies by warps of their own
    ("bf16", 3, 25, 65, 64, 64),      # 150: by everybody
    ("bf16", 3, 25, 130, 128, 64),
])
def test_split_kernels(dtype, B, H, T, dk, dv):
    base = gen.CONFIGS["cfg2"] if dtype == "bf16" else replace(gen.CONFIGS["cfg0"], h0=True, backward=True)
    cfg = replace(base, B=B, H=H, T=T, dk=dk, dv=dv, regime="alpha_slow", seed=211)
    d = gen.make_chunk_inputs(cfg)
    _fwd_check(cfg, d)
    _bwd_check(cfg, d)
    _bwd_check(cfg, d, reuse=True)


@pytest.mark.parametrize("H", [37, 38])      # sequences of d_v = 64: 148 narrow slices, and the first number that takes wide ones
@pytest.mark.parametrize("dtype,dk,dv", [("f32", 64, 64), ("f32", 128, 128), ("bf16", 64, 64), ("bf16", 128, 64), ("bf16", 64, 128)])
def test_edge_between_narrow_and_wide_slices(dtype, dk, dv, H):
    base = gen.CONFIGS["cfg2"] if dtype == "bf16" else replace(gen.CONFIGS["cfg0"], h0=True, backward=True)
    H = H if dv == 64 else H // 2            # 18 and 19 of d_v = 128
    cfg = replace(base, B=1, H=H, T=129, dk=dk, dv=dv, regime="alpha_slow", seed=229)
    d = gen.make_chunk_inputs(cfg)
    _fwd_check(cfg, d)
    _bwd_check(cfg, d)


@pytest.mark.parametrize("T,dk,dv,logits", [(97, 64, 64, False), (64, 128, 64, True), (65, 64, 128, False)])
def test_split_kernels_normalise(T, dk, dv, logits):
    # bf16 with d_k or d_v = 64, q and k normalised in the kernels (their own branch of the chunk backward)
    from oracle import recurrence as orc
    from paper_2606_08804_b200 import binding as qd
    cfg = replace(gen.CONFIGS["cfg2"], B=2, H=3, T=T, dk=dk, dv=dv, regime="alpha_slow", seed=223)
    d = gen.make_chunk_inputs(cfg)
    r = np.random.default_rng(13)
    rnd = lambda x: gen.round_bf16(x.astype(np.float32))
    for n in ("q", "k"):
        d[n] = rnd(d[n] * np.exp(r.normal(0.0, 1.0, d[n].shape[:-1] + (1,))))
    if logits:
        shp = (cfg.B, cfg.T, cfg.H)
        d["beta"], d["alpha"], d["lam"] = rnd(r.normal(0.0, 1.5, shp)), rnd(r.normal(3.0, 1.5, shp)), rnd(r.normal(-0.8, 1.0, shp))
    t = gu.dev_inputs(d, cfg.dtype)
    args = (d["q"], d["k"], d["v"], d["beta"], d["alpha"], d["lam"], d["h0"])
    ro, rh = orc.forward_fused(*args, logits=logits, norm_qk=True)
    ref = orc.backward_fused(*args, d["dO"], d["dhT"], logits=logits, norm_qk=True)
    dev = [t[n] for n in ("q", "k", "v", "beta", "alpha", "lam", "h0")]
    o, hT, ws = qd.chunk_fwd(*dev, save_for_bwd=True, logits=logits, norm_qk=True)
    g = qd.chunk_bwd(*dev, t["dO"], t["dhT"], workspace=ws, reuse_fwd=True, logits=logits, norm_qk=True)
    gu.check("split norm", "o", o, ro, cfg.dtype)
    gu.check("split norm", "hT", hT, rh, cfg.dtype, state=True)
    for n in ("dq", "dk", "dv", "dbeta", "dalpha", "dlam", "dh0"):
        gu.check("split norm", n, g[n], ref[n], cfg.dtype, state=(n == "dh0"))
