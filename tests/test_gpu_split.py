"""The fp32-accurate kernels at the edges of their dispatch: both slice widths of the state chains, every head-dimension
pair, ragged last chunks, against the oracle."""
from dataclasses import replace

import pytest

from paper_2606_08804_b200 import inputs as gen
from test_gpu_chunk import _bwd_check, _fwd_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,B,H,T,dk,dv", [
    ("f32", 4, 15, 65, 64, 64),       # 120 slices of 32 columns: the wide slices, one token in the last chunk
    ("f32", 7, 17, 63, 64, 64),       # 119: narrow slices, one short chunk
    ("f32", 2, 15, 130, 128, 128),    # wide slices, both head dimensions 128
    ("f32", 1, 3, 129, 128, 128),
    ("bf16", 4, 15, 100, 64, 64),
    ("bf16", 1, 2, 1, 64, 64),
    ("bf16", 5, 12, 70, 128, 64),
    ("bf16", 3, 10, 127, 64, 128),
])
def test_split_kernels(dtype, B, H, T, dk, dv):
    base = gen.CONFIGS["cfg2"] if dtype == "bf16" else replace(gen.CONFIGS["cfg0"], h0=True, backward=True)
    cfg = replace(base, B=B, H=H, T=T, dk=dk, dv=dv, regime="alpha_slow", seed=211)
    d = gen.make_chunk_inputs(cfg)
    _fwd_check(cfg, d)
    _bwd_check(cfg, d)
    _bwd_check(cfg, d, reuse=True)
