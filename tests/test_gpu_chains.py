"""The state chains at the edges of their split: 74 sequences (two CTAs each) and 75 (one), one and a few chunks, ragged ends."""
from dataclasses import replace

import pytest

from paper_2606_08804_b200 import inputs as gen
from test_gpu_chunk import _bwd_check, _fwd_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,T", [(2, 37, 65), (3, 25, 65), (1, 4, 33), (1, 2, 64 * 7 + 1), (5, 15, 64 * 5)])
def test_chain_split(B, H, T):
    cfg = replace(gen.CONFIGS["cfg2"], B=B, H=H, T=T, regime="trained_like", seed=227)
    d = gen.make_chunk_inputs(cfg)
    _fwd_check(cfg, d)
    _fwd_check(cfg, d, save=True)
    _bwd_check(cfg, d, reuse=True)
    _bwd_check(cfg, d)
