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


@pytest.mark.parametrize("B,H,T", [(1, 64, 65), (5, 13, 65), (3, 43, 129)])
def test_chunk_order(B, H, T):
    """Work items of the chunk backward: one group of 64 sequences, a second one of one, three; taken from a counter, so a second
    backward over the same forward has to find it at zero again."""
    import torch

    from gpu_util import dev_inputs
    from paper_2606_08804_b200 import binding as qd

    cfg = replace(gen.CONFIGS["cfg2"], B=B, H=H, T=T, regime="trained_like", seed=331)
    d = gen.make_chunk_inputs(cfg)
    _bwd_check(cfg, d, reuse=True)
    t = dev_inputs(d, cfg.dtype)
    a = [t[n] for n in ("q", "k", "v", "beta", "alpha", "lam", "h0")]
    _, _, ws = qd.chunk_fwd(*a, save_for_bwd=True)
    first, second = (qd.chunk_bwd(*a, t["dO"], t["dhT"], workspace=ws, reuse_fwd=True) for _ in range(2))
    for n, x in first.items():
        assert x is None or torch.equal(x, second[n]), n


@pytest.mark.parametrize("T", [1, 63, 64, 66, 129])
def test_preparation_edges(T):
    """One chunk of one token, one short of a whole chunk, whole, a second one of two tokens, a third of one."""
    cfg = replace(gen.CONFIGS["cfg2"], B=1, H=3, T=T, regime="trained_like", seed=401 + T)
    d = gen.make_chunk_inputs(cfg)
    _fwd_check(cfg, d)
    _bwd_check(cfg, d, reuse=True)


@pytest.mark.parametrize("T", [64 * 2, 64 * 3, 64 * 3 + 1, 64 * 4 - 1, 64 * 6 + 17])
@pytest.mark.parametrize("without", ["", "alpha lam", "h0"])
def test_half_chain_edges(T, without):
    """Two CTAs to a sequence, their tiles three deep: as many chunks as that, one fewer, one more, twice around; without a forget gate (one
    copy of Delta^T instead of two); normalised in the kernels too; and a prompt has the bits of a forward with saves."""
    import torch

    import gpu_util as gu
    from gpu_util import dev_inputs
    from oracle import recurrence as orc
    from paper_2606_08804_b200 import binding as qd

    cfg = replace(gen.CONFIGS["cfg2"], B=2, H=3, T=T, regime="trained_like", seed=419 + T)
    d = gen.make_chunk_inputs(cfg)
    for n in without.split():
        d[n] = None
    _fwd_check(cfg, d, save=True)
    _bwd_check(cfg, d, reuse=True)
    t = dev_inputs(d, cfg.dtype)
    a = [t[n] for n in ("q", "k", "v", "beta", "alpha", "lam", "h0")]
    for norm in (False, True):
        (o, hT, _), (p, hP, _) = (qd.chunk_fwd(*a, save_for_bwd=s, norm_qk=norm) for s in (True, False))
        assert torch.equal(o, p) and torch.equal(hT, hP)
        if norm:
            ro, rh = orc.forward_fused(*(d[n] for n in ("q", "k", "v", "beta", "alpha", "lam", "h0")), norm_qk=True)
            gu.check("half chain norm", "o", o, ro, cfg.dtype)
            gu.check("half chain norm", "hT", hT, rh, cfg.dtype, state=True)


@pytest.mark.parametrize("T", [64, 64 * 3 + 1, 64 * 7 - 1])
@pytest.mark.parametrize("norm", [False, True])
def test_half_and_whole_chain_have_the_same_bits(T, norm):
    """74 sequences take two CTAs each, 75 one: what the first 74 of 75 come to does not depend on it, prompts, saves and gradients."""
    import torch

    from gpu_util import dev_inputs
    from paper_2606_08804_b200 import binding as qd

    cfg = replace(gen.CONFIGS["cfg2"], B=75, H=1, T=T, regime="trained_like", seed=617 + T)
    t = dev_inputs(gen.make_chunk_inputs(cfg), cfg.dtype)

    def run(B):
        a = [t[n][:B].contiguous() for n in ("q", "k", "v", "beta", "alpha", "lam", "h0")]
        p, hP, _ = qd.chunk_fwd(*a, save_for_bwd=False, norm_qk=norm)
        o, hT, ws = qd.chunk_fwd(*a, save_for_bwd=True, norm_qk=norm)
        g = qd.chunk_bwd(*a, t["dO"][:B].contiguous(), t["dhT"][:B].contiguous(), workspace=ws, reuse_fwd=True, want_dh0=True, norm_qk=norm)
        assert qd.workspace_status(ws) == 0
        return [p, hP, o, hT] + [x for x in g.values() if x is not None]
    half, whole = run(74), run(75)
    assert len(half) == len(whole) > 10
    for x, y in zip(half, whole):
        assert torch.equal(x, y[:74])


@pytest.mark.parametrize("B,H,T,parts", [(1, 16, 64 * 64, (2, 2)), (2, 20, 64 * 64 + 1, (2, 1)), (1, 4, 64 * 256, (3, 2)),
                                         (1, 1, 64 * 1024 - 63, (3, 2)), (1, 40, 64 * 120 - 1, (2, 2)), (2, 2, 64 * 64, (1, 2)),
                                         (2, 8, 64 * 128 - 5, (2, 3)), (1, 36, 64 * 128, (2, 3)), (1, 32, 64 * 256 + 1, (3, 3))])
def test_in_parts(B, H, T, parts):
    """Long, few sequences are taken in `parts` (forward, backward), unless the kernels are timed one by one: the same bits either way,
    with the state passed on through h_T and (none asked for) through the workspace, replayed from a graph, and close to the oracle."""
    import torch

    from gpu_util import dev_inputs
    from paper_2606_08804_b200 import binding as qd

    cfg = replace(gen.CONFIGS["cfg2"], B=B, H=H, T=T, regime="trained_like", seed=347)
    d = gen.make_chunk_inputs(cfg)
    _fwd_check(cfg, d, pairs=[(0, 0), (B - 1, H - 1)])
    _bwd_check(cfg, d, pairs=[(0, 0), (B - 1, H - 1)], reuse=True)
    t = dev_inputs(d, cfg.dtype)
    a = [t[n] for n in ("q", "k", "v", "beta", "alpha", "lam", "h0")]
    shape = qd.make_shape(t["q"], t["v"], 64)

    def call(logits, norm, save, hT):
        o, h, ws = qd.chunk_fwd(*a, save_for_bwd=save, want_hT=hT, logits=logits, norm_qk=norm)
        g = qd.chunk_bwd(*a, t["dO"], t["dhT"], workspace=ws, reuse_fwd=True, logits=logits, norm_qk=norm) if save else {}
        r = qd.chunk_bwd(*a, t["dO"], t["dhT"], logits=logits, norm_qk=norm) if save else {}
        assert qd.workspace_status(ws) == 0
        return [x for x in (o, h, *g.values(), *r.values()) if x is not None]

    cases = [(False, False, False, True), (False, False, True, True), (False, False, True, False), (True, True, True, True)]
    assert (qd.chunk_parts(shape, False), qd.chunk_parts(shape, True)) == parts
    results = [call(*c) for c in cases]
    for c, x, y in zip(cases, results, _in_one_part(shape, lambda: [call(*c) for c in cases])):
        assert len(x) == len(y) and all(torch.equal(i, j) for i, j in zip(x, y)), c

    o, hT, ws = qd.chunk_fwd(*a, save_for_bwd=True)
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        qd.chunk_fwd(*a, save_for_bwd=True, workspace=ws, o=o, hT=hT)
        g = qd.chunk_bwd(*a, t["dO"], t["dhT"], workspace=ws, reuse_fwd=True)
    o.zero_(), hT.zero_()
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    for x, y in zip((o, hT, *g.values()), results[1]):
        assert torch.equal(x, y)


def _in_one_part(shape, f):
    """f() with the kernels timed one by one, which takes one part."""
    from paper_2606_08804_b200 import binding as qd

    qd.profile_enable(True)
    try:
        assert (qd.chunk_parts(shape, False), qd.chunk_parts(shape, True)) == (1, 1)
        return f()
    finally:
        qd.profile_enable(False)
        qd.profile_read(reset=True)


@pytest.mark.parametrize("without", ["h0", "dhT", "dh0", "h0 dhT dh0", "alpha", "lam", "alpha lam", "alpha lam h0 dhT dh0"])
@pytest.mark.parametrize("B,H,T", [(1, 16, 64 * 128 - 5), (3, 4, 64 * 256)])
def test_in_parts_without(B, H, T, without):
    """Inputs that a call may leave out, and dh0 not asked for, in two and three parts: the bits of one part; and h_T in h0's place."""
    import torch

    from gpu_util import dev_inputs
    from paper_2606_08804_b200 import binding as qd

    cfg = replace(gen.CONFIGS["cfg2"], B=B, H=H, T=T, regime="alpha_slow", seed=353)
    d = gen.make_chunk_inputs(cfg)
    for n in without.split():
        d[n] = None
    t = dev_inputs(d, cfg.dtype)
    a = [t[n] for n in ("q", "k", "v", "beta", "alpha", "lam")]
    shape, want = qd.make_shape(t["q"], t["v"], 64), "dh0" not in without.split()
    assert (qd.chunk_parts(shape, False), qd.chunk_parts(shape, True)) == (2 if T < 64 * 255 else 3, 3)

    def call():
        r = []
        for save in (False, True):
            o, hT, ws = qd.chunk_fwd(*a, t["h0"], save_for_bwd=save)
            r += [o, hT]
        for kw in (dict(workspace=ws, reuse_fwd=True), {}):
            # gradients of coefficients that are absent, on request
            out = {n: torch.full((B, T, H), float("nan"), device="cuda") for n, x in (("dalpha", t["alpha"]), ("dlam", t["lam"])) if x is None}
            for o in ({}, out) if out else ({},):
                g = qd.chunk_bwd(*a, t["h0"], t["dO"], t["dhT"], want_dh0=want, out=dict(o), **kw)
                assert (g["dh0"] is not None) == want
                r += [x for x in g.values() if x is not None]
        if t["h0"] is not None:
            state = t["h0"].clone()
            o, _, ws = qd.chunk_fwd(*a, state, hT=state)
            r += [o, state]
        assert qd.workspace_status(ws) == 0
        return r

    x, y = call(), _in_one_part(shape, call)
    assert len(x) == len(y) and all(torch.equal(i, j) for i, j in zip(x, y))


@pytest.mark.parametrize("B,H,T", [(1, 16, 64 * 128), (1, 4, 64 * 256 - 1)])
def test_in_parts_between_other_kernels(B, H, T):
    """Kernels that write the inputs right before the calls, and overwrite them and the outputs' copies right after, in one stream: the
    preparation and the chunk backward of a part, which do not wait for the chain before them, are ordered with both."""
    import torch

    from gpu_util import dev_inputs
    from paper_2606_08804_b200 import binding as qd

    cfg = replace(gen.CONFIGS["cfg2"], B=B, H=H, T=T, regime="trained_like", seed=359)
    t = dev_inputs(gen.make_chunk_inputs(cfg), cfg.dtype)
    names = ("q", "k", "v", "beta", "alpha", "lam", "h0", "dO", "dhT")
    shape = qd.make_shape(t["q"], t["v"], 64)
    assert qd.chunk_parts(shape, True) > 1

    def pair(x, ws, o, hT, g):
        qd.chunk_fwd(*(x[n] for n in names[:7]), save_for_bwd=True, workspace=ws, o=o, hT=hT)
        qd.chunk_bwd(*(x[n] for n in names[:7]), x["dO"], x["dhT"], workspace=ws, reuse_fwd=True, out=g)

    want = [None, None, {}]
    want[0], want[1], ws = qd.chunk_fwd(*(t[n] for n in names[:7]), save_for_bwd=True)
    want[2] = qd.chunk_bwd(*(t[n] for n in names[:7]), t["dO"], t["dhT"], workspace=ws, reuse_fwd=True)
    o, hT, g = torch.empty_like(want[0]), torch.empty_like(want[1]), {n: torch.empty_like(x) for n, x in want[2].items()}
    outs = [o, hT, *g.values()]
    x = {n: torch.full_like(t[n], float("nan")) for n in names}
    copies = [[] for _ in range(3)]
    for c in copies:
        for n in names:
            x[n].copy_(t[n])                              # the producers
        pair(x, ws, o, hT, g)
        for n in names:
            x[n].fill_(float("nan"))                      # the next user of the buffers
        for y in outs:
            c.append(y.clone())
            y.fill_(float("nan"))
    torch.cuda.synchronize()
    assert qd.workspace_status(ws) == 0
    for c in copies:
        assert all(torch.equal(i, j) for i, j in zip(c, [want[0], want[1], *want[2].values()]))


def test_in_parts_on_two_streams():
    """Two calls in parts at a time, each on its own stream, thread and workspace, with a decode on a third: the bits of one after the other."""
    import threading

    import torch

    from gpu_util import dev_inputs
    from paper_2606_08804_b200 import binding as qd

    work = []
    for H, T, seed in ((16, 64 * 128 - 5, 367), (4, 64 * 256, 373)):
        t = dev_inputs(gen.make_chunk_inputs(replace(gen.CONFIGS["cfg2"], B=1, H=H, T=T, regime="trained_like", seed=seed)), "bf16")
        a = [t[n] for n in ("q", "k", "v", "beta", "alpha", "lam", "h0")]
        ws = qd.alloc_workspace(qd.make_shape(t["q"], t["v"], 64), True, "cuda")
        assert qd.chunk_parts(qd.make_shape(t["q"], t["v"], 64), True) > 1

        def pair(a=a, t=t, ws=ws):
            o, hT, _ = qd.chunk_fwd(*a, save_for_bwd=True, workspace=ws)
            return [o, hT, *qd.chunk_bwd(*a, t["dO"], t["dhT"], workspace=ws, reuse_fwd=True).values()]

        work.append(pair)
    x = [y[:, 0].contiguous() for y in a[:6]]
    work.append(lambda: [qd.recurrent_step(*x, t["h0"].clone())])
    want = [f() for f in work]
    torch.cuda.synchronize()
    got, errors = [[] for _ in work], []

    def run(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(6):
                    got[i].append(work[i]())
                torch.cuda.current_stream().synchronize()
        except Exception as e:          # noqa: BLE001 -- told to the test below
            errors.append(e)

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(work))]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
    for w, rounds in zip(want, got):
        assert len(rounds) == 6 and all(torch.equal(p, q) for r in rounds for p, q in zip(r, w))
