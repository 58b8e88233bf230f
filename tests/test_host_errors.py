"""What goes wrong inside torch on the native host path keeps its Python exception type."""
import pytest
import torch


def test_index_error_of_torch_stays_one():
    from paper_2606_08804_b200 import binding as qd
    z = torch.zeros(1, 2, 64)
    with pytest.raises(IndexError):                  # v without dimensions: torch refuses to give its last one
        qd.recurrent_step(z, z, torch.tensor(0.0), None, None, None, None)


def _inputs(T, H, requires_grad=False):
    g = torch.Generator(device="cuda").manual_seed(5)
    n = lambda *s: torch.randn(*s, device="cuda", generator=g)
    unit = lambda x: torch.nn.functional.normalize(x, dim=-1)
    t = [unit(n(1, T, H, 128)), unit(n(1, T, H, 128)), n(1, T, H, 128)] + [n(1, T, H).sigmoid() for _ in range(3)]
    return [x.bfloat16().requires_grad_(requires_grad) for x in t]


@pytest.mark.gpu
@pytest.mark.parametrize("entry", ["chunk_fwd", "qdelta_chunk", "recurrent_steps"])
def test_out_of_memory_can_be_caught_as_such(entry):
    from paper_2606_08804_b200 import autograd as qa
    from paper_2606_08804_b200 import binding as qd
    t = _inputs(4096, 16, requires_grad=entry == "qdelta_chunk")
    state = torch.zeros(1, 16, 128, 128, device="cuda")
    call = {"chunk_fwd": lambda: qd.chunk_fwd(*t, save_for_bwd=True), "qdelta_chunk": lambda: qa.qdelta_chunk(*t),
            "recurrent_steps": lambda: qd.recurrent_steps(*t, state)}[entry]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # the allocator of this process may hold 2 MB more than it does now: less than the output (16 MB) or the workspace takes
    limit = torch.cuda.memory_reserved() + (2 << 20)
    torch.cuda.set_per_process_memory_fraction(limit / torch.cuda.get_device_properties(0).total_memory)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            call()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    call()
    torch.cuda.synchronize()


@pytest.mark.gpu
def test_exception_of_a_saved_tensor_hook_stays_one():
    from paper_2606_08804_b200 import autograd as qa

    class Stop(Exception):
        pass

    def pack(x):
        raise Stop

    t = _inputs(64, 1, requires_grad=True)
    with torch.autograd.graph.saved_tensors_hooks(pack, lambda x: x), pytest.raises(Stop):
        qa.qdelta_chunk(*t)


@pytest.mark.gpu
def test_checkpointed_call_recomputes_its_forward():
    from torch.utils.checkpoint import checkpoint
    from paper_2606_08804_b200 import autograd as qa
    t = _inputs(130, 2, requires_grad=True)
    o, _ = qa.qdelta_chunk(*t)
    want = torch.autograd.grad(o.float().sum(), t)
    o, _ = checkpoint(qa.qdelta_chunk, *t, use_reentrant=False)
    for x, y in zip(torch.autograd.grad(o.float().sum(), t), want):
        assert torch.equal(x, y)


@pytest.mark.gpu
@pytest.mark.parametrize("change,says", [
    (lambda x: x.cpu(), "contiguous CUDA tensor"),
    (lambda x: x.cpu() if x.dtype == torch.uint8 else x, "contiguous CUDA tensor"),        # the workspace
    (lambda x: x.float() if x.dim() == 4 else x, "dtype"),
    (lambda x: x[:, :1].contiguous() if x.dim() == 3 else x, "shape"),
    (lambda x: x.transpose(1, 2).contiguous().transpose(1, 2) if x.dim() == 4 else x, "contiguous CUDA tensor"),
])
def test_saved_tensors_that_come_back_changed_are_refused(change, says):
    from paper_2606_08804_b200 import autograd as qa
    from paper_2606_08804_b200 import binding as qd
    t = _inputs(130, 2, requires_grad=True)
    with torch.autograd.graph.saved_tensors_hooks(lambda x: x, change):
        o, _ = qa.qdelta_chunk(*t)
    with pytest.raises(qd.QdeltaError, match=says):
        o.float().sum().backward()
    torch.cuda.synchronize()


@pytest.mark.gpu
def test_saved_tensors_kept_on_the_host_give_the_same_gradients():
    from paper_2606_08804_b200 import autograd as qa
    t = _inputs(130, 2, requires_grad=True)
    want = torch.autograd.grad(qa.qdelta_chunk(*t)[0].float().sum(), t)
    with torch.autograd.graph.save_on_cpu():
        o, _ = qa.qdelta_chunk(*t)
    for x, y in zip(torch.autograd.grad(o.float().sum(), t), want):
        assert torch.equal(x, y)
