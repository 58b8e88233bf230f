"""`torch.autograd` front-end of the chunkwise kernels: marshalling only.

    o, hT = qdelta_chunk(q, k, v, beta, alpha, lam, h0, logits=False, norm_qk=False)

q, k [B,T,H,dk], v [B,T,H,dv], beta/alpha/lam [B,T,H] (alpha, lam, h0 may be None), all CUDA tensors; returns the
outputs o [B,T,H,dv] and the final state hT [B,H,dk,dv] (fp32), both differentiable.  The forward runs
`qdelta_chunk_fwd` saving what the backward needs in a workspace that the autograd node keeps; the backward runs
`qdelta_chunk_bwd` on that workspace; the node itself is native (host/host.cpp).  Every number is computed by the library's CUDA kernels.
"""
from . import binding as qd


def qdelta_chunk(q, k, v, beta, alpha=None, lam=None, h0=None, logits=False, norm_qk=False):
    """Differentiable chunkwise Q-Delta: returns (o, hT)."""
    flags = (qd.QD_COEF_LOGITS if logits else 0) | (qd.QD_NORM_QK if norm_qk else 0)
    return qd._host().chunk_autograd(q, k, v, beta, alpha, lam, h0, flags)
