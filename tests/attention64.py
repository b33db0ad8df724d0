"""Block-sparse attention in float64 on the GPU, over the lists a layer's own selection wrote."""
import numpy as np
import torch


def attention64(layer, h):
    """Output [N, 64] of head h of a gpu_harness.Layer."""
    rp, ci = layer.csr()
    keep = np.zeros((layer.nq, layer.nb), bool)
    for i in range(layer.nq):
        at = h * layer.nq + i
        keep[i, ci[rp[at]:rp[at + 1]]] = True
    t = torch.arange(layer.N, device="cuda")
    keep = torch.from_numpy(keep).cuda()[t // layer.q_block][:, t // 64]
    q, k, v = (x[:, h].double() for x in (layer.Q, layer.K, layer.V))
    # the last channel apart: huge numbers in it must not meet the others' rounding
    s = (q[:, :63] @ k[:, :63].T + q[:, 63:] * k[:, 63]) / 8.0
    return torch.softmax(s.masked_fill(~keep, -float("inf")), dim=1) @ v


def errors(layer):
    """Of the layer's bf16 output: the largest error beyond the rounding to bf16 (2^-8 of the
    value), and sum |error| / sum |value|."""
    err = size = worst = 0.0
    for h in range(layer.H):
        want = attention64(layer, h)
        assert bool(torch.isfinite(want).all())
        diff = (layer.buf.O[:, h].double() - want).abs()
        worst = max(worst, float((diff - 2.0 ** -8 * want.abs()).max()))
        err, size = err + float(diff.sum()), size + float(want.abs().sum())
    return worst, err / size
