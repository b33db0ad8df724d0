"""Forwards of small layers, whose attention items are shared by up to 4 CTAs each, dense ones by
more than sparse ones where that shortens the longest share: output against the oracle on every
row, and the host-buffer forward's bits.  The item counts put the layers on each side of the
lines between the ways to share on 152 SMs; budgets of one block leave some CTAs without
entries."""
import pytest

import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,ns,c", [
    (64 * 16, 1, 0, 1),        # 8 items, lists of one or two blocks for 4 CTAs
    (64 * 15 + 1, 2, 3, 5),    # 16 blocks, one token in the last
    (64 * 50 + 30, 3, 35, 9),  # 78 items: 3 CTAs each; two dense blocks
    (64 * 38, 4, 0, 38),       # 76 items: 4 CTAs each, nothing dropped
    (64 * 100 - 7, 3, 0, 2),   # 150 items: 2 CTAs each
    (64 * 77 + 38, 3, 37, 31),  # 117 items: 4 CTAs for the dense ones, 2 for the others
    (64 * 130, 3, 70, 7),      # 195 items: 2 CTAs for the dense ones, one for the others
    (64 * 205, 3, 10, 12),     # 309 items: more than one wave, whole items
])
def test_split_items(N, H, ns, c):
    inp = synth.make_random_layer(N, H, 64 * H, seed=N + H)
    layer = G.Layer(inp, ns, [c] * H, 1).run_forward()
    rows = [(h, i) for h in range(H) for i in range(layer.nq)]
    r = G.compare_attention_bf16(layer, rows)
    assert r["max_abs"] <= G.ATT_MAX_ABS and r["mean_rel"] <= G.ATT_MEAN_REL, r
    b = layer.buf
    want = b.O.clone()
    host = [t.cpu().pin_memory() for t in (layer.Q, layer.K, layer.V)]
    out = torch.empty(N, H, 64, dtype=torch.bfloat16).pin_memory()
    layer.ress.forward_host(layer.d, *host, out, layer.Q, layer.K, layer.V, b.O, b.F, layer.c_h, 1,
                            layer.rho, b.ws, b.row_ptr, b.col_idx, b.J_best)
    torch.cuda.current_stream().synchronize()
    assert torch.equal(out.view(torch.int16), want.cpu().view(torch.int16))
