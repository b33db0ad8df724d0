"""Calls that follow one another in a stream without a synchronisation, each reading what the
one before wrote while the two overlap: the three separate calls of a layer, with fixed and with
variable list lengths, and layers that take the output of the call before as their input.
The results are those of the same calls with a synchronisation between them."""
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,q_block,cdf", [(64 * 41 + 9, 3, 64, 0.0), (64 * 41 + 9, 3, 128, 0.0),
                                             (64 * 150, 4, 64, 0.0), (64 * 60 + 5, 2, 64, 0.9)])
def test_score_restore_attention(N, H, q_block, cdf):
    layers = []
    for seed in (1, 2):
        inp = synth.make_random_layer(N, H, 64 * H, seed=seed)
        layers.append(G.Layer(inp, 11, [9] * H, 0 if cdf else 2, q_block=q_block,
                              variant=O.Variant(cdf=cdf) if cdf else None))
    r, first, b = layers[0].ress, layers[0], layers[0].buf
    v = first.device_variant()
    r.prepare_wo(first.d, first.W, b.F)

    def run(layer, sync):
        calls = (lambda: r.score(first.d, layer.Q, layer.K, layer.V, b.F, first.c_h, b.ws, variant=v),
                 lambda: r.restore(first.d, first.c_h, first.rounds, first.rho, b.ws, b.row_ptr,
                                   b.col_idx, b.J_best, variant=v),
                 lambda: r.sparse_attn(first.d, layer.Q, layer.K, layer.V, b.row_ptr, b.col_idx, b.O,
                                       b.ws))
        for call in calls:
            call()
            if sync:
                torch.cuda.synchronize()
        n = b.row_ptr[-1:].clone()
        return [t.clone() for t in (b.O, b.row_ptr, b.col_idx, b.J_best)], n

    want = [run(x, True) for x in layers]
    got = [run(layers[k], False) for k in (0, 1, 0, 1)]  # lists and outputs differ from call to call
    torch.cuda.synchronize()
    r.status(b.ws)
    for k, (res, n) in enumerate(got):
        ref, count = want[k % 2]
        assert int(n) == int(count)
        for i, (x, y) in enumerate(zip(res, ref)):
            m = int(n) if i == 2 else x.numel()  # the lists' capacity may be larger
            assert torch.equal(x.reshape(-1)[:m], y.reshape(-1)[:m]), (k, i)


@pytest.mark.parametrize("q_block", [64, 128])
def test_layers_that_read_the_output_before(q_block):
    N, H = 64 * 90 + 17, 4
    inp = synth.make_random_layer(N, H, 64 * H, seed=4)
    layer = G.Layer(inp, 30, [12] * H, 1, q_block=q_block)
    r, b = layer.ress, layer.buf
    r.prepare_wo(layer.d, layer.W, b.F)

    def chain(sync):
        x = [layer.Q, layer.K, layer.V]
        outs = [torch.empty_like(layer.Q) for _ in range(6)]
        for k, o in enumerate(outs):
            if k % 2:  # a residual update between the layers
                r.out_proj(layer.d, x[0], layer.W, x[1].view(N, -1), o.view(N, -1), b.ws)
            else:
                r.forward(layer.d, *x, b.F, layer.c_h, layer.rounds, layer.rho, b.ws, b.row_ptr,
                          b.col_idx, o, b.J_best)
            if sync:
                torch.cuda.synchronize()
            x = [o] + x[:2]
        return outs

    want = chain(True)
    for _ in range(3):
        got = chain(False)
        torch.cuda.synchronize()
        r.status(b.ws)
        assert all(torch.equal(p.view(torch.int16), q.view(torch.int16)) for p, q in zip(got, want))
