"""Kept-block lists at the edges of the two ways the CSR kernel writes them (word by word for
short or dense lists, lane by lane for long sparse ones): one mask word, a word with one block,
32 and 33 words, sparse and dense budgets beside dense (special) rows.  Every row lists exactly the
blocks outside its best drop set, ascending; in a forward, every attention item's list is the
union of its rows' lists with the rows' bits."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,ns,c", [
    (64 * 31, 0, 4), (64 * 32 + 1, 1, 30), (64 * 64, 70, 2),
    (64 * 1024 - 9, 3, 60), (64 * 1025, 130, 60), (64 * 1025, 130, 700),
])
@pytest.mark.parametrize("q_block", [64, 128])
def test_lists(N, ns, c, q_block):
    inp = synth.make_random_layer(N, 1, 64, seed=N + c)
    layer = G.Layer(inp, ns, [c], 1, q_block=q_block).run_forward()
    b = layer.buf  # the forward once more: run_forward's last call lists adjacent rows
    layer.ress.forward(layer.d, layer.Q, layer.K, layer.V, b.F, layer.c_h, 1, layer.rho, b.ws,
                       b.row_ptr, b.col_idx, b.O, b.J_best)
    layer.ress.status(b.ws)
    kept = ~layer.drop_sets()
    kept[:, layer.nqc:] = True  # special query rows attend densely
    rows = layer.kept()
    for i in range(layer.nq):
        assert np.array_equal(rows[(0, i)], np.flatnonzero(kept[0, i])), i
    L = b.layout
    items = -(-layer.nb // 2)
    plen = b.ws_view("plen", torch.int32, (items,)).cpu().numpy()
    plist = b.ws_view("t", torch.int32, (layer.nq * L.ld,)).cpu().numpy()
    prow = b.ws_view("prow", torch.int32, (items,)).cpu().numpy()
    rp = b.row_ptr.cpu().numpy()
    for u in range(items):
        if q_block == 128:
            a = z = u
        elif u < layer.nqc // 2:
            a, z = prow[u] & 0xffff, prow[u] >> 16
        else:
            a, z = 2 * u, 2 * u + 1
        first = kept[0, a]
        second = kept[0, z] if z < layer.nq else np.zeros_like(first)
        at = rp[u if q_block == 128 else 2 * u]
        got = plist[at:at + plen[u]]
        want = {int(j): int(first[j]) | int(second[j]) << 1 for j in np.flatnonzero(first | second)}
        assert len(got) == len(want) and {int(e) & 0xffff: int(e) >> 16 for e in got} == want, u
