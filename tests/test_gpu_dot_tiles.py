"""Row-by-block products at the edges of their tiles and of a CTA's run of tiles: one tile, one
block or row more than a tile, fewer and more tiles than SMs (a run then crosses stripes of rows
and heads), and rounds in which some heads swap nothing.  Same acceptance rules as the other
selection tests."""
import pytest

import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,ns,c,R,q_block", [
    (64 * 128, 0, (13,), 1, 64),                       # one tile
    (64 * 129, 0, (13, 1), 2, 64),                     # a row and a block more; head 1 swaps nothing
    (64 * 260 + 1, 65, (1, 1), 1, 128),                # no head swaps
    (64 * 520 + 33, 7, (1, 40, 2, 60, 3, 52) * 2, 2, 128),   # 180 tiles for 152 SMs, gaps
    (64 * 385, 0, (20, 1, 38) * 4, 2, 128),            # 96 tiles; 64 or 32 in a round
])
def test_tiles(N, ns, c, R, q_block):
    H = len(c)
    inp = synth.make_random_layer(N, H, 64 * H, seed=N + H)
    layer = G.Layer(inp, ns, list(c), R, q_block=q_block).run(attention=False)
    G.check_selection(G.compare_selection(layer, layer.oracle_select()))
