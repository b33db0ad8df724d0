"""The pooled map's product summed as ranges of 64-block chunks: the edges of chunks and ranges, two
and three ranges in one CTA, and the sizes on both sides of the rule that gives each range a CTA
of its own.  Same acceptance rules as the other selection tests."""
import pytest

import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,ns,H,q_block", [
    (64 * 64, 0, 2, 64),          # one chunk
    (64 * 64 + 1, 0, 2, 128),     # a block in the second chunk
    (64 * 129, 3, 1, 64),         # three chunks, a block in the last
    (64 * 250 + 40, 70, 2, 64),   # four chunks in three ranges
    (64 * 512 - 7, 0, 1, 128),    # eight chunks: the last size whose ranges share a CTA
    (64 * 513, 5, 1, 128),        # nine: a CTA per range
    (64 * 320, 0, 20, 128),       # 40 stripes: three ranges, five chunks
    (64 * 320, 0, 20, 64),        # 60 stripes: two ranges
])
def test_ranges(N, ns, H, q_block):
    nb = -(-N // 64)
    inp = synth.make_random_layer(N, H, 64 * H, seed=N + H)
    layer = G.Layer(inp, ns, [max(1, nb // 10)] * H, 1, q_block=q_block).run(attention=False)
    G.check_selection(G.compare_selection(layer, layer.oracle_select()))
