"""Row-by-block products on persistent CTAs, which take over above two tiles per SM: tile counts
below, at and just above that line (runs of two and of three tiles), runs that cross stripes of
rows and heads, a row and a block more than a tile, ragged lengths on both query grids, and
rounds in which only some heads swap blocks.  (With at most 32 heads, that many tiles need at
least 4 tiles of blocks, so every stripe of rows is more than one tile.)  The rows at the edges of
every tile and one in between are compared with the oracle; same acceptance rules as the other
selection tests."""
import pytest

import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,ns,q_block,heads,small,R,persistent", [
    (64 * 400, 0, 64, 0, 0, 1, False),            # at most 2 tiles per SM
    (64 * 400, 0, 64, 1, 0, 1, True),             # a head's 16 tiles more
    (64 * 449 + 33, 70, 64, 5, 4, 2, True),       # 4 heads never swap; the line is crossed without them
    (64 * 449 + 33, 70, 64, 1, 3, 2, True),       # the rounds' products fall below the line
    (64 * 513, 0, 64, 1, 2, 1, True),             # a row and a block more than 4 tiles
    (64 * 640 - 5, 3, 128, 1, 5, 2, True),        # 3 x 5 tiles per head
])
def test_runs(N, ns, q_block, heads, small, R, persistent):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nb, nqc = -(-N // 64), (N - ns) // q_block
    per_head = -(-nqc // 128) * -(-nb // 128)
    H = 2 * sms // per_head + heads
    assert (H * per_head > 2 * sms) == persistent and H <= 32
    # budgets of 1 swap nothing; the others 25 to 40 blocks, every few heads a small one
    c = [1 if small and h % (H // small) == 1 else 25 + h % 16 for h in range(H)]
    inp = synth.make_random_layer(N, H, 64 * H, seed=N + H)
    layer = G.Layer(inp, ns, c, R, q_block=q_block).run(attention=False)
    rows = [(h, i) for h in range(H) for s in range(0, nqc, 128)
            for i in sorted({s, min(s + 17 + 5 * h, nqc - 1), min(s + 127, nqc - 1)})]
    G.check_selection(G.compare_selection(layer, layer.oracle_select(rows=rows)))
