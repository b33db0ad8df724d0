"""Every way in which a small forward's attention items are shared by the CTAs of a cluster, with
budgets that differ between the heads: the output against float64 on every row.  The sizes are
for 152 SMs; the rule is restated here and the way it gives asserted, so that a case cannot
quietly stop being what it says.  Heads with small budgets next to one with a large budget have
lists shorter than the CTAs that share them, so some CTAs have no entries at all."""
import pytest

import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402
from attention64 import errors  # noqa: E402

pytestmark = pytest.mark.gpu


def _way(N, ns, c, sms):
    """(CTAs per item with dense query blocks, CTAs per sparse item)."""
    H, nb, nc = len(c), -(-N // 64), (N - ns) // 64
    pairs = (nb + 1) // 2
    dense = H * (pairs - nc // 2)
    sparse = H * pairs - dense
    tiles = min(nb, 29 * max(c) // 20 + nb - nc)

    def longest(split, share):
        return max(-(-nb // split) if dense else 0, -(-tiles // share) if sparse else 0)

    best, length = (1, 1), longest(1, 1) - 3
    for split in (2, 3, 4):
        for share in (s for s in (1, 2, 3, 4) if s <= split and split % s == 0):
            clusters = dense + -(-sparse * share // split)
            if split * clusters <= 2 * sms and longest(split, share) < length:
                best, length = (split, share), longest(split, share)
    return best if dense + sparse <= 2 * sms else (1, 1)


@pytest.mark.parametrize("N,ns,c,way", [
    (64 * 101, 0, (60, 1, 1), (2, 1)),       # 101 blocks: the last pair holds a dense half
    (64 * 95 - 11, 64 * 20, (7, 1, 3, 2, 7), (2, 1)),
    (64 * 130, 0, (40, 1), (2, 2)),
    (64 * 140, 64 * 2, (100, 3), (2, 2)),
    (64 * 65 + 1, 64 * 6, (17, 2, 1, 9, 1), (3, 1)),
    (64 * 100, 0, (70, 1), (3, 3)),          # one entry for three CTAs
    (64 * 80, 0, (8, 2), (3, 3)),
    (64 * 100 - 7, 0, (2, 1, 2), (4, 1)),
    (64 * 120 + 9, 9, (60, 1), (4, 2)),
    (64 * 80, 64 * 3, (50, 2, 1), (4, 2)),
    (64 * 40 + 9, 64 * 4, (20, 1, 2), (4, 4)),
    (64 * 60, 64 * 10, (30, 1), (4, 4)),
    (64 * 38, 0, (38, 1, 1, 2), (4, 4)),     # no dense items, one entry for four CTAs
    (64 * 140, 0, (100, 3, 1), (1, 1)),      # whole items: more would not fit one wave
])
def test_ways(N, ns, c, way):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 152:
        assert _way(N, ns, c, sms) == way
    H = len(c)
    inp = synth.make_random_layer(N, H, 64 * H, seed=N + H)
    layer = G.Layer(inp, ns, list(c), 1).run_forward()
    worst, mean = errors(layer)
    assert worst <= G.ATT_MAX_ABS and mean <= G.ATT_MEAN_REL, (worst, mean)
