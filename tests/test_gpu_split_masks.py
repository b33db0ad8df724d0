"""Small forwards, whose attention items are shared by several CTAs, on keys that a caller masks:
one channel of every query is 1 and the masked keys hold a huge negative number (or -inf)
there.  A masked key's weight is exactly 0, wherever the CTAs' shares of a list begin: the first
tile of a share, or all of it, may be masked.  Same acceptance rules as the other attention
tests, against float64 over the forward's own lists."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402
from attention64 import errors  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [-1e4, -1e30, -3.3895313892515355e38, float("-inf")])
@pytest.mark.parametrize("lo,hi", [(0.6, 1.0), (0.3, 0.7)])
@pytest.mark.parametrize("N,H,ns", [(64 * 38, 4, 200), (64 * 61 + 9, 2, 0), (64 * 77 + 38, 3, 37)])
def test_masked_keys(N, H, ns, lo, hi, value):
    inp = synth.make_random_layer(N, H, 64 * H, seed=N + H)
    inp["Q"][:, :, 63] = synth.bf16_bits(np.float32([1.0]))
    inp["K"][:, :, 63] = 0
    nb = -(-N // 64)
    masked = slice(64 * int(lo * nb), N if hi == 1.0 else 64 * int(hi * nb))
    inp["K"][masked, :, 63] = synth.bf16_bits(np.float32([value]))
    layer = G.Layer(inp, ns, [7] * H, 0).run_forward()  # fewer blocks than stay unmasked
    worst, mean = errors(layer)  # (every row keeps keys that are not masked)
    assert worst <= G.ATT_MAX_ABS and mean <= G.ATT_MEAN_REL, (worst, mean)
