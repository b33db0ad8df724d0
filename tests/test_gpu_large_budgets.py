"""Budgets and swap counts above what the row kernels select lane by lane: c_h > 128 in the
initial selection, m > 64 in a round, and 32 < m <= 64, where the survivors of a round's
selection often overflow their list.  Same acceptance rules as the other selection tests."""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,ns,c,R,q_block,variant", [
    (64 * 270 + 9, 5, (129,), 2, 128, None),        # first budget above 128; m = 32, 16
    (64 * 270 + 9, 5, (133,), 2, 128, None),        # m = 33: first one above 32
    (64 * 271, 0, (257, 2), 2, 128, None),          # nearly all kept: m capped by |D|; c = 2 beside it
    (64 * 520 + 33, 7, (260, 301), 3, 128, None),   # m = 65 and 75, then 32 and 37, then 16 and 18
    (64 * 300 + 1, 3, (280,), 1, 64, O.Variant(maximize="full")),  # m = 20 of 300 (capped), sign flipped
    (64 * 560, 0, (272,), 1, 128, O.Variant(maximize="swap")),     # m = 68, keys of both signs
])
def test_large_budgets(N, ns, c, R, q_block, variant):
    H = len(c)
    inp = synth.make_random_layer(N, H, 64 * H, seed=N + c[0])
    layer = G.Layer(inp, ns, list(c), R, variant=variant, q_block=q_block).run(attention=False)
    G.check_selection(G.compare_selection(layer, layer.oracle_select()))


@pytest.mark.parametrize("c", [129, 200, 299])
def test_equal_keys_beyond_the_tie_list(c):
    """With every key token equal all 300 candidates of a row tie (more than the 128 that the
    selection ranks among themselves): the lowest c indices are kept."""
    N, H = 64 * 300, 1
    inp = synth.make_random_layer(N, H, 64 * H, seed=c)
    inp["K"][:] = inp["K"][0:1]
    layer = G.Layer(inp, 0, [c] * H, 0, variant=O.Variant(key="probability"),
                    q_block=128).run(attention=False)
    want = np.ones(layer.nb, dtype=bool)
    want[:c] = False
    assert (layer.drop_sets()[:, :layer.nqc] == want).all()


@pytest.mark.parametrize("c,R", [(200, 0), (290, 0)])
def test_keys_over_many_octaves(c, R):
    """Keys scaled so that the pooled probabilities of a row span far more than the 16 octaves
    below the largest key that the selection counts first: the c-th key lies beyond them."""
    N, H = 64 * 300, 1
    inp = synth.make_random_layer(N, H, 64 * H, seed=300 + c)
    inp["K"] = synth.bf16_bits(synth.bf16_to_f32(inp["K"]) * np.float32(24.0))
    layer = G.Layer(inp, 0, [c], R, variant=O.Variant(key="probability"), q_block=128).run(attention=False)
    P = layer.ws("P", shape=(H, layer.nq, layer.buf.layout.ld))[0, :layer.nqc, :layer.ncand]
    cth = np.sort(P, axis=1)[:, -c]
    assert np.median(P.max(1) / np.maximum(cth, 1e-30)) > 2.0 ** 16
    # the drop sets alone: a row here drops a pooled mass far below the float32 rounding of its
    # kept mass, from which its net drift is formed, so its J (about 1e-20) has no relative accuracy
    r = G.compare_selection(layer, layer.oracle_select())
    assert r["mismatched"] == 0 and r["near"] <= G.NEAR_FRACTION * (r["exact"] + r["near"]) + 1, r
