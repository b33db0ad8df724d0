"""Selections among keys with many ties, as repeated or featureless frames give: blocks of the
same kind have the same pooled key and value, hence the same keys to the bit, so a selection takes
whole kinds in some order and of the last one its lowest blocks.  The counts make the survivor
lists and the lists of the all-keys selection overflow on one side of the drop set or both; unique
blocks above the ties come one by one.  And what ties cost next to keys that all differ."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402

pytestmark = pytest.mark.gpu


def _layer(nb, c, kind, rounds, heads=2):
    """A layer of nb candidate blocks, block j holding the tokens of kind[j]."""
    inp = synth.make_random_layer(64 * nb, heads, 64 * heads, seed=nb + c)
    first = np.unique(kind, return_index=True)[1]
    tokens = (64 * first[kind][:, None] + np.arange(64)).reshape(-1)
    inp["K"], inp["V"] = inp["K"][tokens], inp["V"][tokens]
    return G.Layer(inp, 0, [c] * heads, rounds)


def _check(chosen, pool, kind, m):
    """chosen is a top m of pool: whole kinds, and the lowest blocks of one more, or of several whose
    keys are equal (with two kinds of as many blocks, P_a sqrt(q_a) = P_b sqrt(q_b) on every row)."""
    assert not (chosen & ~pool).any() and chosen.sum() == m
    taken = np.bincount(kind[chosen], minlength=kind.max() + 1)
    there = np.bincount(kind[pool], minlength=kind.max() + 1)
    cut = ((taken > 0) & (taken < there))[kind] & pool  # blocks of the kinds taken in part
    assert (chosen[cut] == (np.arange(cut.sum()) < chosen[cut].sum())).all()


def _repeat(period):
    return lambda nb: np.arange(nb) % period


def _unique(count):
    return lambda nb: np.where(np.arange(nb) % (nb // count) == 3, 1 + np.arange(nb) // (nb // count), 0)


@pytest.mark.parametrize("nb,c,kinds", [
    (700, 9, _repeat(1)), (700, 9, _repeat(2)), (700, 16, _unique(30)),     # survivor lists
    (700, 60, _repeat(1)), (1400, 120, _repeat(3)), (1400, 200, _repeat(5)),
    (1400, 400, _repeat(2)), (2000, 700, _repeat(12)), (2000, 1500, _repeat(13)),
    (2000, 1990, _repeat(1)), (640, 64, _unique(20)), (4096, 130, _repeat(1)),
])
def test_ties(nb, c, kinds):
    kind = kinds(nb)
    everything = np.ones(nb, bool)
    kept = ~_layer(nb, c, kind, 0).run(attention=False).drop_sets()
    after = ~_layer(nb, c, kind, 1).run(attention=False).drop_sets()
    m = min(c // 4, nb - c, c)
    swapped = 0
    for first, last in zip(kept.reshape(-1, nb), after.reshape(-1, nb)):
        _check(first, everything, kind, c)
        if (first != last).any():  # the round's swap lowered the drift
            _check(last & ~first, ~first, kind, m)
            _check(first & ~last, first, kind, m)
            swapped += 1
    assert m == 0 or swapped > 0 or len(np.unique(kind)) == 1


def test_cost():
    nb, c, heads = 1369, 684, 4
    times = []
    for kind in (np.arange(nb), np.zeros(nb, int)):
        layer = _layer(nb, c, kind, 4, heads).run(attention=False)
        r, b = layer.ress, layer.buf
        best = 1e9
        for _ in range(20):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            r.score(layer.d, layer.Q, layer.K, layer.V, b.F, layer.c_h, b.ws)
            r.restore(layer.d, layer.c_h, 4, layer.rho, b.ws, b.row_ptr, b.col_idx, b.J_best)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1))
        times.append(best)
    # all keys tied against all keys different: 2.0 times as long with a bit-by-bit search for
    # both, 4.0 where only the ties take it
    assert times[1] <= 2.5 * times[0], times
