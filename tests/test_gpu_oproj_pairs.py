"""Residual update and token drift at the edges of the CTA pairs' tiles (256 tokens x 256
channels): fewer rows than one CTA's half, one row past a tile, channel counts that are not a
multiple of a tile, tiles split into 2 and 4 units, stripes shared by 1, 2 and 4 pairs."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,d_model", [
    (1, 1, 64), (128, 3, 192), (129, 2, 256), (256, 4, 320), (257, 5, 1024),
    (2748, 4, 256),     # 11 tiles: all of them split
    (5003, 3, 1088),    # five channel tiles, the last of 64 channels
    (9700, 2, 512),     # 76 tiles: one whole wave of 76 pairs
    (9985, 2, 512),     # two tiles more than a wave
    (14000, 1, 768),    # 165 tiles: 13 past two waves
    (256 * 77 + 1, 2, 256),   # drift: pairs with one stripe and with two
    (256 * 160 - 70, 1, 320), # two and three stripes of two channel tiles
])
def test_pair_tile_edges(N, H, d_model):
    import paper_2609_35593_gb300 as ress
    g = torch.Generator(device="cuda").manual_seed(N)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)

    K = H * 64
    a, x = normal(N, H, 64).bfloat16(), normal(N, d_model).bfloat16()
    b = (a.float() + 0.25 * normal(N, H, 64)).bfloat16()
    W = (normal(d_model, K) / K ** 0.5).bfloat16()
    d = ress.dims(N, H, 0, d_model)
    ws = torch.zeros(ress.workspace_bytes(d), dtype=torch.uint8, device="cuda")
    ref = a.view(N, K).double() @ W.double().T
    # one rounding to bf16 (2^-9 relative) of a float32 sum of K exact products (at most
    # K 2^-24 of the sum of their magnitudes)
    acc = K * 2.0 ** -24 * (a.view(N, K).double().abs() @ W.double().abs().T)
    for res in (x, None):
        want = ref + x.double() if res is not None else ref
        y = torch.full((N, d_model), float("nan"), device="cuda").bfloat16()
        ress.out_proj(d, a, W, res, y, ws)
        ress.status(ws)
        assert bool(((y.double() - want).abs() <= 2.0 ** -8 * want.abs() + 2 * acc).all())
    nb = -(-N // 64)
    drift = torch.full((nb,), float("nan"), device="cuda", dtype=torch.float32)
    ress.token_drift(d, a, b, W, drift, ws)
    ress.status(ws)
    q = ((a.double() - b.double()).view(N, K) @ W.double().T).square().sum(1)
    want = torch.nn.functional.pad(q, (0, nb * 64 - N)).view(nb, 64).sum(1)
    # both products are float32 sums of magnitude about 1 with errors near 2^-22 each, against
    # differences of about 1/4; the block sums average them
    assert bool(((drift.double() - want).abs() <= 1e-4 * want).all())
