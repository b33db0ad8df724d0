"""Token drift at the sizes of whole scenes, where a stripe of 256 tokens goes to a cluster of two or
four CTA pairs or several stripes to one persistent pair, against float64."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,d_model", [
    (8 * 1374, 16, 1024),    # 43 stripes: clusters of four pairs
    (16 * 1374, 16, 1024),   # 86 stripes: clusters of two pairs
    (32 * 1374, 16, 1024),   # 172 stripes: clusters of two pairs
    (32 * 1374, 8, 512),     # persistent pairs, two or three stripes each
])
def test_scene_sizes(N, H, d_model):
    import paper_2609_35593_gb300 as ress
    g = torch.Generator(device="cuda").manual_seed(N + H)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)

    K = H * 64
    a = normal(N, H, 64).bfloat16()
    b = (a.float() + 0.25 * normal(N, H, 64)).bfloat16()
    W = (normal(d_model, K) / K ** 0.5).bfloat16()
    d = ress.dims(N, H, 0, d_model)
    ws = torch.zeros(ress.workspace_bytes(d), dtype=torch.uint8, device="cuda")
    nb = -(-N // 64)
    drift = torch.full((nb,), float("nan"), device="cuda", dtype=torch.float32)
    ress.token_drift(d, a, b, W, drift, ws)
    ress.status(ws)
    q = ((a.double() - b.double()).view(N, K) @ W.double().T).square().sum(1)
    want = torch.nn.functional.pad(q, (0, nb * 64 - N)).view(nb, 64).sum(1)
    # both products are float32 sums of magnitude about 1 with errors near 2^-22 each, against
    # differences of about 1/4; the block sums average them
    assert bool(((drift.double() - want).abs() <= 1e-4 * want).all())
