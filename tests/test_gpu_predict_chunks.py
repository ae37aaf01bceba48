"""Predicted starts do not depend on how the rows fall into inference chunks: a
prediction of more rows than one chunk holds against predictions of its parts."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,m,tiles", [(256, 18, 30000), (256, 7, 75001), (64, 18, 15000)])
def test_chunked_prediction_equals_parts(hidden, m, tiles):
    torch = pytest.importorskip("torch")
    from paper_1710_03732_gb300 import rlt2 as R
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    c = 50 * torch.randn(tiles, m, m, generator=g, device="cuda", dtype=torch.float64)
    prev = 20 * torch.randn(tiles, m, generator=g, device="cuda", dtype=torch.float64)
    net = R.Mlp(hidden=hidden, seed=3)
    whole = torch.empty(tiles, m, device="cuda", dtype=torch.float64)
    net.predict(c, whole, prev_u=prev)
    for a in range(0, tiles, 4999):
        part = torch.empty_like(whole[a:a + 4999])
        net.predict(c[a:a + 4999].contiguous(), part, prev_u=prev[a:a + 4999].contiguous())
        assert torch.equal(part, whole[a:a + 4999])
    net.close()
