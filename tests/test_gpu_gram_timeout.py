"""bakron_gram when a bounded wait runs out: an error, and a sum that is not added to
half-way where the samples were split (the parts are missing then)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# one block or three, split along the samples
@pytest.mark.parametrize("k,d,dtype", [(4096, 64, torch.bfloat16), (4096, 250, torch.bfloat16), (3000, 129, torch.float32)])
def test_split_sum_is_left_alone(k, d, dtype, monkeypatch):
    import paper_2608_06291_gb300 as P
    P.build()
    X = torch.randn(k, d, generator=torch.Generator().manual_seed(k)).to(dtype).cuda()
    G = torch.full((d, d), 3.0, device="cuda")
    ws = torch.full((P.bakron_gram_workspace_bytes(d, 8192),), 0xff, dtype=torch.uint8, device="cuda")   # NaNs
    monkeypatch.setenv("BAKRON_SPIN_CYCLES", "0")
    with pytest.raises(P.BakronError) as e:
        P.bakron_gram(X, alpha=1.0, beta=1.0, G=G, workspace=ws)
    assert e.value.status == 4
    assert torch.all(G == 3.0)
    monkeypatch.delenv("BAKRON_SPIN_CYCLES")
    P.bakron_gram(X, alpha=1.0, beta=1.0, G=G, workspace=ws)
    x = X.double()
    want = x.T @ x + 3.0
    assert torch.all((G.double() - want).abs() <= 2.0 ** -14 * (x.abs().T @ x.abs()) + 2.0 ** -20 * 3.0)
