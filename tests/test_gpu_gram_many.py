"""bakron_gram over many samples: partial sums are added one after the other over a
chunk at most, so their rounding does not grow with the number of samples.

For 262144 bf16 samples of 8192 features (read in place, no split of the samples:
1056 blocks) and the default workspace a chunk is 32768 samples: 128 partial sums of
like size in a register, then 8 chunks in G.  One rounding is off by 2.5e-8 (rms) of
the running sum, so a diagonal entry by 2.5e-8 sqrt(128 / 3 / 8 + 8 / 3) = 0.7e-7; all
1024 in a row give 2.5e-8 sqrt(1024 / 3) = 4.6e-7.  Asked for: 2e-7.  Measured is the
scatter over the features, since what the tensor core loses inside 256 samples has the
same sign for all.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [8192, 64])
def test_scatter_of_the_diagonal(chunk):
    """A small workspace does not bring it back (nor a launch per few samples)."""
    import paper_2608_06291_gb300 as P
    P.build()
    k, d = 262144, 8192
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(k, d, generator=g, device="cuda", dtype=torch.bfloat16)
    G = P.bakron_gram(X, alpha=1.0 / k, chunk=chunk)
    torch.cuda.synchronize()
    want = torch.zeros(d, dtype=torch.float64, device="cuda")
    for part in X.split(16384):
        want += part.double().square().sum(0)
    off = G.diagonal().double() * k / want - 1
    print(f"chunk {chunk}: mean {off.mean().item():.2e} scatter {off.std().item():.2e}")
    assert off.std().item() < 2e-7
