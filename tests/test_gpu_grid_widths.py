"""bakron_grid_symmetric at the widths where its kernel changes how many values a
thread keeps (1, 4, 16, 32 per thread of 256, then none): the scale is a candidate
bit for bit, and the oracle's choice unless the two candidates' errors agree to 1e-5
(the comparison of test_gpu_symmetric.py).
"""
import pytest
import torch

from tests.test_gpu_symmetric import _check_grid, _heavy

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2608_06291_gb300 as P


@pytest.mark.parametrize("n", [255, 256, 257, 1025, 4096, 4097, 8192, 8195])
@pytest.mark.parametrize("K", [0, 50])
def test_grid_symmetric_widths(n, K):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    W = torch.from_numpy(_heavy(5, n, n + K)).to("cuda", torch.float32)
    s, z = P.bakron_grid_symmetric(W, 3, 0, K)
    torch.cuda.synchronize()
    _check_grid(W.cpu().numpy(), s.cpu().numpy(), z.cpu().numpy(), 3, 0, K)
