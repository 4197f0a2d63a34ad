"""bakron_prepare is no further off than an fp64 factorisation, at condition numbers
where that shows through the rounding to fp32.

H = L L^T with L unit lower and entries 0 and +-1/2: H is exact in fp32.  The unit
factor wanted is R^-1 diag(R) with R^T R = H, R lower, and R comes from a QL
factorisation of L^T, which sees the square root of H's condition only.  Measured is
the relative Frobenius error, its geometric mean over 24 matrices, since single ones
scatter tenfold either way; allowed is the fp64 factorisation's own plus one rounding
to fp32, 2^-24.  (The sliced products' own errors are 0.4 of fp64's, by emulation.)
"""
import numpy as np
import pytest
import scipy.linalg
import torch

import oracle as O

pytestmark = pytest.mark.gpu


def _problem(d, density, seed):
    rng = np.random.default_rng(seed)
    L = np.tril((rng.random((d, d)) < density) * rng.choice([-0.5, 0.5], (d, d)), -1) + np.eye(d)
    H = L @ L.T
    assert (H.astype(np.float32) == H).all()
    R = np.linalg.qr(L.T[:, ::-1])[1][::-1, ::-1]
    return H, scipy.linalg.solve_triangular(R, np.diag(np.diag(R)), lower=True)


def _mean(errors):
    return float(np.exp(np.mean(np.log(np.maximum(errors, 1e-300)))))


# condition about 3e2, 3e5, 1e10, 1e12 and 1e14, and 1e10 in fewer rows
@pytest.mark.parametrize("d,density", [(384, 0.02), (384, 0.08), (384, 0.2), (384, 0.25), (384, 0.3), (200, 0.4)])
def test_no_further_off_than_fp64(d, density):
    import paper_2608_06291_gb300 as P
    P.build()
    eye = torch.eye(3, device="cuda")
    ours, fp64 = [], []
    for seed in range(24):
        H, want = _problem(d, density, seed)
        got = P.bakron_get_factors(P.bakron_prepare(torch.from_numpy(H).float().cuda(), eye, 0.0))[0]
        norm = np.linalg.norm(want)
        ours.append(np.linalg.norm(got.double().cpu().numpy() - want) / norm)
        fp64.append(np.linalg.norm(O.prepare(H, np.eye(3), 0.0, via_inverse=False).LA - want) / norm)
    print(f"d {d} density {density}: ours {_mean(ours):.2e} fp64 {_mean(fp64):.2e}")
    assert _mean(ours) <= _mean(fp64) + 2.0 ** -24
