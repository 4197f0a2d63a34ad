"""bakron_prepare's verdict, SPD or not, is that of an fp64 Cholesky on the host.

Indefinite matrices whose pivots, entries of the factor or Schur complements leave
(-1, 1) where the factorisation keeps fixed-point numbers: inside a diagonal block,
from one panel to the next and across 128-row tiles, on either side; and positive
definite ones close to that.  Every matrix is either indefinite or positive definite
by 1e-4 of its diagonal or more, a thousand times fp32's rounding of its entries
and far above both factorisations' errors.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2608_06291_gb300 as P


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.lib()


def _spd(H, damp):
    h = H.astype(np.float64)
    h = h + damp * np.trace(h) / len(h) * np.eye(len(h))
    try:
        np.linalg.cholesky(h)
        return True
    except np.linalg.LinAlgError:
        return False


def _verdict(A, B, damp):
    try:
        P.bakron_prepare(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), damp)
    except P.BakronError as e:
        assert e.status == 2
        return False
    return True


def _check(H, want, damp=0.0):
    """H on either side, the identity on the other."""
    H = np.ascontiguousarray(H, dtype=np.float32)
    assert _spd(H, damp) == want
    eye = np.eye(40, dtype=np.float32)
    assert _verdict(H, eye, damp) == want
    assert _verdict(eye, H, damp) == want


# the scaled diagonal is 1/4 of 1 and 15/16 of 3.75
@pytest.mark.parametrize("scale", [1.0, 3.75])
@pytest.mark.parametrize("value", [0.2, 0.34, 0.36, 0.5, 0.7, 0.9, 1.0])
@pytest.mark.parametrize("d,row,cols", [(16, 0, 8), (16, 15, 0), (64, 3, 40), (130, 0, 60), (200, 0, 150),
                                        (200, 70, 130), (700, 0, 690), (700, 300, 500), (700, 690, 2)])
def test_one_row_against_eight(d, row, cols, value, scale):
    """I with eight entries in one row: definite up to 8 value^2 < 1 (0.353)."""
    H = np.eye(d)
    H[row, cols:cols + 8] = H[cols:cols + 8, row] = value
    _check(scale * H, 8 * value * value < 1)


@pytest.mark.parametrize("scale", [1.0, 3.75])
@pytest.mark.parametrize("d,a,b,r", [(64, 60, 59, 3), (200, 199, 190, 2), (400, 390, 260, 100), (400, 200, 199, 180)])
def test_large_entry_of_the_factor(d, a, b, r, scale):
    """Two rows almost alike, a third that leans on their difference: its entry of
    the factor is -22 (or -0.1, and definite)."""
    for lean, want in ((0.5, False), (0.002, True)):
        H = np.eye(d)
        for i, j, v in ((a, b, 0.999), (a, r, lean), (b, r, -lean)):
            H[i, j] = H[j, i] = v
        _check(scale * H, want)


@pytest.mark.parametrize("scale", [1.0, 3.75])
@pytest.mark.parametrize("d,k,i,j", [(64, 63, 20, 10), (200, 199, 30, 10), (400, 390, 200, 100), (400, 399, 398, 397)])
def test_large_entry_of_a_schur_complement(d, k, i, j, scale):
    """Two rows opposite along a third and alike to each other: 0.97 + 0.94."""
    for sign, want in ((1.0, False), (-1.0, True)):
        H = np.eye(d)
        for p, q, v in ((k, i, 0.97), (k, j, -0.97), (i, j, sign * 0.97)):
            H[p, q] = H[q, p] = v
        _check(scale * H, want)


@pytest.mark.parametrize("d", [16, 65, 129, 300, 700])
@pytest.mark.parametrize("low", [-2.0, -0.5, -1e-2, -1e-3, 1e-3, 1e-2])
def test_random_spectrum(d, low):
    """A random symmetric matrix with eigenvalues low (a few) and up to 3."""
    rng = np.random.default_rng(d)
    q = np.linalg.qr(rng.standard_normal((d, d)))[0]
    w = rng.uniform(0.5, 3.0, d)
    w[: max(1, d // 20)] = low
    H = (q * w) @ q.T
    H = (H + H.T) / 2
    assert H.diagonal().min() > 0
    s = np.exp2(rng.integers(-8, 9, d))
    _check(H, low > 0)
    _check(H * s * s[:, None], low > 0)


@pytest.mark.parametrize("d", [64, 300, 700])
def test_rows_almost_alike(d):
    """Every correlation 1 - 1e-3: sums over a panel come as close to 1 as they do."""
    H = np.full((d, d), 1 - 1e-3)
    np.fill_diagonal(H, 1.0)
    for scale in (1.0, 3.75, 3.8):
        _check(scale * H, True)
    _check(3.75 * H, True, 0.01)
