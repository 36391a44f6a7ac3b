"""How far the prior weights are from 64 bits where the correlation runs as transforms: no bias of
their level, whichever transform size the field takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _psf(K, fwhm):
    y, x = np.mgrid[0:K, 0:K] - K // 2
    s = (1.0 + (x * x + y * y) / (0.5 * fwhm) ** 2 * (2.0 ** (1 / 2.5) - 1.0)) ** -2.5
    return (s / s.sum()).astype(np.float32)


def _weights(N, f, K, J, sigma, s1, n_real, seed):
    import torch
    from paper_2402_08725_gb300.binding import noise_weights
    W, m, _ = noise_weights(N, f, K, J, torch.from_numpy(sigma).cuda(), torch.from_numpy(s1).cuda(), n_real, seed)
    return np.asarray(W, dtype=np.float64), m.cpu().numpy().astype(np.float64).reshape(J - 1, f * N, f * N)


@pytest.mark.parametrize("N,f,K", [
    (37, 1, 21),    # L = 48
    (46, 1, 23),    # L = 64
    (32, 2, 64),    # L = 96
    (72, 1, 36),    # L = 96
    (44, 2, 52),    # L = 128
    (56, 2, 60),    # L = 144
    (64, 2, 64),    # L = 160
])
def test_transforms_do_not_bias_the_level(N, f, K):
    import oracle
    rng = np.random.default_rng(N + K)
    sigma = rng.uniform(3.0, 10.0, (4, N, N)).astype(np.float32)
    s1, J, n_real = _psf(K, 5.0), 3, 24
    _, m = _weights(N, f, K, J, sigma, s1, n_real, 17)
    _, ref = oracle.noise_weights(N, f, K, J, sigma.astype(np.float64), s1.astype(np.float64), n_real, 17)
    ref = np.asarray(ref).reshape(m.shape)
    # the rounding of each value (2^-24) averages out over a plane's pixels: more than half of it left
    # over in the mean is a common factor
    for j in range(J - 1):
        assert abs(np.mean(m[j] / ref[j] - 1.0)) < 2.0 ** -25, j


def _uneven(kind, N, sigma):
    """sigma with what the transforms must not lose: a masked region, noise that rises by orders of
    magnitude across the grid, one epoch-long dead column, and one far better pixel."""
    y = np.arange(N)
    s = sigma.copy()
    if kind == "masked corner":
        s[:, :2 * N // 3, :2 * N // 3] = np.inf
    elif kind == "rising 1e6":
        s *= (10.0 ** (6.0 * y / (N - 1)))[None, None, :].astype(np.float32)
    elif kind == "rising 30":
        s *= (30.0 ** (y / (N - 1)))[None, :, None].astype(np.float32)
    elif kind == "dead column":
        s[:, :, N // 4] = np.inf
    elif kind == "one pixel":
        s[:, N // 3, N // 3] *= 1e-4
    elif kind == "all masked":
        s[:] = np.inf
    elif kind == "tiny":
        s *= 1e-18
    return s.astype(np.float32)


@pytest.mark.parametrize("N,f,K", [(40, 2, 41), (96, 1, 64), (50, 3, 45)])  # one transform tile, one, 2 x 2
@pytest.mark.parametrize("kind", ["masked corner", "rising 1e6", "rising 30", "dead column", "one pixel", "all masked",
                                  "tiny"])
def test_faint_and_masked_pixels_keep_their_accuracy(kind, N, f, K):
    import oracle
    rng = np.random.default_rng(3 * N + K)
    sigma = _uneven(kind, N, rng.uniform(3.0, 10.0, (3, N, N)).astype(np.float32))
    s1, J, n_real = _psf(K, 4.0), 3, 20
    _, m = _weights(N, f, K, J, sigma, s1, n_real, 23)
    _, ref = oracle.noise_weights(N, f, K, J, sigma.astype(np.float64), s1.astype(np.float64), n_real, 23)
    ref = np.asarray(ref).reshape(m.shape)
    # A value of y rounds like the sum of its K^2 products: at most about sqrt(K^2) 2^-24 = 4e-6 of its
    # own level; the planes of details hold a tenth of it, so 4e-5 of a pixel's own value, and 2.5 times that
    # for the smallest of a plane.  A pixel that only masked pixels reach has none.
    assert np.array_equal(m == 0.0, ref == 0.0)
    ok = ref > 0.0
    if ok.any():
        assert np.max(np.abs(m[ok] / ref[ok] - 1.0)) < 1e-4
