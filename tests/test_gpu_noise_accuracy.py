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
