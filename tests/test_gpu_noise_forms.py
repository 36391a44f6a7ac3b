"""The prior weights where the correlation runs as transforms, against the FP64 oracle on the same
random stream: the padded single tile at the edges of its transform sizes, cut into tiles, odd grids
and PSFs, and an odd number of realisations (the last pair has one member)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,f,K,J,n_real", [
    (64, 2, 64, 4, 41),    # L = 160, the padded limit: F + K/2 = L
    (63, 2, 63, 3, 40),    # below it, odd PSF
    (65, 2, 64, 3, 33),    # one pixel pair beyond: 2 x 2 tiles
    (45, 3, 51, 4, 17),    # odd grid, tiles of which the last ones are narrower
    (37, 1, 21, 3, 19),    # the smallest transforms in use
    (24, 1, 64, 3, 12),    # PSF wider than the grid
])
def test_transform_correlation_matches_oracle(N, f, K, J, n_real):
    import oracle
    import torch
    from paper_2402_08725_gb300.binding import noise_weights
    rng = np.random.default_rng(1000 * N + K)
    sigma = rng.uniform(2.0, 8.0, size=(3, N, N)).astype(np.float32)
    sigma[rng.random(sigma.shape) < 0.02] = np.inf
    y, x = np.mgrid[0:K, 0:K] - K // 2
    s1 = np.exp(-0.5 * ((x - 0.7) ** 2 / 9.0 + (y + 0.4) ** 2 / 4.0)) + 0.01 * rng.random((K, K))
    s1 = (s1 / s1.sum()).astype(np.float32)
    W, Wm, _ = noise_weights(N, f, K, J, torch.from_numpy(sigma).cuda(), torch.from_numpy(s1).cuda(), n_real, 11)
    W_ref, Wm_ref = oracle.noise_weights(N, f, K, J, sigma.astype(np.float64), s1.astype(np.float64), n_real, 11)
    # every draw, tap and filter sum carries FP32 rounding (2^-24 each); a coefficient's standard
    # deviation over the realisations averages those of its sums: a few 2^-24 of the plane's level,
    # with the finest detail a tenth of the smoothed image's level, stays below 2e-5
    assert np.max(np.abs(W / W_ref - 1.0)) < 2e-5
    m = Wm.cpu().numpy().reshape(J - 1, -1)
    r = Wm_ref.reshape(J - 1, -1)
    for j in range(J - 1):
        assert np.linalg.norm(m[j] - r[j]) < 2e-5 * np.linalg.norm(r[j])
