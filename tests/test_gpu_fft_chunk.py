"""The per-epoch transform kernel at the edges of its shapes, against the FP64 oracle: every transform
size (both factorisations, odd and even second factors), missing second epochs, no source to four,
one to nine phases, odd stamps, groups of several pairs and of one, and items of more epochs than a
group."""
import numpy as np
import pytest

from _helpers import check_deconv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,f,K,M,E,J,gp", [
    (17, 1, 13, 0, 3, 3, 0),    # L = 24: no source, one phase, odd E
    (21, 2, 30, 1, 9, 3, 0),    # L = 32: groups of four pairs, the last of one epoch
    (27, 3, 33, 4, 4, 3, 0),    # L = 40: nine phases, four sources
    (33, 2, 41, 1, 5, 4, 0),    # L = 48
    (41, 2, 53, 2, 3, 3, 0),    # L = 56: odd stamp, two sources
    (48, 2, 61, 1, 7, 4, 0),    # L = 64
    (55, 1, 31, 3, 2, 4, 0),    # L = 72
    (61, 3, 57, 1, 3, 4, 0),    # L = 80 with nine phases
    (80, 2, 63, 1, 5, 4, 0),    # L = 96: groups of two pairs, the last of one epoch
    (95, 2, 64, 1, 4, 4, 1),    # L = 112, one pair per group
    (111, 2, 64, 0, 3, 4, 0),   # L = 128, no source
    (127, 1, 33, 2, 1, 4, 0),   # L = 144, one epoch alone
])
def test_chunk_kernel_matches_oracle(N, f, K, M, E, J, gp):
    import torch
    from paper_2402_08725_gb300 import synthetic as syn
    from paper_2402_08725_gb300.binding import Batch, Problem
    fd = syn.small_deconv(seed=3000 + 10 * N + f, E=E, N=N, f=f, K=K, M=M, J=J, lam=1.3)
    fd.sigma[:, N // 3, N // 2] = np.inf
    prob = Problem.from_field(fd, conv_mode="fft")
    b = Batch([prob])
    b.set_schedule(16, gp)
    loss, grad = b.loss_and_grad(torch.from_numpy(fd.params).cuda())
    check_deconv(fd, loss, grad.cpu().numpy())
    b.close()
    prob.close()
