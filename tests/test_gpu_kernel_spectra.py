"""The kernel spectra of the transform form, which two epochs share a transform for, against the FP64
oracle where the epochs differ most."""
import numpy as np
import pytest

from _helpers import deconv_blocks, oracle_deconv, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [2.0 ** 20, 3.0e-7, 1.0])
@pytest.mark.parametrize("N,f,K", [(21, 2, 30), (48, 2, 61), (37, 1, 30)])
@pytest.mark.parametrize("batched", [False, True])
def test_epochs_of_unlike_normalisation_keep_their_accuracy(N, f, K, scale, batched):
    """Epoch 0's PSF is scaled, its data masked and its source off, and there is no extended channel:
    epoch 1's model is then its own PSF's alone, at whatever scale the other's is."""
    import torch
    from paper_2402_08725_gb300 import synthetic as syn
    from paper_2402_08725_gb300.binding import Batch, Problem
    fd = syn.small_deconv(seed=77 + N, E=2, N=N, f=f, K=K, M=1, J=3, lam=0.0)
    b = deconv_blocks(2, N, f, 1)
    fd.s[0] *= scale
    fd.sigma[0] = np.inf
    fd.params[b["h"]] = 0.0
    fd.params[b["a"].start] = 0.0
    prob = Problem.from_field(fd, conv_mode="fft")
    P = torch.from_numpy(fd.params).cuda()
    if batched:
        batch = Batch([prob])
        batch.set_psfs(torch.from_numpy(np.ascontiguousarray(fd.s, dtype=np.float32).reshape(-1)).cuda())
        loss, grad = batch.loss_and_grad(P)
        batch.close()
    else:
        loss, grad = prob.loss_and_grad(P)
    prob.close()
    L_ref, _, g_ref, _ = oracle_deconv(fd)
    g = grad.cpu().numpy().astype(np.float64)
    assert abs(loss - L_ref) <= 1e-6 * abs(L_ref)
    for name, epoch1 in (("a", slice(1, 2)), ("delta", slice(2, 4)), ("Gamma", slice(1, 2))):
        assert rel_l2(g[b[name]][epoch1], g_ref[b[name]][epoch1]) <= 1e-4, name


@pytest.mark.parametrize("E", [1, 2, 5])
@pytest.mark.parametrize("N,f,K", [(21, 2, 30), (27, 3, 33), (55, 1, 31)])  # four, nine and one phase
@pytest.mark.parametrize("batched", [False, True])
def test_odd_epochs_pair_their_phases(E, N, f, K, batched):
    """The last epoch of an odd number: its phases share transforms two by two, an odd phase alone."""
    import torch
    from _helpers import check_deconv
    from paper_2402_08725_gb300 import synthetic as syn
    from paper_2402_08725_gb300.binding import Batch, Problem
    fd = syn.small_deconv(seed=510 + N + E, E=E, N=N, f=f, K=K, M=2, J=3, lam=1.1)
    prob = Problem.from_field(fd, conv_mode="fft")
    P = torch.from_numpy(fd.params).cuda()
    if batched:
        batch = Batch([prob])
        batch.set_psfs(torch.from_numpy(np.ascontiguousarray(fd.s, dtype=np.float32).reshape(-1)).cuda())
        loss, grad = batch.loss_and_grad(P)
        batch.close()
    else:
        loss, grad = prob.loss_and_grad(P)
    prob.close()
    check_deconv(fd, loss, grad.cpu().numpy())
