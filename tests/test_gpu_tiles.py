"""The direct form at each tile height (16, 32 and 64 rows, with ragged last tiles): the FP64 oracle's values,
and the same bits whatever the height, so that a field alone and in a batch agree."""
import ctypes

import numpy as np
import pytest

from _helpers import check_deconv

pytestmark = pytest.mark.gpu


def _rows(E, N, n):
    import torch
    from paper_2402_08725_gb300 import _native
    lib = ctypes.CDLL(_native.load()._name)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return lib._ZN2sr9tile_rowsEPKiS1_iii((ctypes.c_int * n)(*[E] * n), (ctypes.c_int * n)(*[N] * n), n, sms, 0)


@pytest.mark.parametrize("frame", ["plain", "shifted", "rotated"])
@pytest.mark.parametrize("E,N,f,K,M", [
    (3, 37, 2, 21, 6),   # one tile across, 5 rows in the last of 16 and of 32
    (2, 70, 2, 13, 2),   # tails of 6 columns and 6 rows
    (2, 52, 3, 11, 1),   # nine phases: three at a time in short tiles
    (4, 16, 1, 9, 3),    # one band, one phase
])
def test_tile_heights_agree_and_match_oracle(E, N, f, K, M, frame):
    import torch
    from paper_2402_08725_gb300 import synthetic as syn
    from paper_2402_08725_gb300.binding import Batch, Problem
    fd = syn.small_deconv(seed=4000 + N + f, E=E, N=N, f=f, K=K, M=M, J=3, lam=1.2)
    fd.sigma[:, N // 2, N // 3] = np.inf
    theta = np.linspace(0.2, 2.5, E) if frame == "rotated" else None

    def problem():
        p = Problem.from_field(fd, conv_mode="direct")
        if frame != "plain":
            p.set_translate_h(True)
        if theta is not None:
            p.set_rotations(theta)
        return p

    P = torch.from_numpy(fd.params).cuda()
    alone = problem()
    loss, grad = alone.loss_and_grad(P)
    grad = grad.clone()
    assert _rows(E, N, 1) == 16
    check_deconv(fd, loss, grad.cpu().numpy(), theta=theta, shifted=frame != "plain")
    for rows in (32, 64):
        n = next(k for k in range(1, 2000) if _rows(E, N, k) == rows)
        probs = [problem() for _ in range(n)]
        batch = Batch(probs)
        losses = torch.empty(n, dtype=torch.float64, device="cuda")
        _, g = batch.loss_and_grad(P.repeat(n), losses=losses)
        g = g.reshape(n, -1)
        for i in (0, n - 1):
            assert losses[i].item() == loss and torch.equal(g[i], grad), rows
        batch.close()
        for p in probs:
            p.close()
    alone.close()


def test_moved_fields_of_unlike_grids_equal_single_ones():
    """The shift gradient's sums are each field's own, whatever the widest field of the table is."""
    import torch
    from paper_2402_08725_gb300 import synthetic as syn
    from paper_2402_08725_gb300.binding import Batch, Problem
    fields = [syn.small_deconv(seed=4500 + N, E=E, N=N, f=2, K=11, M=1, J=3, lam=1.0)
              for E, N in ((3, 10), (2, 33), (4, 47), (1, 70))]

    def problem(fd):
        p = Problem.from_field(fd)
        p.set_translate_h(True)
        return p

    probs = [problem(fd) for fd in fields]
    batch = Batch(probs)
    losses = torch.empty(len(fields), dtype=torch.float64, device="cuda")
    _, g = batch.loss_and_grad(torch.from_numpy(batch.pack([fd.params for fd in fields])).cuda(), losses=losses)
    for i, fd in enumerate(fields):
        alone = problem(fd)
        loss, grad = alone.loss_and_grad(torch.from_numpy(fd.params).cuda())
        o = batch.offsets[i]
        assert losses[i].item() == loss and torch.equal(g[o:o + fd.n_params], grad)
        check_deconv(fd, loss, grad.cpu().numpy(), shifted=True)
        alone.close()
    batch.close()
    for p in probs:
        p.close()
