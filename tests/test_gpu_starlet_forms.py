"""A field's prior has the same bits in a cluster (alone) and level by level (in a batch of many)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,f,J", [(32, 2, 4), (45, 3, 5), (61, 2, 6), (128, 2, 4), (85, 3, 7)])
@pytest.mark.parametrize("term", ["weights", "map", "sources"])
def test_cluster_and_levels_give_the_same_bits(N, f, J, term):
    import torch
    from _helpers import check_deconv
    from paper_2402_08725_gb300 import synthetic as syn
    from paper_2402_08725_gb300.binding import Batch, Problem
    fd = syn.small_deconv(seed=5000 + N, E=2, N=N, f=f, K=15, M=2, J=J, lam=1.3)
    small = syn.small_deconv(seed=5100, E=1, N=32, f=2, K=9, M=2, J=3, lam=1.0)

    def problem(d):
        p = Problem.from_field(d, conv_mode="fft")
        if term == "map":
            G = d.f * d.N
            p.set_weight_map(np.random.default_rng(G).uniform(0.5, 2.0, (d.J - 1, G, G)).astype(np.float32))
        if term == "sources":
            p.set_lambda_pts(0.6)
        return p

    alone = problem(fd)
    loss, grad = alone.loss_and_grad(torch.from_numpy(fd.params).cuda())
    grad = grad.clone()
    if term == "weights":
        check_deconv(fd, loss, grad.cpu().numpy())
    n = 24  # more clusters than run at once: the table goes level by level
    fields = [fd] + [small] * n
    probs = [problem(d) for d in fields]
    batch = Batch(probs)
    losses = torch.empty(n + 1, dtype=torch.float64, device="cuda")
    _, g = batch.loss_and_grad(torch.from_numpy(batch.pack([d.params for d in fields])).cuda(), losses=losses)
    assert losses[0].item() == loss and torch.equal(g[:fd.n_params], grad)
    batch.close()
    for p in probs + [alone]:
        p.close()
