"""The training loss does not depend on the order in which the warps' parts arrive, and is exact to its
FP32 terms: each term is rounded a few times (2^-24 each, independent), their sum once, so the loss of
thousands of terms is within 4 units of 2^-24 of the FP64 mean over the same network outputs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")


@pytest.mark.parametrize("n,masked", [(4096, False), (777, True), (8192, True)])
def test_loss(n, masked):
    from paper_2506_06661_gb300 import guess
    g = torch.Generator().manual_seed(n)
    params = guess.GuessModel.create(seed=3).params
    X = torch.randn(n, guess.NIN, generator=g).cuda()
    Y = torch.randn(n, guess.NOUT, generator=g).cuda()
    mask = (torch.rand(n, generator=g) < 0.7).float().cuda() if masked else None
    out = guess.forward(params, X)
    d2 = (out.double() - Y.double()) ** 2
    ref = float((d2 * mask[:, None].double()).sum() / (mask.sum() * guess.NOUT)) if masked else float(d2.mean())
    losses = {guess.loss_grad(params, X, Y, mask)[0] for _ in range(10)}
    assert len(losses) == 1
    assert abs(losses.pop() - ref) <= 4 * 2.0 ** -24 * ref
