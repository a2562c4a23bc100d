"""The differentiable run's outputs are the caller's own: each has its storage,
and one edited in place before the loss gives the gradients of the same loss
written without the edit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _gradients(edit):
    import torch
    from paper_1907_13088_gb300.adjoint import GaussSourceRun, make_function
    rng = np.random.default_rng(471)
    nx, ny, n = 60, 44, 5
    cxy = np.stack([rng.uniform(0, nx, n), rng.uniform(0, ny, n)], 1)
    run = GaussSourceRun((nx, ny), cxy, rng.uniform(0, 6, n), 4, checkpoint_every=3)
    leaf = lambda a: torch.from_numpy(a).cuda().requires_grad_(True)
    theta = torch.from_numpy(rng.standard_normal(n)).requires_grad_(True)
    E0, B0 = (leaf(0.1 * rng.standard_normal((3, ny, nx)).astype(np.float32)) for _ in range(2))
    win = torch.from_numpy(rng.uniform(0, 1, (1, ny, nx)).astype(np.float32)).cuda()
    EN, BN = make_function().apply(theta, E0, B0, run, False)
    assert EN.untyped_storage().data_ptr() != BN.untyped_storage().data_ptr()
    if edit:
        EN.mul_(win)
        BN[:, 0] = 0.0
        loss = 0.5 * ((EN * EN).sum() + (BN * BN).sum())
    else:
        keep = torch.ones_like(BN)
        keep[:, 0] = 0.0
        loss = 0.5 * (((EN * win) * (EN * win)).sum() + ((BN * keep) * (BN * keep)).sum())
    return [g.cpu().numpy() for g in torch.autograd.grad(loss, (theta, E0, B0))]


def test_outputs_can_be_edited_in_place():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_13088_gb300 import build
    build.build()
    for got, want in zip(_gradients(True), _gradients(False)):
        # the same operations in the same order on either side
        assert np.array_equal(got, want)
