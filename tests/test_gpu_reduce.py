"""The fixed-order sums that finish a call (k_loss_reduce), at the edges of what a block, a cluster and
an unrolled pass of it take."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

J = 2100          # 64^2 frames: four partials each, 8 blocks of 256 threads, four loads in flight: 2048 entries a pass


@pytest.fixture(scope="module")
def stack():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2311_14780_gb300 import Plan
    g = torch.Generator().manual_seed(5)
    pos = torch.randint(0, 17, (1, J, 2), generator=g).numpy().astype(np.int32)
    dev = torch.device("cuda", 0)
    plan = Plan(64, 1, 1, J, [(80, 80)], pos)
    O = torch.randn(80 * 80, generator=g, dtype=torch.complex64).to(dev)
    P = torch.randn(1, 1, 64, 64, generator=g, dtype=torch.complex64).to(dev)
    Im = torch.rand(J, 64, 64, generator=g).to(dev)
    yield plan, O, P, Im
    plan.close()


# fewer partials than threads of the first block (the others have none), one more than a block, a
# cluster and a pass of four, and every position
@pytest.mark.parametrize("n", [1, 2, 64, 65, 512, 513, 2048, 2049, 2100])
def test_loss_of_repeated_frames(stack, n):
    """n times the same frame: n times its loss, up to the FP64 roundings of 4 n additions (each entry's
    partials are the same numbers), and the same bits from every call."""
    plan, O, P, Im = stack
    one = float(plan.loss(O, P, Im, batch=torch.zeros(1, dtype=torch.int32, device=O.device)).item())
    idx = torch.zeros(n, dtype=torch.int32, device=O.device)
    got = [float(plan.loss(O, P, Im, batch=idx).item()) for _ in range(20)]
    assert len(set(got)) == 1
    assert abs(got[0] / (n * one) - 1) <= 4 * n * 2.0 ** -53
    assert plan.status() == 0


# positions per block of the loss pass: one (few of 64^2) and eight (83 of 256^2), the last group of three;
# the frame's place in its group
@pytest.mark.parametrize("F,J,j", [(64, 3, 0), (64, 3, 2), (256, 83, 0), (256, 83, 7), (256, 83, 8), (256, 83, 82)])
def test_loss_keeps_64_bits_over_a_block(F, J, j):
    """Terms of three warps of a block that FP64 adds exactly and a double-float (two FP32 numbers) cannot
    hold: 2^36 + 2^10 + 2^-16.  A zero probe leaves the background alone; every other term is zero."""
    from paper_2311_14780_gb300 import Plan
    dev = torch.device("cuda", 0)
    plan = Plan(F, 1, 1, J, [(F, F)], np.zeros((1, J, 2), np.int32), scratch_bytes=(J + 1) * F * F * 8)
    bg = torch.ones(F, F)
    flat = bg.view(-1)
    flat[0], flat[128], flat[256] = 2.0 ** 36, 2.0 ** 10, 2.0 ** -16
    Im = bg.repeat(J, 1, 1)
    Im[j].view(-1)[[0, 128, 256]] = 0.0
    O = torch.ones(F * F, dtype=torch.complex64, device=dev)
    P = torch.zeros(1, 1, F, F, dtype=torch.complex64, device=dev)
    got = plan.loss(O, P, Im.to(dev), bg=bg.to(dev))
    assert float(got.item()) == 2.0 ** 36 + 2.0 ** 10 + 2.0 ** -16
    plan.close()
