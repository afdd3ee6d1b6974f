"""Plan creation on a GPU with little memory left."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_default_batches_shrink_to_what_is_left():
    """512 positions per batch in three buffer sets take 2 GB; with 1 GB left the plan takes smaller batches, and
    gives what it gives with room."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2311_14780_gb300 import Plan
    dev = torch.device("cuda", 0)
    F, M, J = 64, 40, 1536
    g = torch.Generator().manual_seed(2)
    pos = torch.randint(0, 17, (1, J, 2), generator=g).numpy().astype(np.int32)
    O = torch.randn(80 * 80, generator=g, dtype=torch.complex64).to(dev)
    P = torch.randn(1, M, F, F, generator=g, dtype=torch.complex64).to(dev)
    Im = torch.rand(J, F, F, generator=g).to(dev)
    Plan(F, 1, 1, 2, [(F, F)], np.zeros((1, 2, 2), np.int32)).close()       # the library itself is in memory
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device=dev)
    try:
        small = Plan(F, 1, M, J, [(80, 80)], pos)
    finally:
        del hog
        torch.cuda.empty_cache()
    roomy = Plan(F, 1, M, J, [(80, 80)], pos)
    batch = [p.query(1) for p in (small, roomy)]                            # PTYCHO_QUERY_BATCH_POSITIONS
    assert batch[1] == 512 and 64 <= batch[0] < 512
    a, b = (p.loss(O, P, Im).item() for p in (small, roomy))
    assert abs(a / b - 1) < 1e-6
    small.close()
    roomy.close()
