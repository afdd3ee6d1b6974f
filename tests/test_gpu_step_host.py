"""ptycho_step_host with the measured patterns of a batch copied in several pieces."""
import numpy as np
import pytest
import torch

from synthetic import workloads as syn
from test_gpu_parity import Case, dev, strong_z  # noqa: F401

pytestmark = pytest.mark.gpu


# 21 MB of patterns in one batch: pieces of 32, 32 and 17 positions (one-field and pair passes), 26 MB: 8, 8, 8 and
# 1; batches of 48 and 33: 24 and 24, 24 and 9; 1 MB: one piece; the other form of the one-field columns
@pytest.mark.parametrize("F,L,M,n_side,kw", [(256, 1, 1, 9, {}), (256, 1, 2, 9, {}), (512, 1, 1, 5, {}), (512, 1, 2, 5, {}),
                                             (256, 1, 2, 9, dict(scratch_bytes=48 * 2 * 256 * 256 * 8)),
                                             (128, 2, 2, 4, {}), (256, 1, 1, 9, dict(flags=4)), (512, 1, 1, 5, dict(flags=4))])
def test_pieces_take_the_same_step(dev, F, L, M, n_side, kw):
    from paper_2311_14780_gb300 import AdamState
    w = syn.tiny_workload(F=F, L=L, M=M, n_side=n_side, step=F // 16, seed=38, remap=True, loss="poisson", with_sigma=True,
                          with_bg=True)
    case = Case(w, dev, z=strong_z(F), mask_kind="frame", seed=3)
    plan = case.plan(**kw)
    host = torch.as_tensor(case.Ih).contiguous().pin_memory()
    loss = torch.zeros(1, dtype=torch.float64, device=dev)
    loss_host = torch.zeros(1, dtype=torch.float64).pin_memory()
    out = []
    for on_host in (False, True):
        s = AdamState(plan, 1e-2, 1e-1, lr_sigma=1e-2, lr_bg=1e-1, with_z_gradient=True)
        v = [case.O.clone(), case.P.clone(), case.sig_t.clone(), case.bg_t.clone()]
        for _ in range(2):
            if on_host:
                staging = torch.full_like(case.Im, float("nan"))
                plan.step_host(s, v[0], v[1], host, staging, loss, loss_host, v[2], v[3], case.mask_t)
            else:
                plan.step(s, v[0], v[1], case.Im, v[2], v[3], case.mask_t, loss_out=loss)
            torch.cuda.synchronize()
        out.append(v + [s.mO, s.mP, s.m_sigma, s.m_bg, s.g_z, loss.clone()])
    assert torch.equal(staging, case.Im) and float(loss_host.item()) == float(loss.item())
    assert all(torch.equal(a, b) for a, b in zip(*out))
    assert np.isfinite(float(loss.item())) and plan.status() == 0
    plan.close()
