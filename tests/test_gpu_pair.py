"""The DFT passes over pairs of scan positions (csrc/pair.cuh) at the edges of what they take.

Against the FP64 oracle with the bars of test_gpu_parity.py, and against the one-field passes (any
variant flag selects them; RECOMPUTE_COLUMNS is their default at 256^2 and above): both evaluate the
same operations per field, so predicted patterns and the loss are compared bit for bit when the batches
are the same, and gradients to a few units of the FP32 rounding (2^-23 relative per operation; the
probe gradient's positions and the position batches may be added in another order)."""
import numpy as np
import pytest
import torch

from synthetic import workloads as syn
from test_gpu_parity import (Case, _assert_offsets_ok, _offset_errors, _offsets, assert_ok, check_all, dev,  # noqa: F401
                             max_rel, strong_z)

pytestmark = pytest.mark.gpu

ONE_FIELD = 1        # PTYCHO_FLAG_RECOMPUTE_COLUMNS
GRAD_REORDERED = 4e-6


def _case(dev, F, L, M, n_side, seed, **kw):
    w = syn.tiny_workload(F=F, L=L, M=M, n_side=n_side, step=F // 8, seed=seed, remap=True, loss="poisson",
                          with_sigma=True, with_bg=True, **kw)
    return Case(w, dev, z=strong_z(F), mask_kind="frame", seed=seed)


# positions per batch: even, odd (rounded down by the plan), two, and all nine at once (one empty lane);
# modes: one (a warp per row), three (rows per block rounded to whole warps), ten (at 512^2 two feeding
# warps), eleven (at 256^2 no block fits: the one-field passes)
@pytest.mark.parametrize("F,L,M,B", [(64, 2, 1, 4), (64, 3, 3, 9), (128, 2, 1, 3), (128, 1, 2, 9), (128, 2, 5, 2),
                                     (256, 2, 1, 9), (256, 1, 3, 4), (256, 1, 10, 9), (256, 1, 11, 4),
                                     (512, 2, 1, 9), (512, 1, 3, 2), (512, 1, 10, 5)])
def test_pairs_meet_the_oracle_and_the_one_field_passes(dev, F, L, M, B):
    case = _case(dev, F, L, M, 3, 40 + F + 10 * M + B)
    sb = B * L * M * F * F * 8
    plan = case.plan(scratch_bytes=sb)
    assert_ok(check_all(case, plan))
    assert_ok(check_all(case, plan, frames=[8, 1, 5]))             # an odd subset in any order
    ref = case.plan(scratch_bytes=sb, flags=ONE_FIELD)
    args = (case.O, case.P, case.sig_t, case.bg_t)
    assert max_rel(plan.forward(*args).cpu().numpy(), ref.forward(*args).cpu().numpy()) < 1e-6
    a = plan.adjoint(case.O, case.P, case.Im, case.sig_t, case.bg_t, case.mask_t)
    b = ref.adjoint(case.O, case.P, case.Im, case.sig_t, case.bg_t, case.mask_t)
    assert abs(float(a[0].item()) / float(b[0].item()) - 1) < 1e-6
    for x, y in zip(a[1:], b[1:]):
        assert max_rel(x.cpu().numpy(), y.cpu().numpy()) < GRAD_REORDERED
    again = plan.adjoint(case.O, case.P, case.Im, case.sig_t, case.bg_t, case.mask_t)
    assert all(torch.equal(x, y) for x, y in zip(a, again))
    plan.close()
    ref.close()


@pytest.mark.parametrize("F", [64, 256, 512])
def test_probes_that_are_not_16_byte_aligned(dev, F):
    """Probe rows then arrive by 8-byte copies instead of bulk copies: the same bits."""
    case = _case(dev, F, 1, 2, 3, 7)
    plan = case.plan()
    store = torch.empty(case.P.numel() + 1, dtype=torch.complex64, device=dev)
    shifted = store[1:].view(case.P.shape)
    shifted.copy_(case.P)
    assert shifted.data_ptr() % 16 == 8
    a = plan.adjoint(case.O, case.P, case.Im, case.sig_t, case.bg_t, case.mask_t)
    b = plan.adjoint(case.O, shifted, case.Im, case.sig_t, case.bg_t, case.mask_t)
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    plan.close()


@pytest.mark.parametrize("F,M", [(64, 1), (128, 3), (512, 2)])
@pytest.mark.parametrize("bad", [[4, -1, 2], [-1, 4, 2], [4, 2, 99], [-1, -1, 4, 2]])
def test_a_bad_position_index_leaves_its_partner_alone(dev, F, M, bad):
    """An index out of range is skipped and flagged; the valid position in the other lane of its pair
    gives what the valid positions alone give (their order is the same)."""
    case = _case(dev, F, 2, M, 3, 9)
    good = [j for j in bad if 0 <= j < case.w.J]
    plan = case.plan()
    t = lambda v: torch.tensor(v, dtype=torch.int32, device=dev)  # noqa: E731
    a = plan.adjoint(case.O, case.P, case.Im, case.sig_t, case.bg_t, case.mask_t, t(bad))
    assert plan.status() & 1
    b = plan.adjoint(case.O, case.P, case.Im, case.sig_t, case.bg_t, case.mask_t, t(good))
    assert plan.status() == 0
    assert abs(float(a[0].item()) / float(b[0].item()) - 1) < 1e-12
    for x, y in zip(a[1:], b[1:]):
        assert np.isfinite(x.cpu().numpy()).all()
        assert max_rel(x.cpu().numpy(), y.cpu().numpy()) < GRAD_REORDERED
    plan.close()


# fractional offsets of several pixels and of exactly none, one mode and several, an odd batch (the last
# position's lane of the scratch slot) and positions taken one by one (the one-field slot)
@pytest.mark.parametrize("F,L,M,B", [(64, 2, 1, 9), (128, 1, 3, 3), (256, 1, 2, 1), (512, 1, 2, 2)])
def test_shift_by_axes(dev, F, L, M, B):
    case = _case(dev, F, L, M, 3, 90 + F + B)
    delta = _offsets(case.w, F + B, amp=2.5)
    delta[0, 2] = 0.0
    delta[0, 3, 1] = 0.0
    plan = case.plan(scratch_bytes=B * L * M * F * F * 8)
    _assert_offsets_ok(_offset_errors(case, plan, delta))
    _assert_offsets_ok(_offset_errors(case, plan, delta, [8, 0, 5]))
    plan.close()
