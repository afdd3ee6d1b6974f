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


PAIR_PASSES, BATCH_POSITIONS, ROW_ADJ_SPLITS, COLUMN_GROUPS = range(4)      # PTYCHO_QUERY_* of include/ptycho.h


# the counts beside each line of the rule: one field per position by frame size, modes that fill whole warps
# of a block of 320 threads and the next that do not, one position per batch, flags
@pytest.mark.parametrize("F,L,M,B,flags,pair", [
    (64, 1, 1, 9, 0, 1), (128, 1, 1, 9, 0, 1), (256, 1, 1, 9, 0, 0), (512, 1, 1, 9, 0, 0), (256, 2, 1, 9, 0, 1),
    (512, 2, 1, 9, 0, 1), (512, 1, 10, 2, 0, 1), (512, 1, 11, 2, 0, 0), (256, 1, 11, 4, 0, 0), (256, 1, 20, 4, 0, 1),
    (128, 1, 40, 4, 0, 1), (64, 1, 80, 4, 0, 1), (64, 1, 88, 4, 0, 0), (256, 1, 4, 1, 0, 0), (256, 1, 4, 3, 0, 1),
    (256, 1, 4, 4, ONE_FIELD, 0), (256, 1, 4, 4, 512, 1)])
def test_which_plans_take_the_pair_passes(dev, F, L, M, B, flags, pair):
    from paper_2311_14780_gb300 import Plan
    plan = Plan(F, L, M, 9, [(F, F)] * L, np.zeros((L, 9, 2), np.int32), scratch_bytes=B * L * M * F * F * 8, flags=flags)
    assert plan.query(PAIR_PASSES) == pair
    assert plan.query(BATCH_POSITIONS) == (B - B % 2 if pair else B)   # whole pairs within the budget
    plan.close()


# as many modes as a block of the pair row adjoint takes
@pytest.mark.parametrize("F,M", [(256, 18), (256, 20), (128, 40), (64, 72), (64, 80)])
def test_many_modes(dev, F, M):
    case = _case(dev, F, 1, M, 3, 60 + F + M)
    plan = case.plan()
    assert plan.query(PAIR_PASSES) == 1
    assert_ok(check_all(case, plan))
    assert_ok(check_all(case, plan, frames=[8, 1, 5]))
    plan.close()


@pytest.mark.parametrize("F,L,M", [(64, 2, 1), (64, 1, 80), (128, 2, 5), (128, 1, 1), (256, 1, 3), (256, 2, 10), (512, 2, 1),
                                   (512, 1, 10)])
def test_patterns_and_loss_are_the_one_field_passes_bit_by_bit(dev, F, L, M):
    """With the same positions per batch and one mode group."""
    case = _case(dev, F, L, M, 3, 70 + F + M)
    kw = dict(scratch_bytes=4 * L * M * F * F * 8, col_groups=1)
    plan, ref = case.plan(**kw), case.plan(flags=ONE_FIELD, **kw)
    assert (plan.query(PAIR_PASSES), ref.query(PAIR_PASSES)) == (1, 0)
    assert all(p.query(BATCH_POSITIONS) == 4 and p.query(COLUMN_GROUPS) == 1 for p in (plan, ref))
    args = (case.O, case.P, case.sig_t, case.bg_t)
    assert torch.equal(plan.forward(*args), ref.forward(*args))
    loss = [p.loss(case.O, case.P, case.Im, case.sig_t, case.bg_t, case.mask_t) for p in (plan, ref)]
    assert torch.equal(*loss)
    plan.close()
    ref.close()


def test_a_short_batch_reaches_every_split(dev):
    """One-field passes with as many position splits as positions: every split gets one, so that the probe
    gradient is the sum of the positions' own ones, in their order, bit by bit."""
    case = _case(dev, 64, 1, 1, 3, 91)
    plan = case.plan(scratch_bytes=9 * 64 * 64 * 8, flags=4)             # KEEP_PSI, the one-field default at 64^2
    assert plan.query(PAIR_PASSES) == 0 and plan.query(ROW_ADJ_SPLITS) == plan.query(BATCH_POSITIONS) == 9
    grad = lambda b: plan.adjoint(case.O, case.P, case.Im, case.sig_t, case.bg_t, case.mask_t, b)[2]  # noqa: E731
    total = torch.zeros_like(case.P)
    for j in range(9):
        total = total + grad(torch.tensor([j], dtype=torch.int32, device=dev))
    assert torch.equal(grad(None), total)
    plan.close()


@pytest.mark.parametrize("F,L,M,splits", [(64, 1, 72, 5), (64, 3, 72, 3), (128, 1, 40, 1), (256, 1, 20, 1)])
def test_many_modes_split_their_positions(dev, F, L, M, splits):
    """Blocks of 288 to 320 threads run one per SM: where F L of them leave rounds half empty (64 or 192 on 152
    SMs) the positions are split, as far as there are pairs of them (five here); 128 or 256 fill theirs as well
    unsplit."""
    from paper_2311_14780_gb300 import Plan
    plan = Plan(F, L, M, 9, [(F, F)] * L, np.zeros((L, 9, 2), np.int32))
    assert torch.cuda.get_device_properties(dev).multi_processor_count == 152
    assert plan.query(PAIR_PASSES) == 1
    assert plan.query(ROW_ADJ_SPLITS) == splits
    plan.close()


# the pair and the one-field column passes (plain, TMA, staged, recomputed, one block per SM, without TMA)
@pytest.mark.parametrize("F,M,flags", [(64, 40, 0), (64, 40, 4), (64, 40, 16), (64, 40, 64), (128, 40, 0), (128, 8, 4),
                                       (256, 20, 0), (256, 20, 1), (512, 10, 0), (512, 10, 1), (512, 10, 65536),
                                       (512, 10, 8), (512, 10, 4), (512, 10, 64)])
def test_intensity_sum_rounds_once_per_mode(dev, F, M, flags):
    """Constant objects and probes put all of a mode into the pattern's centre, exactly: |Psi_m|^2 = F^2 |c_m|^2.
    The first mode's 2^24 has a unit of 2 in its last place, so each later one may cost half of it, 1; adding
    the squares of the real and the imaginary part (0.77 each) one after the other would lose both."""
    from paper_2311_14780_gb300 import Plan
    plan = Plan(F, 1, M, 2, [(F, F)], np.zeros((1, 2, 2), np.int32), flags=flags, col_groups=1)
    assert plan.query(COLUMN_GROUPS) == 1
    c = torch.full((1, M, 1, 1), 0.875 + 0.875j, dtype=torch.complex64, device=dev)
    c[0, 0] = 4096.0
    I = plan.forward(torch.ones(F * F, dtype=torch.complex64, device=dev), c.expand(1, M, F, F).contiguous())
    centre = I[:, F // 2, F // 2].double().cpu().numpy() / F ** 2
    assert np.abs(centre - (2.0 ** 24 + (M - 1) * 1.53125)).max() <= M - 1
    assert float(I.double().sum().item()) == float(I[:, F // 2, F // 2].double().sum().item())
    plan.close()


@pytest.mark.parametrize("F,fields,J,batch", [(64, 5, 43, 43), (64, 5, 44, 15), (128, 8, 23, 23), (128, 8, 24, 8), (128, 30, 20, 7),
                                              (64, 8, 768, 128), (512, 1, 8, 8), (512, 1, 9, 3)])
def test_chirp_z_batches(dev, F, fields, J, batch):
    """Chirp-z batches hold 1200 fields (and at least 64 positions); a call is one batch instead of three only with few
    positions and few elements."""
    from paper_2311_14780_gb300 import Plan
    plan = Plan(F, 1, fields, J, [(F, F)], np.zeros((1, J, 2), np.int32), zoom=[1.0])
    assert plan.query(BATCH_POSITIONS) == batch
    plan.close()


@pytest.mark.parametrize("F,L,M,J,splits", [(256, 3, 10, 9, 1), (256, 2, 3, 60, 4), (256, 3, 4, 60, 3), (128, 5, 8, 60, 3)])
def test_splits_follow_the_rounds_of_blocks(dev, F, L, M, J, splits):
    """Several rounds of blocks are split where that saves a tenth of them (768 blocks of 10 modes on 304 places: three
    rounds either way), one round always (256 blocks of three modes)."""
    from paper_2311_14780_gb300 import Plan
    plan = Plan(F, L, M, J, [(F, F)] * L, np.zeros((L, J, 2), np.int32))
    assert torch.cuda.get_device_properties(dev).multi_processor_count == 152
    assert plan.query(ROW_ADJ_SPLITS) == splits
    plan.close()


@pytest.mark.parametrize("F,L,M,flags", [(64, 2, 3, 0), (128, 1, 4, 0), (256, 2, 3, 0), (512, 1, 2, 0), (512, 1, 12, 0),
                                         (64, 1, 1, 0), (256, 1, 4, ONE_FIELD)])
def test_subsets_of_every_size_class(dev, F, L, M, flags):
    """Calls beside the lines where a plan changes its passes and mode groups: one position, the most that take the
    one-field passes and one more, half of the batch and one more, all but one."""
    case = _case(dev, F, L, M, 5, 95 + F + M)
    plan = case.plan(flags=flags)
    order = np.random.default_rng(F).permutation(case.w.J)
    assert case.w.J == 25
    for n in (1, 2, 10, 11, 12, 13, 16, 17, 24):
        assert_ok(check_all(case, plan, frames=[int(j) for j in order[:n]]))
    plan.close()
