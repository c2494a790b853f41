"""The status word of the split form's contractions over a whole call: a give-up recorded by
one class outlives the hand-back of the digit planes before the next, the hand-back makes no
give-up of its own, and the blocks behind a give-up are not written.  QDT_SPLIT_FAIL records the
give-up without a wait running out; QDT_W_BUDGET makes the planes be handed back."""
import numpy as np
import pytest

from paper_2606_04316_gb300 import synth

pytestmark = pytest.mark.gpu
BLOCKS = ("coulomb", "gaunt", "gauge")
TIMEOUT = -6


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def make(qdt, seed=761):
    p = synth.chain_problem(2, 2, seed=seed, shells=(0, 1), nprim=2, blocks=BLOCKS, tau=0.0)
    ctx = qdt.Context(0)
    ctx.set_basis(p.basis)
    ctx.set_coefficients(p.CL, p.CS)
    return ctx, ctx.packed_size(BLOCKS, 0, 2) // 8


# integral rows of the L-S class: 8 x 18 function pairs, three components a side, a ninth more for
# the Gaunt block's; 28 KB above them leaves no room for the digit planes of the Coulomb class
BUDGET = str(int(1.12 * 8 * (3 * 8 * 18) ** 2) + 28000)


def test_status_survives_hand_back_of_planes(torch_cuda, monkeypatch):
    torch = torch_cuda
    from paper_2606_04316_gb300 import qdt
    ctx, n = make(qdt)
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    ctx.transform(BLOCKS, 0, 2, 0.0, qdt.SPLIT, out)
    ref = out.clone()
    monkeypatch.setenv("QDT_W_BUDGET", BUDGET)
    for _ in range(3):
        out.zero_()
        ctx.transform(BLOCKS, 0, 2, 0.0, qdt.SPLIT, out)
        assert torch.equal(out, ref)
        # the Coulomb class's first contraction gives up; the L-S class hands the planes back
        monkeypatch.setenv("QDT_SPLIT_FAIL", "1")
        with pytest.raises(qdt.QdtError) as e:
            ctx.transform(BLOCKS, 0, 2, 0.0, qdt.SPLIT, out)
        assert e.value.code == TIMEOUT
        monkeypatch.delenv("QDT_SPLIT_FAIL")
    ctx.close()


@pytest.mark.parametrize("host", [False, True])
def test_blocks_behind_a_give_up_are_not_written(torch_cuda, monkeypatch, host):
    torch = torch_cuda
    from paper_2606_04316_gb300 import qdt
    ctx, n = make(qdt)
    full = torch.zeros(n, dtype=torch.float64, device="cuda")
    ctx.transform(BLOCKS, 0, 2, 0.0, qdt.SPLIT, full)
    ref, per = full.cpu().numpy(), n // len(BLOCKS)
    # contractions in order: Coulomb first and second half, gauge and Gaunt first halves, Gaunt and
    # gauge second halves; the blocks whose contractions all come before the give-up are complete
    for at, done in ((1, 0), (2, 0), (3, 1), (4, 1), (5, 1), (6, 2)):
        out = np.full(n, -7.0) if host else torch.full((n,), -7.0, dtype=torch.float64, device="cuda")
        monkeypatch.setenv("QDT_SPLIT_FAIL", str(at))
        with pytest.raises(qdt.QdtError) as e:
            ctx.transform(BLOCKS, 0, 2, 0.0, qdt.SPLIT, out)
        assert e.value.code == TIMEOUT
        monkeypatch.delenv("QDT_SPLIT_FAIL")
        got, k = (out, 0) if host else (out.cpu().numpy(), done * per)
        assert np.array_equal(got[:k], ref[:k]) and np.all(got[k:] == -7.0), at
        ctx.transform(BLOCKS, 0, 2, 0.0, qdt.SPLIT, out)            # and the context stays usable
        assert np.array_equal(out if host else out.cpu().numpy(), ref)
    ctx.close()


def test_batch_item_that_gives_up_is_not_written(torch_cuda, monkeypatch):
    """An item whose first contraction gives up keeps its output and fails alone."""
    torch = torch_cuda
    from paper_2606_04316_gb300 import qdt
    made = [make(qdt, seed) for seed in (762, 763)]
    refs = []
    for ctx, n in made:
        out = torch.zeros(n, dtype=torch.float64, device="cuda")
        ctx.transform(BLOCKS, 0, 2, 0.0, qdt.SPLIT, out)
        refs.append(out.cpu().numpy())
    outs = [torch.full((n,), -7.0, dtype=torch.float64, device="cuda") for _, n in made]
    jobs = [(ctx, BLOCKS, 0, 2, 0.0, qdt.SPLIT, o) for (ctx, _), o in zip(made, outs)]
    # a batch clears the status for each class: the first contraction of each gives up
    monkeypatch.setenv("QDT_SPLIT_FAIL", "1")
    status, _ = qdt.transform_batch(jobs, raise_on_error=False)
    assert status == [TIMEOUT, TIMEOUT]
    assert all(np.all(o.cpu().numpy() == -7.0) for o in outs)
    monkeypatch.delenv("QDT_SPLIT_FAIL")
    qdt.transform_batch(jobs)
    for o, r in zip(outs, refs):
        assert np.abs(o.cpu().numpy() - r).max() <= 1e-12
    for ctx, _ in made:
        ctx.close()
