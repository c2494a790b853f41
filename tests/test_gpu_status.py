"""The status word of the split form's contractions over a whole call: a give-up recorded by
one class outlives the hand-back of the digit planes before the next, and the hand-back makes
no give-up of its own.  QDT_SPLIT_FAIL records the give-up without a wait running out;
QDT_W_BUDGET makes the planes be handed back."""
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
