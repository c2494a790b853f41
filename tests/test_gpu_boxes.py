"""Integral tiles over the boxes of non-zero Hermite terms, primitive pairs in
twos: every kind of shell pair (diagonal and not, derivative functions of s, p
and d shells), odd and even numbers of primitive pairs, contractions so long
that the inner primitive pairs run in several parts, and pairs so large that
the function pairs do, against the oracle.

Tolerances are the forms' own: 1e-12 (FP64) and 1e-10 (split) for outputs of at
most 1 at the recipe's coefficient scale."""
import numpy as np
import pytest

from paper_2606_04316_gb300 import synth

pytestmark = pytest.mark.gpu
BLOCKS = ("coulomb", "gaunt", "gauge")


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


# shells of each centre, primitives per shell
@pytest.mark.parametrize("shells,nprim", [
    ((0,), 1),              # one primitive pair: half of a two
    ((1,), 1),
    ((2,), 1),              # derivative functions of d shells: 324 function pairs, cut
    ((2, 0), 2),            # an even number of primitive pairs
    ((0, 1), 3),            # nine primitive pairs: the unrolled case
    ((1,), 5),              # 25 primitive pairs
    ((1,), 9),              # 81 primitive pairs: tensors of order 8 in several parts
])
def test_every_kind_of_pair_against_oracle(oracle, torch_cuda, shells, nprim):
    torch = torch_cuda
    from paper_2606_04316_gb300 import qdt
    p = synth.chain_problem(2, 2, seed=710 + nprim, shells=shells, nprim=nprim, blocks=BLOCKS, tau=0.0)
    ctx = qdt.Context(0)
    ctx.set_basis(p.basis)
    ctx.set_coefficients(p.CL, p.CS)
    out = torch.zeros(ctx.packed_size(BLOCKS, 0, 2) // 8, dtype=torch.float64, device="cuda")
    tr = oracle.Transform(p)
    ref = np.concatenate([tr.packed(b).reshape(-1) for b in BLOCKS])
    for prec, tol in ((qdt.FP64, 1e-12), (qdt.SPLIT, 1e-10)):
        out.zero_()
        ctx.transform(BLOCKS, 0, 2, 0.0, prec, out)
        assert np.abs(out.cpu().numpy() - ref).max() <= tol
    # the Coulomb kernel over L-S pairs too (no gauge block)
    sub = torch.zeros(ctx.packed_size(["gaunt"], 0, 2) // 8, dtype=torch.float64, device="cuda")
    ctx.transform(["gaunt"], 0, 2, 0.0, qdt.FP64, sub)
    n = sub.numel()
    assert np.abs(sub.cpu().numpy() - ref[n: 2 * n]).max() <= 1e-12
