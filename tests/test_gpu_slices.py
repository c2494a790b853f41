"""Digit planes of the split contractions, four elements at a time: rows and columns of
every length modulo four, rows on 8-byte boundaries (odd pitch), zero rows, values
far apart in one row; density and quarter routes, against the oracle at the split
form's tolerance."""
import numpy as np
import pytest

from paper_2606_04316_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("shells,centres,kramers", [((0,), 1, 1), ((0,), 2, 2), ((0,), 3, 3), ((1,), 1, 2),
                                                    ((0, 1), 1, 3), ((1,), 3, 4), ((0, 0, 1), 2, 3)])
@pytest.mark.parametrize("route", ["density", "quarter"])
def test_lengths(oracle, torch_cuda, shells, centres, kramers, route):
    torch = torch_cuda
    from paper_2606_04316_gb300 import qdt
    blocks = ("coulomb", "gaunt", "gauge") if route == "density" else ("coulomb",)
    p = synth.chain_problem(centres, kramers, seed=760 + centres, shells=shells, nprim=2, blocks=blocks, tau=0.0)
    ctx = qdt.Context(0)
    ctx.set_basis(p.basis)
    CL = np.array(p.CL)
    CL[0] = 0.0                       # rows of zeros in the density
    CL[-1] *= 1e-13                   # and of values far below the others
    ctx.set_coefficients(CL, p.CS)
    ctx.set_route(route)
    p.CL = CL
    tr = oracle.Transform(p)
    ref = np.concatenate([tr.packed(b).reshape(-1) for b in blocks])
    out = torch.full((ctx.packed_size(blocks, 0, kramers) // 8,), float("nan"), dtype=torch.float64, device="cuda")
    ctx.transform(blocks, 0, kramers, 0.0, qdt.SPLIT, out)
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-10
