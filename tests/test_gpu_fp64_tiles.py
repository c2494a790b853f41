"""FP64 contractions in small tiles: sizes at the edges of the 16 x 16 tiles, of the
64-wide tiles that the result is defined on and of the split sums over K."""
import numpy as np
import pytest

from paper_2606_04316_gb300 import synth

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 64, 65, 130, 209])
@pytest.mark.parametrize("k", [1, 15, 16, 17, 333])
def test_second_half_tiles(torch_cuda, n, k):
    torch = torch_cuda
    from paper_2606_04316_gb300 import qdt
    rng = np.random.default_rng(1000 * n + k)
    D, V = rng.standard_normal((k, n)), rng.standard_normal((k, n))
    O = torch.full((n, n), float("nan"), dtype=torch.float64, device="cuda")
    qdt.second_half_noalloc(torch.from_numpy(D).cuda(), torch.from_numpy(V).cuda(), O)
    got = O.cpu().numpy()
    # k products and at most 64 partial sums, each rounded once
    bound = (k + 66) * EPS * (np.abs(D).T @ np.abs(V))
    tile = np.arange(n) // 64
    upper = tile[:, None] <= tile[None, :]
    assert np.all((np.abs(got - D.T @ V) <= 2 * bound)[upper])


@pytest.mark.parametrize("centres,kramers", [(1, 1), (2, 2), (3, 3), (3, 5)])
def test_first_half_tiles(oracle, torch_cuda, centres, kramers):
    """4, 12, 24 and 60 columns; rows and ket prefixes that end inside a tile."""
    torch = torch_cuda
    from paper_2606_04316_gb300 import qdt
    p = synth.chain_problem(centres, kramers, seed=730 + kramers, shells=(0, 1), nprim=2, blocks=("coulomb", "gauge"),
                            tau=0.0)
    ctx = qdt.Context(0)
    ctx.set_basis(p.basis)
    ctx.set_coefficients(p.CL, p.CS)
    blocks = ("coulomb", "gauge")
    out = torch.zeros(ctx.packed_size(blocks, 0, kramers) // 8, dtype=torch.float64, device="cuda")
    ctx.transform(blocks, 0, kramers, 0.0, qdt.FP64, out)
    tr = oracle.Transform(p)
    ref = np.concatenate([tr.packed(b).reshape(-1) for b in blocks])
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-12
