"""A call waits for the GPU where it needs a result, not between its stages: more
stages than the context has timing events, both precisions, host and device outputs."""
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


@pytest.mark.parametrize("nb", [0, 1, 5])
@pytest.mark.parametrize("host", [False, True])
def test_many_stages(oracle, torch_cuda, nb, host):
    """MO blocks of one index: 12 row batches and 12 screenings per class."""
    torch = torch_cuda
    from paper_2606_04316_gb300 import qdt
    p = synth.chain_problem(2, 12, seed=741, shells=(0, 1), nprim=2, blocks=BLOCKS, tau=0.0)
    ctx = qdt.Context(0)
    ctx.set_basis(p.basis)
    ctx.set_coefficients(p.CL, p.CS)
    if nb:
        ctx.set_route("mo", nb)
    tr = oracle.Transform(p)
    ref = np.concatenate([tr.packed(b).reshape(-1) for b in BLOCKS])
    n = ctx.packed_size(BLOCKS, 0, 12) // 8
    for prec, tol in ((qdt.FP64, 1e-12), (qdt.SPLIT, 1e-10)):
        out = np.full(n, np.nan) if host else torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        for _ in range(2):
            st = ctx.transform(BLOCKS, 0, 12, 0.0, prec, out)
        got = out if host else out.cpu().numpy()
        assert np.abs(got - ref).max() <= tol
        spans = [st["ms_" + k] for k in ("density", "screen", "eri", "half1", "half2", "pack")]
        assert all(t > 0 for t in spans) and sum(spans) <= st["ms_total"] * 1.001
