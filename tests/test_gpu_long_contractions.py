"""Plain-FP32 integrals of long contractions: the sum over the outer primitive pairs keeps its
rounding errors, so a contraction of many primitives is no further off than one primitive.

The bound: with one primitive per shell an integral's error is that of a single primitive
quartet, e.  The contracted integral is a sum of such quartets with independent errors, which
average (all terms of s shells are of one sign); the inner FP32 sums (n / 2 = npp / 2 terms in
each of two chains, about 0.4 sqrt(n / 6) units of 2^-24 each) average over the outer pairs
as well, and a compensated outer sum adds nothing.  So the ratio stays below the largest e of
the same shells."""
import pytest

from paper_2606_04316_gb300 import synth

pytestmark = pytest.mark.gpu
BLOCKS = ("coulomb", "gaunt", "gauge")
SEEDS = (771, 772, 773)


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def ratio(shells, nprim, seed):
    from paper_2606_04316_gb300 import qdt
    p = synth.chain_problem(2, 2, seed=seed, shells=shells, nprim=nprim, blocks=BLOCKS, tau=0.0)
    ctx = qdt.Context(0)
    ctx.set_basis(p.basis)
    ctx.set_coefficients(p.CL, p.CS)
    r = [*ctx.f32_error_ratio(["coulomb", "gaunt"], 0, 2, 0.0), ctx.f32_error_ratio(["gauge"], 0, 2, 0.0)[1]]
    ctx.close()
    return r


@pytest.mark.parametrize("shells,nprim", [((0,), 16), ((1,), 9)])
def test_outer_sum_adds_no_error(torch_cuda, shells, nprim):
    one = [max(v) for v in zip(*(ratio(shells, 1, s) for s in SEEDS))]
    for seed in SEEDS:
        got = ratio(shells, nprim, seed)
        print(shells, nprim, seed, "ratios", got, "one primitive", one)
        assert max(got) <= max(one)
