"""A batch whose requests live on the caller's own streams, while another thread keeps those
streams busy: what the fused launches read of a request is uploaded on that request's stream,
behind the thread's work, so the launches have to wait for it.  Results as alone."""
import threading

import numpy as np
import pytest

from paper_2606_04316_gb300 import synth

pytestmark = pytest.mark.gpu
BLOCKS = ("coulomb", "gaunt", "gauge")
TOL = 1e-12            # a fused launch may regroup sums (as in the batch tests)


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def test_batch_on_busy_streams(torch_cuda):
    torch = torch_cuda
    from paper_2606_04316_gb300 import qdt
    probs = [(synth.chain_problem(3 + i, 3, seed=781 + i, shells=(0, 1), nprim=2, blocks=BLOCKS, tau=1e-11), i % 2)
             for i in range(4)]
    streams = [torch.cuda.Stream() for _ in probs]
    ctxs, outs, alone = [], [], []
    for (p, prec), s in zip(probs, streams):
        ctx = qdt.Context(0, stream=s)
        ctx.set_basis(p.basis)
        ctx.set_coefficients(p.CL, p.CS)
        out = torch.zeros(ctx.packed_size(BLOCKS, 0, p.nK) // 8, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ctx.transform(BLOCKS, 0, p.nK, p.tau, prec, out)
        alone.append(out.cpu().numpy())
        ctxs.append(ctx)
        outs.append(out)
    load = [torch.zeros(1 << 26, device="cuda") for _ in probs[1:]]      # 256 MB: a pass takes about 0.1 ms
    torch.cuda.synchronize()
    stop = threading.Event()

    def busy():
        flight = []
        while not stop.is_set():
            for s, b in zip(streams[1:], load):
                with torch.cuda.stream(s):
                    for _ in range(4):
                        b.add_(1.0)
                    e = torch.cuda.Event()
                    e.record(s)
                    flight.append(e)
            while len(flight) > 4 * len(load):
                flight.pop(0).synchronize()

    th = threading.Thread(target=busy)
    th.start()
    try:
        for _ in range(5):
            qdt.transform_batch([(c, BLOCKS, 0, p.nK, p.tau, prec, o)
                                 for c, (p, prec), o in zip(ctxs, probs, outs)])
            got = [o.cpu().numpy() for o in outs]
            for a, b in zip(alone, got):
                assert np.abs(a - b).max() <= TOL
    finally:
        stop.set()
        th.join()
        torch.cuda.synchronize()
    for c in ctxs:
        c.close()
