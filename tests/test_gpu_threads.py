"""Host threads that launch the same kernels with different shared-memory sizes
(bins, states, logits) at the same time: no launch is refused."""
import threading

import pytest

torch = pytest.importorskip("torch")

from paper_1709_10187_gb300 import build as B  # noqa: E402
from paper_1709_10187_gb300 import rddmc as R  # noqa: E402
from paper_1709_10187_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _walk(w):
    p = R.Problem(w)
    p.ensure_state(32)
    return lambda: p.launch(32, w.seed, max_steps=4)


def _time(w):
    p, n = R.Problem(w), 32
    state = torch.empty(R.time_state_bytes(n), dtype=torch.uint8, device="cuda")
    bins, path = (torch.zeros(w.ncell * p.J, dtype=torch.int64, device="cuda") for _ in range(2))
    counts = torch.zeros(5, dtype=torch.int64, device="cuda")
    ts = R.TimeStep(w.seed, n, 4, 0.0, 1.0e-3, 1, 0, 0, 0, 0)
    return lambda: R.time_step_launch(p.grid, p.table.data_ptr(), ts, state.data_ptr(), state.numel(),
                                      p.tally.data_ptr(), p.tally.numel() * 8, bins.data_ptr(), path.data_ptr(),
                                      counts.data_ptr(), _stream())


def _network(n_out):
    nA, batch = n_out - 32, 64
    wf = 0.1 * torch.randn(R.mlp_param_count(n_out), device="cuda")
    wb = wf.to(torch.bfloat16)
    X = torch.randn((batch, 16), device="cuda").to(torch.bfloat16)
    t = torch.zeros(batch, dtype=torch.int32, device="cuda")
    work = torch.empty(R.mlp_work_bytes(batch, n_out), dtype=torch.uint8, device="cuda")
    grad, loss = torch.empty_like(wf), torch.zeros(1, device="cuda")
    return lambda: R.mlp_loss_grad(n_out, nA, 32, wf.data_ptr(), wb.data_ptr(), X.data_ptr(), t.data_ptr(),
                                   t.data_ptr(), batch, work.data_ptr(), grad.data_ptr(), loss.data_ptr(), _stream())


@pytest.mark.parametrize("make,small,large,calls", [
    (_walk, W.TINY, W.TINY.with_(J=8000), 20_000),
    (_time, W.TINY, W.P2, 20_000),
    (_network, 48, 544, 4000),
], ids=["walk", "time", "network"])
def test_launches_of_different_sizes_are_not_refused(make, small, large, calls):
    B.build()
    errors, fns = [], [make(small), make(large)]
    torch.cuda.synchronize()

    def work(fn):
        with torch.cuda.stream(torch.cuda.Stream()):
            for i in range(calls):
                try:
                    fn()
                except R.RDDMCError as e:
                    errors.append(str(e))
                if i % 64 == 63:
                    torch.cuda.current_stream().synchronize()

    ts = [threading.Thread(target=work, args=(fn,)) for fn in fns]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not errors, (len(errors), errors[0])
