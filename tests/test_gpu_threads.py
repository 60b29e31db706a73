"""Several host threads share the kernels with networks of different sizes (GPU).

Every network of a precision runs in the same kernel with its own amount of
shared memory. Threads that plan and launch a small network must not take
shared memory away from a launch of a large one in another thread: all calls
succeed, with the results of the same calls from one thread.
"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_10558_gb300 import build as _build  # noqa: E402

_build.build()
from paper_2511_10558_gb300 import carbox, synth  # noqa: E402

YR = synth.YEAR
CALLS = 150


def _caller(kind, net, prec, C, t_end):
    """A function that runs one call of the kind on its own buffers and stream."""
    N = carbox.Network.from_synth(net)
    dev = torch.device("cuda:0")
    phi = torch.tensor(synth.cells(C, seed=5), device=dev)
    x0 = torch.tensor(np.repeat(synth.initial_abundances(net)[:, None], C, axis=1), device=dev).contiguous()
    opt = carbox.options(precision=prec)
    stream = torch.cuda.Stream(dev)
    stream.wait_stream(torch.cuda.current_stream(dev))
    if kind == "grad":
        tape = carbox.Tape(N, C, 400)
        with torch.cuda.stream(stream):
            carbox.solve_record(N, tape, phi, x0, 0.0, t_end, opt)
            cot = torch.ones_like(x0)
        stream.synchronize()

    def call():
        with torch.cuda.stream(stream):
            if kind == "grad":
                out = carbox.grad(tape, cot, C)[0]
            else:
                out = carbox.solve(N, phi, x0, 0.0, t_end, opt)[0]
            stream.synchronize()
            return out.cpu().numpy()

    return call


@pytest.mark.parametrize("kind,prec", [("solve", carbox.CBX_MIXED), ("solve", carbox.CBX_FP64),
                                       ("grad", carbox.CBX_FP64)])
def test_threads_with_networks_of_two_sizes(net32, net150, kind, prec):
    large = _caller(kind, net150, prec, 1, 1.0)
    small = [_caller(kind, net32, prec, 1, 1.0) for _ in range(3)]
    want = large()
    done, failed = threading.Event(), []

    def spin(call):
        first = None
        try:
            while not done.is_set():
                out = call()
                first = out if first is None else first
                np.testing.assert_array_equal(out, first)
        except Exception as e:  # noqa: BLE001 (reported by the test's thread)
            failed.append(e)

    threads = [threading.Thread(target=spin, args=(c,)) for c in small]
    for t in threads:
        t.start()
    try:
        for _ in range(CALLS):
            np.testing.assert_array_equal(large(), want)
    finally:
        done.set()
        for t in threads:
            t.join()
    assert not failed, failed


def test_server_takes_small_requests_while_large_ones_launch(net32, net150):
    opt = carbox.options(precision=carbox.CBX_MIXED)
    nets = [carbox.Network.from_synth(n) for n in (net150, net32)]
    cells = [(synth.cells(1, seed=6), synth.initial_abundances(n)[:, None].copy()) for n in (net150, net32)]
    srv = carbox.Server(mem_budget=1 << 30, n_streams=8)
    ids = [(k % 5 != 0, srv.submit(nets[k % 5 != 0], *cells[k % 5 != 0], 0.0, 1.0 + k, opt)) for k in range(400)]
    outs = [(which, srv.wait(i)) for which, i in ids]
    srv.close()
    assert all(np.all(st == carbox.CBX_CELL_OK) for _, (_, st, _) in outs)
