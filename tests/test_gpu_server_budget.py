"""A server's memory budget, whatever shape its launches take (GPU).

* A request is refused when one cell to an SM does not fit the budget, and
  taken when it does, in the callers' order if there is no room for another.
* Requests whose least reservations fit side by side run side by side.

Reservations are checked through the server's peak: inputs, outputs and end
times of the cells, a workspace per CTA, 8 KB. Results are bitwise those of
cbx_solve.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_10558_gb300 import build as _build  # noqa: E402

_build.build()
from paper_2511_10558_gb300 import carbox, synth  # noqa: E402

YR = synth.YEAR


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _request(net, C, seed):
    return synth.cells(C, seed=seed), np.repeat(synth.initial_abundances(net)[:, None], C, axis=1)


def _bytes(N, C, ctas):
    info = N.info()
    ws = 8 * ((3 * info["R"] + info["nnz_jac"] + 31) // 32 * 32)  # matrix in shared memory
    return C * (40 + 16 * info["S"] + 12) + ctas * ws + 8192


def _check(N, phi, x0, t_end, opt, out):
    want, st, _ = carbox.solve_host(N, phi, x0, 0.0, t_end, opt)
    np.testing.assert_array_equal(out[1], st)
    np.testing.assert_array_equal(out[0], want)
    assert np.all(st == carbox.CBX_CELL_OK)


@pytest.mark.parametrize("S,C", [(32, 1300), (150, 400)])
def test_budget_of_the_least_launch(net32, net150, S, C):
    net = net32 if S == 32 else net150
    N = carbox.Network.from_synth(net)
    opt = carbox.options(precision=carbox.CBX_MIXED)
    phi, x0 = _request(net, C, 3)
    least = _bytes(N, C, _sms())
    srv = carbox.Server(mem_budget=least - 1, n_streams=2, max_ctas=0)
    with pytest.raises(carbox.CarboxError) as e:
        srv.submit(N, phi, x0, 0.0, YR, opt)
    assert e.value.code == carbox.CBX_E_TOO_LARGE
    srv.close()
    srv = carbox.Server(mem_budget=least, n_streams=2, max_ctas=0)
    ids = [srv.submit(N, phi, x0, 0.0, YR, opt) for _ in range(2)]  # the second queues behind the first
    small = srv.submit(N, phi[:3], x0[:, :3].copy(), 0.0, YR, opt)
    for i in ids:
        _check(N, phi, x0, YR, opt, srv.wait(i))
    _check(N, phi[:3], x0[:, :3].copy(), YR, opt, srv.wait(small))
    assert srv.stats()["peak_bytes"] <= least
    srv.close()


def test_room_for_several_cells_on_an_sm_is_used(net32):
    N = carbox.Network.from_synth(net32)
    opt = carbox.options()
    phi, x0 = _request(net32, 2000, 4)
    srv = carbox.Server(mem_budget=1 << 30, n_streams=1, max_ctas=0)
    out = srv.wait(srv.submit(N, phi, x0, 0.0, YR, opt))
    assert srv.stats()["peak_bytes"] >= _bytes(N, 2000, 4 * _sms())
    srv.close()
    _check(N, phi, x0, YR, opt, out)


def test_a_long_queue_leaves_the_shapes(net32, net150):
    # one stream, held by a long cell; behind it a batch that runs several cells to an SM, and forty requests
    # (one cell to an SM whatever they are given) that exceed the budget together but wait for the stream
    net61 = synth.make_network(61, 480)
    N32, N61, N150 = (carbox.Network.from_synth(n) for n in (net32, net61, net150))
    opt = carbox.options()
    phi, x0 = _request(net32, 2000, 6)
    one = _bytes(N61, _sms(), _sms())
    budget = 34 * one
    srv = carbox.Server(mem_budget=budget, n_streams=1, max_ctas=0)
    ids = [srv.submit(N150, *_request(net150, 1, 7), 0.0, 1e7 * YR, opt), srv.submit(N32, phi, x0, 0.0, YR, opt)]
    many = _request(net61, _sms(), 8)
    ids += [srv.submit(N61, *many, float(k), YR, opt) for k in range(40)]  # not merged: different start times
    outs = [srv.wait(i) for i in ids]
    peak = srv.stats()["peak_bytes"]
    srv.close()
    assert _bytes(N32, 2000, 4 * _sms()) <= peak <= budget
    _check(N32, phi, x0, YR, opt, outs[1])
    assert all(np.all(st == carbox.CBX_CELL_OK) for _, st, _ in outs)


def test_requests_run_side_by_side_where_their_least_fits(net150):
    N = carbox.Network.from_synth(net150)
    opt = carbox.options(precision=carbox.CBX_MIXED)
    C, t_end = 304, 1e6 * YR
    phi, x0 = _request(net150, C, 5)
    srv = carbox.Server(mem_budget=2 * _bytes(N, C, _sms()), n_streams=2, max_ctas=0)
    # different start times: not merged; the first runs for tens of milliseconds
    ids = [(t0, srv.submit(N, phi, x0, t0, t_end, opt)) for t0 in (0.0, 1.0)]
    for _, i in ids:
        assert np.all(srv.wait(i)[1] == carbox.CBX_CELL_OK)
    assert srv.stats()["peak_running"] == 2
    srv.close()
