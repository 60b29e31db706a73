"""What a server's limits mean, whatever shape its launches take (GPU).

max_ctas is the most CTAs of a launch, or as many SMs' worth where several CTAs
share an SM (up to eight, of small networks), and may be as large as an int.

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


@pytest.mark.parametrize("prec", [carbox.CBX_FP64, carbox.CBX_MIXED])
@pytest.mark.parametrize("max_ctas", [1, 8, 76, 200])
def test_max_ctas_is_a_share_of_the_device(net32, prec, max_ctas):
    N = carbox.Network.from_synth(net32)
    C, opt = 400, carbox.options(precision=prec)
    phi, x0 = _request(net32, C, 1)
    srv = carbox.Server(mem_budget=1 << 30, n_streams=1, max_ctas=max_ctas)
    out = srv.wait(srv.submit(N, phi, x0, 0.0, 10.0 * YR, opt))
    peak = srv.stats()["peak_bytes"]
    srv.close()
    assert peak <= _bytes(N, C, 8 * max_ctas) + 4 * C  # and the order of the cells
    _check(N, phi, x0, 10.0 * YR, opt, out)


def test_max_ctas_of_any_size(net32):
    N = carbox.Network.from_synth(net32)
    opt = carbox.options()
    phi, x0 = _request(net32, 1300, 2)
    srv = carbox.Server(mem_budget=1 << 30, n_streams=1, max_ctas=2**31 - 1)
    out = srv.wait(srv.submit(N, phi, x0, 0.0, YR, opt))
    srv.close()
    _check(N, phi, x0, YR, opt, out)
