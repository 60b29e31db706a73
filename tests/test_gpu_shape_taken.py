"""The CTA shape that a batch is given (GPU).

Bitwise comparisons between shapes mean something only if the shape under test
ran. The cells' begin and end times tell: those that began before the first one
ended are the launch's CTAs. Expected are the CTAs per SM of the shape that the
plan has for the network, precision, method and cells per SM; the sizes are
those of the bitwise comparisons and both sides of the plan's lines.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_10558_gb300 import build as _build  # noqa: E402

_build.build()
from paper_2511_10558_gb300 import carbox, synth  # noqa: E402

YR = synth.YEAR
FP64, MIXED = carbox.CBX_FP64, carbox.CBX_MIXED
BDF, ESDIRK = carbox.CBX_METHOD_BDF, carbox.CBX_METHOD_ESDIRK


@pytest.mark.parametrize("S,load,prec,method,ctas", [
    (32, 1.0, FP64, BDF, (1, 1)), (33, 2.0, FP64, BDF, (2, 2)), (32, 5.0, MIXED, BDF, (3, 4)),
    (48, 1.05, FP64, ESDIRK, (1, 1)), (48, 6.1, FP64, BDF, (5, 8)), (48, 6.1, MIXED, ESDIRK, (5, 8)),
    (49, 1.4, FP64, BDF, (1, 1)), (49, 1.6, FP64, ESDIRK, (2, 2)), (49, 4.6, MIXED, BDF, (3, 4)),
    (64, 1.6, MIXED, BDF, (2, 2)), (65, 4.1, FP64, ESDIRK, (3, 4)), (96, 4.1, FP64, BDF, (2, 2)),
    (96, 1.6, MIXED, BDF, (2, 2)), (97, 3.9, FP64, BDF, (1, 1)), (97, 4.1, FP64, BDF, (2, 2)),
    (111, 4.1, FP64, BDF, (2, 2)), (112, 4.1, FP64, BDF, (1, 1)), (113, 6.1, MIXED, ESDIRK, (2, 2)),
    (152, 5.9, MIXED, BDF, (1, 1)), (152, 6.1, MIXED, BDF, (2, 2)), (153, 6.1, MIXED, BDF, (2, 2)),
    (154, 6.1, MIXED, BDF, (1, 1)), (150, 8.0, FP64, BDF, (1, 1)), (200, 4.1, FP64, BDF, (2, 2)),
    (257, 1.9, MIXED, BDF, (1, 1)), (257, 2.1, MIXED, ESDIRK, (2, 2)), (257, 2.1, FP64, BDF, (2, 2))])
def test_shape_of_a_batch(S, load, prec, method, ctas):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    C = int(load * sms)
    net = synth.make_network(S, 6 * S)
    N = carbox.Network.from_synth(net)
    dev = torch.device("cuda:0")
    phi = torch.tensor(synth.cells(C, seed=S), device=dev)
    x0 = torch.tensor(np.repeat(synth.initial_abundances(net)[:, None], C, axis=1), device=dev).contiguous()
    stats = carbox.stats_tensor(C, dev)
    _, st, _ = carbox.solve(N, phi, x0, 0.0, 3.0 * YR, carbox.options(precision=prec, method=method), stats=stats)
    assert np.all(st.cpu().numpy() == carbox.CBX_CELL_OK)
    times = stats[:, 10:14].contiguous().view(torch.int64).cpu().numpy()  # begin, end of each cell
    together = int((times[:, 0] < times[:, 1].min()).sum())
    lo, hi = (min(n * sms, C) for n in ctas)
    assert lo <= together <= hi, (together, sms)
