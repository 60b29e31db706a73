"""Networks at the limit of a CTA's shared memory run (GPU).

The FP64 solver keeps its matrix and, where they fit, the sparse pivots' lists
in shared memory. Near the limit a few bytes decide: with the lists the
networks below are exactly at a CTA's dynamic limit (the device's less 64 bytes
of static variables), between the two figures, and just above both. All of them
run, the latter two without the lists.

Both sides run at rtol 1e-7: their global errors (1 to 10 rtol) stay a factor of
ten below the bound, on the species above 1e-12.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_10558_gb300 import build as _build  # noqa: E402

_build.build()
from oracle import bdf  # noqa: E402
from paper_2511_10558_gb300 import carbox, synth  # noqa: E402

YR = synth.YEAR
DEVICE = 227 * 1024  # shared memory a CTA can have
LIMIT = DEVICE - 64


@pytest.mark.parametrize("R,lo,hi", [(1362, LIMIT, LIMIT), (1305, LIMIT + 1, DEVICE), (1307, DEVICE, DEVICE),
                                     (1413, DEVICE + 1, DEVICE + 64)])
def test_networks_at_the_limit(R, lo, hi):
    net = synth.make_network(152, R)
    N = carbox.Network.from_synth(net)
    assert lo <= N.info()["smem_bytes_fp64"] <= hi  # the premise
    dev = torch.device("cuda:0")
    phi = synth.cells(1, seed=R)
    x0 = synth.initial_abundances(net)
    x, st, _ = carbox.solve(N, torch.tensor(phi, device=dev), torch.tensor(x0[:, None].copy(), device=dev), 0.0, YR,
                            carbox.options(rtol=1e-7))
    assert int(st.cpu()[0]) == carbox.CBX_CELL_OK
    ref = bdf.solve_cell(net, phi[0], x0, 0.0, YR, 1e-7, 1e-20).x
    big = ref > 1e-12
    assert np.max(np.abs(x.cpu().numpy()[big, 0] / ref[big] - 1.0)) <= 1e-5
