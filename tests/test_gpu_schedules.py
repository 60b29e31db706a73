"""Schedules of the linear algebra at the sizes where they can go wrong (GPU).

* Runs of independent sparse pivots: a star (every species reacts with the hubs
  alone) is one run from the first pivot to the hubs, which are the last pivot,
  too few pivots for pairs, or a dense tail that the pairs take over; the tail's
  column groups of at most 16 columns come with the sizes.
* The matrix in global memory: one row more than a CTA's threads, a last block
  of 1, 3 and 32 columns, leading panels that are sparse.

Both sides run at rtol 1e-7, where their step programs may differ (a rounding
can flip a decision of the step controller) but their global errors, measured
at 1 to 10 rtol on these networks, stay a factor of ten below the bound.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_10558_gb300 import build as _build  # noqa: E402

_build.build()
from oracle import bdf  # noqa: E402
from paper_2511_10558_gb300 import carbox, synth  # noqa: E402
from tests.nets import tiny  # noqa: E402

YR = synth.YEAR
RTOL, BOUND = 1e-7, 1e-5


def _check(net, S, precision, t_end):
    N = carbox.Network.from_synth(net)
    dev = torch.device("cuda:0")
    phi = synth.cells(1, seed=S)
    x0 = np.linspace(1.0, 0.1, S)[:, None].copy()
    x, st, _ = carbox.solve(N, torch.tensor(phi, device=dev), torch.tensor(x0, device=dev), 0.0, t_end,
                            carbox.options(rtol=RTOL, atol=1e-20, precision=precision))
    assert np.all(st.cpu().numpy() == carbox.CBX_CELL_OK)
    ref = bdf.solve_cell(net, phi[0], x0[:, 0], 0.0, t_end, RTOL, 1e-20).x
    assert np.max(np.abs(x.cpu().numpy()[:, 0] / ref - 1.0)) <= BOUND


@pytest.mark.parametrize("S", [20, 98, 130, 160])
@pytest.mark.parametrize("hubs", [1, 2, 4, 17])
def test_star_against_oracle(S, hubs):
    rx = []
    for i in range(hubs, S):
        for h in range(hubs):
            rx.append((synth.COSMIC_RAY, (i,), (h,), 3.0 + i + h, 0.0, 0.0))
            rx.append((synth.COSMIC_RAY, (h,), (i,), 1.0 + 0.1 * i, 0.0, 0.0))
    for h in range(hubs):
        for g in range(hubs):
            if g != h:
                rx.append((synth.COSMIC_RAY, (h,), (g,), 2.0 + h + g, 0.0, 0.0))
    _check(tiny(S, rx), S, carbox.CBX_FP64, 3e6 * YR)


@pytest.mark.parametrize("S", [257, 259, 288])
@pytest.mark.parametrize("precision", [carbox.CBX_FP64, carbox.CBX_MIXED])
def test_global_matrix_against_oracle(S, precision):
    # a ring beside random exchange: sparse first pivots, a dense tail
    rng = np.random.default_rng(S)
    rx = [(synth.COSMIC_RAY, (i,), ((i + 1) % S,), 5.0 + (i % 11), 0.0, 0.0) for i in range(S)]
    rx += [(synth.COSMIC_RAY, (int(a),), (int(b),), 1.0 + a % 5, 0.0, 0.0)
           for a, b in rng.integers(0, S, (2 * S, 2)) if a != b]
    _check(tiny(S, rx), S, precision, 1e5 * YR)
