"""Cells with tracks are taken by what they meet along them (GPU).

Half of the cells come out of the shade late in their span, the others stay
under some extinction. The former have more photo-reaction times ahead of them
and have to be among the first that a launch takes, although the first knots of
their tracks say otherwise. The order changes no result.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_10558_gb300 import build as _build  # noqa: E402

_build.build()
from paper_2511_10558_gb300 import carbox, synth  # noqa: E402

YR = synth.YEAR


@pytest.mark.parametrize("K", [2, 4, 40])
def test_cells_out_of_the_shade_come_first(net150, K):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    C, t_end = 2 * sms + 91, 3.0 * YR
    N = carbox.Network.from_synth(net150)
    dev = torch.device("cuda:0")
    phi = synth.cells(C, seed=21)
    late = np.arange(C) % 2 == 1
    phi[:, 2] = np.where(late, 20.0, 3.0)
    track = np.empty((C, K, 6))
    s = np.linspace(0.0, 1.0, K)
    track[:, :, 0] = s * t_end
    track[:, :, 1:] = phi[:, None, :]
    track[late, :, 3] = 20.0 * (1.0 - s)
    x0 = np.repeat(synth.initial_abundances(net150)[:, None], C, axis=1)
    stats = carbox.stats_tensor(C, dev)
    x, st, _ = carbox.solve_track(N, torch.tensor(track, device=dev), torch.tensor(x0, device=dev), 0.0, t_end,
                                  stats=stats)
    assert np.all(st.cpu().numpy() == carbox.CBX_CELL_OK)
    begin = stats[:, 10:12].contiguous().view(torch.int64).cpu().numpy()[:, 0]
    first = np.argsort(begin, kind="stable")[:min(sms, int(late.sum()))]  # one CTA an SM: the first wave
    assert late[first].all()
    part = np.arange(60)
    xp, _, _ = carbox.solve_track(N, torch.tensor(track[part], device=dev),
                                  torch.tensor(x0[:, part].copy(), device=dev), 0.0, t_end)
    np.testing.assert_array_equal(x.cpu().numpy()[:, part], xp.cpu().numpy())
