"""The order in which a launch takes its cells changes no result (GPU).

A launch with more cells than CTAs takes the cells by estimated cost. Each
result must be bitwise that of the same cells solved in launches small enough
to have no order (at most one cell a CTA), whatever the environment holds:
zero and infinite fields, not-a-number (a cell that ends as BAD_INPUT), equal
costs, spans from zero up.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_10558_gb300 import build as _build  # noqa: E402

_build.build()
from paper_2511_10558_gb300 import carbox, synth  # noqa: E402

YR = synth.YEAR
PART = 100  # below the number of SMs: one cell a CTA


def _cells(C, odd):
    phi = synth.cells(C, seed=31)
    if odd:
        phi[::7, 3] = 0.0            # no UV field
        phi[1::7, 4] = 0.0           # no cosmic rays
        phi[2::11, 2] = np.nan       # BAD_INPUT
        phi[3::11, 3] = np.inf       # BAD_INPUT
        phi[4::13, 2] = -5.0
        phi[5::13, 2] = 1e4          # exp(-gamma A_V) underflows
        phi[6::17, 2:4] = (3.0, 0.0)
        phi[6::17, 4] = 0.0          # neither field nor cosmic rays
        phi[7::17, 1] = -1.0         # BAD_INPUT
    return phi


@pytest.mark.parametrize("C,odd,prec", [(153, False, carbox.CBX_FP64), (5000, True, carbox.CBX_FP64),
                                        (2600, True, carbox.CBX_MIXED), (3000, False, carbox.CBX_MIXED)])
def test_ordered_solve_is_bitwise_the_parts(net32, C, odd, prec):
    N = carbox.Network.from_synth(net32)
    dev = torch.device("cuda:0")
    phi = _cells(C, odd)
    if not odd:
        phi[:] = phi[0]  # one bucket holds every cell
        phi[:, 0] *= np.linspace(1.0, 2.0, C)
    x0 = np.repeat(synth.initial_abundances(net32)[:, None], C, axis=1)
    opt = carbox.options(precision=prec)

    def solve(sel):
        p = torch.tensor(phi[sel], device=dev)
        x, st, _ = carbox.solve(N, p, torch.tensor(x0[:, sel], device=dev).contiguous(), 0.0, 30.0 * YR, opt)
        return x.cpu().numpy(), st.cpu().numpy()

    x, st = solve(np.arange(C))
    picks = np.arange(C) if C <= 1000 else np.r_[0:200, C // 2:C // 2 + 100, C - 100:C]
    for a in range(0, len(picks), PART):
        xp, sp = solve(picks[a:a + PART])
        np.testing.assert_array_equal(st[picks[a:a + PART]], sp)
        np.testing.assert_array_equal(x[:, picks[a:a + PART]], xp)
    if odd:
        assert (st == carbox.CBX_CELL_BAD_INPUT).sum() > 0


def test_ordered_track_and_reverse_sweep(net32):
    C = 2100
    N = carbox.Network.from_synth(net32)
    dev = torch.device("cuda:0")
    phi = synth.cells(C, seed=32)
    t_end = 100.0 * YR
    track = synth.tracks(phi, t_end, 3)
    x0 = np.repeat(synth.initial_abundances(net32)[:, None], C, axis=1)
    cot = np.zeros((net32.n_species, C))
    cot[net32.index("H")] = np.linspace(-1.0, 1.0, C)

    def sweep(sel):
        tape = carbox.Tape(N, len(sel), 400)
        x, st = carbox.solve_track_record(N, tape, torch.tensor(track[sel], device=dev),
                                          torch.tensor(x0[:, sel], device=dev).contiguous(), 0.0, t_end)
        g = carbox.grad_env(tape, torch.tensor(cot[:, sel], device=dev).contiguous(), len(sel))
        return [x.cpu().numpy(), st.cpu().numpy()] + [t.cpu().numpy() for t in g[1:]]

    whole = sweep(np.arange(C))
    assert np.all(whole[1] == carbox.CBX_CELL_OK)
    for sel in (np.arange(PART), np.arange(C - PART, C)):
        part = sweep(sel)
        np.testing.assert_array_equal(whole[0][:, sel], part[0])
        for a, b in zip(whole[2:], part[2:]):
            np.testing.assert_array_equal(a[sel], b)
