"""CTA shapes and the pair pipeline of the FP64 LU (GPU).

Batches run with several cells on an SM in a shape chosen from the network's
size and the number of cells; small launches run one cell to an SM. A cell's
arithmetic is the same in every shape, so a batch must be bitwise its cells
solved in small launches. The sizes are the edges of the shapes: 48/49, 64/65
and 96/97 species, the last that fit two FP64 cells (111) and two mixed ones
(152) on an SM and the first that do not, the first with the matrix in global
memory and with more rows than a warp set (257).

The dense pivots of the FP64 LU go in pairs through a pipeline of warps: from
one species to past two column groups, linear chains (dense after ordering or
not) must agree with the oracle.
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
FP64, MIXED = carbox.CBX_FP64, carbox.CBX_MIXED
BDF, ESDIRK = carbox.CBX_METHOD_BDF, carbox.CBX_METHOD_ESDIRK
PART = 100  # below the number of SMs: one cell to an SM


@pytest.mark.parametrize("S,C,prec,method", [
    (33, 160, FP64, BDF), (48, 930, FP64, BDF), (48, 930, MIXED, ESDIRK), (49, 240, FP64, ESDIRK),
    (49, 700, MIXED, BDF), (64, 240, MIXED, BDF), (64, 620, FP64, BDF), (65, 620, FP64, ESDIRK), (65, 240, FP64, BDF),
    (96, 620, FP64, BDF), (96, 250, MIXED, BDF), (97, 620, FP64, BDF), (111, 620, FP64, BDF), (112, 620, FP64, BDF),
    (150, 1250, FP64, BDF), (150, 700, FP64, ESDIRK), (154, 700, FP64, BDF), (155, 700, FP64, BDF),
    (113, 930, MIXED, ESDIRK), (152, 930, MIXED, BDF), (153, 930, MIXED, BDF), (200, 620, FP64, BDF),
    (226, 620, MIXED, BDF), (257, 310, MIXED, BDF), (257, 310, FP64, BDF), (257, 310, MIXED, ESDIRK)])
def test_batch_is_bitwise_its_parts(S, C, prec, method):
    net = synth.make_network(S, 6 * S)
    N = carbox.Network.from_synth(net)
    dev = torch.device("cuda:0")
    phi = synth.cells(C, seed=S)
    x0 = np.repeat(synth.initial_abundances(net)[:, None], C, axis=1)
    opt = carbox.options(precision=prec, method=method)

    def solve(sel):
        x, st, _ = carbox.solve(N, torch.tensor(phi[sel], device=dev),
                                torch.tensor(x0[:, sel], device=dev).contiguous(), 0.0, 3.0 * YR, opt)
        return x.cpu().numpy(), st.cpu().numpy()

    x, st = solve(np.arange(C))
    assert np.all(st == carbox.CBX_CELL_OK)
    for sel in (np.arange(PART), np.arange(C - PART, C)):
        xp, _ = solve(sel)
        np.testing.assert_array_equal(x[:, sel], xp)


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 6, 7, 9, 16, 31, 32, 33, 34, 35, 64, 65, 66, 67, 98])
@pytest.mark.parametrize("cells", [1, 400])
def test_chain_against_oracle(S, cells):
    # X0 -> X1 -> ... -> X_{S-1} -> X0 by cosmic rays, and every species back to X0
    rx = [(synth.COSMIC_RAY, (i,), ((i + 1) % S,), 10.0 + 7.0 * i, 0.0, 0.0) for i in range(S if S > 1 else 0)]
    rx += [(synth.COSMIC_RAY, (i,), (0,), 3.0 + i, 0.0, 0.0) for i in range(2, S)]
    rx += [(synth.PHOTO, (0,), (i,), 1e-14 * i, 1.0, 0.0) for i in range(2, S)]
    if S == 1:
        rx = [(synth.COSMIC_RAY, (0,), (0, 0), 1.0, 0.0, 0.0)]
    net = tiny(S, rx)
    N = carbox.Network.from_synth(net)
    dev = torch.device("cuda:0")
    phi = synth.cells(cells, seed=3)
    x0 = np.repeat(np.linspace(1.0, 0.1, S)[:, None], cells, axis=1)
    t_end = 3e6 * YR
    x, st, _ = carbox.solve(N, torch.tensor(phi, device=dev), torch.tensor(x0, device=dev).contiguous(), 0.0, t_end,
                            carbox.options(rtol=1e-7, atol=1e-20))
    assert np.all(st.cpu().numpy() == carbox.CBX_CELL_OK)
    x = x.cpu().numpy()
    # at rtol 1e-4 a rounding can flip a step decision (66 species: 8e-4 apart,
    # both within the method's error); at 1e-7 the methods' errors stay below 1e-6
    for c in (0, cells - 1):
        ref = bdf.solve_cell(net, phi[c], x0[:, c], 0.0, t_end, 1e-7, 1e-20).x
        assert np.max(np.abs(x[:, c] / ref - 1.0)) <= 1e-5
