"""Runs of independent sparse pivots in the FP64 LU (GPU).

Networks shaped as trees on a core of species that all react with each other:
their leaves, then the levels above, are runs of sparse pivots one after
another, of lengths with every remainder of the eight warps, and a dense tail
follows. That each network has such runs and its matrix in shared memory is
asserted from the compiled network (the star networks of test_gpu_schedules
have one run each: 20 species have none, and with 160 the matrix is in global
memory, where there are no runs; a dense tail follows there too). A batch takes
two cells to an SM, where the lists come from the L2, and is bitwise its cells.

Both sides run at rtol 1e-7: their global errors (1 to 10 rtol) stay a factor of
ten below the bound.
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
from tests.test_lu_pipeline import run_ends  # noqa: E402

YR = synth.YEAR


def tree(S, core, depth):
    """S species: a core, each with each, and `depth` levels on it, each species linked to two of the level before."""
    rng = np.random.default_rng(S + core)
    rx = []

    def link(a, b):
        for i, j in ((a, b), (b, a)):
            rx.append((synth.COSMIC_RAY, (int(i),), (int(j),), 10.0 ** rng.uniform(1.0, 4.0), 0.0, 0.0))

    for a in range(core):
        for b in range(a):
            link(a, b)
    level, at = list(range(core)), core
    for d in range(depth):
        n = (S - core) // depth + (d < (S - core) % depth)
        for v in range(at, at + n):
            for u in rng.choice(level, 2, replace=False):
                link(v, u)
        level, at = list(range(at, at + n)), at + n
    return tiny(S, rx)


@pytest.mark.parametrize("S,core,depth,cells", [(60, 40, 3, 1), (90, 20, 3, 300), (97, 30, 4, 1), (120, 40, 3, 1),
                                                (140, 20, 2, 1), (140, 30, 5, 1)])
def test_trees_against_oracle(S, core, depth, cells):
    net = tree(S, core, depth)
    N = carbox.Network.from_synth(net)
    _, F, kd = N.symbolic()
    ends = run_ends(F, kd)
    runs = [e - k for k, e in enumerate(ends) if k == 0 or ends[k - 1] != e]
    assert len(runs) >= 2 and max(runs) > 8 and kd < S - 3 and N.info()["smem_bytes_fp64"] <= 227 * 1024 - 64
    dev = torch.device("cuda:0")
    phi = synth.cells(cells, seed=S)
    x0 = np.linspace(1.0, 0.1, S)[:, None].repeat(cells, axis=1)
    opt = carbox.options(rtol=1e-7, atol=1e-20)

    def solve(n):
        x, st, _ = carbox.solve(N, torch.tensor(phi[:n], device=dev), torch.tensor(x0[:, :n].copy(), device=dev), 0.0,
                                3e6 * YR, opt)
        assert np.all(st.cpu().numpy() == carbox.CBX_CELL_OK)
        return x.cpu().numpy()

    x = solve(cells)
    np.testing.assert_array_equal(x[:, :1], solve(1))
    ref = bdf.solve_cell(net, phi[0], x0[:, 0], 0.0, 3e6 * YR, 1e-7, 1e-20).x
    assert np.max(np.abs(x[:, 0] / ref - 1.0)) <= 1e-5
