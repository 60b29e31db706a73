"""Runs of sparse pivots and the pair pipeline of the FP64 LU, restated (no GPU).

* Runs: consecutive sparse pivots none of which is in another's row or column.
  Their U rows are prepared side by side; then warp w takes the rows i with
  i mod NW = w of every pivot of the run, without a barrier between pivots. In
  whatever order the warps run, the factors are bit for bit those of single
  pivots.
* Pairs: in the dense range warp 0 finishes the next two U rows while the other
  warps (workers; row i belongs to worker i mod (NW - 1)) are still on the rest
  of their rows. Two events replace the block barrier, each a named barrier on
  which one side arrives and the other waits, used in turn by even and odd
  steps. The schedule is run here with its warps interleaved at random: the
  factors are bit for bit those of single pivots, every wait ends, and no
  barrier gets an arrival that belongs to a later step.
"""
import numpy as np
import pytest

from paper_2511_10558_gb300 import synth
from tests.test_dense_range_exact import crout, pattern_and_fill


def run_ends(F, kd):
    """end[k] of the run that holds sparse pivot k, as the host compiler forms it."""
    ends, k = [], 0
    while k < kd:
        e = k + 1
        while e < kd and not any(F[e, p] or F[p, e] for p in range(k, e)):
            e += 1
        ends += [e] * (e - k)
        k = e
    return ends


def crout_runs(A, F, kd, NW, rng):
    """Sparse pivots in runs, warps in a random order; dense pivots singly."""
    M = A.copy()
    S = M.shape[0]
    ends, k = run_ends(F, kd), 0
    while k < S:
        e = ends[k] if k < kd else k + 1
        pivots = [(m, np.arange(m + 1, S), np.arange(m + 1, S)) if m >= kd else
                  (m, np.flatnonzero(F[m + 1:, m]) + m + 1, np.flatnonzero(F[m, m + 1:]) + m + 1)
                  for m in range(k, e)]
        for i in rng.permutation(len(pivots)):  # the U rows, a warp each
            m, _, cols = pivots[i]
            M[m, cols] *= 1.0 / M[m, m]
        for w in rng.permutation(NW):
            for m, rows, cols in pivots:
                for i in rows[rows % NW == w]:
                    M[i, cols] -= M[i, m] * M[m, cols]
        k = e
    return M


def _matrix(P, seed):
    rng = np.random.default_rng(seed)
    S = P.shape[0]
    A = np.where(P, rng.normal(0.0, 1.0, (S, S)), 0.0)
    A[np.diag_indices(S)] = 5.0 + np.abs(A).sum(axis=1)
    return A


@pytest.mark.parametrize("S,R", [(61, 480), (97, 873), (150, 1500)])
def test_runs_bitwise(S, R):
    from paper_2511_10558_gb300 import carbox
    net = synth.make_network(S, R)
    perm, F, kd = carbox.Network.from_synth(net).symbolic()
    ends = run_ends(F, kd)
    assert max(e - k for k, e in enumerate(ends)) >= 3  # the premise: there are runs
    P = pattern_and_fill(net)[0][np.ix_(perm, perm)]
    A = _matrix(P, S)
    want = crout(A, F, kd)
    for seed in range(3):
        np.testing.assert_array_equal(crout_runs(A, F, kd, 8, np.random.default_rng(seed)), want)


class Barrier:
    """A named barrier: `need` threads' worth of arrivals open it once."""

    def __init__(self, need):
        self.need, self.count, self.opened = need, 0, 0

    def arrive(self):
        self.count += 1
        if self.count == self.need:
            self.count, self.opened = 0, self.opened + 1


def _finish(M, p, prev=None):
    if prev is not None:
        M[p, prev + 1:] -= M[p, prev] * M[prev, prev + 1:]
    M[p, p + 1:] *= 1.0 / M[p, p]


def crout_pipeline(A, NW, rng):
    """The dense range from pivot 0 on with NW warps; returns the factors."""
    M = A.copy()
    S = M.shape[0]
    M[0, 1:] *= 1.0 / M[0, 0]
    M[1:, 1:] -= np.outer(M[1:, 0], M[0, 1:])  # pivot 0 alone, rows 1 and 2 finished
    _finish(M, 1)
    if S > 2:
        _finish(M, 2, 1)
    workers = range(1, NW)
    group = {g: [w for w in workers if w % 4 == g] for g in range(4)}
    first = [Barrier(NW), Barrier(NW)]  # every worker and warp 0
    urows = {(g, s): Barrier(1 + len(group[g])) for g in range(4) for s in (0, 1) if group[g]}
    done = {w: -1 for w in range(NW)}   # the last step whose event this warp has sent
    steps = list(enumerate(range(1, S - 2, 2)))

    def pair(i, k):
        a = M[i, k]
        x = M[i, k + 1:] - a * M[k, k + 1:]
        b = x[0]
        x[1:] = x[1:] - b * M[k + 1, k + 2:]
        M[i, k + 1:] = x

    def wait(bar, others, step):
        # (a thread that waits also arrives; it goes on when the barrier opens)
        opened = bar.opened
        bar.arrive()
        while bar.opened == opened:
            yield
        assert all(done[o] >= step for o in others), "opened before the step it stands for"

    def warp0():
        for step, k in steps:
            if step > 0:
                yield from wait(first[(step - 1) & 1], workers, step - 1)
            pair(k + 2, k)
            _finish(M, k + 2)
            if k + 3 < S:
                pair(k + 3, k)
                _finish(M, k + 3, k + 2)
            yield
            done[0] = step
            for g in range(4):
                if group[g]:
                    assert urows[g, step & 1].count < urows[g, step & 1].need
                    urows[g, step & 1].arrive()
        if steps:
            yield from wait(first[steps[-1][0] & 1], workers, steps[-1][0])

    def worker(w):
        nw = NW - 1
        for step, k in steps:
            if step > 0:
                yield from wait(urows[w % 4, (step - 1) & 1], [0], step - 1)
            sent = False
            i = k + 4 + ((w - 1) + nw * S - (k + 4)) % nw
            while i < S:
                for r in (i, i + nw):  # two rows at a time
                    if r < S:
                        pair(r, k)
                if not sent:
                    done[w] = step
                    first[step & 1].arrive()
                    sent = True
                yield
                i += 2 * nw
            if not sent:
                done[w] = step
                first[step & 1].arrive()
        if steps:
            yield from wait(urows[w % 4, steps[-1][0] & 1], [0], steps[-1][0])

    live = [warp0()] + [worker(w) for w in workers]
    turns = 0
    while live:
        t = live[rng.integers(len(live))]
        try:
            next(t)
        except StopIteration:
            live.remove(t)
        turns += 1
        assert turns < 2000 * S, "a wait does not end"
    return M


@pytest.mark.parametrize("NW", [2, 4, 8])
@pytest.mark.parametrize("S", [3, 4, 5, 6, 9, 16, 33, 64, 97])
def test_pair_pipeline_bitwise(S, NW):
    A = _matrix(np.ones((S, S), dtype=bool), S)
    want = crout(A, np.ones((S, S), dtype=bool), 0)
    for seed in range(4):
        np.testing.assert_array_equal(crout_pipeline(A, NW, np.random.default_rng(seed)), want)
