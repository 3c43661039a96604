"""The FP32 tile factor as its launch runs it (host model, no GPU): blocks 0 and 1
take the chain's tile rows in turn and the other CTAs the list of tasks, without
the chain's own.  Block l % 2 waits for tiles (l, l - 2), (l - 1, l - 2) and the
updates of (l, l - 1), applies that tile's last update, solves it against the panels
of L_l-1,l-1 as the other block counts them off, waits for the updates of (l, l),
applies the last one and factors it, counting its own panels.  The launch cannot
deadlock if, with the chain as far on as the finished tasks let it, the next task
of the list has all it waits for: then the first unfinished task is never stuck,
whatever the number of CTAs.  Replaying the tile operations in that order in numpy
(FP64) must give the Cholesky factor."""
import numpy as np
import pytest

from test_chol_tasks import CHAIN_SOLVE, FINAL_DIAG, FINAL_OFF, INV, TILE, UPDATE, tasks


class Chain:
    """Blocks 0 and 1: block b's tile rows b, b + 2, ...; one step of it is the
    part of a row between two waits."""

    def __init__(self, nb, state, panels, ops):
        self.nb, self.state, self.panels, self.ops = nb, state, panels, ops
        self.row = [0, 1]
        self.stage = [0, 0]  # 0: before the solve, 1: solving (panels seen in self.seen), 2: before the factor
        self.seen = [0, 0]

    def step(self, b):
        """Whether block b got on."""
        l, s, nb = self.row[b], self.state, self.nb
        if l >= nb:
            return False
        if self.stage[b] == 0:
            if l >= 2 and not (s[l, l - 2] >= l - 1 and s[l - 1, l - 2] >= l - 1 and s[l, l - 1] >= l - 2):
                return False
            if l >= 2:
                assert s[l, l - 1] == l - 2
                self.ops.append((UPDATE, l, l - 1, l - 2))
            self.stage[b], self.seen[b] = (1 if l else 2), 0
            return True
        if self.stage[b] == 1:
            if self.panels[l - 1] <= self.seen[b]:
                return False
            self.seen[b] += 1
            if self.seen[b] == 4:
                self.ops.append((CHAIN_SOLVE, l, l - 1, l - 1))
                s[l, l - 1] = l
                self.stage[b] = 2
            return True
        if l >= 2 and s[l, l] < l - 1:
            return False
        if self.panels[l] == 0:
            assert l < 2 or s[l, l] == l - 1
            self.ops.append((FINAL_DIAG, l, l, l - 1))
        self.panels[l] += 1
        if self.panels[l] == 4:
            s[l, l] = l + 1
            self.row[b], self.stage[b] = l + 2, 0
        return True

    def run(self):
        while self.step(0) | self.step(1):
            pass


def replay(m, nproc):
    """The operations in the order of the model, or an assertion."""
    nb = -(-m // TILE)
    state, panels, ops = np.zeros((nb, nb), dtype=np.int64), np.zeros(nb, dtype=np.int64), []
    chain = Chain(nb, state, panels, ops)
    for kind, i, l, k in tasks(m, nproc):
        if kind in (FINAL_DIAG, CHAIN_SOLVE) or (kind == UPDATE and k == l - 1):
            continue  # the chain's own
        chain.run()
        if kind == INV:
            assert state[l, l] >= l + 1 and panels[l] == 4
        elif kind == UPDATE:
            assert state[i, k] >= k + 1 and state[l, k] >= k + 1 and state[i, l] == k, (i, l, k)
            state[i, l] = k + 1
        else:
            assert l == 0 or (state[i, l - 1] >= l and state[l, l - 1] >= l and state[i, l] == l - 1), (i, l)
            assert panels[l] == 4, (i, l)
            state[i, l] = l + 1
        ops.append((kind, i, l, k))
    chain.run()
    assert all(state[i, l] == l + 1 for l in range(nb) for i in range(l, nb))
    return ops


@pytest.mark.parametrize("m,nproc", [(1, 304), (128, 152), (129, 1), (300, 2), (513, 3), (1000, 152), (2048, 152),
                                     (4096, 152), (4096, 7), (8192, 152)])
def test_no_task_waits_for_a_later_one(m, nproc):
    nb = -(-m // TILE)
    ops = replay(m, nproc)
    assert len(ops) == len(set(ops)) == nb + nb * (nb + 1) // 2 + sum(
        max(0, l - 1) * (nb - l) for l in range(nb)) + max(0, nb - 2)


@pytest.mark.parametrize("m,nproc", [(300, 3), (700, 152)])
def test_the_order_gives_the_factor(m, nproc):
    rng = np.random.default_rng(m)
    G = rng.standard_normal((m, m + 7))
    M = G @ G.T + m * np.eye(m)
    W = np.tril(M).copy()
    s = lambda t: slice(t * TILE, min(m, (t + 1) * TILE))
    for kind, i, l, k in replay(m, nproc):
        if kind == INV:
            continue
        if kind == CHAIN_SOLVE:
            W[s(i), s(l)] = np.linalg.solve(W[s(l), s(l)], W[s(i), s(l)].T).T
            continue
        if kind == UPDATE or l > 0:
            kk = k if kind == UPDATE else l - 1
            W[s(i), s(l)] -= W[s(i), s(kk)] @ W[s(l), s(kk)].T
        if kind == FINAL_DIAG:
            B = np.tril(W[s(l), s(l)])
            W[s(l), s(l)] = np.linalg.cholesky(B + np.tril(B, -1).T)
        elif kind == FINAL_OFF:
            W[s(i), s(l)] = np.linalg.solve(W[s(l), s(l)], W[s(i), s(l)].T).T
    W = np.tril(W)
    assert np.abs(W - np.linalg.cholesky(M)).max() <= 1e-12 * np.abs(W).max()
