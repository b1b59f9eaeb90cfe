"""The two lists that the dataflow LDL^T kernel is launched with (no GPU): the main tasks and the critical
ones, row tile s on panels s-2 .. s-4, with S(t, k) and U(t, k+1, k) of a critical row in one task. Every
task once, and no deadlock under any schedule of the kernel's groups: those of the main list hold the
next ticket in reserve while a task runs, the critical ones do not; a folded task keeps its group through
both of its parts."""
import ctypes
import random

import numpy as np
import pytest

FB = 16


@pytest.fixture(scope="module")
def lists():
    import __graft_entry__ as g
    g.build()
    from paper_2502_17683_gb300 import _lib, api
    f = _lib.load().thc_cpd_ldl_device_lists
    f.argtypes = [_lib.I, _lib.I, ctypes.POINTER(ctypes.c_short), _lib.I, _lib.IP]

    def get(R, n):
        cap = len(api.thc_cpd_ldl_schedule(R, n))
        out, nmain = np.zeros((cap, 4), np.int16), ctypes.c_int()
        k = f(R, n, out.ctypes.data_as(ctypes.POINTER(ctypes.c_short)), cap, ctypes.byref(nmain))
        assert 0 <= k <= cap
        t = [tuple(int(v) for v in x) for x in out[:k]]
        return api.thc_cpd_ldl_schedule(R, n), t[:nmain.value], t[nmain.value:]

    return get


@pytest.mark.parametrize("R,n", [(720, 100), (80, 5), (17, 1), (5, 4), (33, 40), (100, 0), (256, 1794), (520, 250)])
def test_lists_hold_every_task_once(lists, R, n):
    all_tasks, main, crit = lists(R, n)
    nT = -(-R // FB)
    assert not any(t < nT and k >= t - 4 for _, t, _, k in main)
    assert all(t < nT and k >= t - 4 for _, t, _, k in crit)
    unfolded = [x for ty, t, j, k in main + crit for x in
                ([(0, t, j, k), (1, t, k + 1, k)] if ty == 2 else [(ty, t, j, k)])]
    assert len(unfolded) == len(set(unfolded)) and set(unfolded) == set(map(tuple, all_tasks))


def _run(R, n, main, crit, workers, crit_workers, seed):
    """Random interleaving of the chain and the groups; returns None or what is left when nothing can move."""
    pick = random.Random(seed)
    nT, nM = -(-R // FB), -(-n // FB)
    cnt = np.zeros((nT + nM, nT), int)
    sdone, fdone = np.zeros(nT + nM, int), 0
    queue, nxt = [main, crit], [0, 0]

    def claim(w):
        nxt[w] += 1
        return queue[w][nxt[w] - 1] if nxt[w] <= len(queue[w]) else None

    # a group: [list, current task, reserved one, part of a folded task that is done]
    groups = [[0, claim(0), None, 0] for _ in range(workers)] + [[1, claim(1), None, 0] for _ in range(crit_workers)]
    for g in groups:
        if g[0] == 0 and g[1]:
            g[2] = claim(0)

    def ready(g):
        ty, t, j, k = g[1]
        if ty == 0 or (ty == 2 and g[3] == 0):
            return fdone >= k + 1 and cnt[t, k] >= k
        j = k + 1 if ty == 2 else j
        return sdone[t] >= k + 1 and sdone[j] >= k + 1 and cnt[t, j] >= k

    while True:
        acts = [g for g in groups if g[1] and ready(g)]
        s = fdone
        if s < nT and (s == 0 or (cnt[s, s - 1] >= s - 1 and cnt[s, s] >= s - 1)):
            acts.append(None)
        if not acts:
            left = [g for g in groups if g[1]]
            done = fdone == nT and not left and all(x >= len(q) for x, q in zip(nxt, queue))
            return None if done else (fdone, left)
        g = pick.choice(acts)
        if g is None:
            if s:
                sdone[s] = s
            fdone += 1
            continue
        ty, t, j, k = g[1]
        if ty == 0 or (ty == 2 and g[3] == 0):
            assert sdone[t] == k  # panels in order
            sdone[t] = k + 1
        else:
            j = k + 1 if ty == 2 else j
            assert cnt[t, j] == k
            cnt[t, j] = k + 1
        if ty == 2 and g[3] == 0:
            g[3] = 1
            continue
        g[3] = 0
        if g[0] == 0:
            g[1], g[2] = g[2], None
            if g[1]:
                g[2] = claim(0)
        else:
            g[1] = claim(1)


@pytest.mark.parametrize("R,n", [(70, 21), (129, 35), (16, 40), (200, 0), (300, 20)])
@pytest.mark.parametrize("workers,crit_workers", [(1, 1), (4, 1), (3, 4), (64, 12)])
def test_no_schedule_of_the_lists_deadlocks(lists, R, n, workers, crit_workers):
    _, main, crit = lists(R, n)
    for seed in range(3):
        assert _run(R, n, main, crit, workers, crit_workers, seed) is None


def test_a_missing_task_is_noticed(lists):
    _, main, crit = lists(129, 35)
    assert _run(129, 35, main[1:], crit, 4, 1, 0) is not None
    assert _run(129, 35, main, crit[1:], 4, 1, 0) is not None
