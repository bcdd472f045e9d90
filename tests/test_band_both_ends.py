"""The banded Cholesky's elimination from both ends (BandShape in
csrc/ba_band_sched.h): the task list, printed by a host build, is executed by
blocking workers in two pools with the waits of the device tasks, in random
order among those that may complete.  Every tile's update columns are derived
here from the matrix's block rows alone.  No deadlock, and the factor and the
solution are numpy's of the reordered random banded SPD system."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TB = 4  # the schedule does not depend on the tile size
D, U, T, F, B, INV = 0, 1, 2, 3, 4, 5


@pytest.fixture(scope="module")
def scheduler(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    exe = tmp_path_factory.mktemp("band") / "band_both_ends"
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Wextra", "-Werror", "-I",
                    os.path.join(ROOT, "paper_2409_12190_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "c", "band_both_ends.cpp"), "-o", str(exe)], check=True)

    def run(*argv):
        out = subprocess.run([str(exe), *map(str, argv)], capture_output=True, text=True, check=True).stdout.splitlines()
        return [[int(v) for v in line.split()] for line in out]
    return run


@pytest.mark.parametrize("nb,bwt,s_upd,workers,crit", [
    (3, 1, 1, 8, 2),      # one row at each end, one between
    (4, 1, 1, 3, 1),
    (9, 3, 1, 8, 4),      # as short as the rule takes
    (10, 3, 2, 6, 2),     # segments of two columns, runs of odd length
    (23, 5, 3, 152, 8),
    (40, 2, 1, 12, 4),
    (17, 4, 1, 1, 0),     # one block for everything
    (8, 3, 1, 8, 2),      # too wide: from the top
    (6, 0, 1, 4, 1),      # no coupling
])
def test_both_ends(scheduler, nb, bwt, s_upd, workers, crit):
    (nb, bwt, top, joint, ncrit), row, *tasks = scheduler(nb, bwt, s_upd, workers, crit)
    split = bwt >= 1 and nb >= 3 * bwt and nb >= bwt + 2
    assert split == (top < nb) and sorted(row) == list(range(nb))
    if split:  # the ends are the matrix's, and do not meet
        assert row[:top] == list(range(top)) and row[top:joint] == list(range(nb - 1, nb - 1 - (joint - top), -1))
        assert row[joint:] == list(range(top, top + nb - joint)) and nb - joint >= bwt
    has = lambda I, J: abs(row[I] - row[J]) <= bwt  # noqa: E731
    tiles = [(I, J) for J in range(nb) for I in range(J, nb) if has(I, J)]
    upd = {(I, J): [K for K in range(J) if has(I, K) and has(J, K)] for I, J in tiles}
    for (I, J), ks in upd.items():  # the tile set is closed under elimination
        if I == J and ks and ks[-1] == J - 1:
            ks.pop()                # D_J's
    assert all(has(I, J) for J in range(nb) for K in range(J) for I in range(J, nb) if has(I, K) and has(J, K))
    got = {}
    for x, I, J, Ka, before in tasks:
        if x & 7 == U:
            assert 1 <= x >> 3 <= s_upd
            got.setdefault((I, J), []).append((before, list(range(Ka, Ka + (x >> 3)))))
    for k, ks in upd.items():
        segs = sorted(got.pop(k, []))
        assert sum((c for _, c in segs), []) == ks
        assert [b for b, _ in segs] == [sum(len(c) for _, c in segs[:i]) for i in range(len(segs))]
    assert not got
    assert sorted((I, J) for x, I, J, _, _ in tasks if x & 7 == T) == sorted((I, J) for I, J in tiles if I > J + 1)
    for typ in (D, INV, F, B):
        assert sorted(t[2] for t in tasks if t[0] & 7 == typ) == list(range(nb))

    # the system, in elimination order
    rng = np.random.default_rng(100 * nb + bwt)
    n = nb * TB
    M = np.where(np.abs(np.subtract.outer(np.arange(n) // TB, np.arange(n) // TB)) <= bwt, rng.standard_normal((n, n)), 0)
    A = M + M.T
    A += np.eye(n) * (np.abs(A).sum(1).max() + 1.0)
    perm = np.concatenate([np.arange(TB) + TB * r for r in row])
    A = A[np.ix_(perm, perm)]
    b = rng.standard_normal(n)
    L_ref, x_ref = np.linalg.cholesky(A), np.linalg.solve(A, b)
    blk = lambda I, J: (slice(I * TB, I * TB + TB), slice(J * TB, J * TB + TB))  # noqa: E731
    chain = [0 if J < top else 1 if J < joint else 2 for J in range(nb)]
    begin, end = (0, top, joint), (top, joint, nb)
    for seed in range(3):
        L, y = np.tril(A).copy(), b.copy()
        flag, prog, inv, fwd, bwd = set(), {t: 0 for t in tiles}, set(), [0, 0, 0], [0, 0, 0]

        def ready(t):
            x, I, J, Ka, before = t
            typ = x & 7
            if typ == D:
                chained = J >= 1 and (J, J - 1) in prog
                return not chained or ((J - 1, J - 1) in flag and prog[J, J - 1] >= len(upd[J, J - 1])
                                       and prog[J, J] >= len(upd[J, J]))
            if typ == U:
                return prog[I, J] >= before and all((I, K) in flag and (J, K) in flag for K in range(Ka, Ka + (x >> 3)))
            if typ == T:
                return (J, J) in flag and prog[I, J] >= len(upd[I, J])
            if typ == INV:
                return (J, J) in flag
            if typ == F:
                return J in inv and fwd[chain[J]] >= J - begin[chain[J]] and all(
                    (J, K) in flag and fwd[chain[K]] > K - begin[chain[K]] for K in range(J) if has(J, K))
            c = chain[I]
            return fwd[chain[-1]] >= nb - begin[chain[-1]] and bwd[c] >= end[c] - 1 - I and all(
                bwd[chain[K]] >= end[chain[K]] - K for K in range(I + 1, nb) if has(K, I))

        def run(t):
            x, I, J, Ka, _ = t
            typ = x & 7
            if typ == D:
                if J >= 1 and (J, J - 1) in prog:
                    L[blk(J, J - 1)] = np.linalg.solve(L[blk(J - 1, J - 1)], L[blk(J, J - 1)].T).T
                    flag.add((J, J - 1))
                    L[blk(J, J)] -= np.tril(L[blk(J, J - 1)] @ L[blk(J, J - 1)].T)
                S = L[blk(J, J)]
                L[blk(J, J)] = np.linalg.cholesky(S + np.tril(S, -1).T)
                flag.add((J, J))
            elif typ == U:
                for K in range(Ka, Ka + (x >> 3)):
                    L[blk(I, J)] -= L[blk(I, K)] @ L[blk(J, K)].T
                if I == J:
                    L[blk(I, J)] = np.tril(L[blk(I, J)])
                prog[I, J] += x >> 3
            elif typ == T:
                L[blk(I, J)] = np.linalg.solve(L[blk(J, J)], L[blk(I, J)].T).T
                flag.add((I, J))
            elif typ == INV:
                inv.add(J)
            elif typ == F:
                v = y[J * TB:J * TB + TB] - sum(L[blk(J, K)] @ y[K * TB:K * TB + TB] for K in range(J) if has(J, K))
                y[J * TB:J * TB + TB] = np.linalg.solve(L[blk(J, J)], v)
                fwd[chain[J]] = J - begin[chain[J]] + 1
            else:
                v = y[I * TB:I * TB + TB] - sum(L[blk(K, I)].T @ y[K * TB:K * TB + TB] for K in range(I + 1, nb) if has(K, I))
                y[I * TB:I * TB + TB] = np.linalg.solve(L[blk(I, I)].T, v)
                bwd[chain[I]] = end[chain[I]] - I

        order = np.random.default_rng(seed)
        pools, size = [tasks[ncrit:], tasks[:ncrit]], [workers - crit, crit] if ncrit else [workers, 0]
        held, nxt, done = [[], []], [0, 0], 0
        while done < len(tasks):
            for p in (0, 1):
                while len(held[p]) < size[p] and nxt[p] < len(pools[p]):
                    held[p].append(pools[p][nxt[p]])
                    nxt[p] += 1
            can = [(p, k) for p in (0, 1) for k, t in enumerate(held[p]) if ready(t)]
            assert can, f"deadlock with {done} of {len(tasks)} tasks done"
            p, k = can[order.integers(len(can))]
            run(held[p].pop(k))
            done += 1
        assert np.max(np.abs(L - L_ref)) <= 1e-13 * np.max(np.abs(L_ref))
        assert np.max(np.abs(y - x_ref)) <= 1e-12 * np.max(np.abs(x_ref))
