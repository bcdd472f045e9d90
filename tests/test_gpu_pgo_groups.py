"""The register-resident pose-graph PCG over its range of block layouts: one
node a block, several, a last group that is short, and more blocks than one
round of the exchange's polls takes, against the oracle's iterates."""
import numpy as np
import pytest

import paper_2409_12190_gb300 as ba
import scenegen
from oracle import LMOptions
from oracle import pgo
from paper_2409_12190_gb300.pgo import PoseGraph
from paper_2409_12190_gb300.pgo import synthesize

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 151, 153, 1000, 5200])
def test_iterates_over_the_block_layouts(N):
    """A chain with closures every 7 nodes; 12 iterations.  Bound: 1e-9, the
    bound of the other iterate tests (the iterates agree to rounding)."""
    rng = np.random.default_rng(N)
    ei, ej = np.arange(N - 1), np.arange(1, N)
    far = np.arange(0, max(N - 9, 0), 7)
    ei, ej = np.concatenate([ei, far]).astype(np.int32), np.concatenate([ej, far + 9]).astype(np.int32)
    E = len(ei)
    P7 = np.concatenate([rng.normal(size=(N, 3)) * 5, rng.normal(size=(N, 4))], 1)
    Ts = pgo.poses_to_matrices(P7)
    Tms = np.stack([pgo.se3_exp(rng.normal(size=6) * 0.05) @ pgo.se3_inv(Ts[i]) @ Ts[j] for i, j in zip(ei, ej)])
    infos = np.tile(np.eye(6), (E, 1, 1))
    g = scenegen.PoseGraph(poses_gt=P7, ei=ei, ej=ej, noise=np.zeros((E, 6)),
                           info=np.tile(pgo.info_upper(np.eye(6)), (E, 1)), drift=np.zeros((N, 6)))
    blk = pgo.assemble(Ts, ei, ej, Tms, infos)
    mask = np.zeros(N, bool)
    mask[0] = True
    k = min(12, 3 * (N - 1))
    want, its, _ = pgo.solve_damped(blk, 1e-2, LMOptions(solver="pcg", pcg_tol=0.0, pcg_maxiter=k), mask)
    with PoseGraph(P7, ei, ej, pgo.matrices_to_poses(Tms), g.info, fixed=(0,), options=ba.Options()) as pg:
        dx, gits, _ = pg.damped_solve(1e-2, k, 0.0)
        again, _, _ = pg.damped_solve(1e-2, k, 0.0)
    got = dx.cpu().numpy()
    assert gits == its == k
    assert np.max(np.abs(got - want)) < 1e-9 * np.max(np.abs(want))
    assert np.array_equal(got, again.cpu().numpy())  # fixed order: the same bits


def _graph(g):
    meas, poses0 = synthesize(g.poses_gt, g.ei, g.ej, g.noise, g.drift)
    return PoseGraph(poses0, g.ei, g.ej, meas, g.info, fixed=(0,), options=ba.Options())


def test_a_smaller_graph_leaves_a_larger_one_solvable():
    """The larger graph's blocks hold more shared memory than the smaller one's:
    creating and solving the smaller one in between changes nothing for it."""
    large, small = scenegen.sphere_graph(20, 25, seed=1), scenegen.sphere_graph(2, 3, seed=2)
    with _graph(large) as a:
        want = a.damped_solve(1e-2, 12, 0.0)[0].cpu()
        with _graph(small) as b:
            b.damped_solve(1e-2, 12, 0.0)
            got = a.damped_solve(1e-2, 12, 0.0)[0].cpu()
            b.solve(2)
        a.solve(2)
        assert np.all(np.isfinite(a.poses().cpu().numpy()))
    assert np.array_equal(got.numpy(), want.numpy())
