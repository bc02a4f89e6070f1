"""The counts over observed points (dJ_o, the residual, n_vol) from the cells
about a pose and the pixel windows of Eq. (1), against the oracle, which tests
every point against every pixel: small and large delta, wide and narrow
cameras, coarse images, dense clouds that take several rounds of the list."""
import numpy as np
import pytest

import oracle
from paper_1510_05613_gb300 import perch, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delta", [1e-4, 0.002, 0.01, 0.06, 0.5, 2.0])
@pytest.mark.parametrize("width,f", [(40, 30.0), (160, 140.0), (160, 420.0)])
def test_counts_near_the_poses(width, f, delta):
    base = synth.camera_c1()
    cam = synth.Camera(width, 3 * width // 4, f, 0.9 * f, width / 2 - 0.3, 3 * width / 8 + 0.4, base.T_wc)
    meshes, grid = synth.meshes_c1(), synth.pose_grid(-0.1, 0.05, 5, 4)
    gt = synth.objs([(0, 1, 1, 0), (1, 4, 4, 1)])
    depth = synth.observe(cam, meshes, grid, gt, 0.002, 0.05, 7)
    w = oracle.World(cam, meshes, grid, delta)
    wl = synth.Workload("near", cam, meshes, grid, delta, gt, depth)
    hyps = synth.all_hypotheses(grid, [0, 1])
    parents = [gt[:0], gt[:1], gt[1:], synth.objs([(1, 0, 0, 2)])]
    hp = (np.arange(len(hyps)) % 4).astype(np.int32)
    p = perch.Perch(0)
    p.setup(wl)
    for K in (2, 3):  # with and without the residual
        exp = oracle.eval_batch(w, depth, parents, hp, hyps, K)
        for share in (True, False):
            p.perch_set_share_renders(share)
            for shortcut in (False, True):
                p.perch_set_shortcut(shortcut)
                got = perch.records(p.perch_eval_successors(parents, hp, hyps, K))
                assert np.array_equal(got, exp), (K, share, shortcut)
    p.close()


@pytest.mark.parametrize("volumes", [False, True])
def test_dense_cloud_takes_several_rounds(volumes):
    """About 20000 observed points under the object: the list is filled and
    emptied many times, in single-scene and multi-scene batches."""
    base = synth.camera_c2()
    cam = synth.Camera(320, 240, 1600.0, 1600.0, 159.5, 119.5, base.T_wc)
    meshes, grid = synth.meshes_c1(), synth.pose_grid(-0.02, 0.02, 3, 3)
    gt = synth.objs([(0, 1, 1, 0)])
    depth = synth.observe(cam, meshes, grid, gt, 0.002, 0.05, 3)
    assert (depth > 0).sum() > 15000
    w = oracle.World(cam, meshes, grid, 0.004, exact_volumes=volumes)
    wl = synth.Workload("dense", cam, meshes, grid, 0.004, gt, depth)
    hyps = synth.all_hypotheses(grid, [0, 1])[::7]
    parents = [gt[:0], synth.objs([(1, 2, 2, 0)])]
    hp = (np.arange(len(hyps)) % 2).astype(np.int32)
    exp = oracle.eval_batch(w, depth, parents, hp, hyps, 2)
    p = perch.Perch(0)
    p.setup(wl, exact_volumes=volumes)
    assert np.array_equal(perch.records(p.perch_eval_successors(parents, hp, hyps, 2)), exp)
    p.perch_set_scene(1, depth)
    got = perch.records(p.perch_eval_successors_multi(parents, [1, 1], [2, 2], hp, hyps))
    assert np.array_equal(got, exp)
    p.close()
