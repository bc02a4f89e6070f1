"""The ICP's nearest-point searches (pixel windows, their 4 x 4 blocks, the grid
for a camera whose matrix is no rotation, the two CTA widths) against the
oracle, which scans the whole cloud: image sizes that are no multiple of a
block, wide and narrow cameras, small and large radii."""
import numpy as np
import pytest

import oracle
from paper_1510_05613_gb300 import perch, synth

pytestmark = pytest.mark.gpu


def _case(width, height, f, T=None):
    T = synth.camera_c1().T_wc if T is None else T
    cam = synth.Camera(width, height, f, 0.95 * f, width / 2 - 0.3, height / 2 + 0.4, T)
    meshes, grid = synth.meshes_c1(), synth.pose_grid(-0.1, 0.05, 5, 4)
    gt = synth.objs([(0, 1, 1, 0), (1, 4, 4, 1)])
    jitter = np.array([[0.013, -0.009, 0.2], [-0.011, 0.008, 0.3]])
    depth = synth.observe(cam, meshes, grid, gt, 0.002, 0.05, 11, jitter)
    return synth.Workload("w", cam, meshes, grid, 0.01, gt, depth)


def _compare(wl, hyps, radius, iters):
    parents = [wl.gt[:0], wl.gt[:1], wl.gt[1:]]
    hp = (np.arange(len(hyps)) % 3).astype(np.int32)
    exp = oracle.icp_refine(oracle.World.of(wl), wl.depth, parents, hp, hyps, radius, iters)
    p = perch.Perch(0)
    p.setup(wl)
    got = p.perch_icp_refine(parents, hp, hyps, radius, iters)
    p.close()
    for k in exp.dtype.names:
        assert np.array_equal(got[k], exp[k].astype(got[k].dtype)), (k, np.nonzero(got[k] != exp[k])[0][:5])
    return exp


@pytest.mark.parametrize("radius", [0.0, 0.004, 0.02, 0.06, 0.5])
@pytest.mark.parametrize("width,height,f", [(41, 30, 35.0), (157, 118, 140.0), (163, 121, 400.0)])
def test_windows_of_any_size(width, height, f, radius):
    wl = _case(width, height, f)
    hyps = synth.all_hypotheses(wl.grid, [0, 1])  # 200: more than there are SMs
    exp = _compare(wl, hyps, radius, 8)
    if radius == 0.02 and width > 100:
        assert (exp["n_corr"] > 20).sum() > 20 and (exp["n_corr"] < exp["n_model"]).any()


@pytest.mark.parametrize("n", [1, 2, 3, 100])
def test_few_successors(n):
    wl = _case(157, 118, 140.0)
    _compare(wl, synth.all_hypotheses(wl.grid, [0, 1])[::200 // n][:n], 0.02, 20)


@pytest.mark.parametrize("stretch", [3e-5, 0.02])
def test_camera_matrix_off_a_rotation(stretch):
    """Within the windows' padding, and past it (the grid)."""
    T = synth.camera_c1().T_wc.copy()
    T[:, 1] *= np.float32(1.0 + stretch)
    wl = _case(157, 118, 140.0, T.astype(np.float32))
    _compare(wl, synth.all_hypotheses(wl.grid, [0, 1])[::3], 0.02, 10)


def test_new_observation_and_radius_between_calls():
    """The searched cloud follows the observation and the radius."""
    wl = _case(157, 118, 140.0)
    hyps = synth.all_hypotheses(wl.grid, [0, 1])[::5]
    hp = np.zeros(len(hyps), np.int32)
    p = perch.Perch(0)
    p.setup(wl)
    other = synth.observe(wl.cam, wl.meshes, wl.grid, synth.objs([(0, 3, 2, 1), (1, 0, 3, 2)]), 0.002, 0.05, 5)
    for depth in (wl.depth, other, wl.depth):
        p.perch_set_observation(depth, wl.cam.fxfycxcy, wl.cam.T_wc, wl.delta)
        for radius in (0.02, 0.05, 0.02):
            exp = oracle.icp_refine(oracle.World.of(wl), depth, [wl.gt[:0]], hp, hyps, radius, 4)
            got = p.perch_icp_refine([wl.gt[:0]], hp, hyps, radius, 4)
            for k in exp.dtype.names:
                assert np.array_equal(got[k], exp[k].astype(got[k].dtype)), (k, radius)
    p.close()
