"""Grouping, scans and summed-area tables at their edges: pose counts about a
multiple of 1024 and past 2048 blocks' single units, hypotheses of mixed meshes within a warp, images whose
width is no multiple of four or of a tile, against the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_1510_05613_gb300 import perch, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,n_yaw,width", [(1, 1, 33), (5, 4, 161), (16, 2, 160), (16, 4, 254), (23, 4, 160),
                                            (33, 5, 97), (40, 16, 160)])
def test_groups_and_tables(nx, n_yaw, width):
    base = synth.camera_c1()
    cam = synth.Camera(width, 3 * width // 4, 0.875 * width, 0.9 * width, width / 2 - 0.3, 3 * width / 8 + 0.4,
                       base.T_wc)
    meshes, grid = synth.meshes_c1(), synth.pose_grid(-0.1, 0.2 / nx, nx, n_yaw)
    gt = synth.objs([(0, nx // 4, nx // 4, 0), (1, nx - 1, nx - 1, n_yaw - 1)])
    depth = synth.observe(cam, meshes, grid, gt, 0.002, 0.05, 7)
    rng = np.random.default_rng(nx)
    hyps = synth.all_hypotheses(grid, [0, 1])
    hyps = hyps[rng.choice(len(hyps), min(len(hyps), 301), replace=False)]  # meshes mixed within a warp
    many = [gt[:0], gt[:1], gt[1:]]
    w = oracle.World(cam, meshes, grid, 0.004)
    p = perch.Perch(0)
    p.setup(synth.Workload("groups", cam, meshes, grid, 0.004, gt, depth))
    for parents in (many, many[1:2]):  # grouped by pose, by mesh
        hp = (np.arange(len(hyps)) % len(parents)).astype(np.int32)
        exp = oracle.eval_batch(w, depth, parents, hp, hyps, 3)
        for shortcut in (False, True):
            p.perch_set_shortcut(shortcut)
            got = p.perch_eval_successors(parents, hp, hyps, 3)
            assert np.array_equal(perch.records(got), exp), shortcut
    p.close()
