"""The tile renders' quick path (binary32 edge functions, centres tested two by
two, larger triangles shared by eight lanes) and its general path (integers)
against the oracle, where one could go wrong: edges through pixel centres,
triangle extents about the line between the two paths, boxes cut at every
image border, full queues, meshes whose chunks end anywhere."""
import numpy as np
import pytest

import oracle
from helpers import top_down_camera
from paper_1510_05613_gb300 import perch, synth

pytestmark = pytest.mark.gpu


def _check(cam, meshes, grid, hyps, setup=lambda p: None):
    """Records of the hypotheses over an empty and a one-object parent, by one
    render per hypothesis and by shared renders, against the oracle."""
    w = oracle.World(cam, meshes, grid, 0.01)
    scene = hyps[len(hyps) // 2:len(hyps) // 2 + 1]
    z, _ = oracle.render(w, scene)
    depth = np.where(np.isfinite(z), z, 0.0).astype(np.float32)
    parents = [hyps[:0], hyps[:1]]
    hp = (np.arange(len(hyps)) % 2).astype(np.int32)
    exp = oracle.eval_batch(w, depth, parents, hp, hyps, 2)
    p = perch.Perch(0)
    wl = synth.Workload("t", cam, meshes, grid, 0.01, scene, depth)
    p.setup(wl)
    p.perch_set_shortcut(False)
    setup(p)
    for share in (True, False):
        p.perch_set_share_renders(share)
        got = perch.records(p.perch_eval_successors(parents, hp, hyps, 2))
        bad = np.nonzero((got != exp).any(1))[0]
        assert bad.size == 0, (share, bad.size, hyps[bad[:3]], got[bad[:3]], exp[bad[:3]])
    one = perch.records(p.perch_eval_successors([hyps[:0]], np.zeros(len(hyps), np.int32), hyps, 2))
    assert np.array_equal(one, oracle.eval_batch(w, depth, [hyps[:0]], np.zeros(len(hyps), np.int32), hyps, 2))
    p.close()
    assert (exp[:, 4] > 0).any()


def _sheet(n, step, name="sheet"):
    """n x n quads of side `step` facing up at height 1 (and their underside)."""
    k = np.arange(n + 1)
    v = np.array([((i - n / 2) * step, (j - n / 2) * step, 1.0) for i in k for j in k], np.float32)
    t = []
    for i in range(n):
        for j in range(n):
            a, b, c, d = i * (n + 1) + j, (i + 1) * (n + 1) + j, (i + 1) * (n + 1) + j + 1, i * (n + 1) + j + 1
            t += [(a, b, c), (a, c, d), (c, b, a), (d, c, a)]
    return synth.Mesh(name, v, np.array(t, np.int32), 0.0, 1.0, -1.0)


@pytest.mark.parametrize("step", [1 / 256, 1 / 128, 3 / 256, 1 / 64, 1 / 16, 1 / 4])
def test_edges_through_pixel_centres(step):
    """Vertices on pixel centres and quarter pixels: every edge of the sheet
    passes through centres, and the top-left rule decides each of them."""
    cam = top_down_camera(64, 48, 64.0, 32.0, 24.0)
    grid = synth.PoseGrid(np.array([-0.25, -1 / 128, 0.125], np.float32), np.array([-0.125, 0.0, 1 / 256], np.float32),
                          np.array([[1.0, 0.0], [0.0, 1.0], [0.6, 0.8]], np.float32))
    n = max(1, min(24, int(0.25 / step)))
    _check(cam, [_sheet(n, step)], grid, synth.all_hypotheses(grid, [0]))


@pytest.mark.parametrize("side,n", [(0.10, 1), (0.14, 1), (0.16, 1), (0.16, 2), (0.24, 1), (0.24, 2), (0.24, 3)])
@pytest.mark.parametrize("inline,depth", [(8, 32), (32, 128)])
def test_triangle_extents_about_the_paths_line(side, n, inline, depth):
    """Boxes whose triangles span about 25 to 130 pixels at the nearest and
    farthest poses, so that the poses of one mesh take both paths."""
    cam = synth.camera_c2()
    grid = synth.pose_grid(-0.4, 0.4, 3, 3)

    def setup(p):
        p.perch_set_inline_pixels(inline)
        p.perch_set_bin_depth(depth)

    _check(cam, [synth.box_mesh(side, 0.8 * side, 0.9 * side, n)], grid, synth.all_hypotheses(grid, [0]), setup)


@pytest.mark.parametrize("family", [synth.meshes_c1, synth.meshes_c2])
def test_boxes_cut_at_every_border(family):
    """Poses inside the image, across each of its borders and corners and
    outside; coarse meshes also overflow the queue of larger triangles."""
    cam = synth.camera_c2()
    cam = synth.Camera(200, 150, 525.0, 525.0, 99.5, 74.5, cam.T_wc)
    grid = synth.pose_grid(-0.36, 0.12, 7, 2)
    meshes = family()[:2]

    def setup(p):
        p.perch_set_inline_pixels(8)
        p.perch_set_bin_depth(32)

    _check(cam, meshes, grid, synth.all_hypotheses(grid, [0, 1]), setup)


@pytest.mark.parametrize("n_tri", [1, 2, 31, 33, 255, 257, 511, 1361, 1535, 1537])
def test_meshes_of_any_length(n_tri):
    """Chunks of any number of triangles and vertices: the first n_tri
    triangles of a 10k-triangle box."""
    m = synth.meshes_c2()[0]
    used, idx = np.unique(m.tris[:n_tri], return_inverse=True)
    part = synth.Mesh("part", m.verts[used], idx.reshape(-1, 3).astype(np.int32), 0.01, 0.0, 0.1)
    grid = synth.pose_grid(-0.3, 0.3, 3, 4)
    _check(synth.camera_c2(), [part], grid, synth.all_hypotheses(grid, [0]))
