"""The launches of a phase's meshes side by side on several streams: records
against the CPU oracle's, with fewer and more meshes than streams, meshes without
hypotheses, calls that reuse the buffers at once, and inside a captured graph."""
import numpy as np
import pytest
import torch

import oracle
from paper_1510_05613_gb300 import perch, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_mesh", [1, 2, 5, 8])
@pytest.mark.parametrize("shared", [False, True])
def test_records_with_meshes_side_by_side(n_mesh, shared):
    cam, grid = synth.camera_c1(), synth.pose_grid(-0.1, 0.05, 5, 4)
    base = synth.meshes_c1()
    meshes = [base[i % len(base)] for i in range(n_mesh)]
    gt = synth.objs([(0, 1, 1, 0), (n_mesh - 1, 4, 4, 1)])
    depth = synth.observe(cam, meshes, grid, gt, 0.002, 0.05, 7)
    rng = np.random.default_rng(n_mesh)
    hyps = synth.all_hypotheses(grid, [m for m in range(n_mesh) if m % 3 != 1 or n_mesh == 2])
    hyps = hyps[rng.choice(len(hyps), min(len(hyps), 157), replace=False)]
    parents = [gt[:0], gt[:1]] if shared else [gt[:1]]  # poses shared by parents: k_render and k_cost, else k_eval
    hp = (np.arange(len(hyps)) % len(parents)).astype(np.int32)
    exp = oracle.eval_batch(oracle.World(cam, meshes, grid, 0.004), depth, parents, hp, hyps, 3)
    p = perch.Perch(0)
    p.setup(synth.Workload("streams", cam, meshes, grid, 0.004, gt, depth))
    for _ in range(3):
        got = p.perch_eval_successors(parents, hp, hyps, 3)
        p.perch_eval_successors(parents, hp, hyps[::-1].copy(), 3)  # other records in the same buffers
        assert np.array_equal(perch.records(got), exp)
    P, plen, stride = p.pack_parents(parents)
    t = [torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1)).cuda() for a in (P, plen, hp, hyps)]
    out = torch.zeros((len(hyps), 7), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for _ in range(3):
        out.zero_()
        torch.cuda.synchronize()
        p.perch_eval_graph(t[0], stride, t[1].view(torch.int32), t[2].view(torch.int32), t[3], 3, out)
        torch.cuda.synchronize()
        rec = out.cpu().numpy().view(got.dtype).reshape(-1)
        assert np.array_equal(perch.records(rec), exp)
    p.close()
