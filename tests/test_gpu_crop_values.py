"""Crop values at the edges of bfloat16: depths whose value lies on, just
below and just above a midpoint between two bfloat16 numbers, about zero and the
clamp, and depths that are tiny, far or no depth, bit for bit against the
oracle."""
import numpy as np
import pytest

from oracle import cnn
from paper_1510_05613_gb300 import perch, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0, 1, 2])
def test_crop_values_round_as_in_double(seed):
    wl = synth.workload_c1()
    rng = np.random.default_rng(seed)
    hyp = synth.all_hypotheses(wl.grid, [0, 1])
    hyp = hyp[rng.choice(len(hyp), 5, replace=False)]
    H, W = wl.depth.shape
    depth = np.empty(H * W, np.float32)
    for k, o in enumerate(hyp):  # a fifth of the image for each hypothesis' z_ref
        zr = cnn.crop_centre(wl.cam, wl.meshes[int(o["mesh"])], wl.grid, o)[2]
        n = len(depth[k::5])
        exp = rng.integers(-20, 2, n)  # 2^-20 .. 2^1
        t = (1.0 + (rng.integers(0, 128, n) + 0.5) / 128.0) * 2.0 ** exp * rng.choice([-1.0, 1.0], n)
        t[: n // 8] = rng.choice([0.0, 3.0, -3.0], n // 8)
        d = (zr - t / 10.0).astype(np.float32)
        step = rng.integers(-1, 2, n)
        d = np.where(step < 0, np.nextafter(d, np.float32(0)), np.where(step > 0, np.nextafter(d, np.float32(9)), d))
        depth[k::5] = d
    odd = rng.choice(H * W, 60, replace=False)
    depth[odd] = np.resize(np.float32([0.0, -1.0, np.inf, np.nan, 1e-42, 1e-20, 4.0, -np.inf]), 60)
    depth = depth.reshape(H, W)
    p = perch.Perch(0)
    p.setup(synth.Workload("crops", wl.cam, wl.meshes, wl.grid, wl.delta, wl.gt, depth))
    got, _ = p.perch_cnn_crops([wl.gt[:0]], np.zeros(len(hyp), np.int32), hyp)
    exp, _ = cnn.crops(wl.cam, wl.meshes, wl.grid, depth, np.full((H, W), np.inf, np.float32), hyp)
    got = got.float().cpu().numpy().astype(np.float64)
    bad = np.argwhere(got != exp)
    assert bad.size == 0, (len(bad), bad[:5], got[tuple(bad[0])], exp[tuple(bad[0])])
    p.close()
