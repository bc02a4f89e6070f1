"""Batches large enough for the flags of their records to be looked at on the
device: the same records as in pieces below that size, a failed wait still
reported, a bad hypothesis at either end still refused by name."""
import numpy as np
import pytest

from paper_1510_05613_gb300 import perch, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16383, 16384, 40001])
def test_large_batches(n):
    wl = synth.workload_c1()
    p = perch.Perch(0)
    p.setup(wl)
    all_h = synth.all_hypotheses(wl.grid, [0, 1])
    hyps = all_h[np.arange(n) % len(all_h)]
    parents = [wl.gt[:0], wl.gt[:1]]
    hp = (np.arange(n) // len(all_h) % 2).astype(np.int32)
    got = p.perch_eval_successors(parents, hp, hyps, 3)
    want = np.concatenate([p.perch_eval_successors(parents, hp[k:k + 5000], hyps[k:k + 5000], 3)
                           for k in range(0, n, 5000)])
    assert np.array_equal(got, want)
    p.perch_set_shortcut(False)
    p.perch_set_wait_limit(0)
    with pytest.raises(perch.PerchError) as e:
        p.perch_eval_successors(parents, hp, hyps, 3)
    assert e.value.code == perch.PERCH_E_DEVICE
    p.perch_set_wait_limit(-1)
    assert np.array_equal(p.perch_eval_successors(parents, hp, hyps, 3), got)
    for at in (0, n - 1):
        for field, value in (("mesh", 2), ("ix", -1), ("iy", wl.grid.ny), ("iyaw", wl.grid.n_yaw)):
            bad = hyps.copy()
            bad[field][at] = value
            with pytest.raises(perch.PerchError, match=f"hypothesis {at}: object"):
                p.perch_eval_successors(parents, hp, bad, 3)
        for value in (-1, 2):
            worse = hp.copy()
            worse[at] = value
            with pytest.raises(perch.PerchError, match=f"hypothesis {at}: parent {value} out of range"):
                p.perch_eval_successors(parents, worse, hyps, 3)
    p.close()
