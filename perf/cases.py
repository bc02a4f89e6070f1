"""What this framework is timed on: calls that its users make, over the range
of sizes that they make them at.

A case is a dict of plain values; `kind` says which call it is:
  eval    perch_eval_successors (host arrays) or perch_eval_successors_dev
          (device arrays): one batch of successors of some parents
  frame   a new depth image (perch_set_observation) and the successors near
          the objects' last poses
  label   training pairs of the learned heuristic: successors of many scenes
          (perch_eval_successors_multi) and their crops
  icp     perch_icp_refine of root successors, or perch_refine_scene
  forward predictions of the learned heuristic's network
  train   one epoch of its training and the weights that come out
  search  a new depth image and the search for its scene
Scenes are the seeded synthetic ones of the package: procedural meshes, a
simulated depth sensor with noise and dropout.
"""
import functools
import math

import numpy as np
import torch

from paper_1510_05613_gb300 import heuristic, perch, synth

SIGMA, DROPOUT, DELTA = 0.003, 0.05, 0.01


def listed():
    return [
        # one state expanded on a small camera: the smallest batch that a search issues, where latency counts
        {"name": "eval_small", "kind": "eval", "width": 160, "meshes": "small", "K": 2, "nx": 10, "ny": 10, "yaws": 8,
         "parents": "one", "n": 0, "api": "host", "shortcut": True, "volumes": False},
        # the root expansion of a three-object scene, closed-form volumes
        {"name": "eval_root", "kind": "eval", "width": 640, "meshes": "even", "K": 3, "nx": 50, "ny": 50, "yaws": 16,
         "parents": "root", "n": 0, "api": "host", "shortcut": True, "volumes": True},
        # eight states of a search expanded at once: two levels, poses shared by the parents
        {"name": "eval_states", "kind": "eval", "width": 640, "meshes": "even", "K": 3, "nx": 50, "ny": 50, "yaws": 16,
         "parents": "states", "n": 0, "api": "host", "shortcut": True, "volumes": False},
        # the benchmark's batch: every hypothesis rendered, arrays on the device
        {"name": "eval_full", "kind": "eval", "width": 640, "meshes": "even", "K": 3, "nx": 50, "ny": 50, "yaws": 16,
         "parents": "path", "n": 0, "api": "dev", "shortcut": False, "volumes": False},
        # heavy occlusion: meshes of 2k to 50k triangles added to two others; an odd number of hypotheses
        {"name": "eval_uneven", "kind": "eval", "width": 640, "meshes": "uneven", "K": 5, "nx": 50, "ny": 50,
         "yaws": 16, "parents": "one", "n": 29989, "api": "dev", "shortcut": False, "volumes": False},
        # tracking: a new depth image and the neighbourhood of each object's last pose
        {"name": "frame", "kind": "frame", "width": 640, "meshes": "even", "K": 3, "nx": 50, "ny": 50, "yaws": 16,
         "reach": 3, "volumes": False},
        # labels and inputs of the learned heuristic from eight scenes of two to five objects
        {"name": "label", "kind": "label", "width": 640, "meshes": "uneven", "nx": 25, "ny": 25, "yaws": 8,
         "scenes": 8, "per_parent": 512},
        # the objects of a found scene refined against each other: the smallest refinement
        {"name": "icp_scene", "kind": "icp", "width": 640, "meshes": "uneven", "K": 5, "nx": 50, "ny": 50, "yaws": 16,
         "n": 0, "radius": 0.02, "iters": 20},
        # every successor of the root refined, as the benchmark does
        {"name": "icp_root", "kind": "icp", "width": 640, "meshes": "even", "K": 3, "nx": 50, "ny": 50, "yaws": 16,
         "n": 120000, "radius": 0.02, "iters": 20},
        # predictions for the candidates of a pool of states
        {"name": "forward", "kind": "forward", "n": 2048, "batch": 256, "onehot": 128},
        # an epoch of training on 2048 pairs
        {"name": "train", "kind": "train", "n": 2048, "batch": 256, "onehot": 128},
        # a new depth image searched for its best scene
        {"name": "search", "kind": "search", "width": 640, "meshes": "even", "K": 3, "nx": 50, "ny": 50, "yaws": 16,
         "states": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "frame", "label", "icp", "forward", "train", "search"])
    c = {"kind": kind}
    if kind == "forward":
        return {**c, "n": _log(rng, 1, 2048), "batch": 32 * rng.randint(1, 32), "onehot": rng.randint(1, 200)}
    if kind == "train":
        b = 32 * rng.randint(1, 16)
        return {**c, "n": min(2048, b * rng.randint(1, 8) + rng.randint(0, 31)), "batch": b,
                "onehot": rng.randint(1, 200)}
    width = rng.choice([160, 320, 640]) if kind != "search" else rng.choice([320, 640])
    meshes = rng.choice(["small", "even", "uneven"]) if kind != "search" else "even"
    top = {"small": 2, "even": 3, "uneven": 5}[meshes]
    c.update(width=width, meshes=meshes, nx=rng.randint(20, 50), ny=rng.randint(20, 50), yaws=rng.randint(4, 16))
    if kind == "label":
        return {**c, "scenes": rng.randint(2, 8), "per_parent": _log(rng, 32, 512)}
    if kind == "search":
        return {**c, "K": 3, "nx": rng.randint(25, 50), "ny": rng.randint(25, 50), "states": rng.choice([1, 2, 4, 8])}
    c["K"] = rng.randint(2, top)
    if kind == "frame":
        return {**c, "reach": rng.randint(1, 4), "volumes": rng.random() < 0.5}
    if kind == "icp":
        c["yaws"] = 16
        return {**c, "n": _log(rng, 100, 60000), "radius": round(rng.uniform(0.01, 0.025), 4),
                "iters": rng.randint(4, 20)}
    shortcut = rng.random() < 0.7
    most = 20000 if meshes == "uneven" and not shortcut else 100000
    return {**c, "parents": rng.choice(["one", "root", "states", "path"]), "n": _log(rng, 50, most),
            "api": rng.choice(["host", "dev"]), "shortcut": shortcut, "volumes": rng.random() < 0.5}


# ---------------------------------------------------------------- inputs
@functools.lru_cache(None)
def _meshes(family):
    return {"small": synth.meshes_c1, "even": synth.meshes_c2, "uneven": synth.meshes_c3}[family]()


def _camera(width):
    s = width / 640.0
    c = synth.camera_c2()
    return synth.Camera(width, 3 * width // 4, 525.0 * s, 525.0 * s, width / 2 - 0.5, 3 * width / 8 - 0.5, c.T_wc)


def _grid(case):
    """Poses over a metre of table."""
    xs = np.linspace(-0.49, 0.49, case["nx"]).astype(np.float32)
    ys = np.linspace(-0.49, 0.49, case["ny"]).astype(np.float32)
    return synth.PoseGrid(xs, ys, synth.pose_grid(0.0, 0.1, 2, case["yaws"]).cos_sin)


def _scene(case, seed, k, off_grid=False):
    """A scene of k distinct objects and its depth image."""
    rng = np.random.default_rng(seed)
    meshes, grid, cam = _meshes(case["meshes"]), _grid(case), _camera(case["width"])
    ids = sorted(rng.permutation(len(meshes))[:k].tolist())
    jitter = None
    if off_grid:
        step = [0.98 / (case["nx"] - 1), 0.98 / (case["ny"] - 1), 2.0 * math.pi / case["yaws"]]
        jitter = (rng.random((k, 3)) - 0.5) * np.array(step)
    gt = synth.sample_scene(meshes, grid, ids, seed, margin=0.03 if off_grid else 0.005, max_tries=2000)
    depth = synth.observe(cam, meshes, grid, gt, SIGMA, DROPOUT, seed, jitter)
    return synth.Workload("case", cam, meshes, grid, DELTA, gt, depth, SIGMA, DROPOUT, seed)


def _near(rng, grid, objs, cells, turns):
    """The objects moved by up to `cells` grid cells and `turns` yaw steps."""
    o = objs.copy()
    n = len(o)
    o["ix"] = np.clip(o["ix"] + rng.integers(-cells, cells + 1, n), 0, grid.nx - 1)
    o["iy"] = np.clip(o["iy"] + rng.integers(-cells, cells + 1, n), 0, grid.ny - 1)
    o["iyaw"] = (o["iyaw"].astype(np.int64) + rng.integers(-turns, turns + 1, n)) % grid.n_yaw
    return o


def _batch(case, wl, rng):
    """Parents and successors of one evaluation call."""
    K, order = wl.K, wl.gt[rng.permutation(wl.K)]
    if case["parents"] == "root":
        parents = [order[:0]]
    elif case["parents"] == "one":
        parents = [order[:K // 2]]
    elif case["parents"] == "path":  # the root, a state of every level below it
        parents = [order[:j] for j in range(K)]
    else:  # the states that a search has open at one time: true poses and near misses
        parents = []
        for i in range(8):
            order = wl.gt[rng.permutation(K)]
            parents.append(_near(rng, wl.grid, order[:1 + i % (K - 1)], 1 if i >= 2 else 0, 0))
    hyps, hp = [], []
    for i, par in enumerate(parents):
        left = [m for m in wl.mesh_multiset if m not in set(int(v) for v in par["mesh"])]
        h = synth.all_hypotheses(wl.grid, left)
        hyps.append(h)
        hp.append(np.full(len(h), i, np.int32))
    hyps, hp = np.concatenate(hyps), np.concatenate(hp)
    if 0 < case["n"] < len(hyps):
        keep = np.sort(rng.choice(len(hyps), case["n"], replace=False))
        hyps, hp = hyps[keep], hp[keep]
    return parents, hp, hyps


def _words(records):
    """Records as rows of 32-bit words."""
    return records.view(np.int32).reshape(len(records), -1)


def _pairs(case, seed):
    """Crops, one-hot indices and costs as the learned heuristic meets them:
    near and far successors of the states of one scene."""
    rng = np.random.default_rng(seed)
    c = {"meshes": "even", "nx": 50, "ny": 50, "yaws": 16, "width": 640}
    wl = _scene(c, seed, 3)
    p = perch.Perch(0)
    p.setup(wl)
    p.perch_set_shortcut(False)
    parents = [wl.gt[:j] for j in range(3)]
    n, hp = case["n"], rng.integers(0, 3, case["n"]).astype(np.int32)
    hyps = _near(rng, wl.grid, wl.gt[np.maximum(hp, rng.integers(0, 3, n))], 4, 2)
    far = rng.random(n) < 0.5
    hyps["ix"][far] = rng.integers(0, 50, far.sum())
    hyps["iy"][far] = rng.integers(0, 50, far.sum())
    rec = p.perch_eval_successors(parents, hp, hyps, 3)
    crops, _ = p.perch_cnn_crops(parents, hp, hyps)
    p.close()
    cost = rec["djr"].astype(np.float64) + rec["djo"] + rec["resid"]
    target = torch.tensor(np.log1p(cost), dtype=torch.float32, device="cuda")
    onehot = torch.tensor(rng.integers(0, case["onehot"], n), dtype=torch.int32, device="cuda")
    return crops, onehot, target


def prepare(case, seed):
    kind, rng = case["kind"], np.random.default_rng(seed + 77)
    s = {"case": case}
    if kind in ("forward", "train"):
        s["data"] = _pairs(case, seed)
        s["stream"] = torch.cuda.Stream()
        s["net"] = heuristic.new_network(case["onehot"], case["batch"], seed=seed % 1000, stream=s["stream"])
        torch.cuda.synchronize()
        return s
    p = s["p"] = perch.Perch(0)
    if kind == "label":
        scenes = [_scene(case, seed * 100 + i, 2 + i % (min(5, len(_meshes(case["meshes"]))) - 1))
                  for i in range(case["scenes"])]
        heuristic.setup_scenes(p, scenes)
        parents, pscene, pK, hp, hyps = [], [], [], [], []
        for i, wl in enumerate(scenes):
            order = wl.gt[rng.permutation(wl.K)]
            for j in range(wl.K):
                n = case["per_parent"]
                h = _near(rng, wl.grid, order[rng.integers(j, wl.K, n)], 3, 2)
                far = rng.random(n) < 0.5
                h["ix"][far] = rng.integers(0, wl.grid.nx, far.sum())
                h["iy"][far] = rng.integers(0, wl.grid.ny, far.sum())
                hp.append(np.full(n, len(parents), np.int32))
                hyps.append(h)
                parents.append(order[:j])
                pscene.append(i)
                pK.append(wl.K)
        s.update(parents=parents, pscene=pscene, pK=pK, hp=np.concatenate(hp), hyps=np.concatenate(hyps))
        return s
    wl = s["wl"] = _scene(case, seed, case["K"], off_grid=kind == "icp")
    p.setup(wl, exact_volumes=case.get("volumes", False))
    if kind == "eval":
        p.perch_set_shortcut(case["shortcut"])
        parents, hp, hyps = _batch(case, wl, rng)
        s.update(parents=parents, hp=hp, hyps=hyps)
        if case["api"] == "dev":
            P, plen, s["stride"] = p.pack_parents(parents)
            for name, a in (("parents_t", P), ("plen_t", plen), ("hp_t", hp), ("hyps_t", hyps)):
                s[name] = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1)).cuda()
            s["plen_t"], s["hp_t"] = s["plen_t"].view(torch.int32), s["hp_t"].view(torch.int32)
            s["out_t"] = torch.zeros((len(hyps), 7), dtype=torch.int32, device="cuda")
    elif kind == "frame":
        r = case["reach"]
        dx, dy, yaw = (a.reshape(-1) for a in np.meshgrid(np.arange(-r, r + 1), np.arange(-r, r + 1),
                                                          np.arange(wl.grid.n_yaw), indexing="ij"))
        hyps = np.repeat(wl.gt, len(dx))
        hyps["ix"] = np.clip(hyps["ix"] + np.tile(dx, wl.K), 0, wl.grid.nx - 1)  # a cell again at the table's edge
        hyps["iy"] = np.clip(hyps["iy"] + np.tile(dy, wl.K), 0, wl.grid.ny - 1)
        hyps["iyaw"] = np.tile(yaw, wl.K)
        others = [wl.gt[:0]] + [np.delete(wl.gt, k) for k in range(wl.K)]  # alone, and with the others in place
        which = {int(m): k + 1 for k, m in enumerate(wl.gt["mesh"])}
        hp = np.concatenate([np.zeros(len(hyps), np.int32), np.array([which[int(m)] for m in hyps["mesh"]], np.int32)])
        s.update(parents=others, hp=hp, hyps=np.concatenate([hyps, hyps]))
    elif kind == "icp":
        if case["n"]:
            hyps = synth.all_hypotheses(wl.grid, wl.mesh_multiset)
            hyps = hyps[np.sort(rng.choice(len(hyps), min(case["n"], len(hyps)), replace=False))]
            s.update(parents=[wl.gt[:0]], hp=np.zeros(len(hyps), np.int32), hyps=hyps)
    else:  # search
        p.perch_set_symmetry(wl.meshes)
        p.perch_set_render_cache(True)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- the calls
def _new_image(s):
    wl = s["wl"]
    s["p"].perch_set_observation(wl.depth, wl.cam.fxfycxcy, wl.cam.T_wc, wl.delta)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "forward":
        return s["net"].perch_cnn_forward(s["data"][0], s["data"][1])
    if kind == "train":
        losses, _ = heuristic.train(s["net"], s["data"], epochs=1, batch=case["batch"], stream=s["stream"])
        return {"losses": losses, "params": s["net"].perch_cnn_get_params()}
    p = s["p"]
    if kind == "label":
        rec = p.perch_eval_successors_multi(s["parents"], s["pscene"], s["pK"], s["hp"], s["hyps"])
        crops, onehot = p.perch_cnn_crops(s["parents"], s["hp"], s["hyps"], parent_scene=s["pscene"])
        return {"records": _words(rec), "crops": crops, "onehot": onehot}
    if kind == "icp":
        if case["n"]:
            rec = p.perch_icp_refine(s["parents"], s["hp"], s["hyps"], case["radius"], case["iters"])
        else:
            rec, _ = p.perch_refine_scene(s["wl"].gt, case["radius"], case["iters"])
        return {"motion": rec.view(np.float64).reshape(len(rec), 6)[:, :4], "counts": _words(rec)[:, 8:]}
    if kind == "search":
        _new_image(s)
        r = p.perch_search(s["wl"].mesh_multiset, w=1.0, batch_states=case["states"], max_expansions=400,
                           heuristics=16)
        return {"cost": r["cost"], "proven": r["proven_optimal"], "scene": np.array(r["key"], np.int64)}
    if kind == "frame":
        _new_image(s)
    if case.get("api") == "dev":
        p.perch_eval_successors_dev(s["parents_t"], s["stride"], s["plen_t"], s["hp_t"], s["hyps_t"], case["K"],
                                    s["out_t"])
        return s["out_t"]
    return _words(p.perch_eval_successors(s["parents"], s["hp"], s["hyps"], case["K"]))


# ---------------------------------------------------------------- the least work
PARAMS = sum(int(np.prod(x)) for x in heuristic.param_shapes(0))
FORWARD_FLOPS, TRAIN_FLOPS = 100.7e6, 297.1e6  # per crop: convolutions without padding, FC layers


def _pose_ops(case):
    """Operations of one pose's render (vertices, triangles, covered pixels)
    and the pixels it covers, both as means over the family's meshes."""
    f2 = (525.0 * case["width"] / 640.0) ** 2 / 2.0  # (pixels per metre)^2 at the table's distance
    ops, px = [], []
    for m in _meshes(case["meshes"]):
        d = m.verts.max(0) - m.verts.min(0)
        w = 0.5 * float(d[0] + d[1])
        px.append(f2 * w * 0.7 * (float(d[2]) + 0.79 * w))
        ops.append(40.0 * m.n_verts + 20.0 * m.n_tris + 50.0 * px[-1])
    return float(np.mean(ops)), float(np.mean(px))


def work(case):
    kind = case["kind"]
    if kind == "forward":
        return {"bytes": case["n"] * (16384 + 8) + 2.0 * PARAMS, "flops": case["n"] * FORWARD_FLOPS}
    if kind == "train":
        steps = case["n"] // case["batch"]  # weights, two moments: read and written each step
        n = steps * case["batch"]
        return {"bytes": n * 16392.0 + steps * 24.0 * PARAMS, "flops": n * TRAIN_FLOPS}
    image, poses = 3.0 * case["width"] ** 2, case["nx"] * case["ny"] * case["yaws"]
    ops, px = _pose_ops(case)
    if kind == "label":
        n = case["scenes"] * 3.0 * case["per_parent"]
        return {"bytes": case["scenes"] * image + n * (40 + 16388), "flops": n * ops}
    K = case["K"]
    if kind == "icp":
        n = case["n"] or K
        met = n if not case["n"] else 0.1 * n  # the successors that meet the cloud
        return {"bytes": image + 60.0 * n, "flops": n * ops + met * px * 30.0 * case["iters"]}
    if kind == "frame":
        n = K * (2 * case["reach"] + 1) ** 2 * case["yaws"]
        return {"bytes": image + 80.0 * n, "flops": n * ops + 20.0 * n * px}
    if kind == "search":  # one expansion of each level; a quarter of the poses near what is seen
        n = poses * K * (K + 1) / 2
        return {"bytes": image + 40.0 * n, "flops": 0.25 * poses * K * ops}
    n = {"one": 1, "root": K, "path": K * (K + 1) / 2, "states": 8 * K / 2.0}[case["parents"]] * poses
    n = min(n, case["n"]) if case["n"] else n
    near = 0.25 if case["shortcut"] else 1.0
    return {"bytes": image + 40.0 * n, "flops": near * (min(n, K * poses) * ops + 10.0 * n * px)}


# ---------------------------------------------------------------- in 64 bits
def _shapes(onehot):
    out = []
    for cin, cout in ((2, 32), (32, 64), (64, 128), (128, 128)):
        out += [(cout, 3, 3, cin), (cout,)]
    return out + [(96, 8192 + onehot), (96,), (1, 96), (1,)]


def _predict(params, crops, onehot, width):
    x = crops.double().permute(0, 3, 1, 2)
    for l in range(4):
        w = params[2 * l].permute(0, 3, 1, 2)
        x = torch.relu(torch.nn.functional.conv2d(x, w, params[2 * l + 1], stride=1 if l == 0 else 2, padding=1))
    x = x.permute(0, 2, 3, 1).reshape(x.shape[0], -1)
    x = torch.cat([x, torch.nn.functional.one_hot(onehot.long(), width).double()], 1)
    x = torch.relu(x @ params[8].T + params[9])
    return (x @ params[10].T)[:, 0] + params[11]


def exact(case, seed):
    """The network's outputs from its float32 weights in 64 bits. The other
    kinds return counts, whole numbers that are compared as they are, and
    motions that follow from counts."""
    if case["kind"] not in ("forward", "train"):
        return None
    crops, onehot, target = _pairs(case, seed)
    init = synth.he_normal(_shapes(case["onehot"]), seed % 1000)
    params = [torch.tensor(a, device="cuda").double() for a in init]
    if case["kind"] == "forward":
        with torch.no_grad():
            return torch.cat([_predict(params, crops[i:i + 256], onehot[i:i + 256], case["onehot"])
                              for i in range(0, case["n"], 256)])
    for a in params:
        a.requires_grad_(True)
    b, n = case["batch"], case["n"]
    steps = n // b
    perm = torch.randperm(n, generator=torch.Generator().manual_seed(0)).cuda()
    m, v = [torch.zeros_like(a) for a in params], [torch.zeros_like(a) for a in params]
    losses = []
    for k in range(steps):
        idx = perm[k * b:(k + 1) * b]
        loss = 0.5 * ((_predict(params, crops[idx], onehot[idx], case["onehot"]) - target[idx].double()) ** 2).mean()
        losses.append(loss.item())
        grads = torch.autograd.grad(loss, params)
        lr = 1e-3 * 0.1 ** (k / max(1, steps - 1))
        with torch.no_grad():
            for a, g, mi, vi in zip(params, grads, m, v):
                mi.mul_(0.9).add_(g, alpha=0.1)
                vi.mul_(0.999).addcmul_(g, g, value=0.001)
                a -= lr * (mi / (1 - 0.9 ** (k + 1))) / ((vi / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return {"losses": np.array(losses), "params": torch.cat([a.detach().reshape(-1) for a in params])}
