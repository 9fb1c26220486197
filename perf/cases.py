"""Performance cases: what a user of this library has it do, through its public
entry points, at the sizes of the seeded benchmark configurations
(paper_2304_09953_gb300.workload.CONFIGS) and of their slices.

A case names a `kind` (the stage of the screening workflow), the
configuration its ligands and pocket come from, how many ligands, and the
search parameters.  The kinds:

  dock     a docking run of a prepared plan, poses left on the device
  host     the one-call docking from host arrays to host results
  screen   coarse pass, its best-score quantile as cutoff, full run with it
  triage   descriptors, coarse pass, ensemble ranking, docking of the kept part
  refine   gradient-descent refinement of a run's poses
  rescore  exact rescoring of a run's poses and the best passing pose per ligand
  select   pose features, network prediction, the selector's choice
  train    one epoch of the surrogate network
  rank     descriptors of a library and its ranking by a trained network
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2304_09953_gb300 import docking as D
from paper_2304_09953_gb300 import native as N
from paper_2304_09953_gb300 import selector as SEL
from paper_2304_09953_gb300 import workload as W

ETA0 = 0.1           # initial step of the refinement (A^2 per score unit)
LR = 1e-3            # learning rate of the surrogate
TRIAGE_NETS = 5      # networks of the cross-fitted ensemble


def listed():
    full = dict(orient=256, anchor=32, steps=16, top_k=16)  # the benchmark's search: 8,192 starts
    return [
        # an interactive call: one ligand, a small search (the "tiny" configuration)
        dict(name="dock_one_ligand", kind="dock", config="tiny", ligands=1, mode="fp32", orient=64, anchor=8, steps=8,
             top_k=4),
        # the benchmark's headline: a 10,000-ligand library, BF16 maps, FP32 rescoring of the top 16
        dict(name="dock_library_bf16", kind="dock", config="batched", ligands=10000, mode="bf16", **full),
        # the reference form of the same search: FP32 maps in the plain layout
        dict(name="dock_library_fp32", kind="dock", config="batched", ligands=1000, mode="fp32", **full),
        # a chunk of the large target's library: bigger ligands (up to 80 atoms, 15 bonds), 96^3 maps
        dict(name="dock_target_bf16", kind="dock", config="combined", ligands=1500, mode="bf16", **full),
        # a service request: a few hundred ligands from host memory, odd sampling sizes, FP16 maps
        dict(name="dock_host_arrays_fp16", kind="host", config="batched", ligands=301, mode="fp16", orient=101,
             anchor=17, steps=12, top_k=5),
        # screening for the best 1% of a library, exactly
        dict(name="screen_best_bf16", kind="screen", config="batched", ligands=2000, mode="bf16", frac=0.01, **full),
        # the calibrated triage step: a coarse pass and the ensemble choose what is docked
        dict(name="triage_step_bf16", kind="triage", config="batched", ligands=2000, mode="bf16", keep=0.418, **full),
        # post-docking stages on the top poses of a library
        dict(name="refine_top_poses", kind="refine", config="batched", ligands=1000, mode="bf16", iters=32, orient=64,
             anchor=8, steps=16, top_k=16),
        dict(name="rescore_top_poses", kind="rescore", config="batched", ligands=2000, mode="bf16", orient=64, anchor=8,
             steps=16, top_k=16),
        dict(name="select_poses", kind="select", config="batched", ligands=2000, mode="bf16", orient=64, anchor=8,
             steps=16, top_k=16),
        # the surrogate: an epoch of training, and ranking a large library
        dict(name="train_epoch", kind="train", config="learned_train", ligands=16384, batch=1024),
        dict(name="rank_library", kind="rank", config="learned_train", ligands=100000, keep=0.05),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dock", "dock", "dock", "host", "screen", "triage", "refine", "rescore", "select", "train",
                       "rank"])
    if kind == "train":
        return dict(kind=kind, config="learned_train", ligands=_log(rng, 1100, 16384),
                    batch=rng.choice([256, 512, 1000, 1024]))
    if kind == "rank":
        return dict(kind=kind, config="learned_train", ligands=_log(rng, 700, 100000),
                    keep=rng.choice([0.01, 0.05, 0.2, 0.418]))
    config = rng.choice(["batched", "batched", "combined"])
    steps = rng.choice([8, 12, 16, 16, 16, 18, 24])
    mode = rng.choice(["bf16", "bf16", "fp32", "fp32c", "fp16"])
    c = dict(kind=kind, config=config, mode=mode, steps=steps, top_k=rng.choice([1, 4, 7, 16, 16, 30]))
    # ligands x starts within the listed cases' (a single ligand to a library, 128 to 8,192 starts)
    c["orient"] = _log(rng, 16, 256)
    c["anchor"] = rng.randint(5, 32)
    starts = c["orient"] * c["anchor"]
    if kind in ("dock", "host", "screen", "triage"):
        low = 60 if kind in ("screen", "triage") else 1
        most = 900 * (8192 / starts) * (0.4 if mode == "fp32" else 1.0) * (0.5 if config == "combined" else 1.0)
        c["ligands"] = _log(rng, low, max(low, min(3000, most)))
        if kind == "screen":
            c["frac"] = rng.choice([0.01, 0.02, 0.05])
        if kind == "triage":
            c["keep"] = rng.choice([0.05, 0.1, 0.418])
            c["steps"] = 16
        return c
    c["orient"], c["anchor"] = 32, 8
    c["ligands"] = _log(rng, 20, 1000)
    if kind == "refine":
        c["iters"] = rng.choice([8, 16, 32])
    return c


# --------------------------------------------------------------------------
def _workload(case, seed):
    """Ligands, pocket and sampling of a case, drawn from the seed alone."""
    kw = {}
    if "orient" in case:
        kw = dict(n_orient=case["orient"], n_anchor=case["anchor"], steps=case["steps"], top_k=case["top_k"])
    return W.make_workload(case["config"], n_ligands=case["ligands"], seed=5000 + 2 * seed, pocket_seed=5001 + 2 * seed,
                           **kw)


def _coarse(s):
    """The coarse pass: the first orientations and anchors of the full search, best pose only."""
    return dataclasses.replace(s, quats=s.quats[:32], n_anchor=min(8, s.n_anchor), top_k=1)


def _descriptors(bh, n):
    desc = torch.empty((n, 256), dtype=torch.float32, device="cuda")
    N.ligate_descriptors(bh.h, desc)
    return desc


def _coarse_scores(ph, bh, w):
    """Best scores of a coarse docking pass (training labels), on the device."""
    pl = D.Plan(ph, bh, _coarse(w.sampling), mode="bf16", rescore=False)
    pl.run()
    best = torch.empty(bh.n, dtype=torch.float32, device="cuda")
    N.ligate_plan_best_scores(pl.h, best, 1, 0)
    torch.cuda.synchronize()
    pl.close()
    return best


class _Net:
    def __init__(self, seed):
        self.h = N.ligate_surrogate_create(None, seed)

    def __del__(self):
        if getattr(self, "h", None):
            N.ligate_surrogate_destroy(self.h)
            self.h = None


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case, kind = case, case["kind"]
    w = st.w = _workload(case, seed)
    n = st.n = w.ligands.n
    st.ph = D.PocketHandle(w.pocket)
    if kind == "host":
        prec, layout = D.MODES[case["mode"]]
        st.s = N.make_sampling(w.sampling, prec, layout, prec != N.LIGATE_FP32)
        st.out = np.zeros((n, case["top_k"]), N.POSE_DTYPE)
        return st
    st.bh = D.BatchHandle(w.ligands)
    if kind in ("train", "rank"):
        st.net = _Net(seed)
        m = n if kind == "train" else min(n, 8192)
        sub = st.bh if m == n else D.BatchHandle(w.ligands.subset(np.arange(m)))
        st.train_desc = _descriptors(sub, m)
        st.labels = _coarse_scores(st.ph, sub, w)
        st.epoch = 0
        if kind == "rank":
            N.ligate_surrogate_train(st.net.h, st.train_desc, st.labels, m, 2, min(512, m // 8 * 8), LR, seed)
            st.k = int(math.ceil(n * case["keep"] - 1e-9))
            st.desc = torch.empty((n, 256), dtype=torch.float32, device="cuda")
            st.idx = torch.empty(st.k, dtype=torch.int32, device="cuda")
            st.pred = torch.empty(n, dtype=torch.float32, device="cuda")
        return st
    K = case["top_k"]
    st.plan = D.Plan(st.ph, st.bh, w.sampling, mode=case["mode"])
    if kind in ("dock", "screen"):
        st.out = torch.empty(n * K * N.POSE_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    if kind in ("screen", "triage"):
        st.coarse = D.Plan(st.ph, st.bh, _coarse(w.sampling), mode=case["mode"], rescore=False)
    if kind == "screen":
        st.cut = torch.empty(1, dtype=torch.float32, device="cuda")
        st.plan.set_cutoff(st.cut)
    elif kind == "triage":
        st.k = int(math.ceil(n * case["keep"] - 1e-9))
        st.desc = _descriptors(st.bh, n)
        st.coarse.run()
        N.ligate_plan_best_scores(st.coarse.h, st.desc, 256, 233)
        best = st.desc[:, 233].contiguous()
        b = min(256, n // 8 * 8)
        st.nets = [_Net(seed + f) for f in range(TRIAGE_NETS)]
        for f, net in enumerate(st.nets):
            N.ligate_surrogate_train(net.h, st.desc, best, n, 2, b, LR, seed + f)
        st.idx = torch.empty(st.k, dtype=torch.int32, device="cuda")
        st.pred = torch.empty(n, dtype=torch.float32, device="cuda")
        st.out = torch.empty(st.k * K * N.POSE_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    elif kind in ("refine", "rescore", "select"):
        st.plan.run()
        if kind == "refine":
            st.refined = torch.empty(n * K * N.REFINED_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        else:
            st.rescored = torch.empty(n * K * N.RESCORED_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        if kind == "rescore":
            st.idx = torch.empty(n, dtype=torch.int32, device="cuda")
            st.energy = torch.empty(n, dtype=torch.float32, device="cuda")
        if kind == "select":
            st.feat = torch.empty((n * K, 256), dtype=torch.float32, device="cuda")
            st.pred = torch.empty(n * K, dtype=torch.float32, device="cuda")
            st.idx = torch.empty(n, dtype=torch.int32, device="cuda")
            N.ligate_plan_pose_features(st.plan.h, st.feat)
            N.ligate_plan_rescore(st.plan.h, st.rescored)
            st.train_desc, st.labels = st.feat.clone(), SEL.labels(st.rescored)
            st.net = _Net(seed)
            m = n * K
            N.ligate_surrogate_train(st.net.h, st.train_desc, st.labels, m, 1, max(8, min(1024, m // 8 * 8)), LR, seed)
    torch.cuda.synchronize()
    return st


def _poses(buf, n, K):
    """Scores, start ids and torsion steps of ligate_pose records."""
    if isinstance(buf, np.ndarray):
        return {"score": buf["score"], "start": buf["start_id"], "tors": buf["tors"]}
    r = buf.view(n, K, N.POSE_DTYPE.itemsize)
    return {"score": r[:, :, :4].view(torch.float32)[:, :, 0], "start": r[:, :, 4:8].view(torch.int32)[:, :, 0],
            "tors": r[:, :, 8:]}


def _fields(buf, dtype):
    """Columns of device records of a numpy record type."""
    r = buf.view(-1, dtype.itemsize)
    out = {}
    for name in dtype.names:
        t, off = dtype.fields[name][:2]
        if t.names:
            out.update(_fields(r[:, off:off + t.itemsize].reshape(-1), t))
            continue
        kind = torch.float32 if t.base.kind == "f" else torch.int32
        out[name] = r[:, off:off + t.itemsize].view(kind)
    return out


def run(st):
    case, n = st.case, st.n
    kind, K = case["kind"], case.get("top_k")
    if kind == "dock":
        N.ligate_plan_run(st.plan.h, st.out)
        return _poses(st.out, n, K)
    if kind == "host":
        N.ligate_dock_batch(st.ph.h, st.w.ligands, st.s, st.out)
        return _poses(st.out, n, K)
    if kind == "screen":
        st.coarse.run()
        st.coarse.best_quantile(case["frac"], st.cut)
        N.ligate_plan_run(st.plan.h, st.out)
        return dict(_poses(st.out, n, K), cutoff=st.cut)
    if kind == "triage":
        N.ligate_descriptors(st.bh.h, st.desc)
        st.coarse.run()
        N.ligate_plan_best_scores(st.coarse.h, st.desc, 256, 233)
        N.ligate_surrogate_rank_ensemble([m.h for m in st.nets], st.desc, n, case["keep"], st.idx, st.pred)
        N.ligate_plan_run_subset(st.plan.h, st.idx, st.k, st.out)
        return dict(_poses(st.out, st.k, K), kept=st.idx, pred=st.pred)
    if kind == "refine":
        N.ligate_plan_refine(st.plan.h, case["iters"], ETA0, st.refined)
        return _fields(st.refined, N.REFINED_DTYPE)
    if kind == "rescore":
        N.ligate_plan_rescore(st.plan.h, st.rescored)
        N.ligate_plan_best_passing(st.plan.h, st.rescored, st.idx, st.energy)
        return dict(_fields(st.rescored, N.RESCORED_DTYPE), best=st.idx, best_energy=st.energy)
    if kind == "select":
        N.ligate_plan_pose_features(st.plan.h, st.feat)
        N.ligate_surrogate_predict(st.net.h, st.feat, n * K, st.pred)
        N.ligate_select_poses(st.pred, st.plan.device_output(), n, K, 0.5 * SEL.FAIL_LABEL, st.idx)
        return {"feat": st.feat, "pred": st.pred, "kept": st.idx}
    if kind == "train":
        st.epoch += 1
        loss = N.ligate_surrogate_train(st.net.h, st.train_desc, st.labels, n, 1, case["batch"], LR, st.epoch)
        return {"loss": np.float32(loss), "weights": N.ligate_surrogate_get_weights(st.net.h)}
    N.ligate_descriptors(st.bh.h, st.desc)
    N.ligate_surrogate_rank(st.net.h, st.desc, n, case["keep"], st.idx, st.pred)
    return {"desc": st.desc, "pred": st.pred, "kept": st.idx}


# --------------------------------------------------------------------------
def _tree(xyz, bonds, rotatable):
    """DFS pre-order of a ligand tree from atom 0 (children ascending) and its
    rotatable bonds in sweep order as (u, v, end) in that order."""
    n = len(xyz)
    adj = [[] for _ in range(n)]
    for a, b in bonds:
        adj[a].append(int(b))
        adj[b].append(int(a))
    order, parent, stack = [], {0: -1}, [0]
    while stack:
        a = stack.pop()
        order.append(a)
        for c in sorted(adj[a], reverse=True):
            if c != parent[a]:
                parent[c] = a
                stack.append(c)
    pos = {a: p for p, a in enumerate(order)}
    size = [1] * n
    for a in reversed(order[1:]):
        size[parent[a]] += size[a]
    rot = []
    for (a, b), r in zip(bonds, rotatable):
        if r:
            v = int(b) if parent[int(b)] == int(a) else int(a)
            rot.append((pos[parent[v]], pos[v], pos[v] + size[v]))
    return np.array(order), sorted(rot, key=lambda t: t[1]), adj


def work(case):
    """Input and output bytes and the arithmetic of the stage: map
    interpolations at 50 FLOP, clash or receptor pairs at 12, 2 M N K of a
    contraction; a search counts every unique trial pose of its greedy sweep
    (the screening run: the coarse search and each start's rigid pose)."""
    kind, n = case["kind"], case["ligands"]
    if kind in ("train", "rank"):
        par = 256 * 512 + 2 * 512 * 512 + 512
        if kind == "train":
            rows = n // case["batch"] * case["batch"]
            return {"bytes": rows * 1028 + 16 * par, "flops": 6.0 * rows * par}
        return {"bytes": n * (38 * 16 + 1028) + 4 * par, "flops": 2.0 * n * par}
    cfg = W.CONFIGS[case["config"]]
    w = W.make_workload(case["config"], n_ligands=min(n, 200), pocket=W.Pocket(np.zeros((1, 2, 2, 2), np.float32), 0, 1, 0))
    atoms = moved = pairs = 0.0
    for i in range(w.ligands.n):
        x, _, b, r = w.ligands.ligand(i)
        rot = _tree(x, b, r)[1]
        atoms += len(x)
        moved += sum(e - v - 1 for _, v, e in rot)
        pairs += len(x) * (len(x) - 1) / 2
    atoms, moved, pairs = atoms / w.ligands.n, moved / w.ligands.n, pairs / w.ligands.n
    K, S, starts = case["top_k"], case["steps"], case["orient"] * case["anchor"]
    maps = cfg["n_types"] * cfg["grid"] ** 3 * (2 if case["mode"] in ("bf16", "fp16") else 4)
    base = maps + n * atoms * 24
    search = 50.0 * (atoms + moved * (S - 1)) * n
    if kind in ("dock", "host"):
        return {"bytes": base + n * K * 24, "flops": starts * search}
    coarse = min(32, case["orient"]) * min(8, case["anchor"]) * search
    if kind == "screen":
        return {"bytes": base + n * K * 24, "flops": coarse + starts * 50.0 * atoms * n}
    if kind == "triage":
        return {"bytes": base + n * 1024 + n * case["keep"] * K * 24, "flops": coarse + case["keep"] * starts * search}
    poses = n * K
    if kind == "refine":
        return {"bytes": base + poses * 152, "flops": poses * (case["iters"] + 1) * (100.0 * atoms + 12.0 * pairs)}
    if kind == "rescore":
        # receptor atoms within the 8 A cutoff of a point, uniform in the map's shell
        L = (cfg["grid"] - 1) * cfg["spacing"]
        near = cfg["n_receptor"] * 8.0 ** 3 / ((0.5 * math.sqrt(3) * L) ** 3 - (0.3 * L) ** 3)
        return {"bytes": base + poses * 48, "flops": poses * 12.0 * (atoms * near + pairs)}
    return {"bytes": base + poses * (24 + 1024 + 4) + n * 4,
            "flops": poses * (50.0 * atoms + 12.0 * pairs + 2.0 * (256 * 512 + 2 * 512 * 512 + 512))}


# --------------------------------------------------------------------------
# FP64 values of the outputs, from the same inputs.
def _f64(a):
    return torch.from_numpy(np.asarray(a, np.float64)).cuda()


class _Lig64:
    """A ligand in DFS order: coordinates about the centroid, bonds, pairs at least 4 bonds apart."""

    def __init__(self, lig):
        xyz, typ, bonds, rotatable = lig
        order, self.rot, adj = _tree(xyz, bonds, rotatable)
        x = np.asarray(xyz, np.float64)[order]
        n = len(order)
        self.x = _f64(x - x.mean(0))
        self.type = torch.from_numpy(np.asarray(typ)[order].astype(np.int64)).cuda()
        A = np.zeros((n, n))
        pos = np.argsort(order)
        for a in range(n):
            A[pos[a], pos[adj[a]]] = 1
        near = np.linalg.matrix_power(A + np.eye(n), 3) > 0
        i, j = np.nonzero(np.triu(~near, 1))
        self.i, self.j = torch.from_numpy(i).cuda(), torch.from_numpy(j).cuda()


def _frames64(w):
    q = np.asarray(w.sampling.quats, np.float64)
    q = q / np.linalg.norm(q, axis=1, keepdims=True)
    a, b, c, d = q.T
    R = np.stack([1 - 2 * (c * c + d * d), 2 * (b * c - a * d), 2 * (b * d + a * c),
                  2 * (b * c + a * d), 1 - 2 * (b * b + d * d), 2 * (c * d - a * b),
                  2 * (b * d - a * c), 2 * (c * d + a * b), 1 - 2 * (b * b + c * c)], 1).reshape(-1, 3, 3)
    return _f64(R), _f64(w.pocket.anchors)


def _turn(x, rot, ang):
    """Coordinates [..., n, 3] with the atoms (v, end) turned by ang [...] about u -> v."""
    u, v, end = rot
    p = x[..., v, :]
    k = p - x[..., u, :]
    k = (k / k.norm(dim=-1, keepdim=True)).unsqueeze(-2)
    r = x[..., v + 1:end, :] - p.unsqueeze(-2)
    c, s = torch.cos(ang)[..., None, None], torch.sin(ang)[..., None, None]
    k = k.expand_as(r)
    r = r * c + torch.cross(k, r, dim=-1) * s + k * (k * r).sum(-1, keepdim=True) * (1 - c)
    return torch.cat([x[..., :v + 1, :], r + p.unsqueeze(-2), x[..., end:, :]], -2)


def _maps64(w):
    return _f64(w.pocket.maps)


def _grid64(maps, w, x, typ):
    """Trilinear map values [..., n] at x [..., n, 3] (A), the penalty outside."""
    dims = torch.tensor(w.pocket.dims, device="cuda", dtype=torch.float64)
    u = (x - _f64(w.pocket.origin)) / w.pocket.spacing
    out = ((u < 0) | (u > dims - 1)).any(-1)
    c = torch.minimum(torch.clamp(torch.floor(u), min=0), dims - 2)
    f = torch.clamp(u - c, 0, 1)
    c = c.long()
    val = 0
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                wt = (f[..., 0] if dx else 1 - f[..., 0]) * (f[..., 1] if dy else 1 - f[..., 1]) * \
                     (f[..., 2] if dz else 1 - f[..., 2])
                val = val + wt * maps[typ, c[..., 2] + dz, c[..., 1] + dy, c[..., 0] + dx]
    return torch.where(out, torch.full_like(val, w.sampling.penalty), val)


def _clash64(w, lig, x):
    d2 = (x[..., lig.i, :] - x[..., lig.j, :]).square().sum(-1)
    return w.sampling.clash_weight * torch.clamp(1 - d2 / w.sampling.clash_cutoff ** 2, min=0).square().sum(-1)


def _dock64(w, mode):
    """Top-K scores of every ligand by the greedy search, all starts at once."""
    R, A = _frames64(w)
    maps = _maps64(w)
    S, K = w.sampling.torsion_steps, w.sampling.top_k
    R = R.repeat_interleave(w.sampling.n_anchor, 0)
    A = A[:w.sampling.n_anchor].repeat(w.sampling.n_orient, 1)
    ang = torch.arange(S, device="cuda", dtype=torch.float64) * (2 * math.pi / S)
    scores = []
    for i in range(w.ligands.n):
        lig = _Lig64(w.ligands.ligand(i))
        x = torch.einsum("sab,nb->sna", R, lig.x) + A[:, None, :]

        def energy(y):
            return _grid64(maps, w, y, lig.type).sum(-1) + _clash64(w, lig, y)

        for b in lig.rot:
            trial = _turn(x[:, None].expand(-1, S, -1, -1), b, ang.expand(len(x), S))
            x = trial[torch.arange(len(x), device="cuda"), energy(trial).argmin(1)]
        scores.append(energy(x).sort()[0][:K])
    return torch.stack(scores)


def _poses64(w, poses):
    """(ligand, coordinates [K, n, 3]) of every row of docked poses."""
    R, A = _frames64(w)
    step = 2 * math.pi / w.sampling.torsion_steps
    for i in range(w.ligands.n):
        lig = _Lig64(w.ligands.ligand(i))
        s = torch.from_numpy(poses[i]["start_id"].astype(np.int64)).cuda()
        t = _f64(poses[i]["tors"]) * step
        x = torch.einsum("sab,nb->sna", R[s // w.sampling.n_anchor], lig.x) + A[s % w.sampling.n_anchor][:, None, :]
        for b, rot in enumerate(lig.rot):
            x = _turn(x, rot, t[:, b])
        yield lig, x


def _rescore64(st):
    w, p = st.w, st.w.pocket
    poses = st.plan.output()
    if (poses["start_id"] < 0).any():
        return None
    rec, rt = _f64(np.asarray(p.receptor_xyz, np.float32)), torch.from_numpy(p.receptor_type.astype(np.int64)).cuda()
    rad, eps = _f64(np.asarray(p.type_radius, np.float32)), _f64(np.asarray(p.type_eps, np.float32))
    inter, clash = [], []
    for lig, x in _poses64(w, poses):
        d2 = (x[:, :, None, :] - rec).square().sum(-1)
        r0 = rad[lig.type][:, None] + rad[rt]
        q = (r0 * r0 / torch.clamp(d2, min=p.rmin ** 2)) ** 3
        v = torch.sqrt(eps[lig.type][:, None] * eps[rt]) * (q * q - 2 * q)
        inter.append(torch.where(d2 <= p.cutoff ** 2, v, torch.zeros_like(v)).sum(-1).clamp(max=p.cap).sum(-1))
        clash.append(_clash64(w, lig, x))
    inter, clash = torch.cat(inter)[:, None], torch.cat(clash)[:, None]
    return {"energy": inter + clash, "e_inter": inter, "e_clash": clash, "n_outside": None, "n_capped": None,
            "pass": None, "best": None, "best_energy": None}


def _network64(h, x, train, labels):
    """The trained network in FP64 on rows x, standardised by its training set."""
    p = torch.from_numpy(N.ligate_surrogate_get_weights(h)).cuda().double()
    sd = train.double().std(0, unbiased=False)
    y = (x.double() - train.double().mean(0)) / torch.where(sd > 1e-12, sd, torch.ones_like(sd))
    o = 0
    for a, b in ((256, 512), (512, 512), (512, 512), (512, 1)):
        y = y @ p[o:o + a * b].view(a, b) + p[o + a * b:o + a * b + b]
        o += a * b + b
        if b > 1:
            y = y.clamp(min=0)
    lab = labels.double()
    return y[:, 0] * lab.std(unbiased=False) + lab.mean()


def exact(case, seed):
    kind = case["kind"]
    if kind == "dock" and case["ligands"] <= 2 and case["orient"] * case["anchor"] <= 1024 and \
            case["mode"] in ("fp32", "fp32c"):
        return {"score": _dock64(_workload(case, seed), case["mode"]), "start": None, "tors": None}
    if kind == "rescore":
        return _rescore64(prepare(case, seed))
    if kind == "rank":
        st = prepare(case, seed)
        r = run(st)
        return {"desc": None, "pred": _network64(st.net.h, r["desc"], st.train_desc, st.labels), "kept": None}
    if kind == "select":
        st = prepare(case, seed)
        return {"feat": None, "pred": _network64(st.net.h, st.train_desc, st.train_desc, st.labels), "kept": None}
    return None
