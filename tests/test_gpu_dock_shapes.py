"""The docking kernel's instances and work-item shapes give the same bits:
16-lane instances against the generic ones, small items against large ones,
a plain-layout plan (which searches the pocket's FP32 corner copy) against
one whose pocket has no copy, at torsion steps around the group sizes and
list lengths from one to the limit; and the result is the oracle's."""
import contextlib

import numpy as np
import pytest

from paper_2304_09953_gb300 import docking as D
from paper_2304_09953_gb300 import native as N
from paper_2304_09953_gb300.workload import Sampling, make_ligands
from tests.device_memory import all_but
from tests.parity import Stats, compare_ligand

pytestmark = pytest.mark.gpu


def tile(chunk=0, reg_cap=0, warps=0):
    t = N.ligate_tile()
    t.reg_cap, t.warps_per_cta = reg_cap, warps
    for b in range(N.LIGATE_N_BUCKETS):
        t.starts_per_item[b] = chunk
    return t


@pytest.mark.parametrize("S,K,orient,anchor", [(1, 1, 3, 5), (7, 4, 5, 7), (8, 32, 8, 8), (9, 5, 6, 11), (16, 16, 16, 8),
                                               (16, 1, 1, 1), (17, 7, 4, 9), (32, 32, 9, 7)])
def test_shapes_agree_and_match_the_oracle(batched_small, S, K, orient, anchor):
    w = batched_small
    idx = [i for i in range(w.ligands.n) if w.ligands.n_rot[i] in (0, 1, 2, 5, 12)][:10] + [1, 2, 3]
    ligs = w.ligands.subset(idx)
    samp = Sampling(w.sampling.quats[:orient], anchor, S, K)
    full, plain = D.PocketHandle(w.pocket), D.PocketHandle(w.pocket, mask=0)
    bh = D.BatchHandle(ligs)
    try:
        ref = D.Plan(full, bh, samp, mode="fp32").result()
        for pocket, mode, t in ((full, "fp32", tile(chunk=8)), (full, "fp32", tile(chunk=4096, warps=1)),
                                (full, "fp32", tile(reg_cap=1)), (full, "fp32c", tile(reg_cap=3)),
                                (plain, "fp32", None), (plain, "fp32", tile(chunk=64, reg_cap=2))):
            assert np.array_equal(D.Plan(pocket, bh, samp, mode=mode, tile=t).result(), ref)
        bf = D.Plan(full, bh, samp, mode="bf16").result()
        for t in (tile(chunk=8), tile(reg_cap=1), tile(reg_cap=3, warps=2)):
            assert np.array_equal(D.Plan(full, bh, samp, mode="bf16", tile=t).result(), bf)
    finally:
        bh.close()
        full.close()
        plain.close()
    st = Stats()
    for r in range(0, len(idx), 4):
        if K <= samp.n_starts:
            compare_ligand(ligs.ligand(r), w.pocket, samp, ref[r], K=K, stats=st)
    print(st.line())


@pytest.mark.parametrize("n_atoms", [64, 65, 96, 128])
@pytest.mark.parametrize("S", [1, 2])
def test_large_ligands_at_few_torsion_steps(batched_small, S, n_atoms):
    """The most start groups per warp with the largest ligands, whose slots
    limit the warps of a CTA: a full run, a selection and the one-call docking
    give the oracle's poses."""
    torch = pytest.importorskip("torch")
    w = batched_small
    ligs = make_ligands(17, np.array([n_atoms, 24, n_atoms], np.int32), np.array([8, 3, 16], np.int32),
                        w.pocket.n_types)
    samp = Sampling(w.sampling.quats[:8], 8, S, 4)
    ph, bh = D.PocketHandle(w.pocket), D.BatchHandle(ligs)
    pl = D.Plan(ph, bh, samp, mode="fp32")
    res = pl.result()
    sel = torch.tensor([2, 0], dtype=torch.int32, device="cuda")
    assert np.array_equal(pl.run_subset(sel, result=True), res[[2, 0]])
    out = np.zeros((ligs.n, 4), N.POSE_DTYPE)
    N.ligate_dock_batch(ph.h, ligs, N.make_sampling(samp, *D.MODES["fp32"], False), out)
    assert np.array_equal(out, res)
    st = Stats()
    for r in range(ligs.n):
        compare_ligand(ligs.ligand(r), w.pocket, samp, res[r], K=4, stats=st)
    print(st.line())


def test_clash_tables_give_way_to_memory(batched_small):
    """A plan whose ligands' clash tables (96 MB here) find no room takes
    tables per warp (32 MB) and gives the same bits."""
    torch = pytest.importorskip("torch")
    w = batched_small
    ligs = w.ligands.subset([i % w.ligands.n for i in range(8000)])
    samp = Sampling(w.sampling.quats[:16], 8, 16, 1)
    ph, bh = D.PocketHandle(w.pocket), D.BatchHandle(ligs)
    D.Plan(ph, bh, samp, mode="bf16").result()  # what the first run loads
    torch.cuda.empty_cache()
    res, used = [], []
    for short in (False, True):
        with all_but(64 << 20) if short else contextlib.nullcontext():
            before = torch.cuda.mem_get_info()[0]
            pl = D.Plan(ph, bh, samp, mode="bf16")
            used.append(before - torch.cuda.mem_get_info()[0])
            res.append(pl.result())
            pl.close()
    assert used[0] > 64 << 20 > used[1]
    assert np.array_equal(res[0], res[1])


def test_quantile_captured_after_a_smaller_selection(batched_small):
    """The quantile's scratch, made at its first call on a selection, serves a
    full run: nothing is allocated inside a stream capture."""
    torch = pytest.importorskip("torch")
    w = batched_small
    ph, bh = D.PocketHandle(w.pocket), D.BatchHandle(w.ligands)
    pl = D.Plan(ph, bh, Sampling(w.sampling.quats[:8], 8, 8, 1), mode="fp32")
    cut = torch.zeros(1, dtype=torch.float32, device="cuda")
    pl.run_subset(torch.arange(3, dtype=torch.int32, device="cuda"))
    pl.best_quantile(1.0, cut)
    best = np.sort(pl.result()[:, 0]["score"])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pl.best_quantile(0.5, cut, torch.cuda.current_stream().cuda_stream)
    graph.replay()
    assert cut.item() == best[w.ligands.n // 2 - 1]


@pytest.mark.parametrize("S", [4, 8, 16, 18, 32])
def test_small_runs_stay_below_1024_items(batched_small, S):
    """A run of one ligand spreads its starts over the resident warps in fewer
    than 1,024 items, whose lists one warp merges."""
    w = batched_small
    bh, ph = D.BatchHandle(w.ligands.subset([0])), D.PocketHandle(w.pocket)
    for orient, anchor in ((20, 30), (31, 33), (33, 31), (48, 32), (64, 31), (128, 31)):
        q = np.random.default_rng(orient).normal(size=(orient, 4))
        samp = Sampling(q / np.linalg.norm(q, axis=1, keepdims=True), min(anchor, len(w.pocket.anchors)), S, 4)
        pl = D.Plan(ph, bh, samp, mode="fp32c")
        least = min(pl.tile()[0].starts_per_item)
        assert least > 0 and -(-samp.n_starts // least) < 1024, (samp.n_starts, least)
        pl.close()
