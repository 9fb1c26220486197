"""Descriptors, refinement gradients, exact rescoring and pose features at the
sizes where their kernels change shape: atoms around multiples of 32 and pair
distances on the bins' edges, 1 to 4 atoms per lane, receptors from one atom
to several list steps that reach beyond the box, and rows at a 4-byte
alignment."""
import contextlib

import numpy as np
import pytest

import oracle
from paper_2304_09953_gb300 import docking as D
from paper_2304_09953_gb300 import native as N
from paper_2304_09953_gb300.workload import Pocket, Sampling, make_ligands
from tests.device_memory import all_but
from tests.parity import Geometry, Stats, check_state_energies, rescore_check
from tests.test_gpu_refine import seeded_states, to_dev
from tests.test_gpu_rescore import explicit

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ATOMS = np.array([1, 2, 3, 4, 8, 17, 31, 32, 33, 47, 48, 63, 64, 65, 96, 97, 128, 33], np.int32)


@pytest.mark.parametrize("types", [8, 1])
def test_descriptors_at_edge_sizes(types):
    """Counts are the oracle's, on a lattice of half bin widths where most
    distances lie exactly on an edge; many ligands per warp and unaligned rows
    change nothing."""
    ligs = make_ligands(3, ATOMS, np.minimum(ATOMS // 8, 16).astype(np.int32), types)
    ligs.xyz[:] = np.round(ligs.xyz / 0.75) * 0.75
    n = ligs.n
    bh = D.BatchHandle(ligs)
    out = torch.full((n * 256 + 2,), -1.0, dtype=torch.float32, device="cuda")
    N.ligate_descriptors(bh.h, out[:n * 256])
    got = out.cpu().numpy()
    assert np.all(got[n * 256:] == -1.0)
    for i in range(n):
        want = oracle.descriptor(ligs.ligand(i))
        np.testing.assert_array_equal(np.round(np.expm1(got[256 * i:256 * i + 256])), np.round(np.expm1(want)))
    shifted = torch.full((n * 256 + 2,), -1.0, dtype=torch.float32, device="cuda")
    N.ligate_descriptors(bh.h, shifted.data_ptr() + 4)
    assert torch.equal(shifted[1:-1], out[:-2]) and shifted[0] == -1.0 and shifted[-1] == -1.0
    idx = np.arange(33000) % n  # four ligands per warp, the last block part full
    many = D.BatchHandle(ligs.subset(list(idx)))
    big = torch.empty((len(idx), 256), dtype=torch.float32, device="cuda")
    N.ligate_descriptors(many.h, big)
    assert torch.equal(big, out[:n * 256].reshape(n, 256)[torch.from_numpy(idx).cuda()])


@pytest.mark.parametrize("n_atoms", [30, 32, 33, 64, 96])
def test_gradient_does_not_depend_on_the_batch(tiny, n_atoms):
    """The batch's largest ligand sets the atoms per lane: a ligand's energy
    and gradient are the same bits beside a 128-atom one."""
    own = make_ligands(8, np.array([n_atoms, 128], np.int32), np.array([min(6, n_atoms // 5), 16], np.int32), 4)

    class W:
        pocket, ligands, sampling = tiny.pocket, own, tiny.sampling

    lig, rec, _ = seeded_states(W, np.zeros(1, int), np.random.default_rng(n_atoms), 33)
    ph = D.PocketHandle(tiny.pocket)
    s = N.make_sampling(tiny.sampling, N.LIGATE_FP32, N.LIGATE_LAYOUT_PLAIN, False, None)
    res = []
    for ligs in (own.subset([0]), own):
        bh = D.BatchHandle(ligs)
        e = torch.zeros(len(lig), dtype=torch.float32, device="cuda")
        g = torch.zeros((len(lig), N.LIGATE_GRAD_DIM), dtype=torch.float32, device="cuda")
        N.ligate_pose_gradient(ph.h, bh.h, s, len(lig), torch.from_numpy(lig).cuda(), to_dev(rec), e, g)
        res.append((e.cpu().numpy(), g.cpu().numpy()))
        bh.close()
    ph.close()
    assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])


@pytest.mark.parametrize("n_rec,beyond", [(1, 0.0), (63, 6.0), (65, 0.0), (1500, 12.0)])
def test_rescoring_and_features_over_receptor_sizes(tiny, n_rec, beyond):
    P0 = tiny.pocket
    rng = np.random.default_rng(n_rec)
    lo, hi = np.asarray(P0.origin), np.asarray(P0.origin) + (np.array(P0.dims) - 1) * P0.spacing
    n_types = P0.maps.shape[0]
    P = Pocket(P0.maps, P0.origin, P0.spacing, P0.anchors, rng.uniform(lo - beyond, hi + beyond, size=(n_rec, 3)),
               rng.integers(0, n_types, size=n_rec).astype(np.int32), np.linspace(1.5, 2.0, n_types),
               np.linspace(0.1, 0.3, n_types))

    class W:
        pocket, ligands, sampling = P, tiny.ligands, tiny.sampling

    lig, sid, tors = explicit(W, 64, 5)
    n = len(lig)
    ph, bh = D.PocketHandle(P), D.BatchHandle(W.ligands)
    s = N.make_sampling(W.sampling)
    dev = [torch.from_numpy(a).cuda() for a in (lig, sid, tors)]
    out = torch.zeros(n * N.RESCORED_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    N.ligate_rescore_poses(ph.h, bh.h, s, n, *dev, out)
    r = out.cpu().numpy().view(N.RESCORED_DTYPE)
    geo, st = Geometry(P), Stats()
    for li in np.unique(lig):
        sel = np.nonzero(lig == li)[0]
        rescore_check(geo, W.ligands.ligand(li), P, W.sampling, sid[sel], tors[sel, :int(W.ligands.n_rot[li])],
                      r[sel], st)
    print(st.line())
    f = torch.empty(n * 256, dtype=torch.float32, device="cuda")
    shifted = torch.full((n * 256 + 2,), -1.0, dtype=torch.float32, device="cuda")
    N.ligate_pose_features(ph.h, bh.h, s, n, *dev, f)
    N.ligate_pose_features(ph.h, bh.h, s, n, *dev, shifted.data_ptr() + 4)
    assert torch.equal(shifted[1:-1], f) and shifted[0] == -1.0 and shifted[-1] == -1.0
    bh.close()
    ph.close()


@pytest.mark.parametrize("n_lig,orient,anchor,S,K", [(1, 64, 128, 8, 4), (40, 3, 5, 17, 1)])
def test_docking_many_starts_or_rows(batched_small, n_lig, orient, anchor, S, K):
    """One ligand with thousands of starts, and clash tables by rounds of a
    table or whole tables, give what large items give."""
    w = batched_small
    ligs = w.ligands.subset([i % w.ligands.n for i in range(n_lig)])
    q = np.random.default_rng(1).normal(size=(orient, 4))
    a = np.asarray(w.pocket.anchors)
    P = Pocket(w.pocket.maps, w.pocket.origin, w.pocket.spacing,
               np.ascontiguousarray(a[np.arange(anchor) % len(a)] + 0.01 * np.arange(anchor)[:, None], np.float32),
               w.pocket.receptor_xyz, w.pocket.receptor_type, w.pocket.type_radius, w.pocket.type_eps)
    samp = Sampling((q / np.linalg.norm(q, axis=1, keepdims=True)), anchor, S, K)
    ph, bh = D.PocketHandle(P), D.BatchHandle(ligs)
    t = N.ligate_tile()
    for b in range(N.LIGATE_N_BUCKETS):
        t.starts_per_item[b] = 2048
    ref = D.Plan(ph, bh, samp, mode="fp32", tile=t).result()
    assert np.array_equal(D.Plan(ph, bh, samp, mode="fp32").result(), ref)
    bh.close()
    ph.close()


@pytest.mark.parametrize("length", [1e3, 3e5, 1e6, 3e6])
def test_rescoring_beside_a_receptor_atom_far_away(tiny, length):
    """A receptor atom far from the box makes the cells wide, and a point's
    cell index rounds by up to 1e-7 of the receptor's length: a one-atom
    ligand stepped across the cell boundary beside the receptor's near end
    still sees every receptor atom within the cutoff (FP64 sum)."""
    P0, h, cut = tiny.pocket, tiny.pocket.spacing, 8.0
    near = 0.75 * (P0.dims[0] - 1) * h  # the near end
    worst = 0.0
    for k in range(8):
        far = np.float32(-length * (1 + 0.003 * k))
        lo, mx = np.float32(float(far) / h), np.float32(near / h)
        end = (float(lo) + (float(mx) - float(lo)) * (1 + 1e-6) + 1e-3) * h  # the last cell's boundary
        # a ladder of receptor atoms about the cutoff before the boundary, 0.6 mA apart
        x = np.float32(end - cut - 0.06 + 6e-4 * np.arange(200))
        y = np.full(201, 4.0, np.float32)
        xyz = np.stack([np.append(x, np.float32(near)), y, y], 1)
        xyz = np.vstack([xyz, [[far, 4.0, 4.0]]]).astype(np.float32)
        xyz[-2, 1] = 100.0  # the near end's own atom sits beyond the cutoff
        T = P0.maps.shape[0]
        rad, eps = np.full(T, 1.8), np.full(T, 0.2)
        P = Pocket(P0.maps, np.zeros(3), h, P0.anchors, xyz, np.zeros(len(xyz), np.int32), rad, eps)
        lig = make_ligands(1, np.array([1], np.int32), np.array([0], np.int32), T)
        px = np.float32(end - 0.06 + 6e-4 * np.arange(200) + 3e-4)
        st = np.zeros(len(px), N.STATE_DTYPE)
        st["rot"][:] = np.eye(3, dtype=np.float32).reshape(-1)
        st["trans"][:] = np.stack([px, np.full_like(px, 4.0), np.full_like(px, 4.0)], 1)
        ph, bh = D.PocketHandle(P), D.BatchHandle(lig)
        out = torch.zeros(len(px) * N.RESCORED_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        N.ligate_rescore_states(ph.h, bh.h, N.make_sampling(tiny.sampling), len(px),
                                torch.zeros(len(px), dtype=torch.int32, device="cuda"), to_dev(st), out)
        got = out.cpu().numpy().view(N.RESCORED_DTYPE)["e_inter"].astype(np.float64)
        bh.close()
        ph.close()
        d = np.abs(px.astype(np.float64)[:, None] - x.astype(np.float64))
        q = (3.6 / d) ** 6
        want = np.where(d <= cut, 0.2 * (q * q - 2 * q), 0.0).sum(1)
        worst = max(worst, np.abs(got - want).max())
    # one atom at the cutoff counts 0.0033: positions are half a step off the ladder,
    # so FP32 rounding moves none across it
    assert worst < 5e-4, worst


def test_listed_and_coarse_cells_give_the_same_bits(batched_small):
    """A receptor set while there is no room for its fine cells' lists is
    summed over the coarse cells: poses inside the lists, across their rim and
    outside them (atoms of both kinds side by side) get the same bits."""
    w, P0 = batched_small, batched_small.pocket
    rng = np.random.default_rng(8)
    lo, hi = np.asarray(P0.origin), np.asarray(P0.origin) + (np.array(P0.dims) - 1) * P0.spacing
    n_types = P0.maps.shape[0]
    bare = Pocket(P0.maps, P0.origin, P0.spacing, P0.anchors)
    rec = (rng.uniform(lo - 14.0, hi + 14.0, size=(11000, 3)).astype(np.float32),
           rng.integers(0, n_types, size=11000).astype(np.int32), np.linspace(1.5, 2.0, n_types),
           np.linspace(0.1, 0.3, n_types), 8.0, 10.0, 0.5)

    class W:
        pocket, ligands, sampling = P0, w.ligands, w.sampling

    lig, st, _ = seeded_states(W, np.arange(w.ligands.n), rng, 40, spread=10.0)
    st["trans"][::50] += np.float32(300.0)
    bh, s = D.BatchHandle(w.ligands), N.make_sampling(w.sampling)
    dev = torch.from_numpy(lig).cuda(), to_dev(st)
    outs, used = [], []
    N.ligate_pocket_set_receptor(D.PocketHandle(bare, mask=0).h, *rec)  # what the first call loads
    for short in (False, True):
        ph = D.PocketHandle(bare, mask=0)
        torch.cuda.empty_cache()
        with all_but(4 << 20) if short else contextlib.nullcontext():
            before = torch.cuda.mem_get_info()[0]
            N.ligate_pocket_set_receptor(ph.h, *rec)
            used.append(before - torch.cuda.mem_get_info()[0])
        out = torch.zeros(len(lig) * N.RESCORED_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        N.ligate_rescore_states(ph.h, bh.h, s, len(lig), *dev, out)
        outs.append(out.cpu().numpy().view(N.RESCORED_DTYPE))
        ph.close()
    bh.close()
    assert used[0] > 6 << 20 > used[1], used
    assert np.array_equal(outs[0], outs[1])
    e = outs[0]["e_inter"]
    assert (e == 0).any() and (np.abs(e) > 1).sum() > len(e) // 2


@pytest.mark.parametrize("cutoff", [3.99, 4.01, 4.48, 5.01, 30.0])
def test_gradient_at_wide_clash_cutoffs(tiny, cutoff):
    """Cutoffs from which the pairs that touch are not looked for, which depends
    on the batch's largest ligand: energy and gradient are the same bits beside
    a ligand that takes more atoms per lane, and the oracle's."""
    own = make_ligands(8, np.array([20, 33, 64, 128], np.int32), np.array([3, 5, 6, 16], np.int32), 4)
    samp = Sampling(tiny.sampling.quats, tiny.sampling.n_anchor, tiny.sampling.torsion_steps, tiny.sampling.top_k,
                    clash_cutoff=cutoff)

    class W:
        pocket, ligands, sampling = tiny.pocket, own, samp

    ph = D.PocketHandle(tiny.pocket)
    s = N.make_sampling(samp, N.LIGATE_FP32, N.LIGATE_LAYOUT_PLAIN, False, None)
    for li in range(3):
        lig, rec, st64 = seeded_states(W, [li], np.random.default_rng(li), 17)
        res = []
        for ligs, at in ((own.subset([li]), 0), (own, li)):
            bh = D.BatchHandle(ligs)
            e = torch.zeros(len(lig), dtype=torch.float32, device="cuda")
            g = torch.zeros((len(lig), N.LIGATE_GRAD_DIM), dtype=torch.float32, device="cuda")
            N.ligate_pose_gradient(ph.h, bh.h, s, len(lig), torch.full((len(lig),), at, dtype=torch.int32,
                                                                     device="cuda"), to_dev(rec), e, g)
            res.append((e.cpu().numpy(), g.cpu().numpy()))
            bh.close()
        assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])
        e64, g64, sc, _, face = oracle.pose_grad(own.ligand(li), tiny.pocket, samp, np.array(st64))
        check_state_energies(Geometry(tiny.pocket), own.ligand(li), tiny.pocket, samp, rec, st64, res[0][0], e64)
        for k in np.nonzero(face >= 1e-4)[0]:  # the bar of the gradient's own test
            np.testing.assert_array_less(np.abs(res[0][1][k, :g64.shape[1]] - g64[k]), 2e-4 * np.maximum(sc[k, 1:], 1.0))
    ph.close()
