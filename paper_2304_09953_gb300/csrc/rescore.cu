// Exact rescoring, pose filter and per-pose selector features (paper
// Sec. 2: a more accurate scoring of the generated poses and a filter;
// Sec. 3.5: a high-throughput pose selector).  Poses come from explicit
// (ligand, start, torsion steps) arrays, from a plan's output, or as
// continuous states (refined poses).
#include <math.h>
#include <string.h>

#include <algorithm>

#include "dock_device.cuh"

namespace ligate {

// ---------------------------------------------------------------------------
// Exact rescoring and filter of explicit or planned poses (paper Sec. 2: a
// more accurate scoring of the generated poses, then a filter).  The
// receptor term is the maps' pair potential evaluated at each atom:
// min(cap, sum_j eps_tj ((r0/r)^12 - 2 (r0/r)^6)) over receptor atoms within
// the cutoff, r floored at rmin (grid units throughout); the clash term is
// the docking score's.
//
// The receptor atoms are sorted by cell of a grid whose cells are at least the
// cutoff wide; a warp takes runs of consecutive poses (mostly one ligand's),
// builds each and sums the receptor term atom by atom (receptor_cells defines
// the sum).
//
// What bounds it: issue and latency of the distance tests (65% of active cycles
// issue; waits on fixed latency, L1 and branches).  The 27 cells
// around an atom hold 6.4 times the atoms within the cutoff.  So each coarse
// cell is split into fine cells about 2 A wide, and a fine cell has the
// receptor atoms that can be within the cutoff of a point in it (1.8 times),
// laid out as the 64 columns (lane, accumulator) that receptor_cells gives
// them, in its order: the same terms in the same order, so the same bits, in a
// third of the steps.  16-bit indices keep the lists small (128 bytes per
// step), and the coordinates stay in L1: staged in shared memory (16 B per
// receptor atom and CTA) they left 24 warps per SM at 3,000 receptor atoms and
// 8 at 8,000.  Two atoms run side by side, for the latency of the loads and of
// the warp sums.  32,000 poses of the batched library (3,000 receptor atoms)
// 2,160 -> 955 us, 4,800 of the large target's (8,000) 815 -> 164 us.
// One receptor atom's term at squared distance d2, added to acc.
__device__ __forceinline__ float pair_term(const RecParams &r, const float2 &pp, float d2, float acc) {
  const float q2 = __fdividef(pp.x, fmaxf(d2, r.rmin2));
  const float q6 = q2 * q2 * q2;
  return fmaf(pp.y, fmaf(q6, q6, -2.f * q6), acc);
}

// Coarse cell coordinate of u along one axis, as a float (clamped to two cells
// beyond the grid first, so far or non-finite coordinates give an empty
// neighbourhood or edge cells).
__device__ __forceinline__ float cell_coord(float u, float lo, float inv, int n) {
  return fminf(fmaxf((u - lo) * inv, -2.f), (float)n + 1.f);
}

// This lane's part of the receptor sum at u over the 3 x 3 x 3 coarse cells around
// it (clamped to the grid), for points outside the fine cells: two receptor atoms
// per lane per iteration, an accumulator each.  What bounds it is the latency of
// short rows, so their bounds are loaded side by side and the two points' sums
// over the lanes run together: 20,000 poses over 24 A beside 400 receptor atoms
// with a cutoff of 3 A 510 -> 419 us, 960 poses all outside 344 -> 311 us.
// Warp-collective, u the same in every lane.
__device__ __noinline__ float receptor_cells(const RecParams &r, const float2 *prow, float ux, float uy,
                                             float uz, int lane) {
  const int cx = (int)floorf(cell_coord(ux, r.lox, r.icx, r.ncx)), cy = (int)floorf(cell_coord(uy, r.loy, r.icy, r.ncy)),
            cz = (int)floorf(cell_coord(uz, r.loz, r.icz, r.ncz));
  const int x0 = max(cx - 1, 0), x1 = min(cx + 1, r.ncx - 1);
  const int y0 = max(cy - 1, 0), y1 = min(cy + 1, r.ncy - 1);
  const int z0 = max(cz - 1, 0), z1 = min(cz + 1, r.ncz - 1);
  // lane r has the bounds of row r of the neighbourhood (x fastest, then y, z)
  const int ny = y1 - y0 + 1, rows = x0 <= x1 && ny > 0 ? ny * max(z1 - z0 + 1, 0) : 0;
  int lo = 0, hi = 0;
  if (lane < rows) {
    const int row = ((z0 + lane / ny) * r.ncy + y0 + lane % ny) * r.ncx;
    lo = __ldg(r.cell + row + x0);
    hi = __ldg(r.cell + row + x1 + 1);
  }
  float acc[2] = {0.f, 0.f};
  for (int k = 0; k < rows; ++k) {
    const int j_hi = __shfl_sync(FULL, hi, k);
    for (int j0 = __shfl_sync(FULL, lo, k) + lane; j0 < j_hi; j0 += 64) {
      float4 a[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) a[q] = __ldg(r.rec + min(j0 + 32 * q, j_hi - 1));
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float dx = ux - a[q].x, dy = uy - a[q].y, dz = uz - a[q].z;
        const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        if (j0 + 32 * q < j_hi && d2 <= r.cut2)
          acc[q] = pair_term(r, prow[__float_as_int(a[q].w)], d2, acc[q]);
      }
    }
  }
  return acc[0] + acc[1];
}

// The fine cells' lists, a warp per cell: lane l has the columns l and l + 32
// (positions l, l + 32, l + 64, ... of a row of cells, in turn).  Steps of the
// longest column, or the entries themselves, 0xffff where a column has ended.
// Bound by issue on the distance tests, in FP32 (the reach's margin covers their
// rounding): in FP64, which this device runs at a sixty-fourth of the rate, the
// two passes over 3,000 receptor atoms and 12,167 cells took 360 us each.
__global__ void __launch_bounds__(256) fine_lists_kernel(const FineGrid g, const float4 *__restrict__ rec,
                                                        const int *__restrict__ cell, const int *__restrict__ first,
                                                        int *__restrict__ steps, uint16_t *__restrict__ list) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= g.nf[0] * g.nf[1] * g.nf[2]) return;
  const int fc[3] = {c % g.nf[0], c / g.nf[0] % g.nf[1], c / g.nf[0] / g.nf[1]};
  int k0[3], k1[3];
  float b0[3], b1[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int cc = (g.f0[a] + fc[a] + g.fs[a]) / g.fs[a] - 1;  // from the coarse cell before the grid
    b0[a] = (float)(g.lo[a] + (g.f0[a] + fc[a]) * g.wf[a]);
    b1[a] = (float)(g.lo[a] + (g.f0[a] + fc[a] + 1) * g.wf[a]);
    k0[a] = max(cc - 1, 0);
    k1[a] = min(cc + 1, g.nc[a] - 1);
  }
  const int total = steps ? 0 : first[c + 1] - first[c];
  uint16_t *const out = steps ? nullptr : list + 64 * (size_t)first[c];
  const float reach2 = (float)g.reach2;
  int n[2] = {0, 0};
  if (k0[0] <= k1[0])
    for (int z = k0[2]; z <= k1[2]; ++z)
      for (int y = k0[1]; y <= k1[1]; ++y) {
        const int row = (z * g.nc[1] + y) * g.nc[0], j1 = cell[row + k1[0] + 1];
        for (int j0 = cell[row + k0[0]] + lane; j0 < j1; j0 += 64)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int j = j0 + 32 * q;
            if (j >= j1) continue;
            const float4 v = rec[j];
            const float dx = fmaxf(0.f, fmaxf(b0[0] - v.x, v.x - b1[0])), dy = fmaxf(0.f, fmaxf(b0[1] - v.y, v.y - b1[1])),
                        dz = fmaxf(0.f, fmaxf(b0[2] - v.z, v.z - b1[2]));
            if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) > reach2) continue;
            if (out && n[q] < total) out[64 * n[q] + lane + 32 * q] = (uint16_t)j;
            ++n[q];
          }
      }
  if (steps) {
    const int most = (int)__reduce_max_sync(FULL, (unsigned)max(n[0], n[1]));
    if (lane == 0) steps[c] = most;
  } else {
#pragma unroll
    for (int q = 0; q < 2; ++q)
      for (int k = n[q]; k < total; ++k) out[64 * k + lane + 32 * q] = 0xffff;
  }
}

constexpr int POSE_RUN = 4;  // consecutive poses a warp takes at a time

__global__ void __launch_bounds__(256) rescore_kernel(const __grid_constant__ DockParams p,
                                                     const __grid_constant__ RecParams r, int n_poses,
                                                     const int32_t *__restrict__ lig_idx,
                                                     const int32_t *__restrict__ start_id,
                                                     const uint8_t *__restrict__ tors,
                                                     const PoseOut *__restrict__ poses,
                                                     const int32_t *__restrict__ row_lig,
                                                     const StateSrc ss,
                                                     ligate_rescored *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2 *pair = reinterpret_cast<float2 *>(smem_raw);
  unsigned char *slots = reinterpret_cast<unsigned char *>(pair + ((r.n_types * r.n_types + 1) & ~1));
  for (int j = threadIdx.x; j < r.n_types * r.n_types; j += blockDim.x) pair[j] = r.pair[j];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  // warp slots without a pair list
  const WarpSmem w = warp_smem(slots + (size_t)warp * smem_bytes_per_warp(p.nmax, 0, 1, 0, 0), p.nmax, 1, 0);
  // runs of consecutive poses, shorter when there are few poses per warp
  const int warps = gridDim.x * W;
  const int run = max(1, min(POSE_RUN, n_poses / (8 * warps)));  // at least 8 runs per warp: balance
  int cur = -1;
  LigDesc d;
  for (long long t = (long long)(blockIdx.x * W + warp) * run, s = 0; t < n_poses;
       t = ++s == run ? (s = 0, t + 1 + (long long)(warps - 1) * run) : t + 1) {
    const int pi = (int)t;
    int li, sid;
    uint32_t tt[4] = {0u, 0u, 0u, 0u};
    const unsigned char *st_rec = nullptr;
    if (ss.base) {  // continuous state
      st_rec = ss.base + (size_t)pi * ss.stride;
      li = ss.lig_idx ? ss.lig_idx[pi] : *reinterpret_cast<const int32_t *>(st_rec + ss.lig_offset);
      sid = (ss.score_offset >= 0 && !isfinite(*reinterpret_cast<const float *>(st_rec + ss.score_offset)))
                ? -1 : 0;  // an empty slot of a refined plan output
    } else if (poses) {
      const PoseOut po = poses[pi];
      li = row_lig[pi / p.K];
      sid = po.start_id;
      for (int q = 0; q < 4; ++q) tt[q] = po.tors[q];
    } else {
      li = lig_idx[pi];
      sid = start_id[pi];
      for (int q = 0; q < 16; ++q) tt[q >> 2] |= (uint32_t)tors[(size_t)pi * 16 + q] << (8 * (q & 3));
    }
    if (li < 0 || li >= p.n_ligands || sid < 0 || sid >= p.n_starts) {  // empty slot or bad index
      if (lane == 0) {
        ligate_rescored o;
        o.energy = o.e_inter = o.e_clash = __int_as_float(0x7f800000);
        o.n_outside = o.n_capped = -1;
        o.pass = 0;
        out[pi] = o;
      }
      continue;
    }
    if (li != cur) {
      __syncwarp();
      d = p.lig[li];
      load_coords(p, w, d, lane);
      cur = li;
    }
    if (st_rec) {
      // state (R, t, phi): torsions on the centred input coordinates about
      // the current axes, then x = R y + t (A) and u = (x - origin) / h
      const float *R = reinterpret_cast<const float *>(st_rec);
      build_state(w.ref, w.pose, w.bonds, d, R, R + 9, R + 12, lane);
      for (int i = lane; i < d.n_atoms; i += 32) {
        float4 u = w.pose[i];
        u.x = (u.x - r.ox) * r.inv_h;
        u.y = (u.y - r.oy) * r.inv_h;
        u.z = (u.z - r.oz) * r.inv_h;
        w.pose[i] = u;
      }
      __syncwarp();
    } else {
      build_pose<MODE_F32_PLAIN>(p, w, w.pose, d, sid, tt, lane);
    }
    float e_inter = 0.f;
    int ncap = 0, nout = 0;
    for (int i0 = 0; i0 < d.n_atoms; i0 += 32) {
      // the lanes look up their own atoms' fine cells side by side (steps -1:
      // outside them, 0: no receptor cell around either)
      int lo_l = 0, steps_l = 0;
      bool out_l = false;
      if (i0 + lane < d.n_atoms) {
        const float4 u = w.pose[i0 + lane];
        out_l = !((u.x >= 0.f) & (u.x <= p.g.fx1) & (u.y >= 0.f) & (u.y <= p.g.fy1) & (u.z >= 0.f) & (u.z <= p.g.fz1));
        const float vx = cell_coord(u.x, r.lox, r.icx, r.ncx), vy = cell_coord(u.y, r.loy, r.icy, r.ncy),
                    vz = cell_coord(u.z, r.loz, r.icz, r.ncz);
        const float cx = floorf(vx), cy = floorf(vy), cz = floorf(vz);
        const int fx = (int)cx * r.fsx + min((int)((vx - cx) * (float)r.fsx), r.fsx - 1) - r.fx0,
                  fy = (int)cy * r.fsy + min((int)((vy - cy) * (float)r.fsy), r.fsy - 1) - r.fy0,
                  fz = (int)cz * r.fsz + min((int)((vz - cz) * (float)r.fsz), r.fsz - 1) - r.fz0;
        if (fx >= 0 && fx < r.nfx && fy >= 0 && fy < r.nfy && fz >= 0 && fz < r.nfz) {
          const int *f = r.fine + (fz * r.nfy + fy) * r.nfx + fx;
          lo_l = __ldg(f);
          steps_l = __ldg(f + 1) - lo_l;
        } else if (cx >= -1.f && cx <= (float)r.ncx && cy >= -1.f && cy <= (float)r.ncy && cz >= -1.f && cz <= (float)r.ncz) {
          steps_l = -1;
        }
      }
      nout += __popc(__ballot_sync(FULL, out_l));
      const int i1 = min(32, d.n_atoms - i0);
      for (int i = 0; i < i1; i += 2) {  // two atoms side by side: their chains and loads overlap
        float4 u[2];
        const float2 *prow[2];
        const uint16_t *list[2];
        int steps[2];
        float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
        unsigned nx[2][2];  // the next step's indices
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const int k = min(i + v, i1 - 1);
          u[v] = w.pose[i0 + k];
          prow[v] = pair + __float_as_int(w.ref[i0 + k].w) * r.n_types;
          list[v] = r.list + (size_t)__shfl_sync(FULL, lo_l, k) * 64 + lane;
          steps[v] = __shfl_sync(FULL, steps_l, k);
          if (i + v >= i1) steps[v] = 0;
          nx[v][0] = nx[v][1] = 0xffffu;
          if (steps[v] > 0) { nx[v][0] = __ldg(list[v]); nx[v][1] = __ldg(list[v] + 32); }
        }
        const int top = max(steps[0], steps[1]);
        for (int k = 0; k < top; ++k) {
          unsigned j[2][2];
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            j[v][0] = nx[v][0];
            j[v][1] = nx[v][1];
            list[v] += 64;
            nx[v][0] = nx[v][1] = 0xffffu;
            if (k + 1 < steps[v]) { nx[v][0] = __ldg(list[v]); nx[v][1] = __ldg(list[v] + 32); }
          }
#pragma unroll
          for (int v = 0; v < 2; ++v)
#pragma unroll
            for (int q = 0; q < 2; ++q)
              if (j[v][q] != 0xffffu) {
                const float4 a = __ldg(r.rec + j[v][q]);
                const float dx = u[v].x - a.x, dy = u[v].y - a.y, dz = u[v].z - a.z;
                const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                if (d2 <= r.cut2) acc[v][q] = pair_term(r, prow[v][__float_as_int(a.w)], d2, acc[v][q]);
              }
        }
        float accs[2] = {acc[0][0] + acc[0][1], acc[1][0] + acc[1][1]};
#pragma unroll
        for (int v = 0; v < 2; ++v)
          if (steps[v] < 0) {  // warp-uniform
            const float4 x = w.pose[i0 + i + v];
            accs[v] = receptor_cells(r, pair + __float_as_int(w.ref[i0 + i + v].w) * r.n_types, x.x, x.y, x.z, lane);
          }
        accs[0] = warp_sum(accs[0]);
        accs[1] = warp_sum(accs[1]);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          if (i + v >= i1) continue;  // warp-uniform
          if (accs[v] >= r.cap) { accs[v] = r.cap; ++ncap; }
          e_inter += accs[v];
        }
      }
    }
    float cl = clash_pairs(p, w.pose, d, p.inv_dc2_grid, lane);
    cl = p.clash_w * warp_sum(cl);
    if (lane == 0) {
      ligate_rescored o;
      o.e_inter = e_inter;
      o.e_clash = cl;
      o.energy = e_inter + cl;
      o.n_outside = nout;
      o.n_capped = ncap;
      o.pass = (nout == 0 && ncap == 0) ? 1 : 0;
      out[pi] = o;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Per-pose selector features (paper Sec. 3.5: a high-throughput pose
// selector).  Per pose 256 FP32: [0, 64) log1p of the counts of atoms whose
// FP32 grid value v falls in bin min(63, max(0, floor((v + 4) * 4)));
// [64, 72) mean v per atom type 0..7; [72] docking score / atoms; [73] clash
// term; [74] log1p(atoms); [75] rotatable bonds; [76] log1p(count of
// v >= 9); rest 0.  One warp per pose; the histogram lives in the warp's
// pair-list slot.  An empty or invalid pose gives all zeros.
//
// What bounds it: instruction issue and the map gathers' latency (67% of active
// cycles issue; about 2,500 warp instructions per pose before, against 1 KB
// written).  Counts come from ballots, the per-type sums
// share one butterfly, log1p of the counts comes from a table made by the same
// function, the row is put together in shared memory and stored in 16-byte
// pieces, and a warp takes consecutive poses, mostly of one ligand: 32,000
// poses of the batched library 157 -> 90 us (serialised).
constexpr int FEAT_LOGS = LIGATE_MAX_ATOMS + 1;
constexpr int FEAT_LIST = 36;  // (80 + 64) * 4 / 16 pair-list entries
__global__ void __launch_bounds__(128) pose_features_kernel(const __grid_constant__ DockParams p, int n_poses,
                                                           const int32_t *__restrict__ lig_idx,
                                                           const int32_t *__restrict__ start_id,
                                                           const uint8_t *__restrict__ tors,
                                                           const PoseOut *__restrict__ poses,
                                                           const int32_t *__restrict__ row_lig,
                                                           float *__restrict__ out, int vec) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float logs[FEAT_LOGS];
  for (int q = threadIdx.x; q < FEAT_LOGS; q += blockDim.x) logs[q] = log1pf((float)q);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  // the pair-list slot holds the feature row (80 floats), then the histogram
  const WarpSmem w = warp_smem(smem_raw + (size_t)warp * smem_bytes_per_warp(p.nmax, 0, 1, 0, FEAT_LIST), p.nmax, 1,
                               FEAT_LIST);
  float *const row = reinterpret_cast<float *>(w.list);
  int *const hist = reinterpret_cast<int *>(row + 80);
  const int warps = gridDim.x * W;
  const int run = max(1, min(POSE_RUN, n_poses / (8 * warps)));
  int cur = -1;
  LigDesc d;
  for (long long t = (long long)(blockIdx.x * W + warp) * run, s = 0; t < n_poses;
       t = ++s == run ? (s = 0, t + 1 + (long long)(warps - 1) * run) : t + 1) {
    const int pi = (int)t;
    float *f = out + (size_t)pi * 256;
    int li, sid;
    uint32_t tt[4] = {0u, 0u, 0u, 0u};
    if (poses) {
      const PoseOut po = poses[pi];
      li = row_lig[pi / p.K];
      sid = po.start_id;
      for (int q = 0; q < 4; ++q) tt[q] = po.tors[q];
    } else {
      li = lig_idx[pi];
      sid = start_id[pi];
      for (int q = 0; q < 16; ++q) tt[q >> 2] |= (uint32_t)tors[(size_t)pi * 16 + q] << (8 * (q & 3));
    }
    if (li < 0 || li >= p.n_ligands || sid < 0 || sid >= p.n_starts) {
      for (int k = lane; k < 256; k += 32) f[k] = 0.f;
      continue;
    }
    if (li != cur) {
      __syncwarp();
      d = p.lig[li];
      load_coords(p, w, d, lane);
      cur = li;
    }
    build_pose<MODE_F32_PLAIN>(p, w, w.pose, d, sid, tt, lane);
    for (int b = lane; b < 64; b += 32) hist[b] = 0;
    __syncwarp();
    float e = 0.f, ts[8];
    int high = 0, tn[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) { ts[t] = 0.f; tn[t] = 0; }
    for (int i0 = 0; i0 < d.n_atoms; i0 += 32) {
      const int i = i0 + lane;
      const bool own = i < d.n_atoms;
      float v = 0.f;
      int ty = -1;
      if (own) {
        const float4 u = w.pose[i];
        v = grid_eval<MODE_F32_PLAIN>(p.maps_f32, __float_as_int(u.w), u.x, u.y, u.z, p.g);
        e += v;
        int b = (int)floorf((v + 4.f) * 4.f);
        b = min(63, max(0, b));
        atomicAdd(&hist[b], 1);
        ty = __float_as_int(w.ref[i].w);
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        if (t == ty) ts[t] += v;
        tn[t] += __popc(__ballot_sync(FULL, t == ty));
      }
      high += __popc(__ballot_sync(FULL, own && v >= 9.f));
    }
    float cl = clash_pairs(p, w.pose, d, p.inv_dc2_grid, lane);
    e = warp_sum(e);
    cl = p.clash_w * warp_sum(cl);
    const float t8 = warp_sum8(ts[0], ts[1], ts[2], ts[3], ts[4], ts[5], ts[6], ts[7], lane);  // type lane >> 2
    __syncwarp();
    for (int b = lane; b < 64; b += 32) row[b] = logs[hist[b]];
    if ((lane & 3) == 0) {
      int n = 0;
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (t == lane >> 2) n = tn[t];
      row[64 + (lane >> 2)] = n > 0 ? t8 / (float)n : 0.f;
    }
    if (lane == 0) {
      row[72] = (e + cl) / (float)d.n_atoms;
      row[73] = cl;
      row[74] = logs[d.n_atoms];
      row[75] = (float)d.n_rot;
      row[76] = logs[high];
      row[77] = row[78] = row[79] = 0.f;
    }
    __syncwarp();
    if (vec) {
      float4 *const f4 = reinterpret_cast<float4 *>(f);
      f4[lane] = lane < 20 ? reinterpret_cast<const float4 *>(row)[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
      f4[32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      for (int k = lane; k < 256; k += 32) f[k] = k < 80 ? row[k] : 0.f;
    }
    __syncwarp();
  }
}

cudaError_t launch_pose_features(const DockParams &p, int n_poses, const int32_t *lig_idx,
                                 const int32_t *start_id, const uint8_t *tors, const ligate_pose *poses,
                                 const int32_t *row_lig, float *out, cudaStream_t s) {
  if (n_poses <= 0) return cudaSuccess;
  const int warps = 4;
  const size_t smem = (size_t)warps * smem_bytes_per_warp(p.nmax, 0, 1, 0, FEAT_LIST);
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(pose_features_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, occ = 0;
  if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) ||
      (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, pose_features_kernel, 32 * warps, smem)))
    return e;
  const long long need = (n_poses + warps - 1) / warps;
  const int grid = (int)std::min<long long>(need, (long long)sms * std::max(occ, 1));
  pose_features_kernel<<<grid, 32 * warps, smem, s>>>(p, n_poses, lig_idx, start_id, tors,
                                                      reinterpret_cast<const PoseOut *>(poses), row_lig, out,
                                                      (reinterpret_cast<uintptr_t>(out) & 15) == 0);
  return cudaGetLastError();
}

// Size by which rescoring accepts a receptor: 16 B per atom, the pair table, the
// cell table and a warp's slot within a CTA's 227 KB, about 12,000 atoms.  The
// kernel stages none of the receptor; the limit is the entry points' own.
size_t rescore_smem_bytes(const DockParams &p, const RecParams &r, int warps) {
  const int ncells = r.ncx * r.ncy * r.ncz;
  return (size_t)r.n_rec * 16 + (size_t)((r.n_types * r.n_types + 1) & ~1) * 8 +
         (size_t)((ncells + 1 + 3) & ~3) * 4 + (size_t)warps * smem_bytes_per_warp(p.nmax, 0, 1, 0, 0);
}

cudaError_t launch_rescore(const DockParams &p, const RecParams &r, int n_poses, const int32_t *lig_idx,
                           const int32_t *start_id, const uint8_t *tors, const ligate_pose *poses,
                           const int32_t *row_lig, const StateSrc *states, ligate_rescored *out,
                           cudaStream_t s) {
  if (n_poses <= 0) return cudaSuccess;
  const int warps = 8;
  const size_t smem = (size_t)((r.n_types * r.n_types + 1) & ~1) * 8 + (size_t)warps * smem_bytes_per_warp(p.nmax, 0, 1, 0, 0);
  if (smem > 227 * 1024) return cudaErrorInvalidValue;  // never: 32 KB of pairs and 8 slots of at most 6 KB
  cudaError_t e = cudaFuncSetAttribute(rescore_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, occ = 0;
  if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) ||
      (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, rescore_kernel, 32 * warps, smem)))
    return e;
  const long long need = (n_poses + warps - 1) / warps;
  const int grid = (int)std::min<long long>(need, (long long)sms * std::max(occ, 1));
  StateSrc ss;
  memset(&ss, 0, sizeof(ss));
  if (states) ss = *states;
  rescore_kernel<<<grid, 32 * warps, smem, s>>>(p, r, n_poses, lig_idx, start_id, tors,
                                                reinterpret_cast<const PoseOut *>(poses), row_lig, ss, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Coordinates of continuous states as the refinement and the exact
// rescoring build them (build_state): one warp per state, Angstrom, atoms
// written back in the ligand's input order.
__global__ void __launch_bounds__(256) state_coords_kernel(const DockParams p, const uint8_t *__restrict__ order,
                                                           int n, const int32_t *__restrict__ lig_idx,
                                                           const ligate_pose_state *__restrict__ states,
                                                           float *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const WarpSmem w = warp_smem(smem_raw + (size_t)warp * smem_bytes_per_warp(p.nmax, 0, 1, 0), p.nmax, 1);
  const int pi = blockIdx.x * (blockDim.x >> 5) + warp;
  if (pi >= n) return;
  float *o = out + (size_t)pi * LIGATE_MAX_ATOMS * 3;
  const int li = lig_idx[pi];
  if (li < 0 || li >= p.n_ligands) {  // caller's device data
    for (int q = lane; q < LIGATE_MAX_ATOMS * 3; q += 32) o[q] = __int_as_float(0x7fc00000);
    return;
  }
  const LigDesc d = p.lig[li];
  load_coords(p, w, d, lane);
  const ligate_pose_state &st = states[pi];
  build_state(w.ref, w.pose, w.bonds, d, st.rot, st.trans, st.tors, lane);
  for (int i = lane; i < d.n_atoms; i += 32) {
    const float4 x = w.pose[i];
    float *a = o + 3 * (int)order[d.atom_base + i];
    a[0] = x.x; a[1] = x.y; a[2] = x.z;
  }
}

cudaError_t launch_state_coords(const DockParams &p, const uint8_t *order, int n, const int32_t *lig_idx,
                                const ligate_pose_state *states, float *out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int warps = 4;
  const size_t smem = (size_t)warps * smem_bytes_per_warp(p.nmax, 0, 1, 0);
  cudaError_t e = cudaFuncSetAttribute(state_coords_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       227 * 1024);
  if (e != cudaSuccess) return e;
  state_coords_kernel<<<(n + warps - 1) / warps, 32 * warps, smem, s>>>(p, order, n, lig_idx, states, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Per-ligand result after the filter (paper Sec. 2: docking, then rescoring
// and a filter; a ligand scores as its best surviving pose): one thread per
// row of K rescored poses, the lowest energy among those that pass (ties:
// the smaller slot), or -1 and +inf when none passes.
__global__ void best_passing_kernel(const ligate_rescored *__restrict__ rec, int n, int K,
                                    int32_t *__restrict__ idx, float *__restrict__ energy) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  int best = -1;
  float be = __int_as_float(0x7f800000);
  for (int k = 0; k < K; ++k) {
    const ligate_rescored q = rec[(size_t)r * K + k];
    if (q.pass == 1 && (best < 0 || q.energy < be)) { best = k; be = q.energy; }
  }
  idx[r] = best;
  if (energy) energy[r] = be;
}

// Learned pose selector's rule (paper Sec. 3.5: a pose selector that keeps
// one pose per ligand without rescoring them all): per row of K poses in
// docking order, the first live pose (start id >= 0) whose predicted label
// is below pass_below; else the live pose with the lowest prediction (ties:
// the smaller slot); -1 for a row without a live pose.
__global__ void select_poses_kernel(const float *__restrict__ pred, const PoseOut *__restrict__ poses, int n,
                                    int K, float pass_below, int32_t *__restrict__ idx) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  int first = -1, low = -1;
  float lp = 0.f;
  for (int k = 0; k < K; ++k) {
    if (poses[(size_t)r * K + k].start_id < 0) continue;
    const float v = pred[(size_t)r * K + k];
    if (first < 0 && v < pass_below) first = k;
    if (low < 0 || v < lp) { low = k; lp = v; }
  }
  idx[r] = first >= 0 ? first : low;
}

// Selector training label of a rescored pose: its energy clipped to
// fail_label when it passes the filter, fail_label when it fails (an empty
// slot too).
__global__ void selector_labels_kernel(const ligate_rescored *__restrict__ rec, long long n, float fail_label,
                                       float *__restrict__ out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const ligate_rescored q = rec[i];
  out[i] = q.pass == 1 ? fminf(q.energy, fail_label) : fail_label;
}

cudaError_t launch_best_passing(const ligate_rescored *rec, int n, int K, int32_t *idx, float *energy,
                                cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  best_passing_kernel<<<(n + 127) / 128, 128, 0, s>>>(rec, n, K, idx, energy);
  return cudaGetLastError();
}

cudaError_t launch_select_poses(const float *pred, const ligate_pose *poses, int n, int K, float pass_below,
                                int32_t *idx, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  select_poses_kernel<<<(n + 127) / 128, 128, 0, s>>>(pred, reinterpret_cast<const PoseOut *>(poses), n, K,
                                                      pass_below, idx);
  return cudaGetLastError();
}

cudaError_t launch_selector_labels(const ligate_rescored *rec, long long n, float fail_label, float *out,
                                   cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  selector_labels_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(rec, n, fail_label, out);
  return cudaGetLastError();
}

cudaError_t launch_fine_lists(const FineGrid &g, const float4 *rec, const int *cell, const int *first, int *steps,
                              uint16_t *list) {
  const int cells = g.nf[0] * g.nf[1] * g.nf[2];
  if (cells <= 0) return cudaSuccess;
  fine_lists_kernel<<<(cells + 7) / 8, 256>>>(g, rec, cell, first, steps, list);
  return cudaGetLastError();
}

}  // namespace ligate
