// Docking and explicit-pose kernels behind the C ABI: the clash tables of a
// run, the generic instances of the docking kernel (dock_kernel.cuh), scores
// and coordinates of explicit poses, start frames, and the launchers.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>
#include <string.h>

#include <algorithm>

#include "dock_kernel.cuh"

namespace ligate {

size_t dock_smem_per_warp(int nmax, int S, int G, int rmax) { return smem_bytes_per_warp(nmax, S, G, rmax); }

int dock_memo1_tables(const LigDesc &d, const BondRec *bonds, int) {
  int n = 0;
  for (int b = 2; b < d.n_rot; ++b) n += bonds[b].n_cand1 > 0;
  return n;
}

// The clash tables of every row's ligand, once per run: one warp per (row,
// table) or, when that leaves the chip idle (split), per (row, table, round of G
// steps): 301 ligands 68 -> 39 us.  What a row's work items share is built here once instead of by
// every item's warp, so items can be small (a batch that leaves few starts
// per warp) without paying for the tables again, and a ligand's tables are
// built in parallel.  The same device code builds the tables in the docking
// kernel when the rows' tables do not fit the plan's budget.
__global__ void __launch_bounds__(128) clash_tables_kernel(const __grid_constant__ DockParams p, const int32_t *__restrict__ row_lig,
                                                           int rows, int split) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const WarpSmem w = warp_smem(smem_raw + (size_t)warp * smem_bytes_per_warp(p.nmax, 0, p.G, 0), p.nmax, p.G);
  const int tables = 2 + p.m1max, S = p.S, L = p.L, G = p.G;
  const long long task = (long long)blockIdx.x * (blockDim.x >> 5) + warp, id = task / split;
  const int part = (int)(task % split), row = (int)(id / tables), t = (int)(id % tables);
  const int r0 = split > 1 ? part : 0, r1 = split > 1 ? part + 1 : (S + G - 1) / G;  // rounds of a table
  if (t == 0 && part > 0) return;
  if (row >= rows) return;
  const int li = row_lig[row];
  const LigDesc d = p.lig[li];
  if (d.n_rot == 0 || (t == 1 && (d.n_rot < 2 || memo_bonds(S) < 2))) return;
  int slot_bond = -1;
  if (t >= 2) {  // the bond whose single-separator table has slot t - 2
    bool mine = false;
    if (lane >= 2 && lane < d.n_rot) {
      const BondRec b = p.bonds[d.bond_base + lane];
      mine = b.n_cand1 > 0 && (b.e1 >> 16) == t - 2;
    }
    slot_bond = __ffs(__ballot_sync(FULL, mine)) - 1;
    if (slot_bond < 0) return;
  }
  load_coords(p, w, d, lane);
  const int g = lane / L, k = lane - g * L;
  float4 *pose = w.pose + (size_t)g * (p.nmax + 1);
  float ck = 1.f, sk = 0.f;
  if (k < S) step_cs(p, k, ck, sk);
  float R[9], T[3];
  start_frame(p, 0, R, T);
  float *memo = p.tab + (size_t)row * p.tab_stride, *m1 = memo + memo_floats(S, p.rmax);
  if (t == 0) input_rows(p, w, pose, d, R, T, ck, sk, g, k, L, G, S, memo);
  else if (t == 1) turn_table<false>(p, w, pose, d, w.bonds[0], w.bonds[1], R, T, ck, sk, g, k, L, G, S, memo + S, r0, r1);
  else single_table(p, w, pose, d, w.bonds[slot_bond], R, T, ck, sk, g, k, L, G, S, m1, r0, r1);
}

// ---------------------------------------------------------------------------
// Explicit poses: one warp per pose.
template <int MODE>
__global__ void __launch_bounds__(256) score_poses_kernel(const DockParams p, int n_poses,
                                                          const int32_t *__restrict__ lig_idx,
                                                          const int32_t *__restrict__ start_id,
                                                          const uint8_t *__restrict__ tors,
                                                          float *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const WarpSmem w = warp_smem(smem_raw + (size_t)warp * smem_bytes_per_warp(p.nmax, 0, 1, 0), p.nmax, 1);
  const int pi = blockIdx.x * (blockDim.x >> 5) + warp;
  if (pi >= n_poses) return;
  const int li = lig_idx[pi], sid = start_id[pi];
  if (li < 0 || li >= p.n_ligands || sid < 0 || sid >= p.n_starts) {  // caller's device data
    if (lane == 0) out[pi] = __int_as_float(0x7fc00000);
    return;
  }
  const LigDesc d = p.lig[li];
  load_coords(p, w, d, lane);
  uint32_t tt[4];
  for (int q = 0; q < 4; ++q) {
    const uint8_t *t = tors + (size_t)pi * LIGATE_MAX_ROT + 4 * q;
    tt[q] = (uint32_t)t[0] | ((uint32_t)t[1] << 8) | ((uint32_t)t[2] << 16) | ((uint32_t)t[3] << 24);
  }
  const float e = full_score<MODE>(p, p.maps, w, w.pose, d, sid, tt, lane);
  if (lane == 0) out[pi] = e;
}

// ---------------------------------------------------------------------------
// Explicit poses' coordinates as every kernel builds them: one warp per pose,
// grid units, atoms written back in the ligand's input order.
__global__ void __launch_bounds__(256) pose_coords_kernel(const DockParams p, const uint8_t *__restrict__ order,
                                                          int n_poses, const int32_t *__restrict__ lig_idx,
                                                          const int32_t *__restrict__ start_id,
                                                          const uint8_t *__restrict__ tors,
                                                          float *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const WarpSmem w = warp_smem(smem_raw + (size_t)warp * smem_bytes_per_warp(p.nmax, 0, 1, 0), p.nmax, 1);
  const int pi = blockIdx.x * (blockDim.x >> 5) + warp;
  if (pi >= n_poses) return;
  float *o = out + (size_t)pi * LIGATE_MAX_ATOMS * 3;
  const int li = lig_idx[pi], sid = start_id[pi];
  if (li < 0 || li >= p.n_ligands || sid < 0 || sid >= p.n_starts) {  // caller's device data
    for (int q = lane; q < LIGATE_MAX_ATOMS * 3; q += 32) o[q] = __int_as_float(0x7fc00000);
    return;
  }
  const LigDesc d = p.lig[li];
  load_coords(p, w, d, lane);
  uint32_t tt[4];
  for (int q = 0; q < 4; ++q) {
    const uint8_t *t = tors + (size_t)pi * LIGATE_MAX_ROT + 4 * q;
    tt[q] = (uint32_t)t[0] | ((uint32_t)t[1] << 8) | ((uint32_t)t[2] << 16) | ((uint32_t)t[3] << 24);
  }
  build_pose<MODE_F32_PLAIN>(p, w, w.pose, d, sid, tt, lane);
  for (int i = lane; i < d.n_atoms; i += 32) {
    const float4 x = w.pose[i];
    float *a = o + 3 * (int)order[d.atom_base + i];
    a[0] = x.x; a[1] = x.y; a[2] = x.z;
  }
}

cudaError_t launch_pose_coords(const DockParams &p, const uint8_t *order, int n_poses, const int32_t *lig_idx,
                               const int32_t *start_id, const uint8_t *tors, float *out, cudaStream_t s) {
  if (n_poses <= 0) return cudaSuccess;
  const int warps = 4;
  const size_t smem = (size_t)warps * smem_bytes_per_warp(p.nmax, 0, 1, 0);
  cudaError_t e = cudaFuncSetAttribute(pose_coords_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       227 * 1024);
  if (e != cudaSuccess) return e;
  pose_coords_kernel<<<(n_poses + warps - 1) / warps, 32 * warps, smem, s>>>(p, order, n_poses, lig_idx,
                                                                            start_id, tors, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Start frames: rotation of each orientation quaternion (normalised, rows
// re-orthonormalised by Gram-Schmidt in FP32) scaled by 1/h, and anchors in
// grid units.
__global__ void start_frames_kernel(const float4 *__restrict__ quat, int n_orient,
                                    const float *__restrict__ anchors, int n_anchor, float ox,
                                    float oy, float oz, float inv_h, float *__restrict__ rot,
                                    float *__restrict__ anc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_orient) quat_frame(quat[i], inv_h, rot + 9 * i);
  if (i < n_anchor) {
    anc[3 * i] = (anchors[3 * i] - ox) * inv_h;
    anc[3 * i + 1] = (anchors[3 * i + 1] - oy) * inv_h;
    anc[3 * i + 2] = (anchors[3 * i + 2] - oz) * inv_h;
  }
}

// ---------------------------------------------------------------------------
// Kernel instance of a mode, register cap and lanes per start: reg_cap 1 = at
// most 85 registers (6 CTAs of 128 threads per SM), 2 = at most 102 (5 CTAs),
// 3 = at most 128 (4 CTAs), 0 = the mode's default: 128 for the plain FP32
// layout (eight scalar gathers per interpolation want registers for loads in
// flight), 102 for the corner layouts (one vector gather; occupancy wins).
// 16 lanes per start (9 to 16 torsion steps) have instances of their own,
// with the group arithmetic folded (dock_l16.cu); the 85-register ones spill
// either way and stay generic.
static const void *dock_fn(int mode, int reg_cap, int L) {
  const int minb = reg_cap == 1 ? 6 : reg_cap == 2 ? 5 : reg_cap == 3 ? 4 : (mode == MODE_F32_PLAIN ? 4 : 5);
  if (L == 16 && minb < 6) return dock_fn_l16(mode, minb);
  switch (mode * 3 + (minb - 4)) {
    case 0: return (const void *)dock_kernel<MODE_F32_PLAIN, 4, 0>;
    case 1: return (const void *)dock_kernel<MODE_F32_PLAIN, 5, 0>;
    case 2: return (const void *)dock_kernel<MODE_F32_PLAIN, 6, 0>;
    case 3: return (const void *)dock_kernel<MODE_F32_CORNER, 4, 0>;
    case 4: return (const void *)dock_kernel<MODE_F32_CORNER, 5, 0>;
    case 5: return (const void *)dock_kernel<MODE_F32_CORNER, 6, 0>;
    case 6: return (const void *)dock_kernel<MODE_BF16_CORNER, 4, 0>;
    case 7: return (const void *)dock_kernel<MODE_BF16_CORNER, 5, 0>;
    case 8: return (const void *)dock_kernel<MODE_BF16_CORNER, 6, 0>;
    case 9: return (const void *)dock_kernel<MODE_F16_CORNER, 4, 0>;
    case 10: return (const void *)dock_kernel<MODE_F16_CORNER, 5, 0>;
    default: return (const void *)dock_kernel<MODE_F16_CORNER, 6, 0>;
  }
}

cudaError_t launch_dock(int mode, int reg_cap, const DockParams &p, int grid, int block, size_t smem,
                        cudaStream_t s) {
  void *args[] = {(void *)&p};
  return cudaLaunchKernel(dock_fn(mode, reg_cap, p.L), dim3(grid), dim3(block), args, smem, s);
}

cudaError_t launch_clash_tables(const DockParams &p, const int32_t *row_lig, int rows, cudaStream_t s) {
  if (rows <= 0 || !p.tab || p.rmax == 0) return cudaSuccess;
  // four warps per CTA, fewer where their slots exceed a CTA's shared memory
  // (G = 32 start groups, S = 1, with more than 64 atoms: 79 or 104 KB a warp)
  const size_t per_warp = smem_bytes_per_warp(p.nmax, 0, p.G, 0);
  const int warps = (int)std::min<size_t>(4, (size_t)(227 * 1024) / per_warp);
  const size_t smem = (size_t)warps * per_warp;
  cudaError_t e = cudaFuncSetAttribute(clash_tables_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return e;
  // rounds of a table side by side while that makes few warps per SM
  const int rounds = (p.S + p.G - 1) / p.G;
  long long n = (long long)rows * (2 + p.m1max);
  const int split = n * rounds <= 65536 ? rounds : 1;
  n *= split;
  clash_tables_kernel<<<(unsigned)((n + warps - 1) / warps), 32 * warps, smem, s>>>(p, row_lig, rows, split);
  return cudaGetLastError();
}

size_t dock_tab_stride(int S, int rmax, int m1max) { return (size_t)memo_floats(S, rmax) + ((size_t)m1max * S * S + 3) / 4 * 4; }

size_t dock_kernel_local_bytes(int mode, int reg_cap, int L) {
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, dock_fn(mode, reg_cap, L)) != cudaSuccess) return 0;
  return a.localSizeBytes;
}

int dock_kernel_max_ctas_per_sm(int mode, int reg_cap, int L, int block, size_t smem) {
  int n = 0;
  const void *f = dock_fn(mode, reg_cap, L);
  if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
    return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, block, smem) != cudaSuccess) return 0;
  return n;
}

cudaError_t launch_start_frames(const double *, const float *quat_f32_dev, int n_orient,
                                const float *anchors_dev, int n_anchor, const double origin[3],
                                double h, float *rot_out, float *anc_out, cudaStream_t s) {
  const int n = n_orient > n_anchor ? n_orient : n_anchor;
  start_frames_kernel<<<(n + 127) / 128, 128, 0, s>>>(
      reinterpret_cast<const float4 *>(quat_f32_dev), n_orient, anchors_dev, n_anchor,
      (float)origin[0], (float)origin[1], (float)origin[2], (float)(1.0 / h), rot_out, anc_out);
  return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_score_t(const DockParams &p, int n_poses, const int32_t *lig_idx,
                                  const int32_t *start_id, const uint8_t *tors, float *out,
                                  cudaStream_t s) {
  const int warps = 4;
  const size_t smem = (size_t)warps * smem_bytes_per_warp(p.nmax, 0, 1, 0);
  cudaError_t e = cudaFuncSetAttribute(score_poses_kernel<MODE>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return e;
  score_poses_kernel<MODE><<<(n_poses + warps - 1) / warps, 32 * warps, smem, s>>>(
      p, n_poses, lig_idx, start_id, tors, out);
  return cudaGetLastError();
}

cudaError_t launch_score_poses(int mode, const DockParams &p, int n_poses, const int32_t *lig_idx,
                               const int32_t *start_id, const uint8_t *tors, float *out,
                               cudaStream_t s) {
  if (n_poses <= 0) return cudaSuccess;
  switch (mode) {
    case MODE_F32_PLAIN: return launch_score_t<MODE_F32_PLAIN>(p, n_poses, lig_idx, start_id, tors, out, s);
    case MODE_F32_CORNER: return launch_score_t<MODE_F32_CORNER>(p, n_poses, lig_idx, start_id, tors, out, s);
    case MODE_BF16_CORNER: return launch_score_t<MODE_BF16_CORNER>(p, n_poses, lig_idx, start_id, tors, out, s);
    default: return launch_score_t<MODE_F16_CORNER>(p, n_poses, lig_idx, start_id, tors, out, s);
  }
}

}  // namespace ligate
