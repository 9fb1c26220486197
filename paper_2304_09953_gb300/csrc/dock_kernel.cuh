// Persistent docking kernel for sm_103a: rigid starts (orientation x anchor),
// greedy torsion sweep, trilinear grid score + intramolecular clash term,
// warp-shuffle top-K per ligand, last-arriver merge and optional FP32
// rescoring.  Paper Sec. 2 (multi-restart docking with a geometric score;
// ligand score = best pose; optional re-scoring of the generated poses) and
// Sec. 3.3 (one batch of ligand-pocket pairs per device launch).
//
// Work mapping.  A warp takes work items (ligand, range of starts) from a
// global queue.  Inside the warp, lanes form G = 32 / L groups of L lanes
// (L = S rounded up to a power of two); each group runs one start, and lane
// k of a group evaluates torsion step k of the current bond.  Every lane of
// the warp therefore executes the same bond, the same moved atom and the same
// clash partner at the same time: no divergence, and each pose coordinate is
// a shared-memory broadcast.  Only the moved side of the current bond is
// re-scored (the rest of the score is the same for every k); the k = 0 lane
// re-evaluates the current pose, so E += V(k*) - V(0).
//
// Branch and bound: a start whose lower bound on its final energy exceeds
// the K-th best energy already found stops sweeping (bound_setup,
// beyond_bound); the top-K is unchanged.  The two groups of a warp run in
// lockstep, so a work item visits each orientation's anchors in the plan's
// nearest-neighbour pair order (DockParams::visit): partners sweep nearby
// poses and tend to stop together, and then the warp leaves the bond loop.
#pragma once

#include "dock_device.cuh"

namespace ligate {

// Clash part of the sweep of bond br at this lane's torsion step (ck, sk):
// the sum over the bond's crossing candidate pairs of max(0, 1 - d^2/d_c^2)^2
// on the group's conformation `pose` (grid units; axis n through pv).
// Moved atom i travels on a circle about the axis; with
// u = radial vector of i, m = n x u, w = radial vector of fixed atom
// j, P = u.w, Q = m.w and D0 = |x_i - x_j|^2 at the current pose,
//   d^2(theta) = D0 + 2P (1 - cos theta) - 2Q sin theta,
// whose minimum over the circle is D0 + 2P - 2 sqrt(P^2 + Q^2).  A
// pair whose minimum is beyond d_c contributes exactly zero at every
// step and is dropped; the others are evaluated in closed form.
// Warp-collective: every lane calls it, each with its own group's data; a
// group that is not `alive` (its start was pruned) loads and tests nothing.
__device__ __forceinline__ float clash_sweep(const DockParams &p, const WarpSmem &w, const float4 *pose,
                                             const LigDesc &d, const BondRec &br, float nx, float ny,
                                             float nz, const float4 &pv, float ck, float sk, int g,
                                             int k, int L, int G, unsigned &n_pair,
                                             bool alive = true) {
  if (br.n_cand == 0) return 0.f;  // warp-uniform: every pair was memoised
  float ac = 0.f;
  const int cap = PAIR_WARP / G;  // nearly 6 L
  float4 *list = w.list + g * cap;
  float2 *cab = w.cab + g * p.nmax;  // (axial a, radial distance b) of each atom
  const unsigned lmask = L == 32 ? FULL : ((1u << L) - 1u);
  const unsigned below = (1u << k) - 1u;
  const float omc = 1.f - ck;
  int cnt = 0;
  for (int j = alive ? k : d.n_atoms; j < d.n_atoms; j += L) {
    const float4 xj = pose[j];
    const float fx = xj.x - pv.x, fy = xj.y - pv.y, fz = xj.z - pv.z;
    const float a = fmaf(fx, nx, fmaf(fy, ny, fz * nz));
    const float wx = fmaf(-a, nx, fx), wy = fmaf(-a, ny, fy), wz = fmaf(-a, nz, fz);
    // radial distance by the hardware square-root approximation (relative
    // error ~1e-7): it only feeds the survivor test, whose threshold carries
    // a 1e-4 margin, and the pair coefficients' squared radii
    float rb;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(rb) : "f"(fmaf(wx, wx, fmaf(wy, wy, wz * wz))));
    cab[j] = make_float2(a, rb);
  }
  __syncwarp();
  auto flush = [&]() {
    const int top = __reduce_max_sync(FULL, (unsigned)cnt);
    if (top == 0) return;
    __syncwarp();
    // the group's lanes turn buffered pair indices into closed-form
    // coefficients, one pair per lane
    for (int q = k; q < cnt; q += L) {
      const unsigned pr = __float_as_uint(list[q].w);
      const int i = pr & 0xffu, j = pr >> 8;
      const float2 hi = cab[i], hj = cab[j];
      const float4 xi = pose[i], xj = pose[j];
      // radial vectors about the axis: w = (x - p) - a n
      const float4 ui = make_float4(fmaf(-hi.x, nx, xi.x - pv.x), fmaf(-hi.x, ny, xi.y - pv.y),
                                    fmaf(-hi.x, nz, xi.z - pv.z), 0.f);
      const float4 wj = make_float4(fmaf(-hj.x, nx, xj.x - pv.x), fmaf(-hj.x, ny, xj.y - pv.y),
                                    fmaf(-hj.x, nz, xj.z - pv.z), 0.f);
      const float da = hi.x - hj.x;
      const float P = fmaf(ui.x, wj.x, fmaf(ui.y, wj.y, ui.z * wj.z));
      const float cx = ui.y * wj.z - ui.z * wj.y, cy = ui.z * wj.x - ui.x * wj.z,
                  cz = ui.x * wj.y - ui.y * wj.x;
      const float Q = fmaf(nx, cx, fmaf(ny, cy, nz * cz));  // (n x u).w
      const float D0 = fmaf(da, da, fmaf(hi.y, hi.y, fmaf(hj.y, hj.y, -2.f * P)));
      list[q] = make_float4(fmaf(-D0, p.inv_dc2_grid, 1.f), -2.f * P * p.inv_dc2_grid,
                            2.f * Q * p.inv_dc2_grid, 0.f);
    }
    __syncwarp();
    for (int q = 0; q < top; ++q) {
      if (q < cnt) {
        const float4 e = list[q];
        const float t = fmaxf(0.f, fmaf(e.z, sk, fmaf(e.y, omc, e.x)));
        ac = fmaf(t, t, ac);
      }
    }
    n_pair += cnt;
    cnt = 0;
    __syncwarp();
  };
  // candidates of this bond, L per pass (the first set loaded by the caller);
  // with u = radial vector of the moved atom, the minimum distance over its
  // circle is sqrt(da^2 + (b_j - b_i)^2)
  const uint16_t *cand = p.cand + d.cand_base + br.cand_off;
  // PASSES independent passes of L candidates per iteration: their
  // loads and tests overlap, then the survivors are appended in order
  constexpr int PASSES = 4;
  for (int c0 = 0; c0 < br.n_cand; c0 += PASSES * L) {
    if (c0 > 0 && __any_sync(FULL, cnt > cap - PASSES * L)) flush();
    unsigned pr[PASSES];
    bool surv[PASSES];
#pragma unroll
    for (int u = 0; u < PASSES; ++u) {
      const int c = c0 + u * L + k;
      pr[u] = alive && c < br.n_cand ? __ldg(cand + c) : 0u;
    }
#pragma unroll
    for (int u = 0; u < PASSES; ++u) {
      const float2 hi = cab[pr[u] & 0xffu], hj = cab[pr[u] >> 8];
      const float da = hi.x - hj.x, db = hj.y - hi.y;
      surv[u] = alive && (c0 + u * L + k < br.n_cand) && fmaf(da, da, db * db) < p.dc2_grid_margin;
    }
#pragma unroll
    for (int u = 0; u < PASSES; ++u) {
      const unsigned gm = (__ballot_sync(FULL, surv[u]) >> (g * L)) & lmask;
      if (surv[u]) list[cnt + __popc(gm & below)].w = __uint_as_float(pr[u]);
      cnt += __popc(gm);
    }
  }
  flush();
  return ac;
}

// The input conformation posed by start 0's frame (R, T), where every clash
// table is built (the clash term is invariant under the rigid move).
__device__ __forceinline__ void pose_input(const WarpSmem &w, float4 *pose, const LigDesc &d, const float (&R)[9],
                                           const float (&T)[3], int k, int L) {
  for (int i = k; i < d.n_atoms; i += L) {
    const float4 a = w.ref[i];
    pose[i] = make_float4(fmaf(R[0], a.x, fmaf(R[1], a.y, fmaf(R[2], a.z, T[0]))),
                          fmaf(R[3], a.x, fmaf(R[4], a.y, fmaf(R[5], a.z, T[1]))),
                          fmaf(R[6], a.x, fmaf(R[7], a.y, fmaf(R[8], a.z, T[2]))), 0.f);
  }
  __syncwarp();
}

// Clash sums of the swept candidates of bond bb at every step k after bond be
// alone turned by each step t, out[t S + k], rounds r0 to r1: group g takes t =
// r G + g in round r.
// LAST: stored with an L2 evict-last policy (ahead of streaming data).
// Warp-collective.
template <bool LAST>
__device__ void turn_table(const DockParams &p, const WarpSmem &w, float4 *pose, const LigDesc &d, const BondRec &be,
                           const BondRec &bb, const float (&R)[9], const float (&T)[3], float ck, float sk, int g,
                           int k, int L, int G, int S, float *out, int r0, int r1) {
  unsigned n_pair = 0;  // not counted: once per ligand
  for (int r = r0; r < r1; ++r) {
    const int te = min(r * G + g, S - 1);  // groups past S repeat the last step
    pose_input(w, pose, d, R, T, k, L);
    float ex, ey, ez;
    const float4 ev = pose[be.v];
    bond_axis(pose[be.u], ev, ex, ey, ez);
    float ce, se;
    step_cs(p, te, ce, se);
    Rot re;
    re.make(ce, se, ex, ey, ez, ev.x, ev.y, ev.z);
    __syncwarp();
    for (int i = be.v + 1 + k; i < be.end; i += L) {
      float4 q = pose[i];
      re.apply(q.x, q.y, q.z, q.x, q.y, q.z);
      pose[i] = q;
    }
    __syncwarp();
    float mx, my, mz;
    const float4 qv = pose[bb.v];
    bond_axis(pose[bb.u], qv, mx, my, mz);
    const float a1 = clash_sweep(p, w, pose, d, bb, mx, my, mz, qv, ck, sk, g, k, L, G, n_pair);
    if (r * G + g < S && k < S) {
      if (LAST) {
        uint64_t pol;
        asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
        asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(out + te * S + k), "f"(a1), "l"(pol) : "memory");
      } else {
        out[te * S + k] = a1;
      }
    }
    __syncwarp();
  }
}

// The pairs of bond b >= 2 that bond e1 alone separates, by e1's step.
static __device__ void single_table(const DockParams &p, const WarpSmem &w, float4 *pose, const LigDesc &d, BondRec bb,
                             const float (&R)[9], const float (&T)[3], float ck, float sk, int g, int k, int L, int G,
                             int S, float *m1, int r0, int r1) {
  bb.cand_off += bb.n_cand0;
  bb.n_cand = bb.n_cand1;
  turn_table<true>(p, w, pose, d, w.bonds[bb.e1 & 0xffff], bb, R, T, ck, sk, g, k, L, G, S,
                   m1 + (bb.e1 >> 16) * S * S, r0, r1);
}

// memo[k]: the sums of bond 0's sweep; memo[memo_row0(S) + (b - memo_bonds(S))
// S + k]: of each later bond b, the sums over its first n_cand0 candidates;
// all on the input conformation.
static __device__ void input_rows(const DockParams &p, const WarpSmem &w, float4 *pose, const LigDesc &d, const float (&R)[9],
                           const float (&T)[3], float ck, float sk, int g, int k, int L, int G, int S, float *memo) {
  unsigned n_pair = 0;
  pose_input(w, pose, d, R, T, k, L);
  for (int b = 0; b < d.n_rot; b = b == 0 ? memo_bonds(S) : b + 1) {
    BondRec bb = w.bonds[b];
    if (b > 0) {
      if (bb.n_cand0 == 0) continue;  // warp-uniform
      bb.n_cand = bb.n_cand0;
    }
    float mx, my, mz;
    const float4 qv = pose[bb.v];
    bond_axis(pose[bb.u], qv, mx, my, mz);
    const float a0 = clash_sweep(p, w, pose, d, bb, mx, my, mz, qv, ck, sk, g, k, L, G, n_pair);
    if (g == 0 && k < S) memo[(b == 0 ? 0 : memo_row0(S) + (b - memo_bonds(S)) * S) + k] = a0;
    __syncwarp();
  }
}

// All clash tables of the loaded ligand by one warp: input_rows and bond 1's
// sums after bond 0's step (memo[S + k0 S + k]) into w.memo, the single-
// separator tables into m1 (if given).  For runs without clash_tables_kernel.
// Out of line (once per ligand of a warp): its candidate sweeps would make
// up most of the kernel's inlined code.
static __device__ __noinline__ void build_memo(const DockParams &p, unsigned char *slot, int li, float *m1) {
  const WarpSmem w = warp_smem(slot, p.nmax, p.G);
  const LigDesc d = p.lig[li];
  const int L = p.L, G = p.G, S = p.S, lane = threadIdx.x & 31, g = lane / L, k = lane - g * L;
  float4 *pose = w.pose + (size_t)g * (p.nmax + 1);
  float ck = 1.f, sk = 0.f;
  if (k < S) step_cs(p, k, ck, sk);
  float R[9], T[3];
  start_frame(p, 0, R, T);
  if (m1)
    for (int b = 2; b < d.n_rot; ++b) {
      const BondRec bb = w.bonds[b];
      if (bb.n_cand1 > 0) single_table(p, w, pose, d, bb, R, T, ck, sk, g, k, L, G, S, m1, 0, (S + G - 1) / G);
    }
  input_rows(p, w, pose, d, R, T, ck, sk, g, k, L, G, S, w.memo);
  if (d.n_rot >= 2 && memo_bonds(S) == 2)
    turn_table<false>(p, w, pose, d, w.bonds[0], w.bonds[1], R, T, ck, sk, g, k, L, G, S, w.memo + S, 0,
                      (S + G - 1) / G);
}

// Drops the L2 copies of the whole 128-byte lines inside [lo, hi) without
// writing them back to DRAM: for scratch whose contents are dead (a
// ligand's merged partial lists, a warp's clash tables at exit).  Lines that
// reach outside the range may hold another owner's live data and are left
// alone.  Warp-collective over `lane`; the caller has finished its reads.
// A discard acts as a write of undefined data, so the fence and the warp
// barrier order it before any lane's next write to the same lines.
__device__ __forceinline__ void l2_discard(const void *lo, const void *hi, int lane) {
  const uintptr_t a = ((uintptr_t)lo + 127u) & ~(uintptr_t)127u, b = (uintptr_t)hi & ~(uintptr_t)127u;
  for (uintptr_t q = a + (uintptr_t)lane * 128u; q < b; q += 32u * 128u)
    asm volatile("discard.global.L2 [%0], 128;" ::"l"(q) : "memory");
  __threadfence();
  __syncwarp();
}

// Lower bound of a start's final energy (branch and bound on the sweep).
// A bond turns the DFS range (v, end); atom i is moved by no bond after the
// last one whose range holds it.  Before bond b the atoms with lastb <= b are
// fixed for good, the others can still reach any cell, and the clash term is
// never negative, so the final energy is at least
//   A_b + lbc[b],  A_b = grid energy of the fixed atoms at the current pose,
//   lbc[b] = sum over the atoms a bond >= b moves of their type's map minimum.
// Also per bond: which of its moved atoms it moves for the last time.
// Warp-collective.
static __device__ void bound_setup(const DockParams &p, const WarpSmem &w, const LigDesc &d, int lane) {
  const int W = p.nmax >> 5;
  uint8_t *const lastb = reinterpret_cast<uint8_t *>(w.cab);  // scratch: 1 + the last bond that moves each atom (0: none)
  for (int i0 = 0; i0 < d.n_atoms; i0 += 32) {
    const int i = i0 + lane;
    int last = 0;
    for (int b = 0; b < d.n_rot; ++b) {
      const BondRec &br = w.bonds[b];
      if (i > br.v && i < br.end) last = b + 1;
    }
    if (i < d.n_atoms) lastb[i] = (uint8_t)last;
    const unsigned fx = __ballot_sync(FULL, last == 0);
    if (lane == 0) w.fixm[i0 >> 5] = fx;
  }
  __syncwarp();
  for (int s = 0; s <= d.n_rot; ++s) {
    float a = 0.f;
    for (int i = lane; i < d.n_atoms; i += 32)
      if (lastb[i] > s) a += p.gmin[__float_as_int(w.ref[i].w)];
    a = warp_sum(a);
    if (lane == 0) w.lbc[s] = a;
  }
  for (int b = 0; b < d.n_rot; ++b) {
    const BondRec &br = w.bonds[b];
    for (int i0 = br.v + 1, q = 0; i0 < br.end; i0 += 32, ++q) {
      const int i = i0 + lane;
      const unsigned m = __ballot_sync(FULL, i < br.end && lastb[i < br.end ? i : 0] == b + 1);
      if (lane == 0) w.lastm[b * W + q] = m;
    }
  }
  __syncwarp();
}

// Order-preserving 32-bit key of a float (smaller value, smaller key) and
// its inverse; the argmin of the sweep uses the same map.
__device__ __forceinline__ unsigned value_key(float v) {
  const unsigned b = __float_as_uint(v);
  return b ^ ((unsigned)((int)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ float key_value(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k ^ 0x80000000u) : ~k);
}

// True when a start whose final energy is at least `lb` cannot enter a top-K
// whose K-th best energy is `thr`.  The margin covers the FP32 rounding of
// the running energy and of the bound (sums of at most 128 terms of
// magnitude at most the cap, over at most 16 bonds), so the test holds for
// the kernel's own arithmetic; an empty top-K (thr = inf) prunes nothing.
__device__ __forceinline__ bool beyond_bound(float lb, float thr) {
  return lb > thr + 1.f + (fabsf(thr) + fabsf(lb)) * (1.f / 1024.f);
}

// ---------------------------------------------------------------------------
// CTAs of at most 128 threads; MINB of them must fit on one SM: 4 caps the
// registers at 128 (16 resident warps), 5 at 102 (20 warps), 6 at 85 (24
// warps).  Bytes of frame, spill stores and spill loads: BF16 with 16 lanes per
// start 16/0/0 at 128 registers and 80/52/92 at 96 (the call of build_memo holds
// registers across it), generic 128/164/296 at 80.
// Latency of the map gathers is covered by resident warps, so occupancy
// matters more than per-thread registers here.
template <int MODE, int MINB, int LT>
__global__ void __launch_bounds__(128, MINB) dock_kernel(const __grid_constant__ DockParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char *const slot = smem_raw + (size_t)warp * smem_bytes_per_warp(p.nmax, p.S, p.G, p.rmax);
  const WarpSmem w = warp_smem(slot, p.nmax, p.G);
  const int L = LT ? LT : p.L, G = LT ? 32 / LT : p.G, S = p.S, K = p.K;
  const int g = lane / L, k = lane - g * L;
  const int glead = g * L;
  float4 *pose = w.pose + (size_t)g * (p.nmax + 1);
  uint8_t *const steps = w.steps + LIGATE_MAX_ROT * g;
  float ck = 1.f, sk = 0.f;
  if (k < S) step_cs(p, k, ck, sk);
  const int ts = type_stride(MODE, p.g);
  const unsigned bias = cell_bias<MODE>(p.g);
  const GridConst &gc = p.g;
  const float INF = __int_as_float(0x7f800000);
  // single-separator tables: the row's (p.tab), or this warp's own scratch
  float *const m1w = p.memo1 ? p.memo1 + ((size_t)blockIdx.x * (blockDim.x >> 5) + warp) * p.m1max * S * S
                             : nullptr;
  const float *m1 = m1w;

  const int n_items = p.n_items_dev ? __ldcg(p.n_items_dev) : p.n_items;
  int cur = -1, n_memo = 0;
  LigDesc d;
  float clash_ref = 0.f;

  for (;;) {
    int it = 0;
    if (lane == 0) it = atomicAdd(p.queue, 1);
    it = __shfl_sync(FULL, it, 0);
    if (it >= n_items) {
      if (m1w) {  // this warp's clash tables are dead: no write-back
        __syncwarp();
        l2_discard(m1w, m1w + (size_t)p.m1max * S * S, lane);
      }
      break;
    }
    const Item item = p.items[it];
    if (item.ligand != cur) {
      __syncwarp();
      if (m1w && cur >= 0) l2_discard(m1w, m1w + (size_t)p.m1max * S * S, lane);  // the last ligand's tables
      clash_ref = load_ligand(p, w, item.ligand, d, lane);
      cur = item.ligand;
      n_memo = min(d.n_rot, memo_bonds(S));
      if (p.tab) {  // clash_tables_kernel's rows
        const float4 *src = reinterpret_cast<const float4 *>(p.tab + (size_t)item.row * p.tab_stride);
        const int nf = n_memo > 0 ? memo_floats(S, d.n_rot) / 4 : 0;
        for (int q = lane; q < nf; q += 32) reinterpret_cast<float4 *>(w.memo)[q] = __ldg(src + q);
        m1 = p.tab + (size_t)item.row * p.tab_stride + memo_floats(S, p.rmax);
      } else if (n_memo > 0) {
        build_memo(p, slot, item.ligand, m1w);
      }
      bound_setup(p, w, d, lane);
    }
    TopSlots top;
    top.clear(lane);
    float thr = INF;  // K-th best energy of the item so far: a start bounded above it stops
    float thr_pub = INF;  // the last value this warp shared with the row's other items
    unsigned *const row_thr = p.lig_thr ? p.lig_thr + item.row : nullptr;
    const float cut = p.cut ? __ldcg(p.cut) : INF;  // screening cutoff (the same for every ligand)
    // work counters: surviving pairs of this lane's group, and how many starts
    // swept how many bonds (w.swept), which gives all others at the item's end
    unsigned n_pair = 0;
    if (lane < LIGATE_MAX_ROT + 2) w.swept[lane] = 0;
    __syncwarp();

    for (int s0 = item.s0; s0 < item.s1; s0 += G) {
      // visit index (a group past the end repeats the last one) -> start id:
      // each orientation's anchors in the plan's visiting order
      const int vi = min(s0 + g, item.s1 - 1);
      const int sid = p.visit ? vi - vi % p.n_anchor + p.visit[vi % p.n_anchor] : vi;
      // the row's shared K-th best (any item's is at least the row's final
      // one, so it bounds as safely as this item's own), loaded now and used
      // after the rigid stage's gathers
      unsigned shared_key = 0;
      if (row_thr && lane == 0) shared_key = __ldcg(row_thr);
      // -- rigid start: pose = R_o (x - c) / h + (a - origin) / h
      float R[9], T[3];
      start_frame(p, sid, R, T);
      float e = 0.f, ef = 0.f;  // ef: the atoms no bond moves
      for (int i = k; i < d.n_atoms; i += L) {
        const float4 r = w.ref[i];
        float4 u;
        u.x = fmaf(R[0], r.x, fmaf(R[1], r.y, fmaf(R[2], r.z, T[0])));
        u.y = fmaf(R[3], r.x, fmaf(R[4], r.y, fmaf(R[5], r.z, T[1])));
        u.z = fmaf(R[6], r.x, fmaf(R[7], r.y, fmaf(R[8], r.z, T[2])));
        const unsigned off = __float_as_uint(r.w) * (unsigned)ts + bias;
        u.w = __uint_as_float(off);
        pose[i] = u;
        const float gi = sweep_eval<MODE>(p.maps, off, u.x, u.y, u.z, gc);
        e += gi;
        if (w.fixm[i >> 5] >> (i & 31) & 1u) ef += gi;
      }
      for (int o = L >> 1; o > 0; o >>= 1) {
        e += __shfl_xor_sync(FULL, e, o);
        ef += __shfl_xor_sync(FULL, ef, o);
      }
      float E = fmaf(p.clash_w, clash_ref, e);
      float A = ef;  // grid energy of the atoms fixed for good (the bound's first part)
      shared_key = __shfl_sync(FULL, shared_key, 0);
      const float thr_use = fminf(fminf(thr, cut), shared_key ? key_value(~shared_key) : INF);
      // a group past the item's end, or a start bounded above the K-th best, sweeps nothing
      bool alive = s0 + g < item.s1 && !beyond_bound(A + w.lbc[0], thr_use);
      int nb = alive ? LIGATE_MAX_ROT + 1 : 0;  // bonds swept before the bound stopped the start
      if (k == 0) *reinterpret_cast<uint4 *>(steps) = make_uint4(0, 0, 0, 0);
      __syncwarp();

      // -- greedy torsion sweep
      for (int b = 0; b < d.n_rot; ++b) {
        if (!__any_sync(FULL, alive)) break;  // every start of the warp is pruned
        const BondRec br = w.bonds[b];
        const float4 pv = pose[br.v];
        float nx, ny, nz;
        bond_axis(pose[br.u], pv, nx, ny, nz);
        Rot rot;
        rot.make(ck, sk, nx, ny, nz, pv.x, pv.y, pv.z);
        // from bond n_memo on: the pairs whose geometry earlier steps change
        // are swept live after the grid part, and the pairs bond e1 alone
        // separates come from their table by e1's chosen step, loaded here so
        // that the grid part hides its way from L2 (the candidates too would
        // cost two registers over the grid part: 2.7% slower)
        BondRec live = br;
        float c1 = 0.f;
        if (b >= n_memo) {
          const bool has1 = m1 && b >= 2 && br.n_cand1 > 0;  // warp-uniform
          if (alive && has1 && k < S) {
            const int te = steps[br.e1 & 0xffff];
            uint64_t pol;  // the tables stay in L2 ahead of streaming data (evict-last policy)
            asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
            asm volatile("ld.global.cg.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(c1)
                         : "l"(m1 + ((br.e1 >> 16) * S + te) * S + k), "l"(pol));
          }
          const int skip = br.n_cand0 + (has1 ? br.n_cand1 : 0);
          live.cand_off += skip;
          live.n_cand -= skip;
        }
        // grid part: every moved atom at this lane's torsion step, two atoms
        // per iteration: two map gathers in flight per lane, and the rotation
        // and interpolation arithmetic of the pair in packed FP32 (FFMA2);
        // agf: the atoms this bond moves for the last time (fixed after it).
        float ag = 0.f, ag2 = 0.f, agf = 0.f;
        const int bb = b + 1, iend = alive ? br.end : 0;  // a pruned group evaluates nothing
        {
          const uint32_t *lm = w.lastm + b * (p.nmax >> 5);
          int i = br.v + 1;
          uint32_t m = 0;
          for (int q0 = 0; i < iend; q0 += 32) {
            m = lm[q0 >> 5];
            const int e = min(iend, br.v + 1 + q0 + 32);
            for (; i + 1 < e; i += 2) {
              const float4 q = pose[i], q2 = pose[i + 1];
              float2 v;
              if (MODE == MODE_F32_PLAIN) {  // eight scalar gathers each: registers go to loads in flight
                float yx, yy, yz, zx, zy, zz;
                rot.apply(q.x, q.y, q.z, yx, yy, yz);
                rot.apply(q2.x, q2.y, q2.z, zx, zy, zz);
                v.x = sweep_eval<MODE>(p.maps, __float_as_uint(q.w), yx, yy, yz, gc);
                v.y = sweep_eval<MODE>(p.maps, __float_as_uint(q2.w), zx, zy, zz, gc);
              } else {
                float2 ox, oy, oz;
                rot.apply(q.x, q.y, q.z, ox.x, oy.x, oz.x);
                rot.apply(q2.x, q2.y, q2.z, ox.y, oy.y, oz.y);
                v = sweep_eval2<MODE>(p.maps, __float_as_uint(q.w), __float_as_uint(q2.w), ox, oy, oz, gc);
              }
              ag += v.x;
              ag2 += v.y;
              if (m & 1u) agf += v.x;
              if (m & 2u) agf += v.y;
              m >>= 2;
            }
            if (i < e) {  // the last atom of an odd range
              const float4 q = pose[i];
              float yx, yy, yz;
              rot.apply(q.x, q.y, q.z, yx, yy, yz);
              const float ga = sweep_eval<MODE>(p.maps, __float_as_uint(q.w), yx, yy, yz, gc);
              ag += ga;
              if (m & 1u) agf += ga;
              ++i;
            }
          }
        }
        ag += ag2;
        float ac;
        if (b < n_memo) {  // looked up: bond 0, or bond 1 after bond 0's step
          ac = k < S ? w.memo[b == 0 ? k : S + (int)steps[0] * S + k] : 0.f;
        } else {  // pairs whose geometry earlier steps change, swept live, + the memoised rest
          ac = clash_sweep(p, w, pose, d, live, nx, ny, nz, pv, ck, sk, g, k, L, G, n_pair, alive);
          if (br.n_cand0 > 0 && k < S) ac += w.memo[memo_row0(S) + (b - memo_bonds(S)) * S + k];
          ac += c1;
        }
        const float V = (k < S) ? fmaf(p.clash_w, ac, ag) + 0.f : INF;  // + 0: -0 becomes +0
        // argmin over the group's lanes (ties: smaller k) by one min-reduction
        // of an order-preserving integer key and one ballot
        const unsigned vb = __float_as_uint(V);
        const unsigned key = vb ^ ((unsigned)((int)vb >> 31) | 0x80000000u);
        const unsigned gmask = L == 32 ? FULL : (((1u << L) - 1u) << glead);
        const unsigned kmin = __reduce_min_sync(gmask, key);
        const int bk1 = __ffs(__ballot_sync(FULL, key == kmin) & gmask) - 1 - glead;
        const int bk = alive ? bk1 : 0;  // a pruned group keeps its pose
        const float best = __uint_as_float((kmin & 0x80000000u) ? (kmin ^ 0x80000000u) : ~kmin);
        const float V0 = __shfl_sync(FULL, V, glead);
        const float cb = __shfl_sync(FULL, ck, glead + bk);
        const float sb = __shfl_sync(FULL, sk, glead + bk);
        E += best - V0;
        // the atoms fixed from now on at the chosen step join the bound's
        // first part; the rest may still reach their map minimum
        A += __shfl_sync(FULL, agf, glead + bk);
        if (alive && bb < d.n_rot && beyond_bound(A + w.lbc[bb], thr_use)) { alive = false; nb = bb; }
        if (k == 0) steps[b] = (uint8_t)bk;
        __syncwarp();
        if (__any_sync(FULL, bk != 0)) {  // a group whose step is 0 applies the identity exactly
          Rot rb;
          rb.make(cb, sb, nx, ny, nz, pv.x, pv.y, pv.z);
          for (int i = br.v + 1 + k; i < br.end; i += L) {
            float4 q = pose[i];
            rb.apply(q.x, q.y, q.z, q.x, q.y, q.z);
            pose[i] = q;
          }
        }
        __syncwarp();
      }

      if (k == 0 && s0 + g < item.s1) atomicAdd(w.swept + nb, 1u);

      // -- candidates of this start group into the warp's top-K (a pruned
      // start's energy exceeds the K-th best: it could not enter)
      for (int gg = 0; gg < G; ++gg) {
        const int src = gg * L;
        const float ce = __shfl_sync(FULL, E, src);
        const bool live = __shfl_sync(FULL, alive, src);
        const int cs = __shfl_sync(FULL, sid, src);
        if (!live) continue;
        const int at = top.insert(ce, cs, K, lane);
        if (at >= 0 && lane == 0) {
          const uint4 t = reinterpret_cast<const uint4 *>(w.steps)[gg];
          uint2 *const o = reinterpret_cast<uint2 *>(p.partial[(size_t)item.slot * K + at].tors);
          o[0] = make_uint2(t.x, t.y);
          o[1] = make_uint2(t.z, t.w);
        }
      }
      thr = __shfl_sync(FULL, top.e, K - 1);
      if (row_thr && thr < thr_pub) {  // share an improved K-th best with the row's other items
        if (lane == 0) atomicMax(row_thr, ~value_key(thr));
        thr_pub = thr;
      }
    }

    if (p.stats) {
      // lane b holds the starts that swept bond b (all those not pruned before
      // it); the work of a bond's sweep is the same for each of them
      __syncwarp();
      unsigned long long at = 0, ct = 0, tt = 0, sw = 0;
      const unsigned mine = lane < LIGATE_MAX_ROT + 2 ? w.swept[lane] : 0u;
      unsigned starts = mine, pruned = lane <= LIGATE_MAX_ROT ? mine : 0u;
      for (int o = 16; o > 0; o >>= 1) {
        starts += __shfl_xor_sync(FULL, starts, o);
        pruned += __shfl_xor_sync(FULL, pruned, o);
      }
      unsigned upto = mine;  // starts pruned after at most `lane` bonds
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(FULL, upto, o);
        if (lane >= o) upto += t;
      }
      if (lane < d.n_rot) {
        const BondRec br = w.bonds[lane];
        const unsigned long long c = starts - upto;
        at = c * (unsigned)(br.end - br.v - 1) * (unsigned)S;
        ct = c * (unsigned)br.n_cand;
        sw = c;
        if (lane >= n_memo) tt = c * (unsigned)(br.n_cand - br.n_cand0 - (m1 && lane >= 2 ? br.n_cand1 : 0));
      }
      unsigned long long q = k == 0 ? n_pair : 0;
      for (int o = 16; o > 0; o >>= 1) {
        at += __shfl_xor_sync(FULL, at, o);
        tt += __shfl_xor_sync(FULL, tt, o);
        q += __shfl_xor_sync(FULL, q, o);
        ct += __shfl_xor_sync(FULL, ct, o);
        sw += __shfl_xor_sync(FULL, sw, o);
      }
      if (lane == 0) {
        atomicAdd(p.stats + 0, at + (unsigned long long)starts * d.n_atoms);
        atomicAdd(p.stats + 1, tt);
        atomicAdd(p.stats + 2, q);
        atomicAdd(p.stats + 3, ct);
        atomicAdd(p.stats + 4, (unsigned long long)pruned);
        atomicAdd(p.stats + 5, sw);
      }
    }

    // -- publish this item's list (each entry's steps move from their slot to
    // the entry's rank); the last item of the ligand merges
    __syncwarp();
    PoseOut *const mine = p.partial + (size_t)item.slot * K;
    uint2 ta = make_uint2(0, 0), tb = make_uint2(0, 0);
    if (lane < K && top.s != EMPTY_SID) {
      const uint2 *o = reinterpret_cast<const uint2 *>(mine[top.at].tors);
      ta = __ldcg(o);
      tb = __ldcg(o + 1);
    }
    __syncwarp();
    if (lane < K) {
      PoseOut o;
      o.score = top.e; o.start_id = top.s;
      o.tors[0] = ta.x; o.tors[1] = ta.y; o.tors[2] = tb.x; o.tors[3] = tb.y;
      mine[lane] = o;
    }
    __threadfence();
    __syncwarp();
    int prev = 0;
    if (lane == 0) prev = atomicAdd(p.done + item.row, 1);
    prev = __shfl_sync(FULL, prev, 0);
    if (prev != p.lig_items[item.row] - 1) continue;
    __threadfence();

    // merge: 8 lists' energies and starts in flight; a list ascends, so past
    // its first loser nothing of it enters; an entry's slot is its place in
    // the row's lists, where its steps are read at the end
    TopSlots all;
    all.clear(0);
    const int slot0 = p.lig_slot0[item.row], nit = p.lig_items[item.row];
    const PoseOut *const lists = p.partial + (size_t)slot0 * K;
    constexpr int AHEAD = 8;
    for (int c0 = 0; c0 < nit; c0 += AHEAD) {
      float pe[AHEAD];
      int ps[AHEAD];
#pragma unroll
      for (int u = 0; u < AHEAD; ++u) {
        const bool in = lane < K && c0 + u < nit;
        const float2 es = in ? __ldcg(reinterpret_cast<const float2 *>(lists + (size_t)(c0 + u) * K + lane))
                             : make_float2(INF, __int_as_float(EMPTY_SID));
        pe[u] = es.x;
        ps[u] = __float_as_int(es.y);
      }
#pragma unroll
      for (int u = 0; u < AHEAD; ++u)
        for (int j = 0; j < K; ++j) {
          const float ce = __shfl_sync(FULL, pe[u], j);
          const int cs = __shfl_sync(FULL, ps[u], j);
          if (cs == EMPTY_SID || all.insert(ce, cs, K, lane) < 0) break;
          if (all.e == ce && all.s == cs) all.at = (c0 + u) * K + j;  // the one lane that took it
        }
    }
    uint32_t tt[4] = {0u, 0u, 0u, 0u};  // this entry's steps
    if (lane < K && all.s != EMPTY_SID) {
      const uint2 *o = reinterpret_cast<const uint2 *>(lists[all.at].tors);
      const uint2 x = __ldcg(o), y = __ldcg(o + 1);
      tt[0] = x.x; tt[1] = x.y; tt[2] = y.x; tt[3] = y.y;
    }
    __syncwarp();  // the ligand's partial lists are merged and dead: no write-back
    l2_discard(p.partial + (size_t)slot0 * K, p.partial + (size_t)(slot0 + nit) * K, lane);
    int rank = lane;
    if (p.rescore) {
      for (int j = 0; j < K; ++j) {
        const int cs = __shfl_sync(FULL, all.s, j);
        if (cs == EMPTY_SID) break;
        uint32_t tj[4];
        for (int q = 0; q < 4; ++q) tj[q] = __shfl_sync(FULL, tt[q], j);
        const float en = full_score<MODE_F32_PLAIN>(p, p.maps_f32, w, w.pose, d, cs, tj, lane);
        if (lane == j) all.e = en;
      }
      rank = 0;  // equal keys (empty slots) keep their lane order
      for (int j = 0; j < K; ++j) {
        const float oe = __shfl_sync(FULL, all.e, j);
        const int os = __shfl_sync(FULL, all.s, j);
        if (pose_less(oe, os, all.e, all.s) || (j < lane && !pose_less(all.e, all.s, oe, os))) ++rank;
      }
    }
    if (lane < K) {
      PoseOut o;
      o.score = all.e;
      o.start_id = all.s == EMPTY_SID ? -1 : all.s;
      for (int q = 0; q < 4; ++q) o.tors[q] = tt[q];
      p.out[(size_t)item.row * K + rank] = o;
    }
  }
}

}  // namespace ligate
