// Pose refinement by gradient descent (paper Sec. 2: the docking search is
// a gradient descent from multiple restarts; the greedy sweep's best poses
// are the restarts and a local descent refines each of them).
//
// State q = (R, t, phi): x_i = R (y_i - c) + t, y the input conformation
// after torsion angle phi_b is applied to each rotatable bond in sweep order
// about its current axis u -> v (c the input centroid; t in Angstrom).  The
// energy is the docking score on the FP32 maps.  Its generalised gradient is
//   F = sum_i g_i,  tau = sum_i (x_i - t) x g_i,
//   psi_b = n_b . sum_{i moved by b} (x_i - x_v) x g_i,
// the derivatives along a translation, a rotation about t and a turn of
// bond b, with g_i = dE/dx_i (trilinear derivative in the atom's cell / h,
// zero for penalty atoms; clash -4 w t (x_i - x_j) / d_c^2 per pair with
// t = 1 - d^2/d_c^2 > 0).  Descent: the trial t - eta F / N,
// GS(exp([-eta tau / I_R]x) R), phi - eta psi / I_b (I_R, I_b the moments
// 1 + sum |r|^2 about t and about each bond axis) is accepted when it lowers
// E (eta *= 1.25), else rejected (eta *= 0.5), for a fixed iteration count.
//
// One warp per pose: lanes over atoms for the coordinate build, the
// per-atom gradient (each lane sums the pair forces on its own atoms, so no
// atomics) and the moment sums; warp reductions give the warp-uniform
// energy and gradient.
//
// What bounds it: instruction issue (73% of active cycles), 33 evaluations of
// about 2,500 warp instructions per pose.  So work that the whole warp did alike or one lane did
// alone is spread over the lanes: sines and cosines of the torsions and the
// trial's torsion steps by a lane per bond, the pairs that touch found by one
// ballot per atom (the forces then visit those only), eight sums in one
// butterfly, and the bonds' torque sums laid out several to a pass
// (bond_segments).  Two state slots take turns instead of copies.  Every sum
// keeps its terms and its tree, so the descent, which is chaotic in its last
// bits, takes the same steps.  16,000 poses of the batched library, 32
// iterations: 2,279 -> 1,585 us.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "dock_device.cuh"

namespace ligate {
namespace {

constexpr unsigned FULLM = 0xffffffffu;
constexpr int NG = 6 + LIGATE_MAX_ROT;  // gradient components
constexpr int NI = 1 + LIGATE_MAX_ROT;  // moments
// Squared clash cutoff (A^2), by atoms per lane, from which enough pairs of a
// ligand touch that finding them costs more than it saves (us with the search
// and without, 16 iterations: 4,800 poses of the batched library at cutoffs of 3,
// 4 and 8 A 342/358, 376/362, 481/362; 2,400 poses of 80 atoms at 4, 4.5 and 8 A
// 482/502, 516/504, 632/506; of 120 atoms at 4, 5 and 8 A 768/870, 895/874,
// 1085/876).
constexpr float NEAR2_ALL[4] = {16.f, 16.f, 20.f, 25.f};
constexpr uint32_t SEG_IDLE = 1u << 31;  // bond segment entry of a lane without a bond

struct State {
  float R[9], t[3], phi[LIGATE_MAX_ROT];
};
static_assert(sizeof(State) == sizeof(ligate_pose_state), "state layout");
static_assert(sizeof(ligate_refined) == sizeof(State) + 16, "refined layout");

// Per-warp shared memory.
struct RSmem {
  float4 *ref;  // [nmax] input coordinates - centroid (A), .w = atom type (int bits)
  float4 *x;    // [nmax] coordinates of the state being evaluated
  float4 *g;    // [nmax] dE/dx
  BondRec *bonds;
  State *q;     // [2]: current, trial
  float *G;     // [2][NG]
  float *I;     // [2][NI]
  uint32_t *seg;  // [32 LIGATE_MAX_ROT] bond segments (bond_segments)
  uint16_t *uv;   // [LIGATE_MAX_ROT] u | v << 8 of each bond
  int passes;
};

// Rounded up to 16 bytes: every warp's float4 arrays must stay 16-byte aligned.
__host__ __device__ inline size_t refine_smem_per_warp(int nmax) {
  const size_t b = (size_t)nmax * 48 + sizeof(BondRec) * LIGATE_MAX_ROT + 2 * sizeof(State) +
                   2 * NG * sizeof(float) + 2 * NI * sizeof(float) +
                   32 * LIGATE_MAX_ROT * sizeof(uint32_t) + LIGATE_MAX_ROT * sizeof(uint16_t);
  return (b + 15) / 16 * 16;
}

__device__ __forceinline__ RSmem rsmem(unsigned char *base, int nmax) {
  RSmem w;
  w.ref = reinterpret_cast<float4 *>(base);
  w.x = w.ref + nmax;
  w.g = w.x + nmax;
  w.bonds = reinterpret_cast<BondRec *>(w.g + nmax);
  w.q = reinterpret_cast<State *>(w.bonds + LIGATE_MAX_ROT);
  w.G = reinterpret_cast<float *>(w.q + 2);
  w.I = w.G + 2 * NG;
  w.seg = reinterpret_cast<uint32_t *>(w.I + 2 * NI);
  w.uv = reinterpret_cast<uint16_t *>(w.seg + 32 * LIGATE_MAX_ROT);
  w.passes = 0;
  return w;
}

__device__ __forceinline__ float wsum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULLM, v, o);
  return v;
}

__device__ __forceinline__ void unit_axis(const float4 &a, const float4 &b, float &nx, float &ny,
                                          float &nz) {
  nx = b.x - a.x; ny = b.y - a.y; nz = b.z - a.z;
  const float inv = rsqrtf(nx * nx + ny * ny + nz * nz);
  nx *= inv; ny *= inv; nz *= inv;
}

// Trilinear value of an atom type's FP32 map at grid coordinates u (from the
// corner copy when the pocket has one) and its derivative with respect to u (zero outside [0, n-1], where the value is
// the penalty).
__device__ __forceinline__ float map_value_grad(const float *__restrict__ maps, const float4 *__restrict__ corner,
                                                int type, float ux, float uy, float uz, const GridConst &g, float &dx,
                                                float &dy, float &dz) {
  dx = dy = dz = 0.f;
  if (!((min3_nan(ux, uy, uz) >= 0.f) & (ux <= g.fx1) & (uy <= g.fy1) & (uz <= g.fz1))) return g.penalty;
  const float tx = fminf(__fadd_rd(ux, CELL_M), g.cx), ty = fminf(__fadd_rd(uy, CELL_M), g.cy),
              tz = fminf(__fadd_rd(uz, CELL_M), g.cz);
  const int ix = __float_as_int(tx) - (int)CELL_MB, iy = __float_as_int(ty) - (int)CELL_MB,
            iz = __float_as_int(tz) - (int)CELL_MB;
  const float fx = ux - (tx - CELL_M), fy = uy - (ty - CELL_M), fz = uz - (tz - CELL_M);
  float v0, v1, v2, v3, v4, v5, v6, v7;
  if (corner) {  // the same values, one 32-byte cell
    const float4 *m = corner + 2 * (size_t)(((type * (g.nz - 1) + iz) * (g.ny - 1) + iy) * (g.nx - 1) + ix);
    const float4 a = __ldg(m), b = __ldg(m + 1);
    v0 = a.x; v1 = a.y; v2 = a.z; v3 = a.w; v4 = b.x; v5 = b.y; v6 = b.z; v7 = b.w;
  } else {
    const float *m = maps + ((type * g.nz + iz) * g.ny + iy) * g.nx + ix;
    const int sy = g.nx, sz = g.nx * g.ny;
    v0 = __ldg(m); v1 = __ldg(m + 1); v2 = __ldg(m + sy); v3 = __ldg(m + sy + 1);
    v4 = __ldg(m + sz); v5 = __ldg(m + sz + 1); v6 = __ldg(m + sz + sy); v7 = __ldg(m + sz + sy + 1);
  }
  const float d0 = v1 - v0, d1 = v3 - v2, d2 = v5 - v4, d3 = v7 - v6;
  const float y0z0 = fmaf(fx, d0, v0), y1z0 = fmaf(fx, d1, v2);
  const float y0z1 = fmaf(fx, d2, v4), y1z1 = fmaf(fx, d3, v6);
  const float z0 = fmaf(fy, y1z0 - y0z0, y0z0), z1 = fmaf(fy, y1z1 - y0z1, y0z1);
  const float e0 = fmaf(fy, d1 - d0, d0), e1 = fmaf(fy, d3 - d2, d2);
  dx = fmaf(fz, e1 - e0, e0);
  const float c0 = y1z0 - y0z0, c1 = y1z1 - y0z1;
  dy = fmaf(fz, c1 - c0, c0);
  dz = z1 - z0;
  return fmaf(fz, z1 - z0, z0);
}

struct RefineArgs {
  DockParams p;
  float ox, oy, oz, h, inv_h;
  int n;
  const int32_t *lig_idx;      // state/eval modes: ligand of each pose
  const State *init;           // state/eval modes
  const PoseOut *poses;        // plan mode: [rows][K]
  const int32_t *row_lig;      // plan mode: ligand of each row
  int iters;
  float eta0;
  ligate_refined *out;         // refine modes
  float *energy, *grad;        // eval mode
};

// Energy and generalised gradient of state w.q[s] into w.G[s], w.I[s].  HW:
// atoms per lane (n_atoms <= 32 HW).  FIND: the pairs that may touch are found
// first (clash cutoffs below NEAR2_ALL's), else every pair is visited; pairs that
// do not touch add nothing, so the values are the same.
template <int HW, bool FIND>
__device__ float eval_state(const RefineArgs &a, const RSmem &w, const LigDesc &d, int s, int lane) {
  const DockParams &p = a.p;
  const State &q = w.q[s];
  build_state(w.ref, w.x, w.bonds, d, q.R, q.t, q.phi, lane);
  const float fcl = -4.f * p.clash_w * p.inv_dc2_ang;
  // which pairs may touch (distance below d_c, with a margin), a ballot per
  // atom over the lanes' own atoms: the pair forces then visit only those, in
  // the same order
  const float near2 = 1.0001f / p.inv_dc2_ang;
  uint32_t hit[HW][HW];  // [own atom lane + 32 h][word of partners]
#pragma unroll
  for (int h = 0; h < HW; ++h)
#pragma unroll
    for (int wd = 0; wd < HW; ++wd) hit[h][wd] = FIND || wd >= d.n_words ? 0u : ~0u;
  if (FIND) {
    float4 own[HW];
#pragma unroll
    for (int h = 0; h < HW; ++h)
      own[h] = lane + 32 * h < d.n_atoms ? w.x[lane + 32 * h] : make_float4(__int_as_float(0x7f800000), 0.f, 0.f, 0.f);  // touches nothing
#pragma unroll
    for (int h = 0; h < HW; ++h) {
      const int i1 = min(d.n_atoms, 32 * h + 32);
      for (int i = 32 * h; i < i1; ++i) {
        const float4 xi = w.x[i];
        const bool mine = lane == i - 32 * h;
#pragma unroll
        for (int wd = 0; wd + 1 < HW; wd += 2) {  // two of the lane's atoms in packed FP32
          const float2 rx = sub2(make_float2(xi.x, xi.x), make_float2(own[wd].x, own[wd + 1].x)),
                       ry = sub2(make_float2(xi.y, xi.y), make_float2(own[wd].y, own[wd + 1].y)),
                       rz = sub2(make_float2(xi.z, xi.z), make_float2(own[wd].z, own[wd + 1].z));
          const float2 d2 = __ffma2_rn(rx, rx, __ffma2_rn(ry, ry, __fmul2_rn(rz, rz)));
          const unsigned m0 = __ballot_sync(FULLM, d2.x < near2), m1 = __ballot_sync(FULLM, d2.y < near2);
          if (mine) { hit[h][wd] = m0; hit[h][wd + 1] = m1; }
        }
        if (HW & 1) {
          const float rx = xi.x - own[HW - 1].x, ry = xi.y - own[HW - 1].y, rz = xi.z - own[HW - 1].z;
          const unsigned m = __ballot_sync(FULLM, fmaf(rx, rx, fmaf(ry, ry, rz * rz)) < near2);
          if (mine) hit[h][HW - 1] = m;
        }
      }
    }
  }
  float e = 0.f, cl = 0.f, F0 = 0.f, F1 = 0.f, F2 = 0.f, T0 = 0.f, T1 = 0.f, T2 = 0.f, IR = 0.f;
#pragma unroll
  for (int h = 0; h < HW; ++h) {
    const int i = lane + 32 * h;
    if (i >= d.n_atoms) break;
    const float4 xi = w.x[i];
    float dx, dy, dz;
    e += map_value_grad(p.maps_f32, p.maps_f32c, __float_as_int(xi.w), (xi.x - a.ox) * a.inv_h,
                        (xi.y - a.oy) * a.inv_h, (xi.z - a.oz) * a.inv_h, p.g, dx, dy, dz);
    float gx = dx * a.inv_h, gy = dy * a.inv_h, gz = dz * a.inv_h;
#pragma unroll
    for (int wd = 0; wd < HW; ++wd) {
      uint32_t m = hit[h][wd];
      if (m) m &= __ldg(p.elig + d.elig_base + i * d.n_words + wd);
      while (m) {
        const int j = 32 * wd + __ffs(m) - 1;
        m &= m - 1;
        const float4 xj = w.x[j];
        const float rx = xi.x - xj.x, ry = xi.y - xj.y, rz = xi.z - xj.z;
        const float tt = fmaf(-fmaf(rx, rx, fmaf(ry, ry, rz * rz)), p.inv_dc2_ang, 1.f);
        if (tt > 0.f) {
          if (j > i) cl = fmaf(tt, tt, cl);
          const float f = fcl * tt;
          gx = fmaf(f, rx, gx); gy = fmaf(f, ry, gy); gz = fmaf(f, rz, gz);
        }
      }
    }
    w.g[i] = make_float4(gx, gy, gz, 0.f);
    const float rx = xi.x - q.t[0], ry = xi.y - q.t[1], rz = xi.z - q.t[2];
    F0 += gx; F1 += gy; F2 += gz;
    T0 += ry * gz - rz * gy; T1 += rz * gx - rx * gz; T2 += rx * gy - ry * gx;
    IR += rx * rx + ry * ry + rz * rz;
  }
  const float s8 = warp_sum8(fmaf(p.clash_w, cl, e), F0, F1, F2, T0, T1, T2, IR, lane);  // value lane >> 2 of the eight
  const float E = __shfl_sync(FULLM, s8, 0);
  float *G = w.G + s * NG, *I = w.I + s * NI;
  __syncwarp();
  for (int q = 0; q < w.passes; ++q) {
    const uint32_t sg = w.seg[32 * q + lane];  // bond | first atom << 8 | atom past the range << 16 | log2 width << 24
    const int b = sg & 0xff, end = sg >> 16 & 0xff, width = 1 << (sg >> 24 & 7);
    const int u = w.uv[b] & 0xff, v = w.uv[b] >> 8;
    const float4 pu = w.x[u], pv = w.x[v];
    float nx, ny, nz;
    unit_axis(pu, pv, nx, ny, nz);
    float ps = 0.f, ib = 0.f;
    for (int i = sg >> 8 & 0xff; i < end; i += 32) {
      const float4 xi = w.x[i], gi = w.g[i];
      const float rx = xi.x - pv.x, ry = xi.y - pv.y, rz = xi.z - pv.z;
      ps += nx * (ry * gi.z - rz * gi.y) + ny * (rz * gi.x - rx * gi.z) + nz * (rx * gi.y - ry * gi.x);
      const float ra = rx * nx + ry * ny + rz * nz;
      ib += rx * rx + ry * ry + rz * rz - ra * ra;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float p2 = __shfl_xor_sync(FULLM, ps, o), i2 = __shfl_xor_sync(FULLM, ib, o);
      if (o < width) { ps += p2; ib += i2; }
    }
    if ((lane & (width - 1)) == 0 && !(sg & SEG_IDLE)) { G[6 + b] = ps; I[1 + b] = 1.f + ib; }
  }
  if ((lane & 3) == 0 && lane > 0) {
    if (lane < 28) G[(lane >> 2) - 1] = s8;
    else I[0] = 1.f + s8;
  }
  if (lane >= d.n_rot && lane < LIGATE_MAX_ROT) { G[6 + lane] = 0.f; I[1 + lane] = 1.f; }
  __syncwarp();
  return E;
}

// Lays the bonds' moved atoms out over the lanes, several bonds to a pass: a
// bond of m moved atoms takes an aligned segment of the least power of two of
// lanes (at most 32) that holds them, its atoms in order from the segment's
// first lane (a lane of a bond with more than 32 also takes the atoms 32
// further).  Widest segments first, so the segments pack without holes.  The
// sums over a segment are then wsum's: the lanes outside it hold zeros there.
__device__ int bond_segments(const RSmem &w, const LigDesc &d, int lane) {
  for (int q = lane; q < 32 * LIGATE_MAX_ROT; q += 32) w.seg[q] = SEG_IDLE;  // bond 0, no atoms, width 1
  int v = 0, m = 0, lw = 0;
  if (lane < d.n_rot) {
    const BondRec &br = w.bonds[lane];
    v = br.v;
    m = br.end - br.v - 1;
    while (lw < 5 && (1 << lw) < m) ++lw;
    w.uv[lane] = (uint16_t)(br.u | br.v << 8);
  }
  __syncwarp();
  int pos = 0;
  for (int k = 5; k >= 0; --k)
    for (unsigned set = __ballot_sync(FULLM, lane < d.n_rot && lw == k); set; set &= set - 1) {
      const int b = __ffs(set) - 1;
      const int bv = __shfl_sync(FULLM, v, b), bm = __shfl_sync(FULLM, m, b);
      if (lane < (1 << k))
        w.seg[pos + lane] = (uint32_t)b | (uint32_t)(bv + 1 + lane) << 8 | (uint32_t)(bv + 1 + bm) << 16 | (uint32_t)k << 24;
      pos += 1 << k;
    }
  __syncwarp();
  return (pos + 31) / 32;
}

// Trial state from w.q[c] with gradient w.G + c NG and moments w.I + c NI into
// w.q[1 - c]: the rotation by every lane alike, the translation and the
// torsions by a lane per component.
__device__ void make_trial(const RSmem &w, int c, int n_atoms, int n_rot, float eta, int lane) {
  const State &q = w.q[c];
  State &t = w.q[1 - c];
  const float *G = w.G + c * NG, *I = w.I + c * NI;
  const float sN = eta / (float)n_atoms, sR = -eta / I[0];
  if (lane < 3) t.t[lane] = q.t[lane] - sN * G[lane];
  const float wx = sR * G[3], wy = sR * G[4], wz = sR * G[5];
  const float th = sqrtf(wx * wx + wy * wy + wz * wz);
  float M[9] = {1.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f, 1.f};
  if (th > 0.f) {
    const float nx = wx / th, ny = wy / th, nz = wz / th;
    float sn, c;
    sincosf(th, &sn, &c);
    const float o = 1.f - c;
    M[0] = c + o * nx * nx;      M[1] = o * nx * ny - sn * nz; M[2] = o * nx * nz + sn * ny;
    M[3] = o * ny * nx + sn * nz; M[4] = c + o * ny * ny;      M[5] = o * ny * nz - sn * nx;
    M[6] = o * nz * nx - sn * ny; M[7] = o * nz * ny + sn * nx; M[8] = c + o * nz * nz;
  }
  float R[9];
  for (int r = 0; r < 3; ++r)
    for (int cc = 0; cc < 3; ++cc)
      R[3 * r + cc] = M[3 * r] * q.R[cc] + M[3 * r + 1] * q.R[3 + cc] + M[3 * r + 2] * q.R[6 + cc];
  // Gram-Schmidt on the rows, r2 = r0 x r1
  const float l0 = rsqrtf(R[0] * R[0] + R[1] * R[1] + R[2] * R[2]);
  R[0] *= l0; R[1] *= l0; R[2] *= l0;
  const float dp = R[0] * R[3] + R[1] * R[4] + R[2] * R[5];
  R[3] -= dp * R[0]; R[4] -= dp * R[1]; R[5] -= dp * R[2];
  const float l1 = rsqrtf(R[3] * R[3] + R[4] * R[4] + R[5] * R[5]);
  R[3] *= l1; R[4] *= l1; R[5] *= l1;
  R[6] = R[1] * R[5] - R[2] * R[4];
  R[7] = R[2] * R[3] - R[0] * R[5];
  R[8] = R[0] * R[4] - R[1] * R[3];
  if (lane == 0)
    for (int k = 0; k < 9; ++k) t.R[k] = R[k];
  if (lane < LIGATE_MAX_ROT) t.phi[lane] = lane < n_rot ? q.phi[lane] - eta * G[6 + lane] / I[1 + lane] : 0.f;
}

// MODE 0: energy + gradient of explicit states; 1: refine explicit states;
// 2: refine the plan's top-K poses.
template <int MODE, int HW, bool FIND>
__global__ void __launch_bounds__(128) refine_kernel(const __grid_constant__ RefineArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const DockParams &p = a.p;
  RSmem w = rsmem(smem_raw + (size_t)warp * refine_smem_per_warp(p.nmax), p.nmax);
  const int pi = blockIdx.x * (blockDim.x >> 5) + warp;
  if (pi >= a.n) return;
  int li;
  if (MODE == 2) {
    const PoseOut po = a.poses[pi];
    li = a.row_lig[pi / p.K];
    if (po.start_id < 0) {  // empty slot: nothing to refine
      if (lane == 0) {
        ligate_refined r;
        memset(&r, 0, sizeof(r));
        r.score_in = r.score = po.score;
        r.ligand = li;
        a.out[pi] = r;
      }
      return;
    }
    if (lane == 0) {  // state of docked pose (start, tors) in Angstrom
      State &q = w.q[0];
      const int o = po.start_id / p.n_anchor, an = po.start_id - o * p.n_anchor;
      for (int k = 0; k < 9; ++k) q.R[k] = p.rot[9 * o + k] * a.h;
      q.t[0] = fmaf(p.anc[3 * an], a.h, a.ox);
      q.t[1] = fmaf(p.anc[3 * an + 1], a.h, a.oy);
      q.t[2] = fmaf(p.anc[3 * an + 2], a.h, a.oz);
      const float step = 6.283185307179586f / (float)p.S;
      for (int b = 0; b < LIGATE_MAX_ROT; ++b) {
        const int kb = (po.tors[b >> 2] >> (8 * (b & 3))) & 0xff;
        q.phi[b] = (float)(kb % p.S) * step;
      }
    }
  } else {
    li = a.lig_idx[pi];
    if (li < 0 || li >= p.n_ligands) {  // caller's device data
      if (lane == 0) {
        if (MODE == 0) a.energy[pi] = __int_as_float(0x7fc00000);
        else { ligate_refined r; memset(&r, 0, sizeof(r)); r.score_in = r.score = __int_as_float(0x7fc00000); r.ligand = li; a.out[pi] = r; }
      }
      return;
    }
    if (lane == 0) w.q[0] = a.init[pi];
  }
  const LigDesc d = p.lig[li];
  // input coordinates about their centroid
  float sx = 0.f, sy = 0.f, sz = 0.f;
  for (int i = lane; i < d.n_atoms; i += 32) {
    const float4 v = __ldg(p.atoms + d.atom_base + i);
    w.ref[i] = v;
    sx += v.x; sy += v.y; sz += v.z;
  }
  sx = wsum(sx); sy = wsum(sy); sz = wsum(sz);
  const float inv_n = 1.f / (float)d.n_atoms;
  const float cx = sx * inv_n, cy = sy * inv_n, cz = sz * inv_n;
  __syncwarp();
  for (int i = lane; i < d.n_atoms; i += 32) {
    float4 v = w.ref[i];
    v.x -= cx; v.y -= cy; v.z -= cz;
    w.ref[i] = v;
  }
  for (int b = lane; b < d.n_rot; b += 32) w.bonds[b] = p.bonds[d.bond_base + b];
  __syncwarp();
  w.passes = bond_segments(w, d, lane);

  float E = eval_state<HW, FIND>(a, w, d, 0, lane);
  if (MODE == 0) {
    if (lane == 0) a.energy[pi] = E;
    for (int k = lane; k < NG; k += 32) a.grad[(size_t)pi * NG + k] = w.G[k];
    return;
  }
  const float e_in = E;
  float eta = a.eta0;
  uint32_t mask = 0;
  int cur = 0;  // the slot of the accepted state
  for (int it = 0; it < a.iters; ++it) {
    make_trial(w, cur, d.n_atoms, d.n_rot, eta, lane);
    __syncwarp();
    const float Et = eval_state<HW, FIND>(a, w, d, 1 - cur, lane);
    if (Et < E) {
      cur = 1 - cur;
      E = Et;
      eta *= 1.25f;
      mask |= 1u << it;
    } else {
      eta *= 0.5f;
    }
    __syncwarp();
  }
  if (lane == 0) {
    ligate_refined r;
    memcpy(&r.state, &w.q[cur], sizeof(State));
    r.score_in = e_in;
    r.score = E;
    r.accepted = mask;
    r.ligand = li;
    a.out[pi] = r;
  }
}

}  // namespace

size_t refine_smem_bytes(int nmax) { return refine_smem_per_warp(nmax); }

namespace {
template <bool FIND>
const void *refine_fn(int mode, int hw) {
  const void *const fns[3][4] = {
      {(const void *)refine_kernel<0, 1, FIND>, (const void *)refine_kernel<0, 2, FIND>,
       (const void *)refine_kernel<0, 3, FIND>, (const void *)refine_kernel<0, 4, FIND>},
      {(const void *)refine_kernel<1, 1, FIND>, (const void *)refine_kernel<1, 2, FIND>,
       (const void *)refine_kernel<1, 3, FIND>, (const void *)refine_kernel<1, 4, FIND>},
      {(const void *)refine_kernel<2, 1, FIND>, (const void *)refine_kernel<2, 2, FIND>,
       (const void *)refine_kernel<2, 3, FIND>, (const void *)refine_kernel<2, 4, FIND>}};
  return fns[mode][hw - 1];
}
}  // namespace

cudaError_t launch_refine(int mode, const DockParams &p, const double origin[3], double h, int n,
                          const int32_t *lig_idx, const ligate_pose_state *init, const ligate_pose *poses,
                          const int32_t *row_lig, int iters, float eta0, ligate_refined *out,
                          float *energy, float *grad, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  RefineArgs a;
  memset(&a, 0, sizeof(a));
  a.p = p;
  a.ox = (float)origin[0]; a.oy = (float)origin[1]; a.oz = (float)origin[2];
  a.h = (float)h; a.inv_h = (float)(1.0 / h);
  a.n = n;
  a.lig_idx = lig_idx;
  a.init = reinterpret_cast<const State *>(init);
  a.poses = reinterpret_cast<const PoseOut *>(poses);
  a.row_lig = row_lig;
  a.iters = iters;
  a.eta0 = eta0;
  a.out = out;
  a.energy = energy;
  a.grad = grad;
  const int warps = 4;
  const size_t smem = refine_smem_per_warp(p.nmax) * warps;
  const int hw = p.nmax > 32 ? (p.nmax + 31) / 32 : 1;  // atoms per lane: 1 to 4
  const int m = mode == 0 ? 0 : mode == 1 ? 1 : 2;
  const void *fn = 1.f / p.inv_dc2_ang < NEAR2_ALL[hw - 1] ? refine_fn<true>(m, hw) : refine_fn<false>(m, hw);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  void *args[] = {&a};
  return cudaLaunchKernel(fn, dim3((n + warps - 1) / warps), dim3(32 * warps), args, smem, s);
}

}  // namespace ligate
