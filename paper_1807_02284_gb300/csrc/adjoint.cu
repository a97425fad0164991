// Reverse-mode (adjoint) stepping with checkpointing: gradients of a loss of the final scalar
// (and velocity) field with respect to the initial velocity field.  Not in the paper.
//
// Forward step n -> n+1 at a fluid node x:
//   d_in = pull(D^n);  (rho, u) = moments(d_in);  phi = phi(|grad U^n|(x));
//   D^{n+1}(x) = collide(d_in, u, phi);  U^{n+1}(x) = u;  C^{n+1}(x) = trilinear(C^n, x - u).
// Reverse step, given the adjoints (Lam, Ups, Gam) of (D^{n+1}, U^{n+1}, C^{n+1}):
//   pass A (per fluid node x): recompute the forward at x, then the exact transpose of every
//     stage; the population adjoints go to the pull sources (the pull, with bounce-back, reads
//     every fluid slot exactly once, so these stores never collide), and the adjoint of the
//     adaptive factor becomes one per-node number ms: the adjoint of the velocity difference
//     diff_ab = U_a(x+e_b) - U_a(x-e_b) is mu_ab = ms diff_ab;
//   pass B (per node y): Ups^n_a(y) = sum_b mu_ab(y - e_b) - mu_ab(y + e_b), the differences
//     formed again from U^n, and
//     Gam^n(y) = sum over the nodes x whose departure cell touches y of w_{x->y} Gam^{n+1}(x)
//     (a gather over the 27 neighbours: deterministic, no atomics).
// Initial state: D^0 = f^eq(rho_0, u_0) - w and U^0 = u_0, so
//   dL/du_0 = Ups^0 + (dD^0/du_0)^T Lam^0.
// Inflow nodes: D^{n+1} = f^eq(1, U^n) - w and U^{n+1} = U^n, so their pulled populations get
// a zero adjoint and the adjoint of U^n collects the equilibrium's Jacobian, the copy and the
// scalar's departure-point term; dL/du_0 at an inflow node is then the gradient with respect
// to its (constant) inflow velocity.
// Open faces copy the nearest in-block node, so a slot of a face node can be read by up to 8
// pulls: the one pull that reads it without clamping (or the node's own bounce-back) stores
// into the slot, every clamped pull stores its adjoint in a side buffer indexed by the reading
// node and direction, and k_face_gather then adds those to the slots in a fixed order (no
// atomics: the gradients are bit-reproducible).  Pass B's lagged-velocity gather uses the
// clamped differences (a face node's own difference involves itself), and the scalar gather
// counts a clamped repeat of the node once.
// Scope: blocks with >= 3 nodes per axis, FP32 or FP16-shifted storage (the checkpoints of
// an FP16 run hold its deviations widened to FP32; replays and transposes run in FP32), and
// continuous-scale domains of refined and far-field blocks (the reversed Algorithm 1
// schedule further below).
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "lbm_adjoint.cuh"
#include "lbm_cell.cuh"
#include "runtime.h"

namespace lbm {

struct AdjArgs {
  BlockView fwd;        // D^n, U^n, C^n in (d_out, u_out, c_out unused)
  const float* lam_in;  // Lam^{n+1}: 27 planes (cube order)
  const float* ups_in;  // Ups^{n+1}: 3 planes
  const float* gam_in;  // Gam^{n+1}
  const float* u_next;  // U^{n+1}: 3 planes (scalar gather)
  float* lam_out;       // Lam^n
  float* ups_out;       // Ups^n
  float* gam_out;       // Gam^n
  float* ms;            // adjoint of the gradient norm over 4 |grad|: dL/d(diff_ab) = ms diff_ab
  float* side;          // open faces: adjoints of the clamped pulls (FaceSide layout)
};

// Adjoint of the scalar step with respect to the departure velocity: C^{n+1}(x) is the
// trilinear interpolant of C^n at x - u, so ub -= gam * d(interpolant)/d(fraction) per axis
// (the fraction grows with the displacement -u).  The derivative is 0 where the sample does
// not move with u: a displacement clamped at one node, or a departure point below an open
// face's first node (the forward pins the sample to that node; at the upper face both
// corners already coincide).
__device__ __forceinline__ void scalar_u_vjp(const BlockView& v, const ScalarCell& sc, int x, int y,
                                             int z, float ux, float uy, float uz, float gam,
                                             float (&ub)[3]) {
  if (gam == 0.0f) return;
  const float tx = sc.tx, ty = sc.ty, tz = sc.tz;
  const float dtx = (1 - ty) * (1 - tz) * (sc.c[1] - sc.c[0]) + ty * (1 - tz) * (sc.c[3] - sc.c[2]) +
                    (1 - ty) * tz * (sc.c[5] - sc.c[4]) + ty * tz * (sc.c[7] - sc.c[6]);
  const float dty = (1 - tx) * (1 - tz) * (sc.c[2] - sc.c[0]) + tx * (1 - tz) * (sc.c[3] - sc.c[1]) +
                    (1 - tx) * tz * (sc.c[6] - sc.c[4]) + tx * tz * (sc.c[7] - sc.c[5]);
  const float dtz = (1 - tx) * (1 - ty) * (sc.c[4] - sc.c[0]) + tx * (1 - ty) * (sc.c[5] - sc.c[1]) +
                    (1 - tx) * ty * (sc.c[6] - sc.c[2]) + tx * ty * (sc.c[7] - sc.c[3]);
  const bool lx = !v.per[0] && x == 0 && ux > 0.0f;
  const bool ly = !v.per[1] && y == 0 && uy > 0.0f;
  const bool lz = !v.per[2] && z == 0 && uz > 0.0f;
  if (fabsf(ux) < 1.0f && !lx) ub[0] -= gam * dtx;
  if (fabsf(uy) < 1.0f && !ly) ub[1] -= gam * dty;
  if (fabsf(uz) < 1.0f && !lz) ub[2] -= gam * dtz;
}

// A float copied asynchronously from global to shared memory.
__device__ __forceinline__ void copy_async4(float* smem, const float* g) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(g) : "memory");
}

// Open faces.  A pull whose source x - e_K lies outside the block along a non-periodic axis
// reads the nearest in-block node instead (the clamped copy), so a face node's slot can be
// read by several pulls.  Bits 2a / 2a + 1 of a node's clamp mask say that the node lies on
// the open lower / upper face of axis a; the pull of direction K is clamped on axis a when
// e_K,a = +1 and bit 2a is set, or e_K,a = -1 and bit 2a + 1 is set.
using ClampMask = uint32_t;

template <bool OPEN>
__device__ __forceinline__ ClampMask clamp_mask(const BlockView& v, int x, int y, int z) {
  if constexpr (!OPEN) return 0u;
  const int c[3] = {x, y, z}, nn[3] = {v.nx, v.ny, v.nz};
  ClampMask m = 0u;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (v.per[a]) continue;
    if (c[a] == 0) m |= 1u << (2 * a);
    if (c[a] == nn[a] - 1) m |= 2u << (2 * a);
  }
  return m;
}

// Side buffer of the clamped pulls: one entry per (reading node, direction), filed under the
// lowest axis a0 on which the pull is clamped.  That node lies on face (a0, lower / upper),
// and the direction has e_K,a0 = +1 / -1, so 9 directions remain, numbered by the other two
// components (b < c): j = 3 (e_b + 1) + (e_c + 1).  Face (a0, side) holds 9 planes of its
// area n_b n_c, the position x_b + n_b x_c; faces follow in the order x-, x+, y-, y+, z-, z+.
// 9 * 2 * (ny nz + nx nz + nx ny) floats per block.
__host__ __device__ __forceinline__ size_t face_side_floats(int nx, int ny, int nz) {
  return (size_t)18 * ((size_t)ny * nz + (size_t)nx * nz + (size_t)nx * ny);
}

__device__ __forceinline__ uint32_t face_side_index(int nx, int ny, int nz, int a0, int hi,
                                                    const int (&p)[3], const int (&e)[3]) {
  const uint32_t A0 = (uint32_t)ny * nz, A1 = (uint32_t)nx * nz, A2 = (uint32_t)nx * ny;
  const uint32_t area = a0 == 0 ? A0 : (a0 == 1 ? A1 : A2);
  const uint32_t off = 9u * (a0 == 0 ? 0u : (a0 == 1 ? 2u * A0 : 2u * (A0 + A1))) + 9u * hi * area;
  const int b = a0 == 0 ? 1 : 0, c = a0 == 2 ? 1 : 2;
  const int nb = b == 0 ? nx : ny;
  const uint32_t pos = (uint32_t)p[b] + (uint32_t)nb * (uint32_t)p[c];
  const uint32_t j = (uint32_t)(3 * (e[b] + 1) + (e[c] + 1));
  return off + j * area + pos;
}

// ACC: add to the adjoint already held by the slot (the reverse of a multi-block schedule,
// where a level is read by several operations) instead of storing it.  Every slot has at most
// one unclamped reader or bounce-back writer, so the plain store / add never collides; a
// clamped pull goes to the side buffer (its own entry) and k_face_gather adds it later.
template <bool OPEN, bool ACC, int K = 0>
__device__ __forceinline__ void push_all(const float (&A)[27], float* __restrict__ lam,
                                         uint32_t N, const Nbr<uint32_t>& n, uint32_t idx,
                                         const uint8_t* __restrict__ flags, bool near,
                                         ClampMask cm, const BlockView& v, int x, int y, int z,
                                         float* __restrict__ side) {
  if constexpr (K < 27) {
    constexpr int cx = cxk(K), cy = cyk(K), cz = czk(K);
    const uint32_t src = pull_src<K>(n);
    uint32_t slot = (uint32_t)K * N + src;
    const bool bb = K != 13 && near && (__ldg(flags + src) & F_SOLID);
    if (bb) slot = (uint32_t)(26 - K) * N + idx;
    bool stored = false;
    if constexpr (OPEN) {
      constexpr ClampMask kb = (cx == 1 ? 1u : cx == -1 ? 2u : 0u) |
                               (cy == 1 ? 4u : cy == -1 ? 8u : 0u) |
                               (cz == 1 ? 16u : cz == -1 ? 32u : 0u);
      const ClampMask hit = cm & kb;
      if (hit != 0u && !bb) {
        const int a0 = (hit & 3u) ? 0 : ((hit & 12u) ? 1 : 2);
        const int hi = (hit >> (2 * a0)) & 2u ? 1 : 0;
        const int p[3] = {x, y, z}, e[3] = {cx, cy, cz};
        side[face_side_index(v.nx, v.ny, v.nz, a0, hi, p, e)] = A[K];
        stored = true;
      }
    }
    if (!stored) {
      if (ACC) lam[slot] += A[K];
      else lam[slot] = A[K];
    }
    push_all<OPEN, ACC, K + 1>(A, lam, N, n, idx, flags, near, cm, v, x, y, z, side);
  }
}

// Transpose of the collision (and of the scale mapping, which is the same relaxation with
// other keep factors): K holds the central moments before relaxation at velocity u, A the
// adjoint of the post-collision populations on entry and the adjoint of
// the pre-collision populations on return; the velocity terms are added to ub and the
// adjoint of the keep factors of the high-order groups to kbar.
// With `local` set (the strain-rate mode of the adaptive factor), the factor's input g is
// local_strain of the central moments K, so the keep factors' adjoint flows back into K, rho
// and u here (between the relaxation's transpose and the shifts').  late(ub) adds velocity
// terms that are wanted only before u's own transpose (their loads are in flight until then).
template <typename Late>
__device__ __forceinline__ void collide_vjp(const float (&K)[27], float (&A)[27], float drho, float ux,
                                            float uy, float uz, float inv, const Keep& kf,
                                            float (&ub)[3], float (&kbar)[4],
                                            const RelaxParams* local, float g, Late late) {
  // adjoint of the post-collision raw moments, and those moments themselves
  raw_inverse_vjp<1>(A);
  raw_inverse_vjp<3>(A);
  raw_inverse_vjp<9>(A);
  {
    float T[27];
#pragma unroll
    for (int k = 0; k < 27; ++k) T[k] = K[k];
    relax_to_equilibrium(T, drho, ux, uy, uz, kf);
    unshift_axis<9>(T, uz);
    unshift_axis<3>(T, uy);
    unshift_axis<1>(T, ux);
    ub[0] += shift_dot<1>(A, T);
    ub[1] += shift_dot<3>(A, T);
    ub[2] += shift_dot<9>(A, T);
  }
  unshift_axis_vjp<1>(A, ux);
  unshift_axis_vjp<3>(A, uy);
  unshift_axis_vjp<9>(A, uz);            // A = adjoint of the relaxed central moments
  float bar[4] = {0.f, 0.f, 0.f, 0.f};     // d/d(rho - 1), d/du
  relax_vjp(K, A, drho, ux, uy, uz, kf, bar, kbar);
  ub[0] += bar[1];
  ub[1] += bar[2];
  ub[2] += bar[3];
  float drhob = bar[0];
  if (local && g > 0.0f && g * local->inv_gmax < 1.0f) {
    // g = (3 S_nu / (2 rho)) sqrt(2 ss), ss = |P|^2 of the non-equilibrium second central
    // moments P_ab = K_ab - K^eq_ab (see local_strain): dg/dP_aa = g P_aa / ss,
    // dg/dP_ab = 2 g P_ab / ss (a != b), dg/d(rho - 1) = -g / rho - sum_a dg/dP_aa / 3,
    // dg/du_a = sum_b dg/dP_ab dP_ab/du_a
    float phib = 0.0f;
#pragma unroll
    for (int gi = 0; gi < 4; ++gi) {
      const float S = 1.0f - kf.g[gi];
      phib = fmaf(kbar[gi], local->nuh3[gi] * S * S, phib);
    }
    const float gb = phib * local->a * local->inv_gmax;   // phi = a g / g_max + b below the clamp
    const float dr3 = drho * (1.0f / 3.0f);
    const float pxx = K[kap(2, 0, 0)] - (dr3 - ux * ux);
    const float pyy = K[kap(0, 2, 0)] - (dr3 - uy * uy);
    const float pzz = K[kap(0, 0, 2)] - (dr3 - uz * uz);
    const float pxy = K[kap(1, 1, 0)] + ux * uy;
    const float pxz = K[kap(1, 0, 1)] + ux * uz;
    const float pyz = K[kap(0, 1, 1)] + uy * uz;
    const float ss = fmaf(pxx, pxx, fmaf(pyy, pyy, pzz * pzz)) +
                     2.0f * fmaf(pxy, pxy, fmaf(pxz, pxz, pyz * pyz));
    if (ss > 0.0f) {
      const float c = gb * g / ss;
      A[kap(2, 0, 0)] = fmaf(c, pxx, A[kap(2, 0, 0)]);
      A[kap(0, 2, 0)] = fmaf(c, pyy, A[kap(0, 2, 0)]);
      A[kap(0, 0, 2)] = fmaf(c, pzz, A[kap(0, 0, 2)]);
      A[kap(1, 1, 0)] = fmaf(2.0f * c, pxy, A[kap(1, 1, 0)]);
      A[kap(1, 0, 1)] = fmaf(2.0f * c, pxz, A[kap(1, 0, 1)]);
      A[kap(0, 1, 1)] = fmaf(2.0f * c, pyz, A[kap(0, 1, 1)]);
      drhob -= c * (pxx + pyy + pzz) * (1.0f / 3.0f) + gb * g * inv;
      ub[0] += 2.0f * c * (ux * pxx + uy * pxy + uz * pxz);
      ub[1] += 2.0f * c * (uy * pyy + ux * pxy + uz * pyz);
      ub[2] += 2.0f * c * (uz * pzz + ux * pxz + uy * pyz);
    }
  }
  ub[0] -= shift_dot<1>(A, K);
  ub[1] -= shift_dot<3>(A, K);
  ub[2] -= shift_dot<9>(A, K);
  unshift_axis_vjp<1>(A, -ux);
  unshift_axis_vjp<3>(A, -uy);
  unshift_axis_vjp<9>(A, -uz);           // A = adjoint of the raw moments of the pulled set
  late(ub);
  // u = j / rho with rho = 1 + r_000, j = (r_100, r_010, r_001)
  drhob -= (ub[0] * ux + ub[1] * uy + ub[2] * uz) * inv;
  A[kap(0, 0, 0)] += drhob;
  A[kap(1, 0, 0)] += ub[0] * inv;
  A[kap(0, 1, 0)] += ub[1] * inv;
  A[kap(0, 0, 1)] += ub[2] * inv;
  raw_axis_vjp<9>(A);
  raw_axis_vjp<3>(A);
  raw_axis_vjp<1>(A);                    // A = adjoint of the pulled populations
}

// The nodes of a block's open faces, each once: thread t walks the open faces in the order
// x-, x+, y-, y+, z-, z+ and skips a node that an earlier open face already holds.
__device__ __forceinline__ bool open_face_node(uint32_t t, const int (&nn)[3], const int (&per)[3],
                                               int (&p)[3]) {
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    const int a = f >> 1;
    if (per[a]) continue;
    const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;
    const uint32_t area = (uint32_t)nn[b] * (uint32_t)nn[c];
    if (t >= area) {
      t -= area;
      continue;
    }
    p[a] = (f & 1) ? nn[a] - 1 : 0;
    const uint32_t q = t / (uint32_t)nn[b];
    p[b] = (int)(t - q * (uint32_t)nn[b]);
    p[c] = (int)q;
#pragma unroll
    for (int a2 = 0; a2 < 3; ++a2)
      if (a2 < a && !per[a2] && (p[a2] == 0 || p[a2] == nn[a2] - 1)) return false;
    return true;
  }
  return false;
}

__host__ __device__ __forceinline__ uint32_t open_face_threads(int nx, int ny, int nz, const int (&per)[3]) {
  return (per[0] ? 0u : 2u * (uint32_t)ny * (uint32_t)nz) + (per[1] ? 0u : 2u * (uint32_t)nx * (uint32_t)nz) +
         (per[2] ? 0u : 2u * (uint32_t)nx * (uint32_t)ny);
}

// After pass A: every open-face slot (k, s) adds the adjoints of the clamped pulls that read
// it, in a fixed order, and clears their side entries (each is read by exactly this slot, so
// the buffer is all zeros again for the next launch).  The readers x of (k, s) have, per axis
// a, either x_a = s_a + e_k,a (unclamped) or x_a = s_a where s_a is the face that the pull
// leaves (e_k,a = +1 at s_a = 0, -1 at s_a = n_a - 1); the combinations with at least one
// clamped axis are taken in the order of their axis bits.
// zero (may be null): the buffer pass A read, whose face slots are cleared for the next step,
// where it is pass A's output and a slot that no pull reads unclamped only receives this sum.
// One thread per face node and direction (grid.y): a loop over the 27 directions in one thread
// was a chain of 27 dependent rounds of loads (72 x 60 x 51: 51 us, and 5 us more for clearing
// the slots in a launch of its own).
__global__ void __launch_bounds__(256) k_face_gather(float* __restrict__ lam, float* __restrict__ side,
                                                     float* __restrict__ zero, int nx, int ny,
                                                     int nz, int px, int py, int pz) {
  const int per[3] = {px, py, pz}, nn[3] = {nx, ny, nz};
  const uint32_t t = blockIdx.x * 256u + threadIdx.x;
  if (t >= open_face_threads(nx, ny, nz, per)) return;
  int s[3];
  if (!open_face_node(t, nn, per, s)) return;
  const int k = blockIdx.y;
  const int e[3] = {k % 3 - 1, (k / 3) % 3 - 1, k / 9 - 1};
  const size_t slot = (size_t)k * ((size_t)nx * ny * nz) + ((size_t)s[2] * ny + s[1]) * nx + s[0];
  if (zero) zero[slot] = 0.0f;
  int can = 0;                              // axes on which a reader's pull can be clamped
  bool in[3];                               // whether s + e lies in the block on that axis
  int q[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (!per[a] && ((e[a] == 1 && s[a] == 0) || (e[a] == -1 && s[a] == nn[a] - 1))) can |= 1 << a;
    q[a] = s[a] + e[a];
    if (per[a]) q[a] = q[a] < 0 ? q[a] + nn[a] : (q[a] >= nn[a] ? q[a] - nn[a] : q[a]);
    in[a] = q[a] >= 0 && q[a] < nn[a];
  }
  if (!can) return;
  float sum = 0.0f;
  bool any = false;
#pragma unroll
  for (int combo = 1; combo < 8; ++combo) {
    if ((combo & can) != combo) continue;
    int xr[3];
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const bool clamped = (combo >> a) & 1;
      xr[a] = clamped ? s[a] : q[a];
      ok = ok && (clamped || in[a]);
    }
    if (!ok) continue;
    const int a0 = (combo & 1) ? 0 : ((combo & 2) ? 1 : 2);
    const uint32_t si = face_side_index(nx, ny, nz, a0, e[a0] == -1 ? 1 : 0, xr, e);
    sum += side[si];
    side[si] = 0.0f;
    any = true;
  }
  if (any) lam[slot] += sum;
}

static void launch_face_gather(float* lam, float* side, float* zero, const BlockView& v,
                               cudaStream_t s) {
  const int per[3] = {v.per[0], v.per[1], v.per[2]};
  const unsigned g = (open_face_threads(v.nx, v.ny, v.nz, per) + 255) / 256;
  if (g == 0) return;
  k_face_gather<<<dim3(g, 27, 1), 256, 0, s>>>(lam, side, zero, v.nx, v.ny, v.nz, per[0], per[1], per[2]);
}

// The populations of a wall node (face wall or obstacle surface) pulled from beyond the wall:
// the set wall_regularize completes (same tests).
template <typename IT>
__device__ __forceinline__ unsigned wall_unknowns(const BlockView& v, int x, int y, int z,
                                                  uint8_t fl, const Nbr<IT>& n) {
  const bool lo[3] = {(v.walls & 1) && x == 0, (v.walls & 4) && y == 0, (v.walls & 16) && z == 0};
  const bool hi[3] = {(v.walls & 2) && x == v.nx - 1, (v.walls & 8) && y == v.ny - 1,
                      (v.walls & 32) && z == v.nz - 1};
  unsigned unk = 0u;
#pragma unroll
  for (int k = 0; k < 27; ++k) {
    const int c[3] = {cxk(k), cyk(k), czk(k)};
    bool u = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) u |= (lo[a] && c[a] == 1) || (hi[a] && c[a] == -1);
    if (u) unk |= 1u << k;
  }
  if (fl & F_OBST_WALL) unk |= solid_sources<IT>(v.flags, n);
  return unk;
}

// Transpose of wall_regularize (a linear map of the pulled populations for a fixed unknown
// set): A holds the adjoint of the rebuilt populations on entry and of the pulled ones on
// return.  Forward: d'_k = d_k (known), d_opp(k) (unknown, opposite known), excluded (both
// unknown, weight wb); drho = sum d' / (1 - wb); neq_k = d'_k - w_k drho (0 when both);
// Pi = sum c c neq; out_k = w_k (drho + 4.5 (c c : Pi - tr(Pi) / 3)).
template <typename IT>
__device__ __forceinline__ void wall_regularize_vjp(float (&A)[27], const BlockView& v, int x,
                                                    int y, int z, uint8_t fl, const Nbr<IT>& n) {
  const unsigned unk = wall_unknowns<IT>(v, x, y, z, fl, n);
  float wb = 0.0f, drb = 0.0f;
  float pxx = 0.f, pyy = 0.f, pzz = 0.f, pxy = 0.f, pxz = 0.f, pyz = 0.f;   // adjoint of Pi
  const float third = 1.0f / 3.0f;
#pragma unroll
  for (int k = 0; k < 27; ++k) {
    if (((unk >> k) & 1u) && ((unk >> (26 - k)) & 1u)) wb += wk(k);
    const float cx = (float)cxk(k), cy = (float)cyk(k), cz = (float)czk(k);
    const float a = A[k];
    drb = fmaf(wk(k), a, drb);
    const float q = 4.5f * wk(k) * a;
    pxx = fmaf(q, cx * cx - third, pxx);
    pyy = fmaf(q, cy * cy - third, pyy);
    pzz = fmaf(q, cz * cz - third, pzz);
    pxy = fmaf(q, 2.0f * cx * cy, pxy);
    pxz = fmaf(q, 2.0f * cx * cz, pxz);
    pyz = fmaf(q, 2.0f * cy * cz, pyz);
  }
  float db[27];                          // adjoint of the completed set d'
#pragma unroll
  for (int k = 0; k < 27; ++k) {
    const bool both = ((unk >> k) & 1u) && ((unk >> (26 - k)) & 1u);
    const float cx = (float)cxk(k), cy = (float)cyk(k), cz = (float)czk(k);
    const float nb = cx * cx * pxx + cy * cy * pyy + cz * cz * pzz + cx * cy * pxy +
                     cx * cz * pxz + cy * cz * pyz;
    db[k] = both ? 0.0f : nb;
    if (!both) drb = fmaf(-wk(k), nb, drb);
  }
  const float sb = drb / (1.0f - wb);
#pragma unroll
  for (int k = 0; k < 27; ++k) A[k] = 0.0f;
#pragma unroll
  for (int k = 0; k < 27; ++k) {
    const bool uk = (unk >> k) & 1u, uo = (unk >> (26 - k)) & 1u;
    if (uk && uo) continue;
    const float g = db[k] + sb;
    if (uk) A[26 - k] += g;              // taken from the opposite population
    else A[k] += g;
  }
}

// Pushes the adjoint of a node's pulled populations to their sources when none of them is
// wrapped, clamped or bounced back along y or z: the offsets of pull_inner.
template <bool ACC, int K = 0>
__device__ __forceinline__ void push_inner(const float (&A)[27], float* __restrict__ lam, uint32_t N,
                                           uint32_t nx, uint32_t nxy, uint32_t am, uint32_t a0,
                                           uint32_t ap) {
  if constexpr (K < 27) {
    constexpr int cx = cxk(K), cy = cyk(K), cz = czk(K);
    const uint32_t slot = ((uint32_t)K * N - (uint32_t)cz * nxy - (uint32_t)cy * nx) +
                          (cx > 0 ? am : cx < 0 ? ap : a0);
    if (ACC) lam[slot] += A[K];
    else lam[slot] = A[K];
    push_inner<ACC, K + 1>(A, lam, N, nx, nxy, am, a0, ap);
  }
}

constexpr int ADJ_THREADS = 128;

// Pass A.  OPEN: some face of the block is open (clamped pulls go to the side buffer).  ACC:
// the adjoints of the input level are added to (multi-block reverse), and scale-boundary
// (ghost) nodes, which the step does not update, are left to the mapping that wrote them.
// WALLS: the block has wall faces or obstacle-surface walls (wall_regularize and its
// transpose).
// One thread per node, consecutive threads over the nodes of a plane (no idle lanes when nx is
// not a multiple of the CTA).  Three 27-arrays are live in the transposed collision, which
// holds the kernel at 16 warps per SM, too few to hide its chain of dependent loads; so
// everything known from the node index alone is requested first (the pull and the velocity
// neighbourhood in registers, the 31 adjoints by cp.async into this thread's shared-memory
// column, 4 bytes each), the scalar corners as soon as u is known, and each is waited for
// only where it is used.  128^3: 245 -> 169 us (1995 instructions per node, 61 % of issue slots,
// 52 % of DRAM peak; before, the flags, the pull, the corners and the adjoints waited for one
// another in turn and 19 words per node went to pass B), 72 x 60 x 51 with open faces
// 64 -> 34 us (rows of 72 nodes left 44 % of a 128-thread row's lanes idle).
// 4 CTAs per SM (128 registers, no spills) against 3: 169 against 192 us at 128^3.
template <bool OPEN, bool ACC, bool WALLS>
__global__ void __launch_bounds__(ADJ_THREADS, 4) k_adj_a(AdjArgs a) {
  __shared__ float sadj[31][ADJ_THREADS];     // lam, ups, gam of the node
  __shared__ float scor[8][ADJ_THREADS];      // scalar corners of its departure cell
  const BlockView& v = a.fwd;
  const int t = threadIdx.x;
  const uint32_t nx = (uint32_t)v.nx, nxy = nx * (uint32_t)v.ny;
  const uint32_t i = blockIdx.x * ADJ_THREADS + t;
  if (i >= nxy) return;
  const int y = (int)(i / nx), x = (int)(i - (uint32_t)y * nx), z = blockIdx.y;
  const uint32_t N = (uint32_t)v.N;
  const uint32_t idx = nxy * (uint32_t)z + i;
#pragma unroll
  for (int k = 0; k < 27; ++k) copy_async4(&sadj[k][t], a.lam_in + ((uint32_t)k * N + idx));
#pragma unroll
  for (int c = 0; c < 3; ++c) copy_async4(&sadj[27 + c][t], a.ups_in + ((uint32_t)c * N + idx));
  copy_async4(&sadj[30][t], a.gam_in + idx);
  asm volatile("cp.async.commit_group;" ::: "memory");
  const uint8_t fl = __ldg(v.flags + idx);
  const bool inner = inner_yz(v, y, z);
  const float* __restrict__ din = static_cast<const float*>(v.d_in);
  const uint32_t row = idx - (uint32_t)x;
  const uint32_t am = row + (uint32_t)nbr(x, -1, v.nx, v.per[0]);
  const uint32_t ap = row + (uint32_t)nbr(x, 1, v.nx, v.per[0]);
  const bool local = v.rp.adaptive && v.rp.local;
  const bool lagged = v.rp.adaptive && !local;
  float K[27], g = 0.0f;
  if (inner) {
    pull_inner<float, uint32_t>(K, din, N, nx, nxy, am, idx, ap);
    if (lagged) g = grad_norm_inner<uint32_t>(v.u_in, N, nx, nxy, idx, am, ap);
  } else {
    const Nbr<uint32_t> n = neighbours<uint32_t>(v, x, y, z);
    pull_all<float, uint32_t>(K, din, N, n);
    if (lagged) g = grad_norm<uint32_t>(v.u_in, N, n);
  }
  if ((fl & F_SOLID) || (ACC && (fl & F_GHOST))) {
    a.ms[idx] = 0.0f;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    return;
  }
  if (fl & F_INFLOW) {
    // D^{n+1} = f^eq(1, U^n) - w, U^{n+1} = U^n, C^{n+1} sampled at x - U^n: the pulled
    // populations are unused (their slots get a zero adjoint) and every adjoint goes to U^n,
    // which pass B completes with the lagged-gradient terms of the neighbours
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const float u[3] = {v.u_in[idx], v.u_in[N + idx], v.u_in[2 * N + idx]};
    float ub[3] = {sadj[27][t], sadj[28][t], sadj[29][t]};
    if (!(fl & F_SCALAR_SRC))
      scalar_u_vjp(v, scalar_corners<uint32_t>(v, x, y, z, u[0], u[1], u[2]), x, y, z, u[0], u[1],
                   u[2], sadj[30][t], ub);
#pragma unroll
    for (int k = 0; k < 27; ++k) {
      const float c[3] = {(float)cxk(k), (float)cyk(k), (float)czk(k)};
      const float cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2];
      const float l = sadj[k][t] * wk(k);
#pragma unroll
      for (int a2 = 0; a2 < 3; ++a2) ub[a2] = fmaf(l, 3.0f * c[a2] + 9.0f * cu * c[a2] - 3.0f * u[a2], ub[a2]);
    }
    if (ACC) {
      a.ups_out[idx] += ub[0];
      a.ups_out[N + idx] += ub[1];
      a.ups_out[2 * N + idx] += ub[2];
    } else {
      a.ups_out[idx] = ub[0];
      a.ups_out[N + idx] = ub[1];
      a.ups_out[2 * N + idx] = ub[2];
      float Z[27];
#pragma unroll
      for (int k = 0; k < 27; ++k) Z[k] = 0.0f;
      push_all<OPEN, false>(Z, a.lam_out, N, neighbours<uint32_t>(v, x, y, z), idx, v.flags,
                            (fl & F_NEAR_SOLID) != 0, clamp_mask<OPEN>(v, x, y, z), v, x, y, z, a.side);
    }
    a.ms[idx] = 0.0f;
    return;
  }

  // ---- forward recompute up to the central moments
  // as in cell_update: an obstacle wall node completes what comes from inside the obstacle
  // itself (no bounce-back), every wall node is regularized before the collision
  const bool near = (fl & F_NEAR_SOLID) != 0 && !(WALLS && (fl & F_OBST_WALL));
  if (near) bounce_back<float, uint32_t>(K, din, N, v.flags, neighbours<uint32_t>(v, x, y, z), idx);
  const bool wall = WALLS && (fl & (F_WALL | F_OBST_WALL));
  if constexpr (WALLS) {
    if (wall) wall_regularize<uint32_t>(K, v, x, y, z, fl, neighbours<uint32_t>(v, x, y, z));
  }
  raw_moments(K);
  const float drho = K[kap(0, 0, 0)];
  const float inv = fast_rcp(1.0f + drho);
  const float ux = K[kap(1, 0, 0)] * inv, uy = K[kap(0, 1, 0)] * inv, uz = K[kap(0, 0, 1)] * inv;
  const bool src = (fl & F_SCALAR_SRC) != 0;
  if (!src) scalar_corners_async<uint32_t>(v, x, y, z, ux, uy, uz, &scor[0][t], ADJ_THREADS);
  asm volatile("cp.async.commit_group;" ::: "memory");
  central_from_raw(K, ux, uy, uz);       // K = central moments before relaxation
  if (local) g = local_strain(K, drho, ux, uy, uz, v.rp.s_nu);
  const Keep kf = keep_factors(v.rp, g);

  // ---- adjoint of the collision, of the stored velocity and of the scalar step
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  float A[27];
#pragma unroll
  for (int k = 0; k < 27; ++k) A[k] = sadj[k][t];
  float ub[3] = {sadj[27][t], sadj[28][t], sadj[29][t]};
  float kbar[4] = {0.f, 0.f, 0.f, 0.f};    // d/d(keep factor) of the high-order groups
  collide_vjp(K, A, drho, ux, uy, uz, inv, kf, ub, kbar, local ? &v.rp : nullptr, g,
              [&](float (&b)[3]) {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                if (src) return;
                ScalarCell sc;
#pragma unroll
                for (int c = 0; c < 8; ++c) sc.c[c] = scor[c][t];
                sc.tx = sl_axis(x, ux, v.nx, v.per[0]).t;
                sc.ty = sl_axis(y, uy, v.ny, v.per[1]).t;
                sc.tz = sl_axis(z, uz, v.nz, v.per[2]).t;
                scalar_u_vjp(v, sc, x, y, z, ux, uy, uz, sadj[30][t], b);
              });
  if constexpr (WALLS) {
    if (wall) wall_regularize_vjp<uint32_t>(A, v, x, y, z, fl, neighbours<uint32_t>(v, x, y, z));
  }
  const ClampMask cm = clamp_mask<OPEN>(v, x, y, z);
  if (inner && !near && cm == 0u)
    push_inner<ACC>(A, a.lam_out, N, nx, nxy, am, idx, ap);
  else
    push_all<OPEN, ACC>(A, a.lam_out, N, neighbours<uint32_t>(v, x, y, z), idx, v.flags, near, cm, v,
                        x, y, z, a.side);

  // ---- adjoint of the adaptive factor: K_g = 1 - 1/(phi nu3_g + 1/2)
  float ms = 0.0f;                // (the local-strain mode has no lagged-velocity dependence)
  if (lagged && g > 0.0f && g * v.rp.inv_gmax < 1.0f) {
    float phib = 0.0f;
#pragma unroll
    for (int gi = 0; gi < 4; ++gi) {
      const float S = 1.0f - kf.g[gi];
      phib = fmaf(kbar[gi], v.rp.nuh3[gi] * S * S, phib);
    }
    const float gb = phib * v.rp.a * v.rp.inv_gmax;   // phi = a g / g_max + b below the clamp
    ms = gb * 0.25f / g;                              // dg/d(diff) = diff / (4 g)
  }
  a.ms[idx] = ms;
}

// A node as sender of the scalar gather along one axis: its departure sample sits dsp =
// clamp(-u, -1, 1) away and is shared between two neighbouring nodes by the hat weights
// max(0, -dsp), 1 - |dsp|, max(0, dsp) of the nodes -1, 0, +1 away.  On an open face a sample
// beyond the face is pinned to the face's node: dsp is bounded by 0 on that side.
struct SenderAxis {
  float lo, hi;
};
__device__ __forceinline__ SenderAxis sender_axis(int c, int n, int periodic) {
  return SenderAxis{!periodic && c == 0 ? 0.0f : -1.0f, !periodic && c == n - 1 ? 0.0f : 1.0f};
}
__device__ __forceinline__ void sender_weights(const SenderAxis& s, float u, float (&w)[3]) {
  const float dsp = fminf(fmaxf(-u, s.lo), s.hi);
  w[0] = fmaxf(-dsp, 0.0f);
  w[1] = 1.0f - fabsf(dsp);
  w[2] = fmaxf(dsp, 0.0f);
}

// The nodes -2, -1, +1, +2 away along one axis as wrapped or clamped indices, and the signs of
// the neighbours' difference adjoints: node q's difference along the axis is U(q+1) - U(q-1) with
// the indices wrapped or clamped, so node c receives +mu(c - 1) and -mu(c + 1) where those nodes
// exist, and on an open face also its own +mu (upper: its + neighbour is itself) or -mu (lower).
struct AxisStar {
  int m2, m1, p1, p2;
  float wm, wp, own;
};
__device__ __forceinline__ AxisStar axis_star(int c, int n, int periodic) {
  AxisStar s;
  s.m1 = nbr(c, -1, n, periodic);
  s.p1 = nbr(c, 1, n, periodic);
  s.m2 = nbr(s.m1, -1, n, periodic);
  s.p2 = nbr(s.p1, 1, n, periodic);
  s.wm = periodic || c > 0 ? 1.0f : 0.0f;
  s.wp = periodic || c < n - 1 ? 1.0f : 0.0f;
  s.own = periodic ? 0.0f : (c == 0 ? -1.0f : (c == n - 1 ? 1.0f : 0.0f));
  return s;
}

constexpr int ADJ_BX = 32, ADJ_BY = 8;                     // receivers of one plane of a CTA
constexpr int ADJ_SX = ADJ_BX + 2, ADJ_SENDERS = ADJ_SX * (ADJ_BY + 2);

// A column of senders (fixed x, y): its offset in a plane, its bounds along x and y, and
// whether it lies in the block (a tile may reach past nx or ny, or beyond an open face).
struct SenderColumn {
  uint32_t off;
  SenderAxis x, y;
  bool in;
};
// What a sender holds: its scalar adjoint (0 where it sends nothing: obstacle, scalar source,
// scale boundary, outside the block) and its departure velocity.
struct Sender {
  float g, u[3];
};

__device__ __forceinline__ SenderColumn sender_column(const BlockView& v, int x, int y) {
  if (v.per[0]) x += x < 0 ? v.nx : (x == v.nx ? -v.nx : 0);
  if (v.per[1]) y += y < 0 ? v.ny : (y == v.ny ? -v.ny : 0);
  SenderColumn c;
  c.in = x >= 0 && x < v.nx && y >= 0 && y < v.ny;
  c.off = c.in ? (uint32_t)y * (uint32_t)v.nx + (uint32_t)x : 0u;
  c.x = sender_axis(x, v.nx, v.per[0]);
  c.y = sender_axis(y, v.ny, v.per[1]);
  return c;
}

__device__ __forceinline__ Sender load_sender(const AdjArgs& a, const SenderColumn& c, int z) {
  const BlockView& v = a.fwd;
  Sender s{0.0f, {0.0f, 0.0f, 0.0f}};
  if (v.per[2]) z += z < 0 ? v.nz : (z >= v.nz ? -v.nz : 0);
  if (c.in && z >= 0 && z < v.nz) {
    const uint32_t N = (uint32_t)v.N;
    const uint32_t j = (uint32_t)z * ((uint32_t)v.nx * (uint32_t)v.ny) + c.off;
    const float g = __ldg(a.gam_in + j);
    s.g = (__ldg(v.flags + j) & (F_SOLID | F_SCALAR_SRC | F_GHOST)) ? 0.0f : g;
    s.u[0] = __ldg(a.u_next + j);
    s.u[1] = __ldg(a.u_next + (N + j));
    s.u[2] = __ldg(a.u_next + (2 * N + j));
  }
  return s;
}

// The lagged velocity's adjoint at one node: the six neighbours' (and on an open face its own)
// difference adjoints.  Inflow nodes add it to what pass A left there.  INNER: the node is at
// least two nodes from both ends along y and z, so those neighbours are plain offsets.
template <bool ACC, bool INNER>
__device__ __forceinline__ void lagged_adjoint(const AdjArgs& a, int x, int y, int z, uint32_t idx) {
  const BlockView& v = a.fwd;
  const uint32_t N = (uint32_t)v.N, nx = (uint32_t)v.nx, nxy = nx * (uint32_t)v.ny;
  const AxisStar ax = axis_star(x, v.nx, v.per[0]);
  const uint32_t row = idx - (uint32_t)x;
  const uint32_t xm2 = row + ax.m2, xm1 = row + ax.m1, xp1 = row + ax.p1, xp2 = row + ax.p2;
  uint32_t ym2, ym1, yp1, yp2, zm2, zm1, zp1, zp2;
  AxisStar ay, az;
  if constexpr (INNER) {
    ym2 = idx - 2 * nx; ym1 = idx - nx; yp1 = idx + nx; yp2 = idx + 2 * nx;
    zm2 = idx - 2 * nxy; zm1 = idx - nxy; zp1 = idx + nxy; zp2 = idx + 2 * nxy;
    ay.wm = ay.wp = az.wm = az.wp = 1.0f;
    ay.own = az.own = 0.0f;
  } else {
    ay = axis_star(y, v.ny, v.per[1]);
    az = axis_star(z, v.nz, v.per[2]);
    const uint32_t oy = idx - nx * (uint32_t)y, oz = idx - nxy * (uint32_t)z;
    ym2 = oy + nx * (uint32_t)ay.m2; ym1 = oy + nx * (uint32_t)ay.m1;
    yp1 = oy + nx * (uint32_t)ay.p1; yp2 = oy + nx * (uint32_t)ay.p2;
    zm2 = oz + nxy * (uint32_t)az.m2; zm1 = oz + nxy * (uint32_t)az.m1;
    zp1 = oz + nxy * (uint32_t)az.p1; zp2 = oz + nxy * (uint32_t)az.p2;
  }
  const float* __restrict__ ms = a.ms;
  const float mx = ax.wm * __ldg(ms + xm1), px = ax.wp * __ldg(ms + xp1);
  const float my = ay.wm * __ldg(ms + ym1), py = ay.wp * __ldg(ms + yp1);
  const float mz = az.wm * __ldg(ms + zm1), pz = az.wp * __ldg(ms + zp1);
  const bool face = ax.own != 0.0f || ay.own != 0.0f || az.own != 0.0f;
  const bool keep = ACC || (__ldg(v.flags + idx) & (F_INFLOW | F_SOLID)) == F_INFLOW;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float* __restrict__ U = v.u_in + (uint32_t)k * N;
    const float c = __ldg(U + idx);
    float sum = mx * (c - __ldg(U + xm2));
    sum = fmaf(-px, __ldg(U + xp2) - c, sum);
    sum = fmaf(my, c - __ldg(U + ym2), sum);
    sum = fmaf(-py, __ldg(U + yp2) - c, sum);
    sum = fmaf(mz, c - __ldg(U + zm2), sum);
    sum = fmaf(-pz, __ldg(U + zp2) - c, sum);
    if (face) {
      const float own = __ldg(ms + idx);
      sum = fmaf(own * ax.own, __ldg(U + xp1) - __ldg(U + xm1), sum);
      sum = fmaf(own * ay.own, __ldg(U + yp1) - __ldg(U + ym1), sum);
      sum = fmaf(own * az.own, __ldg(U + zp1) - __ldg(U + zm1), sum);
    }
    float* o = a.ups_out + ((uint32_t)k * N + idx);
    *o = keep ? *o + sum : sum;
  }
}

// Pass B, lagged velocity (only where the adaptive factor depends on it): one thread per node
// without shared memory, so that enough warps are resident to cover its 27 loads (as part of
// the marching kernel below they were waited for plane by plane: 128^3 76 us together, 33 + 33
// us apart; 90 us before the two were rewritten).
template <bool ACC>
__global__ void __launch_bounds__(256, 6) k_adj_lagged(AdjArgs a) {
  const BlockView& v = a.fwd;
  const uint32_t nx = (uint32_t)v.nx, nxy = nx * (uint32_t)v.ny;
  const uint32_t i = blockIdx.x * 256u + threadIdx.x;
  if (i >= nxy) return;
  const int z = blockIdx.y, y = (int)(i / nx), x = (int)(i - nx * (uint32_t)y);
  const uint32_t idx = nxy * (uint32_t)z + i;
  if (y >= 2 && y < v.ny - 2 && z >= 2 && z < v.nz - 2) lagged_adjoint<ACC, true>(a, x, y, z, idx);
  else lagged_adjoint<ACC, false>(a, x, y, z, idx);
}

// Pass B, scalar.  A CTA covers 32 x 8 receivers and marches `zc` planes in z.  Every node of
// the tile and its halo is a sender: its three weights along x and the nine products of its y
// and z weights with its scalar adjoint go to shared memory once per plane (a ring of three
// planes, 48 KB), and a receiver adds 27 products of two shared-memory values.  Before, pass A
// stored nine weights per node and every receiver fetched four values from each of its 27
// neighbours through L1 (923 instructions per node, latency-bound).  The next plane's senders
// are loaded into registers before the current plane's sums.  LAGGED false: no k_adj_lagged
// ran, so ups_out is set here.
template <bool ACC, bool LAGGED>
__global__ void __launch_bounds__(ADJ_BX * ADJ_BY) k_adj_b(AdjArgs a, int zc) {
  __shared__ float ring[3][12][ADJ_SENDERS];     // wx(-1, 0, +1), then wy wz g: 3 ez + ey
  const BlockView& v = a.fwd;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * ADJ_BX + tx;
  const int x0 = blockIdx.x * ADJ_BX, y0 = blockIdx.y * ADJ_BY;
  const int x = x0 + tx, y = y0 + ty;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, v.nz);
  const bool mine = x < v.nx && y < v.ny;
  const uint32_t N = (uint32_t)v.N, nx = (uint32_t)v.nx, nxy = nx * (uint32_t)v.ny;
  // this thread's senders of a plane: slots tid and tid + 256 (the latter for tid < 84)
  const int sb = tid + ADJ_BX * ADJ_BY;
  const bool two = sb < ADJ_SENDERS;
  const SenderColumn ca = sender_column(v, x0 - 1 + tid % ADJ_SX, y0 - 1 + tid / ADJ_SX);
  const SenderColumn cb = sender_column(v, x0 - 1 + sb % ADJ_SX, y0 - 1 + sb / ADJ_SX);
  auto put = [&](int slot, int at, const SenderColumn& c, int z, const Sender& s) {
    float wx[3], wy[3], wz[3];
    sender_weights(c.x, s.u[0], wx);
    sender_weights(c.y, s.u[1], wy);
    sender_weights(sender_axis(z, v.nz, v.per[2]), s.u[2], wz);
    float* o = &ring[slot][0][at];
#pragma unroll
    for (int e = 0; e < 3; ++e) o[e * ADJ_SENDERS] = wx[e];
#pragma unroll
    for (int ez = 0; ez < 3; ++ez) {
      const float gz = wz[ez] * s.g;
#pragma unroll
      for (int ey = 0; ey < 3; ++ey) o[(3 + 3 * ez + ey) * ADJ_SENDERS] = wy[ey] * gz;
    }
  };
  for (int p = -1; p <= 0; ++p) {
    put(p + 1, tid, ca, z0 + p, load_sender(a, ca, z0 + p));
    if (two) put(p + 1, sb, cb, z0 + p, load_sender(a, cb, z0 + p));
  }
  Sender na = load_sender(a, ca, z0 + 1), nb{};
  if (two) nb = load_sender(a, cb, z0 + 1);
  int lo = 0;                                    // ring slot of plane z - 1
  for (int z = z0; z < z1; ++z) {
    const int mid = lo == 2 ? 0 : lo + 1, hi = mid == 2 ? 0 : mid + 1;
    put(hi, tid, ca, z + 1, na);
    if (two) put(hi, sb, cb, z + 1, nb);
    __syncthreads();
    if (z + 1 < z1) {
      na = load_sender(a, ca, z + 2);
      if (two) nb = load_sender(a, cb, z + 2);
    }
    if (mine) {
      const uint32_t idx = nxy * (uint32_t)z + nx * (uint32_t)y + (uint32_t)x;
      if constexpr (!LAGGED && !ACC) {
        if ((__ldg(v.flags + idx) & (F_INFLOW | F_SOLID)) != F_INFLOW) {
#pragma unroll
          for (int k = 0; k < 3; ++k) a.ups_out[(uint32_t)k * N + idx] = 0.0f;
        }
      }
      // scalar adjoint: the sender at offset (dx, dy, dz) sends to offset -d
      float part[3] = {0.0f, 0.0f, 0.0f};        // one chain per plane
      const int at = (ty + 1) * ADJ_SX + tx + 1;
#pragma unroll
      for (int dz = -1; dz <= 1; ++dz) {
        const float(*R)[ADJ_SENDERS] = ring[dz < 0 ? lo : (dz == 0 ? mid : hi)];
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
          for (int dx = -1; dx <= 1; ++dx) {
            const int s = at + dy * ADJ_SX + dx;
            part[dz + 1] = fmaf(R[1 - dx][s], R[3 + 3 * (1 - dz) + (1 - dy)][s], part[dz + 1]);
          }
      }
      const float gam = (part[0] + part[1]) + part[2];
      a.gam_out[idx] = ACC ? a.gam_out[idx] + gam : gam;
    }
    __syncthreads();                             // plane z - 1's slot is overwritten next
    lo = mid;
  }
}

// Grids of the two passes.
static dim3 pass_a_grid(const BlockView& v) {
  return dim3((unsigned)(((size_t)v.nx * v.ny + ADJ_THREADS - 1) / ADJ_THREADS), (unsigned)v.nz, 1);
}

template <bool WALLS>
static void launch_pass_a_t(const AdjArgs& a, bool open, bool acc, cudaStream_t s) {
  const dim3 grd = pass_a_grid(a.fwd), blk(ADJ_THREADS, 1, 1);
  if (acc) {   // multi-block reverse
    if (open) k_adj_a<true, true, WALLS><<<grd, blk, 0, s>>>(a);
    else k_adj_a<false, true, WALLS><<<grd, blk, 0, s>>>(a);
  } else {
    if (open) k_adj_a<true, false, WALLS><<<grd, blk, 0, s>>>(a);
    else k_adj_a<false, false, WALLS><<<grd, blk, 0, s>>>(a);
  }
}

static void launch_pass_a(const AdjArgs& a, bool open, bool acc, cudaStream_t s) {
  if (a.fwd.walls) launch_pass_a_t<true>(a, open, acc, s);
  else launch_pass_a_t<false>(a, open, acc, s);
}

template <bool ACC>
static void launch_pass_b(const AdjArgs& a, cudaStream_t s) {
  const BlockView& v = a.fwd;
  const unsigned gx = (unsigned)(v.nx + ADJ_BX - 1) / ADJ_BX, gy = (unsigned)(v.ny + ADJ_BY - 1) / ADJ_BY;
  // planes per CTA: the waves of 4 CTAs on each of 152 SMs times the sender planes of a CTA
  int zc = 1;
  size_t best = ~(size_t)0;
  for (int c = 2; c <= 32; ++c) {
    const size_t ctas = (size_t)gx * gy * ((v.nz + c - 1) / c);
    const size_t cost = (ctas + 607) / 608 * (size_t)(c + 2);
    if (cost < best) { best = cost; zc = c; }
  }
  const dim3 grd(gx, gy, (unsigned)((v.nz + zc - 1) / zc)), blk(ADJ_BX, ADJ_BY, 1);
  if (v.rp.adaptive && !v.rp.local) {
    k_adj_lagged<ACC><<<dim3((unsigned)(((size_t)v.nx * v.ny + 255) / 256), (unsigned)v.nz, 1), 256, 0, s>>>(a);
    k_adj_b<ACC, true><<<grd, blk, 0, s>>>(a, zc);
  } else {
    k_adj_b<ACC, false><<<grd, blk, 0, s>>>(a, zc);
  }
}

// dL/du_0 = Ups^0 + (dD^0/du_0)^T Lam^0 with D^0_k = w_k (drho + rho (3 cu + 9/2 cu^2 - 3/2 u^2)).
__global__ void k_adj_init(const float* __restrict__ d0, const float* __restrict__ u0,
                           const uint8_t* __restrict__ flags, const float* __restrict__ lam,
                           const float* __restrict__ ups, float* __restrict__ out, uint32_t N) {
  for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += gridDim.x * blockDim.x) {
    if (flags[idx] & (F_SOLID | F_OBST_WALL)) {   // obstacle voxels start at rest
      out[idx] = out[N + idx] = out[2 * N + idx] = 0.0f;
      continue;
    }
    float drho = 0.0f;
#pragma unroll
    for (int k = 0; k < 27; ++k) drho += d0[(uint32_t)k * N + idx];
    const float rho = 1.0f + drho;
    const float u[3] = {u0[idx], u0[N + idx], u0[2 * N + idx]};
    float gsum[3] = {ups[idx], ups[N + idx], ups[2 * N + idx]};
#pragma unroll
    for (int k = 0; k < 27; ++k) {
      const float c[3] = {(float)cxk(k), (float)cyk(k), (float)czk(k)};
      const float cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2];
      const float l = lam[(uint32_t)k * N + idx] * wk(k) * rho;
#pragma unroll
      for (int a2 = 0; a2 < 3; ++a2) gsum[a2] = fmaf(l, 3.0f * c[a2] + 9.0f * cu * c[a2] - 3.0f * u[a2], gsum[a2]);
    }
    out[idx] = gsum[0];
    out[N + idx] = gsum[1];
    out[2 * N + idx] = gsum[2];
  }
}

// ---------------------------------------------------------------- multi-block reverse

// Adjoint buffers of one time level of a block (27 planes of populations, 3 of velocity, 1 of
// scalar).
struct AdjLevel {
  float* f = nullptr;
  float* u = nullptr;
  float* c = nullptr;
};

// Transpose of one scale mapping (Sec. 3.2): per table entry the forward interpolation is
// recomputed, the adjoint of the mapped node (populations, its velocity, its scalar) goes
// back through the relaxation with keep factor K_hat and then, with the trilinear weights,
// to the source corners at the two time levels (added atomically: corners are shared).  The
// mapped node's adjoint is then cleared, since the mapping overwrote its previous value.
// 32 entries per CTA of four warps: the interpolation and the scatter, 8 corners times 28 values
// (twice between two time levels), are shared by the four warps (values k = w, w + 4, ... of
// every entry, lanes over entries), the transposed relaxation runs on one.  With one thread per
// entry all of it was one chain in a few warps per SM: 31 -> 18.9 us, mean over the mappings of
// blocks of 64^3, 48^3 and 32^3 nodes.
constexpr int VJP_LD = 29;
__global__ void __launch_bounds__(128) k_map_vjp(MapArgs a, AdjLevel dst, AdjLevel lo, AdjLevel hi) {
  __shared__ float sK[32 * VJP_LD], sA[32 * VJP_LD];   // interpolant; adjoints (27: scalar)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  const bool live = e < a.n;
  const MapEntry m = live ? a.table[e] : MapEntry{0u, 0u, 0.0f, 0.0f, 0.0f};
  const bool act = live && !(a.dst_flags[m.dst] & a.skip_mask);
  const uint32_t sN = (uint32_t)a.sN, sy = (uint32_t)a.snx, sz = (uint32_t)a.snx * (uint32_t)a.sny;
  uint32_t sc[8];
  float w[8];
  float wsum = 0.0f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    sc[c] = m.src + (c & 1) + ((c >> 1) & 1) * sy + (c >> 2) * sz;
    const float wc = ((c & 1) ? m.tx : 1.0f - m.tx) * (((c >> 1) & 1) ? m.ty : 1.0f - m.ty) *
                     ((c >> 2) ? m.tz : 1.0f - m.tz);
    w[c] = !act || (__ldg(a.src_flags + sc[c]) & F_SOLID) ? 0.0f : wc;
    wsum += w[c];
  }
  const uint32_t dN = (uint32_t)a.dN, d = m.dst;
  const bool mapped = wsum > 0.0f;
  // the rest state written where every corner is an obstacle depends on nothing
  const bool rest = act && !mapped && a.rest_if_empty;
  const float inv_w = mapped ? 1.0f / wsum : 0.0f;
  const float th = a.theta <= 0.0f ? 0.0f : (a.theta >= 1.0f ? 1.0f : a.theta);
  const float* __restrict__ flo = static_cast<const float*>(a.f_lo);
  const float* __restrict__ fhi = static_cast<const float*>(a.f_hi);
#pragma unroll
  for (int i = 0; i < 7; ++i) {
    const int k = wid + 4 * i;
    float v = 0.0f, adj = 0.0f;
    if (k < 27) {
      if (mapped) {
        float g[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint32_t at = (uint32_t)k * sN + sc[c];
          const float fl = th < 1.0f ? __ldg(flo + at) : 0.0f;
          const float fh = th > 0.0f ? __ldg(fhi + at) : 0.0f;
          g[c] = th > 0.0f ? fmaf(th, fh - fl, fl) : fl;
        }
        adj = dst.f[(uint32_t)k * dN + d];
#pragma unroll
        for (int c = 0; c < 8; ++c) v = fmaf(w[c], g[c], v);
      }
      if (mapped || rest) dst.f[(uint32_t)k * dN + d] = 0.0f;
    } else if (mapped || rest) {
      adj = rest ? 0.0f : dst.c[d];
      dst.c[d] = 0.0f;
    }
    sK[lane * VJP_LD + k] = v * inv_w;
    sA[lane * VJP_LD + k] = adj;
  }
  __syncthreads();
  if (wid == 0 && (mapped || rest)) {
    float ub[3] = {dst.u[d], dst.u[dN + d], dst.u[2 * dN + d]};
    dst.u[d] = dst.u[dN + d] = dst.u[2 * dN + d] = 0.0f;
    if (mapped) {
      float K[27], A[27];
#pragma unroll
      for (int k = 0; k < 27; ++k) {
        K[k] = sK[lane * VJP_LD + k];
        A[k] = sA[lane * VJP_LD + k];
      }
      raw_moments(K);
      const float drho = K[kap(0, 0, 0)];
      const float inv = 1.0f / (1.0f + drho);
      const float ux = K[kap(1, 0, 0)] * inv, uy = K[kap(0, 1, 0)] * inv, uz = K[kap(0, 0, 1)] * inv;
      central_from_raw(K, ux, uy, uz);
      Keep kf;
      kf.nu = a.khat;
      kf.g[0] = kf.g[1] = kf.g[2] = kf.g[3] = 1.0f;
      float kbar[4] = {0.f, 0.f, 0.f, 0.f};
      collide_vjp(K, A, drho, ux, uy, uz, inv, kf, ub, kbar, nullptr, 0.0f, [](float (&)[3]) {});
#pragma unroll
      for (int k = 0; k < 27; ++k) sA[lane * VJP_LD + k] = A[k];   // adjoint of the interpolant
    }
  }
  __syncthreads();
  if (!mapped) return;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float wc = w[c] * inv_w;
    if (wc == 0.0f) continue;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
      const int k = wid + 4 * i;
      const float x = wc * sA[lane * VJP_LD + k];
      float* pl = k < 27 ? lo.f + ((uint32_t)k * sN + sc[c]) : lo.c + sc[c];
      float* ph = k < 27 ? hi.f + ((uint32_t)k * sN + sc[c]) : hi.c + sc[c];
      if (th < 1.0f) atomicAdd(pl, (1.0f - th) * x);
      if (th > 0.0f) atomicAdd(ph, th * x);
    }
  }
}

// Before the transpose of an aligned sub-step (out = al0 f(t_n) + al1 in + al2 step(in), the
// stored velocity recomputed from out): the velocity adjoint is turned into population
// adjoints, the al0 and al1 shares go to the t_n level and to the input level node by node,
// and the al2 share is left in the output level for the step's own transpose (whose stored
// velocity was not kept).  Obstacle, inflow and ghost nodes are not aligned and are skipped.
// SAME: the t_n level is the input level (a far-field block's step), which takes al0 + al1.
// One node per thread, the loads of nine populations before the first of their stores (one at
// a time the adds of the three levels waited for one another: 31 -> 11.3 us, mean over blocks of
// 48^3 and 32^3 nodes).
template <bool SAME>
__global__ void __launch_bounds__(128) k_align_vjp_pre(BlockView v, AdjLevel out, AdjLevel L,
                                                       AdjLevel in, float al0, float al1, float al2) {
  const uint32_t N = (uint32_t)v.N;
  const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= N || (v.flags[idx] & (F_SOLID | F_INFLOW | F_GHOST))) return;
  const float* __restrict__ D = static_cast<const float*>(v.d_out);
  const float ub[3] = {out.u[idx], out.u[N + idx], out.u[2 * N + idx]};
  float d[27];
#pragma unroll
  for (int k = 0; k < 27; ++k) d[k] = __ldg(D + ((uint32_t)k * N + idx));
  float s, j[3];
  macros(d, s, j[0], j[1], j[2]);
  const float ia = 1.0f / (1.0f + s);
  const float u[3] = {j[0] * ia, j[1] * ia, j[2] * ia};
  const float a1 = SAME ? al0 + al1 : al1;
#pragma unroll
  for (int k0 = 0; k0 < 27; k0 += 9) {
    float lp[9], l0[9], l1[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const uint32_t at = (uint32_t)(k0 + i) * N + idx;
      lp[i] = out.f[at];
      if constexpr (!SAME) l0[i] = L.f[at];
      l1[i] = in.f[at];
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int k = k0 + i;
      const uint32_t at = (uint32_t)k * N + idx;
      const float p = lp[i] + ia * (ub[0] * (cxk(k) - u[0]) + ub[1] * (cyk(k) - u[1]) + ub[2] * (czk(k) - u[2]));
      if constexpr (!SAME) L.f[at] = fmaf(al0, p, l0[i]);
      in.f[at] = fmaf(a1, p, l1[i]);
      out.f[at] = al2 * p;
    }
  }
  out.u[idx] = out.u[N + idx] = out.u[2 * N + idx] = 0.0f;
  const float cb = out.c[idx];
  if constexpr (!SAME) L.c[idx] += al0 * cb;
  in.c[idx] += a1 * cb;
  out.c[idx] = al2 * cb;
}

// Clears the adjoint of the nodes a collide-stream step wrote (all but the ghost nodes).
__global__ void k_zero_stepped(AdjLevel out, const uint8_t* __restrict__ flags, uint32_t N) {
  for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += gridDim.x * blockDim.x) {
    if (flags[idx] & F_GHOST) continue;
#pragma unroll
    for (int k = 0; k < 27; ++k) out.f[(uint32_t)k * N + idx] = 0.0f;
    out.u[idx] = out.u[N + idx] = out.u[2 * N + idx] = 0.0f;
    out.c[idx] = 0.0f;
  }
}

// The inflow velocity of a node is its stored velocity, carried unchanged from step to step
// and set with u_0, so the gradient with respect to it is dL/du_0 at inflow nodes.
__global__ void k_inflow_grad(const float* __restrict__ du0, const uint8_t* __restrict__ flags,
                              float* __restrict__ out, uint32_t N) {
  for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += gridDim.x * blockDim.x) {
    const bool in = (flags[idx] & (F_INFLOW | F_SOLID)) == F_INFLOW;
    out[idx] = in ? du0[idx] : 0.0f;
    out[N + idx] = in ? du0[N + idx] : 0.0f;
    out[2 * N + idx] = in ? du0[2 * N + idx] : 0.0f;
  }
}

struct TapeState {
  int every = 0;
  std::vector<Level> ckpt;    // states at steps 0, every, 2 every, ...
  std::vector<Level> seg;     // recompute levels 1..every of one segment
  std::vector<void*> buffers;       // device memory of everything below (tape_buffer)
  std::vector<long long> changed;   // step counts at which the caller wrote into the live state
  float* lam[2] = {nullptr, nullptr};
  float* ups[2] = {nullptr, nullptr};
  float* gam[2] = {nullptr, nullptr};
  float* ms = nullptr;
  float* side = nullptr;      // clamped pulls of open faces (all zeros between launches)
  // continuous-scale domains (several blocks)
  bool multi = false;
  std::vector<std::vector<Level>> mck;        // [checkpoint][block]: state at the step start
  std::vector<std::vector<Level>> snap;       // [step of the segment][block]
  std::vector<std::vector<Level>> ver;        // [block]: versions 1.. of the block's levels (MsOp)
  std::vector<Level> spare;                   // [block]: a plain step's result (aligned steps)
  std::vector<std::vector<AdjLevel>> lamb;    // [block][level]: adjoints of the replay levels
  std::vector<float*> grad;                   // [block]: dL/du_0 of the block
};

}  // namespace lbm

using namespace lbm;

// A tape's memory goes back with the tape (the next lbm_init_macro or lbm_set_tape), in few pieces: a
// level, or all that one reverse sweep works on, is one allocation, since a call into the caller's
// allocator takes about 2 us of host time (three arrays a level were 26 allocations and as many
// releases per gradient of a 12-step plume, about 100 us of 1850).
void release_tape(lbm_domain* dom) {
  TapeState* t = dom->tape;
  if (!t) return;
  for (void* p : t->buffers) dom->dev_free(p);
  delete t;
  dom->tape = nullptr;
}

// FP32 arrays one after another in a buffer, each from a 256-byte boundary on.
struct Carve {
  float* base = nullptr;     // null: only adds up the size
  size_t floats = 0;
  float* take(size_t n) {
    float* p = base ? base + floats : nullptr;
    floats += (n + 63) / 64 * 64;
    return p;
  }
  Level level(size_t N) {
    Level L;
    L.f = take(27 * N);
    L.u = take(3 * N);
    L.c = take(N);
    return L;
  }
};

// One allocation of the tape for the arrays that layout(Carve&) takes; false (and the arrays
// null) when there is no memory.
template <typename Layout>
static bool tape_buffer(lbm_domain* dom, const Layout& layout) {
  Carve size;
  layout(size);
  Carve place;
  place.base = static_cast<float*>(dom->dev_alloc(size.floats * sizeof(float)));
  if (!place.base) return false;
  dom->tape->buffers.push_back(place.base);
  layout(place);
  return true;
}

void tape_state_changed(lbm_domain* dom) {
  TapeState* t = dom->tape;
  if (t && (t->changed.empty() || t->changed.back() != dom->steps)) t->changed.push_back(dom->steps);
}

static BlockView view_of(lbm_domain* dom, const Level& from, const Level& to) {
  BlockView v = dom->view(0, 0, 0);
  v.d_in = from.f;
  v.u_in = from.u;
  v.c_in = from.c;
  v.d_out = to.f;
  v.u_out = to.u;
  v.c_out = to.c;
  return v;
}

// Copies or clears several arrays of floats in one launch: a level is three arrays, a state one
// level per block.  Bound by DRAM for large levels, by the launches for small ones: three
// blocks of 64^3, 48^3, 32^3 took 49 copies and 49 memsets per rollout and gradient of two
// steps, 268 us of device time and a call each on the host (now 19 launches, 160 us; 2755 ->
// 2471 us as a whole).  One grid row per array, four 16-byte words in flight per thread (arrays
// off 16 bytes: one float at a time).
struct Pieces {
  static constexpr int MAX = 12;
  float* dst[MAX];
  const float* src[MAX];       // null: clear
  size_t n[MAX];
};

__global__ void __launch_bounds__(256) k_pieces(Pieces p) {
  float* __restrict__ dst = p.dst[blockIdx.y];
  const float* __restrict__ src = p.src[blockIdx.y];
  const size_t n = p.n[blockIdx.y];
  const size_t i0 = blockIdx.x * (size_t)256 + threadIdx.x, T = gridDim.x * (size_t)256;
  const bool wide = ((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src)) & 15) == 0;
  const size_t n4 = wide ? n / 4 : 0;
  float4* __restrict__ d4 = reinterpret_cast<float4*>(dst);
  const float4* __restrict__ s4 = reinterpret_cast<const float4*>(src);
  for (size_t i = i0; i < n4; i += 4 * T) {
    float4 x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      x[j] = src && i + j * T < n4 ? __ldg(s4 + i + j * T) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i + j * T < n4) d4[i + j * T] = x[j];
  }
  for (size_t i = 4 * n4 + i0; i < n; i += T) dst[i] = src ? src[i] : 0.0f;
}

struct PieceList {             // collects pieces and launches them MAX at a time
  Pieces p{};
  int count = 0;
  cudaStream_t s;
  cudaError_t e = cudaSuccess;
  explicit PieceList(cudaStream_t stream) : s(stream) {}
  void add(float* dst, const float* src, size_t n) {
    if (count == Pieces::MAX) flush();
    p.dst[count] = dst;
    p.src[count] = src;
    p.n[count++] = n;
  }
  void level(const Level& D, const Level& S, size_t N) {
    add(static_cast<float*>(D.f), static_cast<const float*>(S.f), 27 * N);
    add(D.u, S.u, 3 * N);
    add(D.c, S.c, N);
  }
  cudaError_t flush() {
    if (count == 0 || e != cudaSuccess) return e;
    size_t n = 1;
    for (int i = 0; i < count; ++i) n = std::max(n, p.n[i]);
    const size_t ctas = std::min<size_t>((n + 4095) / 4096, (size_t)152 * 8);
    k_pieces<<<dim3((unsigned)ctas, (unsigned)count), 256, 0, s>>>(p);
    count = 0;
    return e = cudaGetLastError();
  }
};

static cudaError_t copy_level(const Level& D, const Level& S, size_t N, cudaStream_t s) {
  PieceList list(s);
  list.level(D, S, N);
  return list.flush();
}

// FP16-shifted storage keeps the deviations d = f - w in half precision; a checkpoint holds
// them widened (exactly) to FP32, and the segment replays and transposes run on FP32 levels.
__global__ void k_widen(const __half* __restrict__ in, float* __restrict__ out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    out[i] = __half2float(in[i]);
}

// Records a checkpoint of the current state every `every` steps since the last init.
lbm_status tape_before_step(lbm_domain* dom) {
  TapeState* t = dom->tape;
  if (!t) return LBM_OK;
  if (dom->steps % t->every != 0) return LBM_OK;
  const size_t i = (size_t)(dom->steps / t->every);
  if (t->multi) {    // every block's state at the step start
    while (t->mck.size() <= i) {
      std::vector<Level> v(dom->blocks.size());
      if (!tape_buffer(dom, [&](Carve& m) {
            for (size_t b = 0; b < v.size(); ++b) v[b] = m.level(dom->blocks[b].N);
          }))
        return dom->fail(LBM_ERR_OOM, "checkpoint allocation failed");
      t->mck.push_back(v);
    }
    PieceList list(dom->stream);
    for (size_t b = 0; b < dom->blocks.size(); ++b) {
      const Block& B = dom->blocks[b];
      list.level(t->mck[i][b], B.lv[B.cur], B.N);
    }
    const cudaError_t e = list.flush();
    if (e != cudaSuccess) return dom->cuda_fail(e, "checkpoint copy");
    return LBM_OK;
  }
  Block& B = dom->blocks[0];
  while (t->ckpt.size() <= i) {
    Level L;
    if (!tape_buffer(dom, [&](Carve& m) { L = m.level(B.N); }))
      return dom->fail(LBM_ERR_OOM, "checkpoint allocation failed");
    t->ckpt.push_back(L);
  }
  const Level& S = B.lv[B.cur];
  Level& D = t->ckpt[i];
  cudaError_t e;
  if (dom->desc.storage == LBM_FP16_SHIFTED) {
    const size_t n = B.N * 27;
    const int grid = (int)std::min<size_t>((n + 255) / 256, (size_t)152 * 16);
    k_widen<<<grid, 256, 0, dom->stream>>>(static_cast<const __half*>(S.f),
                                           static_cast<float*>(D.f), n);
    e = cudaGetLastError();
    PieceList list(dom->stream);
    list.add(D.u, S.u, 3 * B.N);
    list.add(D.c, S.c, B.N);
    if (e == cudaSuccess) e = list.flush();
  } else {
    e = copy_level(D, S, B.N, dom->stream);
  }
  if (e != cudaSuccess) return dom->cuda_fail(e, "checkpoint copy");
  return LBM_OK;
}

static lbm_status adjoint_supported(lbm_domain* dom) {
  const Block& B = dom->blocks[0];
  if (B.nx < 3 || B.ny < 3 || B.nz < 3) return dom->fail(LBM_ERR_UNSUPPORTED, "the adjoint needs >= 3 nodes per axis");
  if (27ull * B.N >= 0xFFFFFFFFull) return dom->fail(LBM_ERR_UNSUPPORTED, "block too large for the adjoint");
  if (dom->blocks.size() > 1 && (dom->walls & WALLS_OBSTACLES))
    return dom->fail(LBM_ERR_UNSUPPORTED, "the adjoint of obstacle-surface walls covers single-block domains");
  return LBM_OK;
}

extern "C" lbm_status lbm_set_tape(lbm_domain* dom, int32_t every) {
  if (!dom) return LBM_ERR_INVALID_ARG;
  cudaSetDevice(dom->desc.device);
  if (every < 0) return dom->fail(LBM_ERR_INVALID_ARG, "checkpoint_every must be >= 0");
  release_tape(dom);
  if (every == 0) return LBM_OK;
  if (dom->steps != 0)
    return dom->fail(LBM_ERR_STATE, "the tape must be enabled right after lbm_init_macro");
  lbm_status st = adjoint_supported(dom);
  if (st != LBM_OK) return st;
  dom->tape = new TapeState();
  dom->tape->every = every;
  dom->tape->multi = dom->blocks.size() > 1;
  dom->invalidate_graphs();
  return LBM_OK;
}

// One operation of the Algorithm 1 schedule of a continuous-scale domain, on replay levels
// numbered from a canonical start (every block's state at t_n in level 0).  The adjoints live
// on these levels.  The values an operation reads and writes have versions (v_...): a step
// writes a version of its own, a mapping into a version that the reverse sweep still needs
// first copies it (copy_from), so after one replay of a reference step every operation's inputs
// are there to reverse it.  Version 0 of a block is its state at t_n.
struct MsOp {
  int kind = 0;                       // 0 collide-stream, 1 aligned collide-stream, 2 mapping
  int b = 0, in = 0, out = 0, al = 0; // block and levels of a (aligned) collide-stream
  float al0 = 0.f, al1 = 0.f, al2 = 0.f;
  const MapTable* t = nullptr;        // mapping: table, source block / levels, destination
  int src = 0, lo = 0, hi = 0, dst = 0, dlv = 0;
  float theta = 0.f;
  uint8_t skip = 0;
  bool opens = false;                 // a scale boundary written before the step into its level
  int v_in = 0, v_out = 0, v_al = 0, v_lo = 0, v_hi = 0, v_dst = 0, copy_from = -1;
};

// Versions of the operations' values; versions[b] receives the number of block b's versions,
// last[b] the one holding its state at the end of the step.
static void ms_versions(std::vector<MsOp>& ops, const std::vector<int>& cur_end,
                        std::vector<int>& versions, std::vector<int>& last) {
  const int nb = (int)cur_end.size();
  versions.assign(nb, 1);
  std::vector<std::vector<int>> at(nb, std::vector<int>{0, -1, -1});   // [block][level]
  std::vector<std::vector<char>> needed(nb, std::vector<char>{1});     // [block][version]
  std::vector<char> open(nb, 0);       // the level's version was opened by its scale boundary
  auto fresh = [&](int b, int level) {
    needed[b].push_back(0);
    return at[b][level] = versions[b]++;
  };
  for (MsOp& o : ops) {
    if (o.kind != 2) {
      o.v_in = at[o.b][o.in];
      if (o.kind == 1) o.v_al = at[o.b][o.al];
      needed[o.b][o.v_in] = 1;
      if (o.kind == 1) needed[o.b][o.v_al] = 1;
      o.v_out = open[o.b] ? at[o.b][o.out] : fresh(o.b, o.out);
      open[o.b] = 0;
      needed[o.b][o.v_out] = 1;        // its velocity (and an aligned step's populations)
      continue;
    }
    o.v_lo = at[o.src][o.lo];
    o.v_hi = at[o.src][o.hi];
    needed[o.src][o.v_lo] = needed[o.src][o.v_hi] = 1;
    if (o.opens) {
      o.v_dst = fresh(o.dst, o.dlv);
      open[o.dst] = 1;
      continue;
    }
    o.v_dst = at[o.dst][o.dlv];
    // (the scale boundary at t_n, into version 0, is written before anything reads it and
    // comes out the same on every replay)
    const bool refresh = o.v_dst == 0;
    if (needed[o.dst][o.v_dst] && !refresh) {
      o.copy_from = o.v_dst;
      o.v_dst = fresh(o.dst, o.dlv);
    }
  }
  last.resize(nb);
  for (int b = 0; b < nb; ++b) last[b] = at[b][cur_end[b]];
}

// The operations of one reference step in the order multiscale_step issues them (its forked
// mappings write nodes disjoint from the concurrent collide-stream, so this sequential order
// computes the same values); `cur` receives every block's level at the end of the step.
static std::vector<MsOp> ms_ops(const lbm_domain* dom, std::vector<int>& cur) {
  const int nb = (int)dom->blocks.size();
  cur.assign(nb, 0);
  std::vector<int> saved(nb, 0);
  std::vector<MsOp> ops;
  MsOp s0;
  s0.kind = 0; s0.b = 0; s0.in = 0; s0.out = 1;
  ops.push_back(s0);
  cur[0] = 1;
  // far-field blocks (Sec. 4.2.4-4.2.5): their aligned steps, then inner to outer the nodes
  // inside each child's interior from the child, then outer to inner each child's outer
  // layer from its far block (the refined blocks' operations below read only levels these
  // leave alone, so the sequential order computes the forward's values)
  std::vector<int> far;
  for (int b = 1; b < nb; ++b)
    if (dom->blocks[b].far) far.push_back(b);
  for (int f : far) {
    const Block& F = dom->blocks[f];
    MsOp s;
    s.kind = 1; s.b = f; s.in = 0; s.out = 1; s.al = 0;
    s.al0 = 0.0f;
    s.al1 = (float)(1.0 - 1.0 / F.h);
    s.al2 = (float)(1.0 / F.h);
    ops.push_back(s);
    cur[f] = 1;
  }
  for (int f : far) {
    const MapTable& t = dom->blocks[f].far_in;
    MsOp m;
    m.kind = 2; m.t = &t; m.src = t.src; m.lo = m.hi = cur[t.src]; m.theta = 0.0f;
    m.dst = f; m.dlv = cur[f]; m.skip = F_SOLID | F_GHOST;
    ops.push_back(m);
  }
  for (size_t k = far.size(); k-- > 0;) {
    const MapTable& t = dom->blocks[far[k]].far_out;
    MsOp m;
    m.kind = 2; m.t = &t; m.src = far[k]; m.lo = m.hi = cur[far[k]]; m.theta = 0.0f;
    m.dst = t.dst; m.dlv = cur[t.dst]; m.skip = F_SOLID | F_INFLOW;
    ops.push_back(m);
  }
  for (int b = 1; b < nb; ++b) {
    const Block& B = dom->blocks[b];
    if (B.far) continue;
    const int P = B.prior.src, L = 0, A = 1, Bv = 2;
    const bool exact = B.integer_ratio && std::fabs(B.substeps * B.h - 1.0) < 1e-9;
    auto prior = [&](float theta, int dlv) {
      MsOp m;
      m.kind = 2; m.t = &B.prior; m.src = P; m.lo = saved[P]; m.hi = cur[P]; m.theta = theta;
      m.dst = b; m.dlv = dlv; m.skip = F_SOLID;
      return m;
    };
    ops.push_back(prior(0.0f, L));
    int c = L;
    for (int j = 1; j <= B.substeps; ++j) {
      const int out = (j == 1) ? A : (c == A ? Bv : A);
      ops.push_back(prior(j < B.substeps ? (float)(j * B.h) : 1.0f, out));
      ops.back().opens = true;
      MsOp s;
      s.b = b; s.in = c; s.out = out;
      if (j == B.substeps && !exact) {
        const double t1 = (B.substeps - 1) * B.h, t2 = B.substeps * B.h, T = 1.0;
        s.kind = 1; s.al = L;
        s.al0 = (float)((T - t1) * (T - t2) / ((0.0 - t1) * (0.0 - t2)));
        s.al1 = (float)((T - 0.0) * (T - t2) / ((t1 - 0.0) * (t1 - t2)));
        s.al2 = (float)((T - 0.0) * (T - t1) / ((t2 - 0.0) * (t2 - t1)));
      }
      ops.push_back(s);
      c = out;
    }
    cur[b] = c;
    for (const MapTable& t : B.post) {
      MsOp m;
      m.kind = 2; m.t = &t; m.src = b; m.lo = m.hi = cur[b]; m.theta = 0.0f;
      m.dst = t.dst; m.dlv = cur[t.dst]; m.skip = F_SOLID | F_GHOST;
      ops.push_back(m);
    }
  }
  return ops;
}

// The values of one reference step: `start` holds every block's version 0.
struct MsStep {
  lbm_domain* dom;
  TapeState* t;
  std::vector<Level>* start;
  const Level& at(int b, int version) const {
    return version == 0 ? (*start)[b] : t->ver[b][version - 1];
  }
  BlockView view(int b, const Level& F, const Level& T) const {
    BlockView v = dom->view(b, 0, 0);   // geometry, flags, rates, error word
    v.d_in = F.f; v.u_in = F.u; v.c_in = F.c;
    v.d_out = T.f; v.u_out = T.u; v.c_out = T.c;
    return v;
  }
  MapArgs map_args(const MsOp& o) const {
    const Block& S = dom->blocks[o.src];
    const Block& D = dom->blocks[o.dst];
    const Level &lo = at(o.src, o.v_lo), &hi = at(o.src, o.v_hi), &to = at(o.dst, o.v_dst);
    MapArgs a{};
    a.table = o.t->d;
    a.n = o.t->n;
    a.f_lo = lo.f;
    a.f_hi = hi.f;
    a.c_lo = lo.c;
    a.c_hi = hi.c;
    a.theta = o.theta;
    a.src_flags = S.flags;
    a.snx = S.nx; a.sny = S.ny; a.snz = S.nz; a.sN = S.N;
    a.f_dst = to.f;
    a.u_dst = to.u;
    a.c_dst = to.c;
    a.dst_flags = D.flags;
    a.skip_mask = o.skip;
    a.dN = D.N;
    a.khat = o.t->khat;
    a.rest_if_empty = (o.skip & F_GHOST) ? 0 : 1;   // prior maps write scale boundaries
    return a;
  }
};

static cudaError_t ms_forward_op(const MsStep& m, const MsOp& o, cudaStream_t s) {
  if (o.kind == 2) {
    if (o.copy_from >= 0) {
      const cudaError_t e = copy_level(m.at(o.dst, o.v_dst), m.at(o.dst, o.copy_from),
                                       m.dom->blocks[o.dst].N, s);
      if (e != cudaSuccess) return e;
    }
    return launch_map(m.map_args(o), ST_FP32, s);
  }
  const Block& B = m.dom->blocks[o.b];
  BlockView v = m.view(o.b, m.at(o.b, o.v_in), m.at(o.b, o.v_out));
  if (o.kind == 1) {
    const Level& al = m.at(o.b, o.v_al);
    v.f_al0 = al.f;
    v.c_al0 = al.c;
    v.al0 = o.al0; v.al1 = o.al1; v.al2 = o.al2;
    return launch_step_align(v, B.bx, B.by, s, B.minb);
  }
  return launch_step(v, ST_FP32, B.bx, B.by, s, B.minb);
}

// Transpose of one operation, with its forward values in their versions.
static cudaError_t ms_reverse_op(const MsStep& m, const MsOp& o, cudaStream_t s) {
  lbm_domain* dom = m.dom;
  TapeState* t = m.t;
  if (o.kind == 2) {
    const MapArgs a = m.map_args(o);
    if (a.n > 0)
      k_map_vjp<<<(a.n + 31) / 32, 128, 0, s>>>(a, t->lamb[o.dst][o.dlv], t->lamb[o.src][o.lo],
                                                    t->lamb[o.src][o.hi]);
    return cudaGetLastError();
  }
  const Block& B = dom->blocks[o.b];
  const uint32_t N = (uint32_t)B.N;
  const int g = (int)std::min<size_t>((B.N + 255) / 256, 16384);
  AdjLevel lin = t->lamb[o.b][o.in], lout = t->lamb[o.b][o.out];
  const Level &in = m.at(o.b, o.v_in), &out = m.at(o.b, o.v_out);
  const float* u_next = out.u;
  if (o.kind == 1) {
    // the sub-step's own velocity (the scalar's departure velocity) is not stored by an
    // aligned step: recompute the plain step into the spare level
    const Level& spare = t->spare[o.b];
    cudaError_t e = launch_step(m.view(o.b, in, spare), ST_FP32, B.bx, B.by, s, B.minb);
    if (e != cudaSuccess) return e;
    u_next = spare.u;
    const BlockView v = m.view(o.b, out, out);
    const unsigned ga = (unsigned)((B.N + 127) / 128);
    if (o.al == o.in)
      k_align_vjp_pre<true><<<ga, 128, 0, s>>>(v, lout, lin, lin, o.al0, o.al1, o.al2);
    else
      k_align_vjp_pre<false><<<ga, 128, 0, s>>>(v, lout, t->lamb[o.b][o.al], lin, o.al0, o.al1, o.al2);
  }
  AdjArgs a;
  a.fwd = m.view(o.b, in, in);
  a.lam_in = lout.f; a.ups_in = lout.u; a.gam_in = lout.c;
  a.u_next = u_next;
  a.lam_out = lin.f; a.ups_out = lin.u; a.gam_out = lin.c;
  a.ms = t->ms;
  a.side = t->side;
  const bool open = o.b != 0 || !dom->desc.periodic[0] || !dom->desc.periodic[1] || !dom->desc.periodic[2];
  launch_pass_a(a, open, true, s);
  if (open) launch_face_gather(lin.f, t->side, nullptr, a.fwd, s);
  launch_pass_b<true>(a, s);
  k_zero_stepped<<<g, 256, 0, s>>>(lout, B.flags, N);
  return cudaGetLastError();
}

// The buffers of a reverse sweep over blocks with `versions` value versions each, all of them or
// (a failed allocation) none.
static lbm_status alloc_sweep(lbm_domain* dom, TapeState* t, const std::vector<int>& versions) {
  const int nb = (int)dom->blocks.size();
  size_t nmax = 0, side = 0;
  for (const Block& B : dom->blocks) {
    nmax = std::max(nmax, B.N);
    side = std::max(side, face_side_floats(B.nx, B.ny, B.nz));
  }
  t->ver.resize(nb);
  t->spare.resize(nb);
  t->lamb.resize(nb);
  t->grad.resize(nb);
  for (int b = 0; b < nb; ++b) {
    t->ver[b].resize(versions[b] - 1);
    t->lamb[b].resize(b == 0 ? 2 : 3);
  }
  const bool ok = tape_buffer(dom, [&](Carve& m) {
    for (int b = 0; b < nb; ++b) {
      const size_t N = dom->blocks[b].N;
      for (Level& L : t->ver[b]) L = m.level(N);
      if (b) t->spare[b] = m.level(N);
      for (AdjLevel& A : t->lamb[b]) A = AdjLevel{m.take(27 * N), m.take(3 * N), m.take(N)};
      t->grad[b] = m.take(3 * N);
    }
    t->ms = m.take(nmax);
    t->side = m.take(side);
  });
  cudaError_t e = cudaSuccess;
  if (ok) {
    PieceList zero(dom->stream);
    // (a scale boundary that no one has written yet is read with weight 0: keep it finite)
    for (int b = 0; b < nb; ++b)
      for (Level& L : t->ver[b]) zero.level(L, Level{}, dom->blocks[b].N);
    zero.add(t->side, nullptr, side);
    e = zero.flush();
    if (e == cudaSuccess) return LBM_OK;
  }
  t->ver.clear();
  t->spare.clear();
  t->lamb.clear();
  t->grad.clear();
  return ok ? dom->cuda_fail(e, "adjoint buffers") : dom->fail(LBM_ERR_OOM, "adjoint buffers");
}

// Reverse sweep of a continuous-scale domain: the recorded reference steps are reversed last
// to first; each segment between checkpoints is replayed once to record every step's start
// state, and each step once more from there, keeping a version of every value that its
// operations read (MsOp), before the operations are reversed one after another.  (Replaying
// the operations before each one from the step's start would take K (K + 1) / 2 operations and K
// copies of every block for K operations per step, 120 and 48 for a three-block domain of 1/1.5
// and 1/2.25; a domain of 64^3, 48^3 and 32^3 nodes over two steps, that alone: 7.6 -> 3.3 ms.)
static lbm_status adjoint_multiblock(lbm_domain* dom, int n_steps, const float* dL_dc,
                                     const float* dL_du, float* dL_du0, float* dL_dinflow) {
  TapeState* t = dom->tape;
  cudaStream_t s = dom->stream;
  const int nb = (int)dom->blocks.size();
  std::vector<int> cur_end, versions, last;
  std::vector<MsOp> ops = ms_ops(dom, cur_end);
  ms_versions(ops, cur_end, versions, last);
  if (t->lamb.empty()) {
    const lbm_status st = alloc_sweep(dom, t, versions);
    if (st != LBM_OK) return st;
  }
  const int seg_len = std::min(t->every, std::max(1, n_steps));
  while ((int)t->snap.size() < seg_len) {
    std::vector<Level> v(nb);
    if (!tape_buffer(dom, [&](Carve& m) {
          for (int b = 0; b < nb; ++b) v[b] = m.level(dom->blocks[b].N);
        }))
      return dom->fail(LBM_ERR_OOM, "adjoint step snapshots");
    t->snap.push_back(v);
  }
  if (t->mck.empty()) {
    lbm_status st = tape_before_step(dom);
    if (st != LBM_OK) return st;
  }
  PieceList start(s);
  for (int b = 0; b < nb; ++b)
    for (const AdjLevel& A : t->lamb[b]) start.level(Level{A.f, A.u, A.c}, Level{}, dom->blocks[b].N);
  cudaError_t e = start.flush();
  // the loss depends on the reference block's final scalar (and velocity)
  const size_t N0 = dom->blocks[0].N;
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(t->lamb[0][cur_end[0]].c, dL_dc, N0 * sizeof(float), cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && dL_du)
    e = cudaMemcpyAsync(t->lamb[0][cur_end[0]].u, dL_du, N0 * 3 * sizeof(float), cudaMemcpyDeviceToDevice, s);
  if (e != cudaSuccess) return dom->cuda_fail(e, "adjoint initialisation");

  const int n_seg = (n_steps + t->every - 1) / t->every;
  for (int sg = n_seg - 1; sg >= 0 && e == cudaSuccess; --sg) {
    const int len = std::min(t->every, n_steps - sg * t->every);
    auto replay = [&](int i) {
      const MsStep m{dom, t, &t->snap[i]};
      cudaError_t e = cudaSuccess;
      for (const MsOp& o : ops)
        if (e == cudaSuccess) e = ms_forward_op(m, o, s);
      return e;
    };
    PieceList first(s);
    for (int b = 0; b < nb; ++b) first.level(t->snap[0][b], t->mck[sg][b], dom->blocks[b].N);
    e = first.flush();
    for (int i = 0; i + 1 < len && e == cudaSuccess; ++i) {
      e = replay(i);
      const MsStep m{dom, t, &t->snap[i]};
      PieceList next(s);
      for (int b = 0; b < nb; ++b) next.level(t->snap[i + 1][b], m.at(b, last[b]), dom->blocks[b].N);
      if (e == cudaSuccess) e = next.flush();
    }
    for (int i = len - 1; i >= 0 && e == cudaSuccess; --i) {
      const MsStep m{dom, t, &t->snap[i]};
      e = replay(i);
      for (int k = (int)ops.size() - 1; k >= 0 && e == cudaSuccess; --k) e = ms_reverse_op(m, ops[k], s);
      // the adjoint of this step's start state is in level 0: it is the adjoint of the end
      // state of the step before, whose replay ends in the levels cur_end
      if (!(sg == 0 && i == 0))
        for (int b = 0; b < nb; ++b) std::swap(t->lamb[b][0], t->lamb[b][cur_end[b]]);
    }
  }
  if (e != cudaSuccess) return dom->cuda_fail(e, "multi-block adjoint");
  for (int b = 0; b < nb; ++b) {
    const Block& B = dom->blocks[b];
    const int g = (int)std::min<size_t>((B.N + 255) / 256, 16384);
    k_adj_init<<<g, 256, 0, s>>>(static_cast<const float*>(t->mck[0][b].f), t->mck[0][b].u, B.flags,
                                 t->lamb[b][0].f, t->lamb[b][0].u, t->grad[b], (uint32_t)B.N);
  }
  e = cudaMemcpyAsync(dL_du0, t->grad[0], N0 * 3 * sizeof(float), cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && dL_dinflow) {
    const int g = (int)std::min<size_t>((N0 + 255) / 256, 16384);
    k_inflow_grad<<<g, 256, 0, s>>>(dL_du0, dom->blocks[0].flags, dL_dinflow, (uint32_t)N0);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return dom->cuda_fail(e, "initial-state adjoint");
  dom->post_error_probe();
  return LBM_OK;
}

extern "C" lbm_status lbm_adjoint_block_grad(lbm_domain* dom, int32_t block_id, float* dL_du0) {
  if (!dom) return LBM_ERR_INVALID_ARG;
  cudaSetDevice(dom->desc.device);
  lbm_status st = dom->check_block(block_id);
  if (st != LBM_OK) return st;
  if (!dL_du0) return dom->fail(LBM_ERR_INVALID_ARG, "null output");
  TapeState* t = dom->tape;
  if (!t || (int)t->grad.size() <= block_id || !t->grad[block_id])
    return dom->fail(LBM_ERR_STATE, "no multi-block reverse sweep has run");
  const size_t N = dom->blocks[block_id].N;
  const cudaError_t e = cudaMemcpyAsync(dL_du0, t->grad[block_id], N * 3 * sizeof(float),
                                        cudaMemcpyDeviceToDevice, dom->stream);
  if (e != cudaSuccess) return dom->cuda_fail(e, "gradient copy");
  return dom->sync_and_check();
}

extern "C" lbm_status lbm_adjoint_step(lbm_domain* dom, int32_t n_steps, const float* dL_dc,
                                       const float* dL_du, float* dL_du0, float* dL_dinflow) {
  if (!dom) return LBM_ERR_INVALID_ARG;
  cudaSetDevice(dom->desc.device);
  TapeState* t = dom->tape;
  if (!t) return dom->fail(LBM_ERR_STATE, "no tape: call lbm_set_tape after lbm_init_macro");
  if (n_steps < 0 || n_steps != dom->steps)
    return dom->fail(LBM_ERR_INVALID_ARG, "n_steps must equal the steps recorded since lbm_init_macro");
  if (!dL_dc || !dL_du0) return dom->fail(LBM_ERR_INVALID_ARG, "dL_dscalar_final and dL_du0 are required");
  if (t->multi) return adjoint_multiblock(dom, n_steps, dL_dc, dL_du, dL_du0, dL_dinflow);
  Block& B = dom->blocks[0];
  const size_t N = B.N;
  cudaStream_t s = dom->stream;
  // buffers
  if (!t->ms) {
    const size_t side = face_side_floats(B.nx, B.ny, B.nz);
    if (!tape_buffer(dom, [&](Carve& m) {
          for (int i = 0; i < 2; ++i) {
            t->lam[i] = m.take(27 * N);
            t->ups[i] = m.take(3 * N);
            t->gam[i] = m.take(N);
          }
          t->ms = m.take(N);
          t->side = m.take(side);
        }))
      return dom->fail(LBM_ERR_OOM, "adjoint buffers");
    const cudaError_t e = cudaMemsetAsync(t->side, 0, side * sizeof(float), s);
    if (e != cudaSuccess) return dom->cuda_fail(e, "adjoint buffers");
  }
  const int n_seg = (n_steps + t->every - 1) / t->every;
  // Steps of segment sg that are replayed.  The last one's result is wanted for its velocity
  // alone, which the forward kept: it is the next checkpoint's, or the domain's current one, bit
  // for bit what the replay computes with FP32 storage.  Not where the caller has written into
  // that state since (inflow records of the next frame, node boxes), and not with FP16 storage,
  // whose replay follows unrounded states: there the replay's own result is taken.
  auto replayed = [&](int sg) {
    const int end = std::min((sg + 1) * t->every, n_steps);
    const bool kept = dom->desc.storage == LBM_FP32 &&
                      std::find(t->changed.begin(), t->changed.end(), (long long)end) == t->changed.end();
    return end - sg * t->every - (kept ? 1 : 0);
  };
  int seg_len = 0;
  for (int sg = 0; sg < n_seg; ++sg) seg_len = std::max(seg_len, replayed(sg));
  // (levels of small blocks share an allocation of at most 256 MB)
  const size_t group = std::max<size_t>(1, ((size_t)256 << 20) / (31 * N * sizeof(float)));
  while ((int)t->seg.size() < seg_len) {
    std::vector<Level> v(std::min(group, (size_t)seg_len - t->seg.size()));
    if (!tape_buffer(dom, [&](Carve& m) {
          for (Level& L : v) L = m.level(N);
        }))
      return dom->fail(LBM_ERR_OOM, "recompute levels");
    t->seg.insert(t->seg.end(), v.begin(), v.end());
  }
  if (t->ckpt.empty()) {  // no step was taken: the checkpoint of step 0 is the current state
    lbm_status st = tape_before_step(dom);
    if (st != LBM_OK) return st;
  }
  int c = 0;
  PieceList start(s);
  start.add(t->lam[0], nullptr, 27 * N);
  start.add(t->lam[1], nullptr, 27 * N);
  if (!dL_du) start.add(t->ups[0], nullptr, 3 * N);
  cudaError_t e = start.flush();
  if (e == cudaSuccess && dL_du)
    e = cudaMemcpyAsync(t->ups[0], dL_du, N * 3 * sizeof(float), cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(t->gam[0], dL_dc, N * sizeof(float), cudaMemcpyDeviceToDevice, s);
  if (e != cudaSuccess) return dom->cuda_fail(e, "adjoint initialisation");

  const bool open_faces = !dom->desc.periodic[0] || !dom->desc.periodic[1] || !dom->desc.periodic[2];
  for (int sg = n_seg - 1; sg >= 0; --sg) {
    const int s0 = sg * t->every;
    const int len = std::min(t->every, n_steps - s0);
    // recompute the segment's states 1..n_replay from its checkpoint
    auto level = [&](int i) -> const Level& { return i == 0 ? t->ckpt[sg] : t->seg[i - 1]; };
    const int n_replay = replayed(sg);
    const float* u_end = n_replay == len ? nullptr : sg == n_seg - 1 ? B.lv[B.cur].u : t->ckpt[sg + 1].u;
    for (int i = 0; i < n_replay; ++i) {
      e = launch_step(view_of(dom, level(i), level(i + 1)), ST_FP32, B.bx, B.by, s, B.minb);
      if (e != cudaSuccess) return dom->cuda_fail(e, "adjoint recompute");
    }
    for (int i = len - 1; i >= 0; --i) {
      AdjArgs a;
      a.fwd = view_of(dom, level(i), level(i));
      a.lam_in = t->lam[c];
      a.ups_in = t->ups[c];
      a.gam_in = t->gam[c];
      a.u_next = i + 1 <= n_replay ? level(i + 1).u : u_end;
      a.lam_out = t->lam[c ^ 1];
      a.ups_out = t->ups[c ^ 1];
      a.gam_out = t->gam[c ^ 1];
      a.ms = t->ms;
      a.side = t->side;
      launch_pass_a(a, open_faces, false, s);
      if (open_faces) launch_face_gather(a.lam_out, t->side, t->lam[c], a.fwd, s);
      launch_pass_b<false>(a, s);
      e = cudaGetLastError();
      if (e != cudaSuccess) return dom->cuda_fail(e, "adjoint step");
      c ^= 1;
    }
  }
  const int g = (int)std::min<size_t>((N + 255) / 256, 16384);
  k_adj_init<<<g, 256, 0, s>>>(static_cast<const float*>(t->ckpt[0].f), t->ckpt[0].u, B.flags,
                               t->lam[c], t->ups[c], dL_du0, (uint32_t)N);
  if (dL_dinflow) k_inflow_grad<<<g, 256, 0, s>>>(dL_du0, B.flags, dL_dinflow, (uint32_t)N);
  e = cudaGetLastError();
  if (e != cudaSuccess) return dom->cuda_fail(e, "initial-state adjoint");
  dom->post_error_probe();
  return LBM_OK;
}
