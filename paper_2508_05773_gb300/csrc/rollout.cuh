// rollout.cuh -- device code of BR-MPPI solves for sm_103a.
//
// Paper: "GPU-Accelerated Barrier-Rate Guided MPPI Control for
// Tractor-Trailer Systems" (arXiv 2508.05773).  One solve (Sec. II-B MPPI
// with the BR-MPPI rollout of Sec. IV-A):
//
//   for each sample s, step tau:
//     noise        Philox4x32-10 + Box-Muller (noise.cuh), recomputed (never
//                  stored in HBM): in registers where it is used, or by
//                  noise warps into shared memory (the latency shapes)
//     sample       z_des = clip(U_nom + sigma n), u^alpha_des = clip(sigma_a n)
//     rows         barrier-rate equality per constraint (Eq. cbf_equality):
//                  hitch (Eq. hitch_angle_barrier) and obstacles
//                  (Eq. barrier_function) through the second-order expansion
//                  of Eq. barrier_function_approx (optionally third order for
//                  obstacles; moving and e = 4 obstacles, footprint discs, the
//                  jerk-input model: the extended instantiations)
//     projection   Eq. closed-form_projection in Woodbury form (below)
//     apply        u = clip(z*_u), alpha += z*_alpha
//     dynamics     explicit Euler (Eq. tt_discrete_kinematics)
//     cost         Eq. cost_function_contour at the new state
//   softmin + update (Eq. MPPI_update_rule) as per-tile partials of a
//   max-subtracted log-sum-exp, merged in tile order by the CTA that
//   finishes an instance's last tile.
//
// Launch model.  A work item is (instance, sample tile); a tile is the
// samples one CTA rolls out together.  A plain solve runs one CTA per tile;
// a batch runs a persistent grid that pulls items from a longest-first list
// with an atomic counter.  Partials are per tile and merged in tile order,
// so a solve gives the same bits alone or inside any batch with the same
// launch shape.
//
// Team decomposition: TPS consecutive lanes own one sample (or two, NS = 2,
// in packed registers).  Every lane of a team computes the hitch row (its
// terms enter the team sums once); the obstacle rows are spread over the team
// (row j on lane j % TPS of the latency shapes, a Philox block's four rows on
// one lane elsewhere), each with its noise normal 4 + j.  The rank-2
// structure of the projection makes the cross-lane exchange five floats per
// step.  The step is written in Vec<NS> (vec.cuh), every rounding explicit: a
// sample has the same bits with one sample a team and with two (of one width,
// both drawing their noise themselves), so a batch may run pairs when it fills
// the GPU and not when it does not.  Other widths, and teams with noise warps, add
// the rows' or the cost's terms in another order.
//
// What bounds it (measured on GB300, before this layout -> with it): the
// throughput shapes are bound by issue slots and the FMA pipe.  48 solves of
// 4096 samples, H = 50, 8 ellipses: 493 -> 387 us, 1359 -> 740 thread
// instructions a rollout-step (packed pairs, table-driven normals, the first
// Philox rounds shared, rows as linear forms in (Q d, Q), no subnormal
// scaling around the MUFU); 256 uneven solves 2567 -> 1802 us; S = 65536,
// H = 100, 64 ellipses 2030 -> 1482 us (FMA pipe 51% and ALU pipe 36% busy,
// 2.8 warps a scheduler).  The latency shapes are bound by one compute
// warp's dependency chain: S = 4096, H = 50, 8 ellipses 39.6 -> 31.7 us.
//
// Projection in Woodbury form.  A = [A_u | diag(h~)] where only the a and
// omega columns of A_u are non-zero, M = diag(m_u, m_alpha):
//   K = A M^-1 A^T = D + A_u M_u^-1 A_u^T,  D = diag(h~^2 / m_alpha),
//   S2 = M_u + A_u^T D^-1 A_u (2x2),  g = A_u^T D^-1 r,  y = S2^-1 g,
//   r  = A M^-1 p - b,  lambda = D^-1 (r - A_u y),
//   z*_u = M_u^-1 p_u - y,  z*_alpha_i = p_alpha_i/m_alpha - (r_i - a_i.y)/h~_i,
// algebraically identical to M^-1 [p - A^T K^-1 (A M^-1 p - b)].  With
// u_i = a_i / h~_i and rho_i = r_i / h~_i (one reciprocal per row):
//   S2 = M_u + m_alpha sum u_i u_i^T,  g = m_alpha sum u_i rho_i,
// so the rows accumulate the sums and m_alpha is applied once.
//
// Numerics: states are carried in the frame of the initial pose (position
// along and across the initial heading, angles and progress relative to it)
// so that binary32 rounding is relative to the few metres a rollout travels;
// position, speed, progress and the cost sum are compensated pairs (TwoSum),
// the path table holds low parts; the softmin works on pair differences.
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>
#include <math_constants.h>

#include "noise.cuh"
#include "trig.cuh"
#include "vec.cuh"

namespace brmppi {

// ------------------------------------------------------------ descriptors
// Method constants shared by every instance of a launch.
struct KConst {
  int proj;
  int coll, obs8, abuf;  // collision cost, moving / e = 4 obstacle rows, buffer cost
  float Ts, hTs2, Ts2, inv_lambda;  // Ts, Ts^2 / 2, Ts^2
  float inv_l1, inv_l2, k_hitch, dtheta_max, kappa, r_inflate;
  float Qc, Ql, Qth, R0, R1, R2, mu, nu_bar;
  int iso;         // Qc == Ql: the contouring cost needs no path direction
  float khl2;      // k_hitch / l2
  float zlo0, zlo1, zlo2, zhi0, zhi1, zhi2;
  float alpha0;
  // sampled inputs in the projection's coordinates, M_u^-1 p_u = clip(qa
  // U_nom + qb + qs n, qlo, qhi) with qa = W_u / M_u, qb = rho (hi + lo) /
  // (2 M_u) (without the projection qa = 1, qb = 0), and p_alpha / m_alpha =
  // clip(ps n + pc_am, pam_lo, pam_hi)
  float qa[3], qb[3], qs[3], qlo[3], qhi[3];
  float ps, pc_am, pam_lo, pam_hi;
  float m_u0, m_u1, m_a;  // M_u = W_u + rho, m_alpha = W_alpha + rho
  float h_floor;
  float q_coll, q_abuf, inv_hbuf;
  float alpha_stab, inv_qs0, inv_qs1;  // hitch stabilizer: CBF rate, Q_h^-1
  int nd, discs;                       // footprint discs; non-default footprint
  int third;                           // obstacle rows to third order (rear-axle point only)
  int jerk;                            // jerk-input model: a is a state (x0[7]), input 0 the jerk
  float Ts3_6;                         // Ts^3 / 6
  float inv_nd;
  float disc_e1[8], disc_e2[8];        // disc m at p + disc_e1[m] e1 + disc_e2[m] e2
};

// One solve of a launch (all pointers device memory).
struct Inst {
  const double* x0;
  const float* U_nom;
  const float* obs;
  const float* path;
  float* U_out;
  float* traj_out;   // may be null
  float* J_out;      // may be null
  float* U_next;     // may be null
  int32_t* status;   // may be null
  float* states_out;  // may be null: every sample's states, S x (H+1) x 7
  float* u_safe;      // may be null: stabilized U*[0] (a, omega, nu, slack), written
                      // by the stabilizer launch that follows the solve
  float* inputs_out;  // may be null: every sample's applied inputs, S x H x 3
  float* J_lo_out;    // may be null: low parts of the compensated costs (J_out the high parts)
  float* part;       // tiles * part_stride floats
  unsigned int* sync;  // [0] finished tiles, [1] error bits
  int S, H, n_obs, n_pts, tiles, part_stride;
  float ds, inv_ds, inv_ds_l;  // 1 / ds and its low part
  double inv_ds_d;   // 1 / ds in FP64 (path cell of psi0)
  uint32_t key0, key1, ctr;
  int P;             // Philox blocks per step, ceil((4 + n_obs) / 4)
  int tile_base;     // single launches: tile index of the first CTA (a rank's share of the tiles)
  int no_merge;      // 1: write the tile partials (at part + (tile - tile_base) * part_stride) and
                     // stop; the instance's tiles are merged by merge_tiles_kernel
};

constexpr int kMaxBlocks = 32;  // Philox blocks a step: 3 inputs, the hitch and at most 124 rows

// Shared-memory capacities of a launch (floats).
// Every region is a multiple of 4 floats (16 bytes): float4 accesses stay
// aligned.
struct SmemCaps {
  int obs, path, unom, ustar;
  int noise_per_team;  // teams wider than one lane: staged normals, 2 steps x P blocks x 4
  int uh_per_team;     // 3 H when the applied-input history stays in shared memory, else 0
  int rows_per_team;   // variants without producer warps: floats of row state a sample
  int merge;           // > 0: room for an instance's tile partials (merged in shared memory)
  __host__ __device__ static int pad4(int n) { return (n + 3) & ~3; }
  __host__ __device__ int total(int spb) const {
    // noise and history, or row state; then the partials
    const int tail = (noise_per_team + rows_per_team) * spb + pad4(uh_per_team * spb);
    return obs + path + unom + ustar + pad4(3 * spb) + 256 + 16 + kNoiseTableFloats + 4 * kMaxBlocks + (tail > merge ? tail : merge);
  }
};

struct LaunchDesc {
  Inst single;          // used when work == nullptr (tile = blockIdx.x)
  const Inst* inst;     // batch: instance table
  const int2* work;     // batch: (instance, tile) items, longest first
  int n_work;
  unsigned int* work_ctr;  // [0] next item, [1] CTAs that ran out of work
  float* uh;            // per-CTA applied-input history: gridDim.x * uh_stride floats
                        // (unused by the exact-rows variants: their history is in shared memory)
  int uh_stride;        // 3 * H_max * samples per CTA
  int noise_warps;      // teams wider than one lane: warps that produce the noise
  int rows;             // > 0: the instantiation with exactly this many rows a lane
  SmemCaps caps;
};

enum : unsigned { ERR_EXPONENT = 1u, ERR_NONFINITE_X0 = 2u, ERR_PATH_TURN = 4u };

// Largest heading change between consecutive path rows (rad): the interface
// refuses wider turns, whose linear interpolation is too coarse to follow (no
// arithmetic below depends on it).
constexpr float kMaxPathTurn = 0.78539816339744831f;  // pi / 4

__device__ __forceinline__ float clampf(float v, float lo, float hi) { return fminf(fmaxf(v, lo), hi); }


// the value held by lane `src` mod TPS of the team
template <int TPS, int N>
__device__ __forceinline__ Vec<N> team_take(Vec<N> v, int src) {
  if constexpr (TPS == 1) return v;
  return vmap(v, [=](float x) { return __shfl_sync(0xffffffffu, x, src & (TPS - 1), TPS); });
}

template <int TPS, int N>
__device__ __forceinline__ Vec<N> team_sum(Vec<N> v) {
#pragma unroll
  for (int m = 1; m < TPS; m <<= 1) v = v + vshfl_xor(v, m);
  return v;
}

// (h, l) pairs: lexicographic order of normalised pairs
__device__ __forceinline__ bool pair_less(float ah, float al, float bh, float bl) {
  return ah < bh || (ah == bh && al < bl);
}

// x = hi + lo with hi = fl(x)
__device__ __forceinline__ void split_double(double x, float& hi, float& lo) {
  hi = static_cast<float>(x);
  lo = static_cast<float>(x - static_cast<double>(hi));
}

// Barrier-rate row of the hitch barrier h = dtheta_max - kappa v - |Delta|,
// Delta = theta2 - theta1 (Eq. hitch_angle_barrier), through the
// second-order expansion of Eq. barrier_function_approx: the increment
// Ts hdot + Ts^2/2 hddot along the field with the input held is
// Aa a + Aw omega + c0 (progress never enters).  sp, cp = sin, cos of
// phi = -Delta; tn = tan(delta).
struct HitchRow {
  float h, Aa, Aw, c0;
};
__device__ __forceinline__ HitchRow hitch_row(const KConst& k, float Delta, float sp, float cp, float tn,
                                              float vv, float th1dot) {
  const float sg = Delta >= 0.f ? 1.f : -1.f;
  const float G = sp - k.k_hitch * cp * tn;
  const float th2dot = vv * G * k.inv_l2;
  const float phidot = th1dot - th2dot;
  const float sec2 = 1.f + tn * tn;
  HitchRow r;
  r.h = k.dtheta_max - k.kappa * vv - sg * Delta;
  r.Aa = -k.Ts * k.kappa - k.hTs2 * sg * (G * k.inv_l2 - tn * k.inv_l1);
  r.Aw = k.hTs2 * sg * vv * sec2 * (k.k_hitch * cp * k.inv_l2 + k.inv_l1);
  r.c0 = -k.Ts * sg * (th2dot - th1dot) - k.hTs2 * sg * vv * k.inv_l2 * (cp + k.k_hitch * tn * sp) * phidot;
  return r;
}

// Hitch-angle stabilizer (Sec. IV-D, Eq. hitch_angle_qp): the (a, omega)
// (jerk-input model: (jerk, omega)) nearest the reference in the diag(q_stab) norm, inside the input box,
// whose hitch increment g.u + c0 meets the discrete CBF condition
// (Eq. barrier_constraint_prelim, sign of Eq. cbf_equality)
//   g.u >= rhs = -alpha_stab h - c0.
// KKT with a diagonal weight and a box: the box projection of the reference
// if it meets the condition; else u(mu) = clip(u_ref + mu Q^-1 g) at the
// mu > 0 where g.u(mu) = rhs.  g.u(mu) is piecewise linear and
// non-decreasing with breaks where a coordinate meets a bound, so the root is
// found exactly on the segment that crosses rhs.  No crossing: the box
// corner that maximises the increment.  out = (a, omega, nu, slack).
__device__ __forceinline__ void hitch_stabilize(const KConst& k, float Delta, float vv, float dl, float acc, float ua,
                                                float uw, float un, float* out) {
  float sp, cp;
  sincosf(-Delta, &sp, &cp);
  const float tn = tanf(dl);
  HitchRow r = hitch_row(k, Delta, sp, cp, tn, vv, vv * tn * k.inv_l1);
  if (k.jerk) {  // jerk-input model: (jerk, omega), the acceleration acc a state
    r.c0 += acc * r.Aa;
    r.Aa = -k.hTs2 * k.kappa;
  }
  const float g0 = r.Aa, g1 = r.Aw;
  const float rhs = -k.alpha_stab * r.h - r.c0;
  float a = clampf(ua, k.zlo0, k.zhi0), w = clampf(uw, k.zlo1, k.zhi1);
  const float f0 = g0 * a + g1 * w;
  if (f0 < rhs) {
    const float d0 = g0 * k.inv_qs0, d1 = g1 * k.inv_qs1;
    // breakpoints: the mu > 0 where a coordinate meets a bound (+inf: none)
    auto brk = [](float ref, float d, float bound) {
      const float m = (bound - ref) / d;
      return (d != 0.f && m > 0.f) ? m : CUDART_INF_F;
    };
    float b0 = brk(ua, d0, k.zlo0), b1 = brk(ua, d0, k.zhi0);
    float b2 = brk(uw, d1, k.zlo1), b3 = brk(uw, d1, k.zhi1);
    auto cswap = [](float& x, float& y) {
      const float lo = fminf(x, y), hi = fmaxf(x, y);
      x = lo;
      y = hi;
    };
    cswap(b0, b1);  // sorting network for four keys
    cswap(b2, b3);
    cswap(b0, b2);
    cswap(b1, b3);
    cswap(b1, b2);
    float m_prev = 0.f, f_prev = f0;
    bool crossed = false;
    const float bs[4] = {b0, b1, b2, b3};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float m = bs[i];
      if (crossed || !(m < CUDART_INF_F)) continue;
      const float f = g0 * clampf(ua + m * d0, k.zlo0, k.zhi0) + g1 * clampf(uw + m * d1, k.zlo1, k.zhi1);
      if (f >= rhs) {
        const float mu = m_prev + (rhs - f_prev) * (m - m_prev) / (f - f_prev);
        a = clampf(ua + mu * d0, k.zlo0, k.zhi0);
        w = clampf(uw + mu * d1, k.zlo1, k.zhi1);
        crossed = true;
      }
      m_prev = m;
      f_prev = f;
    }
    if (!crossed) {
      if (d0 != 0.f) a = d0 > 0.f ? k.zhi0 : k.zlo0;
      if (d1 != 0.f) w = d1 > 0.f ? k.zhi1 : k.zlo1;
    }
  }
  out[0] = a;
  out[1] = w;
  out[2] = un;
  out[3] = (g0 * a + g1 * w) - rhs;
}

// Frame of one solve: origin and heading of the tractor at x0.  Rollouts run
// in it: x along the initial heading, angles relative to it, so neither the
// step nor the cost turns by the initial heading, and the rounding of its cos
// / sin (3e-8, the same at every step, so a drift of the whole rollout) enters
// nowhere.  Doubles of x0 enter as unevaluated float pairs (hi + lo).
struct Frame {
  float ox_h, ox_l, oy_h, oy_l, oth_h, oth_l;  // origin (px0, py0, theta1_0)
  float c0, s0, c0l, s0l;                      // cos / sin of theta1_0, and their low parts
  float t2, v_h, v_l, dl;                      // theta2 - theta1_0, speed, steer angle
  float a0;                                    // acceleration (jerk-input model)
  float qf0;                                   // path cell of psi0 less i0
  int i0;                                      // integer path cell of psi0, within kMaxFirstCell
  float psi_h, psi_l;                          // psi0
  double psi0;
};

// sin and cos of the frame's heading hi + lo as float pairs, to about 2e-9:
// Cody-Waite reduction by pi/2 in three parts, then the Taylor series with its
// leading terms in pairs (one lane a CTA; in FP64 it took 0.4 us).
__device__ __forceinline__ void frame_sincos(float hi, float lo, float* s, float* sl, float* c, float* cl) {
  if (!(fabsf(hi) < 1.0e6f)) {  // (NaN too) a float's accuracy
    sincosf(hi, s, c);
    *sl = *c * lo;
    *cl = -*s * lo;
    return;
  }
  const float k = rintf(hi * 0.636619746685028f);
  const float r0 = __fmaf_rn(-k, 1.5707963705062866f, hi);  // exact
  const float r = __fmaf_rn(k, 4.371138828673793e-08f, r0);
  const float rl = __fmaf_rn(k, 4.371138828673793e-08f, __fsub_rn(r0, r)) + fmaf(k, 1.7151245100058e-15f, lo);
  const float z = __fmul_rn(r, r), zl = __fmaf_rn(r, r, -z);  // of r alone: rl turns the result below
  // sin = r + r w, w = z (-1/6 + z/120 - ...)
  const float A = fmaf(z, fmaf(z, fmaf(z, 2.7557319e-06f, -1.9841270e-04f), 8.3333333e-03f), -0.16666667f);
  const float w = __fmul_rn(z, A), wl = __fmaf_rn(z, A, -w) + zl * A;
  const float p = __fmul_rn(r, w), pl = __fmaf_rn(r, w, -p) + r * wl;
  const float sh = __fadd_rn(r, p), se = __fadd_rn(__fsub_rn(r, sh), p) + pl;  // |r| >= |p|
  // cos = 1 - z/2 + z^2 (1/24 - z/720 + ...)
  const float C = fmaf(z, fmaf(z, fmaf(z, -2.7557319e-07f, 2.4801587e-05f), -1.3888889e-03f), 0.041666667f);
  const float ch = __fmaf_rn(-0.5f, z, 1.f);
  const float ce = __fmaf_rn(-0.5f, z, __fsub_rn(1.f, ch)) + fmaf(z * z, C, -0.5f * zl);
  const float sl_ = fmaf(ch, rl, se), cl_ = fmaf(-sh, rl, ce);
  const float s1 = __fadd_rn(sh, sl_), s1l = __fadd_rn(__fsub_rn(sh, s1), sl_);
  const float c1 = __fadd_rn(ch, cl_), c1l = __fadd_rn(__fsub_rn(ch, c1), cl_);
  const int q = static_cast<int>(k);
  const bool odd = q & 1, sneg = q & 2, cneg = (q + 1) & 2;
  const float ss = odd ? c1 : s1, ssl = odd ? c1l : s1l, cc = odd ? s1 : c1, ccl = odd ? s1l : c1l;
  *s = sneg ? -ss : ss;
  *sl = sneg ? -ssl : ssl;
  *c = cneg ? -cc : cc;
  *cl = cneg ? -ccl : ccl;
}

// Path cells are counted from a reference cell of at most this size, as floats
// within +- 2 kMaxFirstCell (stage_cost): every row of a path (8192 at most) is
// within that range of the reference.
constexpr double kMaxFirstCell = 1.0e6;

// The frame of x0, built by warp 0: lane j takes state component j, so the
// FP64 work runs side by side; the path cell of psi0 uses the host's FP64
// reciprocal of ds (no device division).
__device__ __forceinline__ void make_frame_warp(const double* x0, double inv_ds, unsigned int* err, Frame& fr,
                                                bool jerk) {
  const int lane = threadIdx.x & 31;
  if (lane >= (jerk ? 8 : 7)) {
    if (lane == 7) fr.a0 = 0.f;
    return;
  }
  const double x = x0[lane];
  if (!isfinite(x)) atomicOr(err, ERR_NONFINITE_X0);
  float hi, lo;
  split_double(x, hi, lo);
  switch (lane) {
    case 0: fr.ox_h = hi; fr.ox_l = lo; break;
    case 1: fr.oy_h = hi; fr.oy_l = lo; break;
    case 2: {
      fr.oth_h = hi;
      fr.oth_l = lo;
      frame_sincos(hi, lo, &fr.s0, &fr.s0l, &fr.c0, &fr.c0l);
      break;
    }
    case 3: fr.t2 = static_cast<float>(x - x0[2]); break;
    case 4: fr.v_h = hi; fr.v_l = lo; break;
    case 5: fr.dl = static_cast<float>(x); break;
    case 6: {
      fr.psi0 = x;
      fr.psi_h = hi;
      fr.psi_l = lo;
      const double q0 = x * inv_ds;
      // within the range of stage_cost's cell count, so that a cell on the path
      // is counted from here wherever psi0 is
      const double fq = fmin(fmax(floor(q0), -kMaxFirstCell), kMaxFirstCell);
      fr.i0 = static_cast<int>(fq);
      fr.qf0 = static_cast<float>(q0 - fq);
      break;
    }
    default: fr.a0 = static_cast<float>(x); break;  // lane 7: acceleration (jerk-input model)
  }
}

// Shared memory of a CTA (offsets into the dynamic buffer, floats).
struct Smem {
  float* obs;    // 8 per obstacle.  Plain family (parked ellipses): cx, cy,
                 // Qxx, Qxy, Qyy, 0, 0, 0 (the world-axis quadratic form of
                 // h).  Family with the optional terms: cx, cy, cos, sin, kx,
                 // ky, vx', vy' with k = 1/A^2 (e = 2) or 1/A^4 (e = 4, kx
                 // stored negated) and the velocity in the obstacle frame
                 // (zero unless moving)
  float* path;   // 4 per row: x, y, heading in the frame, low parts of x and y
  float* unom;   // 3H: the nominal inputs in the projection's coordinates
  float* ustar;  // 3H + 1 (merge)
  float* jh;     // spb
  float* jl;     // spb
  float* w;      // spb
  float* chunk;  // 256
  float* disc;   // 16: lever arms (along e1, along e2) of the footprint discs
  float* tab;    // NoiseTables
  uint4* blk;    // kMaxBlocks: the Philox blocks' shared words
  float* noise;  // spb x noise_per_team, then (exact-rows variants) the
                 // applied-input history, 3H x spb
  int noise_per_team;
  __device__ Smem(float* base, const SmemCaps& c, int spb) {
    obs = base;
    path = obs + c.obs;
    unom = path + c.path;
    ustar = unom + c.unom;
    jh = ustar + c.ustar;
    jl = jh + spb;
    w = jl + spb;
    chunk = jh + SmemCaps::pad4(3 * spb);
    disc = chunk + 256;
    tab = disc + 16;
    blk = reinterpret_cast<uint4*>(tab + kNoiseTableFloats);
    noise = tab + kNoiseTableFloats + 4 * kMaxBlocks;
    noise_per_team = c.noise_per_team;
  }
};

struct Shared {
  Frame fr;
  float red_h[2], red_l[2];
  float wred_h[16], wred_l[16];  // per-warp pair minima (merge)
  int item;
  int last;
  unsigned err;  // the instance's error bits (merge)
};

// Asynchronous 4-byte copy global -> shared (cp.async): the copies of a
// loop stay in flight together instead of one load-store round trip each.
__device__ __forceinline__ void cp_async4(float* smem_dst, const float* gmem_src) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gmem_src) : "memory");
}
// 16-byte asynchronous copy global -> shared through L2 (cp.async.cg).
__device__ __forceinline__ void cp_async16(float* smem_dst, const float* gmem_src) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// L2 prefetch of a global address (no value; null-safe).  Issued early for
// the outputs that the last CTA writes at the very end, it takes their
// address translation and line allocation off the solve's tail.
__device__ __forceinline__ void prefetch_l2(const void* p) {
  if (p) asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Barrier of the whole CTA that its roles reach at different places.
__device__ __forceinline__ void staging_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }

// Threads of a CTA that roll out samples: all of them with one lane per
// sample; with wider teams the last noise_warps warps produce the noise.
template <int TPS>
__device__ __forceinline__ int compute_threads(int noise_warps) {
  return static_cast<int>(blockDim.x) - 32 * noise_warps;
}

// Variants whose noise comes from producer warps: wider teams with at most
// two Philox blocks per lane.
template <int TPS, int BPT, int NS>
constexpr bool kNoiseWarps = TPS > 1 && BPT <= 2 && NS == 1;

__device__ __forceinline__ void store_pair(float* d, Vec<1> a) { *d = a.x; }
__device__ __forceinline__ void store_pair(float* d, Vec<2> a) { *reinterpret_cast<float2*>(d) = a.x; }

// (hi, lo) = (x, y) - origin in the frame's axes: c dx + s dy as a float pair
// (for the y axis, called with (dy, -dx)).
__device__ __forceinline__ void frame_axis(const Frame& fr, float dxh, float dxl, float dyh, float dyl, float& hi,
                                           float& lo) {
  const float p = __fmul_rn(fr.c0, dxh), q = __fmul_rn(fr.s0, dyh);
  const float pe = __fmaf_rn(fr.c0, dxh, -p), qe = __fmaf_rn(fr.s0, dyh, -q);
  const float sum = __fadd_rn(p, q), bp = __fsub_rn(sum, p);
  const float se = __fadd_rn(__fsub_rn(p, __fsub_rn(sum, bp)), __fsub_rn(q, bp));
  const float l = (se + (pe + qe)) + fmaf(fr.c0, dxl, fmaf(fr.s0, dyl, fmaf(fr.c0l, dxh, fr.s0l * dyh)));
  hi = __fadd_rn(sum, l);
  lo = __fadd_rn(__fsub_rn(sum, hi), l);
}
// a - (oh + ol) as a float pair
__device__ __forceinline__ void minus_origin(float a, float oh, float ol, float& hi, float& lo) {
  hi = __fsub_rn(a, oh);
  const float bp = __fsub_rn(hi, a);
  lo = __fsub_rn(__fsub_rn(__fsub_rn(a, __fsub_rn(hi, bp)), __fadd_rn(oh, bp)), ol);
}
__device__ __forceinline__ void into_frame(const Frame& fr, float x, float y, float& xh, float& xl, float& yh, float& yl) {
  float dxh, dxl, dyh, dyl;
  minus_origin(x, fr.ox_h, fr.ox_l, dxh, dxl);
  minus_origin(y, fr.oy_h, fr.oy_l, dyh, dyl);
  frame_axis(fr, dxh, dxl, dyh, dyl, xh, xl);
  frame_axis(fr, dyh, dyl, -dxh, -dxl, yh, yl);
}

// The reference path into shared memory, one float4 a row: x, y, heading in
// the frame, and the low parts of x and y (bfloat16 each, in one word): at
// 15 m a float's half ulp is 5e-7 m, and the softmin sees the costs of errors
// of that size.  First the raw rows in flight, then (after a barrier) their
// move into the frame.
__device__ __forceinline__ void stage_path(const Inst& in, const Smem& S) {
  for (int j = threadIdx.x; j < 3 * in.n_pts; j += blockDim.x) cp_async4(S.path + j + j / 3, in.path + j);
}
__device__ __forceinline__ void shift_path(const Inst& in, const Smem& S, const Frame& fr, int threads) {
  for (int j = threadIdx.x; j < in.n_pts; j += threads) {
    float4* d = reinterpret_cast<float4*>(S.path) + j;
    const float4 raw = *d;
    float xh, xl, yh, yl;
    into_frame(fr, raw.x, raw.y, xh, xl, yh, yl);
    const uint32_t lo = ((__float_as_uint(xl) + 0x8000u) >> 16) | ((__float_as_uint(yl) + 0x8000u) & 0xffff0000u);
    *d = make_float4(xh, yh, (raw.z - fr.oth_h) - fr.oth_l, __uint_as_float(lo));
  }
}

// The noise's tables (once a CTA).
__device__ __forceinline__ void stage_tables(const Smem& S) {
  const float* t = reinterpret_cast<const float*>(&kNoiseTables);
  for (int j = 4 * static_cast<int>(threadIdx.x); j < kNoiseTableFloats; j += 4 * static_cast<int>(blockDim.x))
    cp_async16(S.tab + j, t + j);
}

// The Philox blocks' shared words.
__device__ __forceinline__ void stage_blocks(const Inst& in, const Smem& S) {
  for (int b = threadIdx.x; b < in.P; b += blockDim.x) {
    const PhiloxBlock pb = philox_block(static_cast<uint32_t>(b), in.ctr, in.key0, in.key1);
    S.blk[b] = make_uint4(pb.a, pb.b, pb.c, 0u);
  }
}
__device__ __forceinline__ PhiloxBlock load_block(const Smem& S, int b) {
  const uint4 v = S.blk[b];
  return {v.x, v.y, v.z, v.w};
}

// The per-step hand-over between the noise warp and the compute warps
// (named barrier 1, every thread of the CTA; whole warps take one role).
__device__ __forceinline__ void step_barrier() { asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory"); }

// A row's state between steps (variants without producer warps): its rate
// less the part in y, and its columns u and (W) w.
template <bool W, int NS>
constexpr int kRowFloats = W ? 4 * NS : 2 * NS;
constexpr int kMaxRowSlots = 32;  // a lane's rows: 4 per Philox block, at most 8 blocks
// A lane's rows where they are in local memory (N floats), aligned for the
// vector accesses of store_row and load_row.
template <int N>
struct alignas(16) LocalRows {
  float v[N];
};
static_assert(alignof(LocalRows<1>) >= 16, "rows are read and written as float4");
template <bool W, int NS>
__device__ __forceinline__ void store_row(float* p, Vec<NS> al, Vec<NS> u, Vec<NS> w) {
  if constexpr (NS == 1) {
    if constexpr (W) *reinterpret_cast<float4*>(p) = make_float4(al.x, u.x, w.x, 0.f);
    else *reinterpret_cast<float2*>(p) = make_float2(al.x, u.x);
  } else {
    *reinterpret_cast<float4*>(p) = make_float4(al.x.x, al.x.y, u.x.x, u.x.y);
    if constexpr (W) *reinterpret_cast<float2*>(p + 4) = w.x;
  }
}
template <bool W, int NS>
__device__ __forceinline__ void load_row(const float* p, Vec<NS>& al, Vec<NS>& u, Vec<NS>& w) {
  if constexpr (NS == 1) {
    if constexpr (W) {
      const float4 v = *reinterpret_cast<const float4*>(p);
      al = v.x;
      u = v.y;
      w = v.z;
    } else {
      const float2 v = *reinterpret_cast<const float2*>(p);
      al = v.x;
      u = v.y;
    }
  } else {
    const float4 v = *reinterpret_cast<const float4*>(p);
    al = Vec<NS>(make_float2(v.x, v.y));
    u = Vec<NS>(make_float2(v.z, v.w));
    if constexpr (W) w = Vec<NS>(*reinterpret_cast<const float2*>(p + 4));
  }
}

// Sampled augmented input in the projection's coordinates.  The projection
// starts from M^-1 p with p = W z_des + rho/2 (z_hi + z_lo) and
// z_des = clip(U_nom + sigma n): a rising affine map of a clip is the clip of
// the mapped value between the mapped bounds, so one fused multiply-add and
// a clip give it, from the nominal input mapped once while it is staged.
// The rate inputs' p_alpha / m_alpha likewise.  Without the projection the
// map is the identity (KConst::qa, qb).
template <int N>
__device__ __forceinline__ Vec<N> sampled_input(const KConst& k, int j, float q_nom, Vec<N> n) {
  return vclamp(fma(Vec<N>(k.qs[j]), n, Vec<N>(q_nom)), k.qlo[j], k.qhi[j]);
}
template <int N>
__device__ __forceinline__ Vec<N> sampled_rate(const KConst& k, Vec<N> n) {
  return vclamp(fma(Vec<N>(k.ps), n, Vec<N>(k.pc_am)), k.pam_lo, k.pam_hi);
}

// Families of instantiations, by the terms they compile in.  A term that a
// step does not have costs it: its uniform branch splits the step into separately
// scheduled parts, its operands hold registers, its code fills the
// instruction cache.
//   kPlain   parked ellipses;
//   kDiscs   every optional term: any footprint, and all below;
//   kPoint   the rear-axle disc only: third-order rows, jerk-input model, buffer
//            cost, and all below;
//   kMoving  moving and e = 4 obstacles, collision cost.
// S = 4096, H = 50, 8 moving rows: 49.7 / 35.0 us on kDiscs / kMoving; third
// order and jerk, S = 3001, H = 61, 61.5 / 50.7 us on kDiscs / kPoint.
enum Family : int { kPlain = 0, kDiscs = 1, kPoint = 2, kMoving = 3 };

// ----------------------------------------------------------- one sample tile
// NS: samples a team rolls out together (Vec<NS>).
// LOCAL: the rows' state in local memory (in place of shared memory).
template <int TPS, int BPT, int EXT, int ROWS, int NS, bool LOCAL>
__device__ void run_tile(const KConst& k, const Inst& in, int tile, float* uh, const Smem& S,
                         Shared& sh, int noise_warps) {
  using T = Vec<NS>;
  constexpr bool DISCS = EXT == kDiscs, TERMS = EXT == kDiscs || EXT == kPoint;
  // Teams wider than one lane run with extra warps (the last ones) that
  // produce every team's normals a step ahead (warp specialisation: the
  // noise leaves the compute warps' dependency chain).
  const int nc = compute_threads<TPS>(noise_warps);
  const int spb = nc / TPS * NS;
  constexpr bool PRODUCED = kNoiseWarps<TPS, BPT, NS>;
  const bool producer = PRODUCED && static_cast<int>(threadIdx.x) >= nc;
  const int team = producer ? 0 : static_cast<int>(threadIdx.x) / TPS;
  const int lt = threadIdx.x % TPS;
  const int s = tile * spb + team * NS;  // the team's first sample
  const int H = in.H;
  const int n_rows = DISCS ? in.n_obs * k.nd : in.n_obs;  // obstacle rows (obstacle x disc)

  if (threadIdx.x == 32) {  // warm the outputs' translations (any CTA may merge)
    prefetch_l2(in.U_out);
    prefetch_l2(in.traj_out);
    prefetch_l2(in.U_next);
    prefetch_l2(in.status);
    prefetch_l2(in.part + static_cast<size_t>(tile - in.tile_base) * in.part_stride);
    if (in.J_out) prefetch_l2(in.J_out + static_cast<size_t>(tile) * spb);
  }
  // --- frame and staging (tables in shared memory, relative coordinates).
  // The raw path, the nominal inputs and each thread's first obstacle are
  // loaded first, so that their global loads overlap warp 0's frame; the
  // shift into the frame follows the barrier.
  const bool obs8 = EXT && k.obs8;
  const int ostride = obs8 ? 8 : 6;
  stage_path(in, S);
  stage_blocks(in, S);
  for (int j = threadIdx.x; j < 3 * H; j += blockDim.x) cp_async4(S.unom + j, in.U_nom + j);
  // obstacles by the compute threads after warp 0 (which builds the frame)
  const int n_stage = PRODUCED ? nc : static_cast<int>(blockDim.x);
  const int o0_ = static_cast<int>(threadIdx.x) - 32;
  const bool has_ob0 = !producer && o0_ >= 0 && o0_ < in.n_obs;
  float ob0[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) ob0[q] = (has_ob0 && q < ostride) ? in.obs[ostride * o0_ + q] : 0.f;
  if (threadIdx.x < 32) make_frame_warp(in.x0, in.inv_ds_d, in.sync + 1, sh.fr, TERMS && k.jerk);
  float sin0 = 0.f, cos0 = 0.f;
  if (has_ob0) sincosf(ob0[4], &sin0, &cos0);
  cp_async_wait_all();
  __syncthreads();
  const Frame& fr = sh.fr;
  auto stage_obstacle = [&](int o, float cx, float cy, float ax, float ay, float sw, float cw_, float e, float vx,
                            float vy) {
    float* d = S.obs + 8 * o;
    const bool e4 = obs8 && e == 4.0f;
    if (e != 2.0f && !e4) atomicOr(in.sync + 1, ERR_EXPONENT);
    const float Ax = ax + k.r_inflate, Ay = ay + k.r_inflate;
    float cxl, cyl;
    into_frame(fr, cx, cy, d[0], cxl, d[1], cyl);
    // the obstacle's axes in the frame
    const float co = fmaf(fr.c0, cw_, fr.s0 * sw), so = fmaf(fr.c0, sw, -(fr.s0 * cw_));
    const float ix = 1.0f / (Ax * Ax), iy = 1.0f / (Ay * Ay);
    if constexpr (!EXT) {
      // parked ellipses: h = d^T Q d - 1 with d the offset in the frame and
      // Q = R^T diag(ix, iy) R (R the rotation into the obstacle's axes):
      // (Qxx, Qxy) in place of (cos, sin), Qyy in slot 4
      const float c2 = co * co, s2 = so * so;
      d[2] = fmaf(c2, ix, s2 * iy);
      d[3] = (co * so) * (ix - iy);
      d[4] = fmaf(s2, ix, c2 * iy);
      d[5] = d[6] = d[7] = 0.f;
    } else {
      d[2] = co;
      d[3] = so;
      d[4] = e4 ? -(ix * ix) : ix;
      d[5] = e4 ? iy * iy : iy;
      d[6] = cw_ * vx + sw * vy;
      d[7] = cw_ * vy - sw * vx;
    }
  };
  // nominal inputs in the projection's coordinates (threads `first`,
  // first + stride, ...)
  auto map_inputs = [&](int first, int stride) {
    for (int j = first; j < 3 * H; j += stride) {
      const int q = j % 3;
      S.unom[j] = fmaf(k.qa[q], S.unom[j], k.qb[q]);
    }
  };
  // Producer warps (latency shapes): while the compute warps move the tables
  // into the frame, they map the nominal inputs and draw the first step.
  const int P_drawn = k.proj ? in.P : 1;  // standard MPPI needs the input normals only
  const int pl = static_cast<int>(threadIdx.x) - nc;
  const int n_blocks = spb * P_drawn, n_prod = 32 * noise_warps;
  // what block b's normals sample: block 0 the inputs (around the nominal
  // ones) and the hitch's rate, others four rows' rates
  struct Draw {
    PhiloxBlock pb;
    PhiloxSample smp;
    float s0, s1, s2, lo0, lo1, lo2, hi0, hi1, hi2;
    const float* nom;
    int nom_stride;
    float* dst;
  };
  auto make_draw = [&](int i) {
    const int tm = i / P_drawn, b = i - tm * P_drawn;
    const bool first = b == 0;
    Draw d;
    d.pb = load_block(S, b);
    d.smp = philox_sample(static_cast<uint32_t>(tile * spb + tm));
    d.s0 = first ? k.qs[0] : k.ps;
    d.s1 = first ? k.qs[1] : k.ps;
    d.s2 = first ? k.qs[2] : k.ps;
    d.lo0 = first ? k.qlo[0] : k.pam_lo;
    d.lo1 = first ? k.qlo[1] : k.pam_lo;
    d.lo2 = first ? k.qlo[2] : k.pam_lo;
    d.hi0 = first ? k.qhi[0] : k.pam_hi;
    d.hi1 = first ? k.qhi[1] : k.pam_hi;
    d.hi2 = first ? k.qhi[2] : k.pam_hi;
    d.nom = first ? S.unom : S.chunk;
    d.nom_stride = first ? 3 : 0;
    d.dst = S.noise + tm * S.noise_per_team + 4 * b;
    return d;
  };
  auto produce = [&](const Draw& d, int tau_d) {
    const uint4 w = philox_words(d.pb, d.smp, philox_step(d.smp, static_cast<uint32_t>(tau_d), in.key0, in.key1),
                                 in.key0, in.key1);
    const float* nom = d.nom + tau_d * d.nom_stride;
    Vec<1> g0, g1, g2, g3;
    box_muller<1>(&w.x, &w.y, S.tab, g0, g1);
    box_muller<1>(&w.z, &w.w, S.tab, g2, g3);
    g0 = vclamp(fma(Vec<1>(d.s0), g0, Vec<1>(nom[0])), d.lo0, d.hi0);
    g1 = vclamp(fma(Vec<1>(d.s1), g1, Vec<1>(nom[1])), d.lo1, d.hi1);
    g2 = vclamp(fma(Vec<1>(d.s2), g2, Vec<1>(nom[2])), d.lo2, d.hi2);
    g3 = sampled_rate(k, g3);
    *reinterpret_cast<float4*>(d.dst + (tau_d & 1) * 4 * in.P) = make_float4(g0.x, g1.x, g2.x, g3.x);
  };
  // Step tau's barrier hands its draws over; the first draws are made before
  // the staging barrier.
  if (producer) {
    map_inputs(pl, n_prod);
    if (pl < 4) S.chunk[pl] = k.pc_am;  // (free until the merge)
    asm volatile("bar.sync 2, %0;" ::"r"(n_prod) : "memory");
    if (n_blocks <= n_prod) {
      // at most one block a thread (the usual case): what the steps share
      // stays in registers
      const Draw d = make_draw(min(pl, n_blocks - 1));
      for (int tau = 0; tau < H; ++tau) {
        if ((pl & ~31) < n_blocks) produce(d, tau);  // (a warp's threads past the last block draw it again)
        if (tau == 0) staging_barrier();
        step_barrier();
      }
    } else {
      for (int tau = 0; tau < H; ++tau) {
        for (int i = pl; i < n_blocks; i += n_prod) produce(make_draw(i), tau);
        if (tau == 0) staging_barrier();
        step_barrier();
      }
    }
  }
  if (!producer) {
    // one row past the obstacles: h = -1 everywhere with no gradient, so a
    // padding slot that reads it adds exactly nothing to the projection's sums
    if (threadIdx.x < 8) S.obs[8 * in.n_obs + threadIdx.x] = 0.f;
    if (has_ob0) stage_obstacle(o0_, ob0[0], ob0[1], ob0[2], ob0[3], sin0, cos0, ob0[5], ob0[6], ob0[7]);
    for (int o = o0_ + n_stage - 32; o0_ >= 0 && o < in.n_obs; o += n_stage - 32) {
      const float* ob = in.obs + ostride * o;
      float so, co;
      sincosf(ob[4], &so, &co);
      stage_obstacle(o, ob[0], ob[1], ob[2], ob[3], so, co, ob[5], obs8 ? ob[6] : 0.f, obs8 ? ob[7] : 0.f);
    }
    shift_path(in, S, fr, n_stage);
    if constexpr (!PRODUCED) map_inputs(threadIdx.x, blockDim.x);
    if constexpr (DISCS) {
#pragma unroll
      for (int m = 0; m < 8; ++m)
        if (static_cast<int>(threadIdx.x) == m) {
          S.disc[2 * m] = k.disc_e1[m];
          S.disc[2 * m + 1] = k.disc_e2[m];
        }
    }
    staging_barrier();
  }

  // --- per-sample state (relative frame)
  T acc = fr.a0;  // acceleration state of the jerk-input model
  T px = 0.f, pxl = 0.f, py = 0.f, pyl = 0.f, t1 = 0.f, t2 = fr.t2, v = fr.v_h, vl = fr.v_l, dl = fr.dl, ps = 0.f,
    psl = 0.f;
  // obstacle slots per lane of the producer variants: 4 BPT; ROWS > 0: exactly
  // ROWS
  static_assert(ROWS == 0 || kNoiseWarps<TPS, BPT, NS>, "exact row slots need the noise-warp variants");
  constexpr int OBS_SLOTS = !PRODUCED ? 1 : (ROWS > 0 ? ROWS : 4 * BPT);
  T alpha_h = k.alpha0;  // the hitch's barrier rate (same on every lane)
  T alpha[OBS_SLOTS];    // the rows' rates (producer variants: in registers)
#pragma unroll
  for (int q = 0; q < OBS_SLOTS; ++q) alpha[q] = k.alpha0;
  // Other variants keep a row's state (its rate without the part in y, and
  // its columns u, w of the step before) in shared memory, one float4 a row
  // and lane (EXT: also the w column): the pass over the team's Philox blocks is then a loop of one body
  // for any number of rows.  Rows in registers need it unrolled: at 16 rows
  // a lane the step was 50 KB of code and waited for instructions (stall 0.8
  // an issue), and 64 registers more a lane cost a third of the warps.
  LocalRows<LOCAL ? kRowFloats<TERMS, NS> * kMaxRowSlots : 1> local_rows;
  const int row_stride = LOCAL ? kRowFloats<TERMS, NS> : kRowFloats<TERMS, NS> * static_cast<int>(blockDim.x);
  float* rows = LOCAL ? local_rows.v : S.noise + kRowFloats<TERMS, NS> * static_cast<int>(threadIdx.x);
  const int passes = (in.P - 1 + TPS - 1) / TPS;  // Philox blocks 1 .. P - 1 over the team's lanes
  if constexpr (!PRODUCED)
    for (int q = 0; q < 4 * passes; ++q) store_row<TERMS, NS>(rows + q * row_stride, T(k.alpha0), T(0.f), T(0.f));
  T ya_p = 0.f, yw_p = 0.f;  // the step before's y
  // exact-rows variants: a lane's rows are the same at every step, so their
  // table entries stay in registers
  float4 row_a[ROWS > 0 ? ROWS : 1], row_b[ROWS > 0 ? ROWS : 1];
  if constexpr (ROWS > 0 && !DISCS) {
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
      const int j = min(lt + TPS * q, n_rows);
      row_a[q] = *reinterpret_cast<const float4*>(S.obs + 8 * j);
      row_b[q] = *reinterpret_cast<const float4*>(S.obs + 8 * j + 4);
    }
  }
  T Jh = 0.f, Jl = 0.f;
  T ua = 0.f, uw = 0.f, un = 0.f;  // applied input of the previous step
  const uint32_t sid = static_cast<uint32_t>(s);
  const int n_pts = in.n_pts;
  const T qf0 = fr.qf0;
  const int i0 = fr.i0;

  // the four normals of Philox block b, given the step's words of the samples
  PhiloxSample smp[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) smp[i] = philox_sample(sid + i);
  struct StepWords {
    PhiloxStep w[NS];
  };
  auto step_words = [&](int tau) {
    StepWords r;
#pragma unroll
    for (int i = 0; i < NS; ++i) r.w[i] = philox_step(smp[i], static_cast<uint32_t>(tau), in.key0, in.key1);
    return r;
  };
  auto draw_block = [&](int b, const StepWords& st, T* out) {
    const PhiloxBlock pb = load_block(S, b);
    uint32_t x[NS], y[NS], z[NS], w[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const uint4 v = philox_words(pb, smp[i], st.w[i], in.key0, in.key1);
      x[i] = v.x;
      y[i] = v.y;
      z[i] = v.z;
      w[i] = v.w;
    }
    box_muller<NS>(x, y, S.tab, out[0], out[1]);
    box_muller<NS>(z, w, S.tab, out[2], out[3]);
  };

  // barrier of constraint row j (obstacle o seen from footprint disc m) at
  // the current state and time t (Eq. barrier_function; moving centres at
  // c + t v); (ce1, se1) and (ce2, se2) the unit headings of the state
  auto row_h = [&](int j, float t, T ce1, T se1, T ce2, T se2) -> T {
    int o = j;
    T dx, dy;
    if constexpr (DISCS) {
      o = (k.nd == 1) ? j : __float2int_rz((static_cast<float>(j) + 0.5f) * k.inv_nd);
    }
    const float4 o0 = *reinterpret_cast<const float4*>(S.obs + 8 * o);
    const float4 o1 = *reinterpret_cast<const float4*>(S.obs + 8 * o + 4);
    dx = (px - T(o0.x)) + pxl;
    dy = (py - T(o0.y)) + pyl;
    if constexpr (DISCS) {
      const float2 lv = *reinterpret_cast<const float2*>(S.disc + 2 * (j - o * k.nd));
      dx = fma(T(lv.y), ce2, fma(T(lv.x), ce1, dx));
      dy = fma(T(lv.y), se2, fma(T(lv.x), se1, dy));
    }
    const T xp = fma(T(o0.z), dx, fma(T(o0.w), dy, T(-t * o1.z)));
    const T yp = fma(T(o0.z), dy, fma(T(-o0.w), dx, T(-t * o1.w)));
    const bool e4 = o1.x < 0.f;
    const T kx = fabsf(o1.x), ky = o1.y;
    const T x2 = xp * xp, y2 = yp * yp;
    const T X = e4 ? x2 * kx : kx, Y = e4 ? y2 * ky : ky;
    return fma(x2, X, fma(y2, Y, T(-1.f)));
  };

  // Stage cost of state (px .. psl) reached with input (ua, uw, un).  With
  // equal contour and lag weights (KConst::iso, the default)
  // Qc e_c^2 + Ql e_l^2 is the weighted distance to the path point, whatever
  // the path's direction there: no sin / cos in the cost.
  struct Visit {
    T px, pxl, py, pyl, t1, t2, ps, psl, ua, uw, un;
  };
  auto stage_cost = [&](const Visit& x) -> T {
    // path cell: floor of qf by the 1.5 * 2^23 shifter on qf - 1/2 (an exact
    // integer may take the cell below with ff = 1, the same point); the
    // clamp keeps the shifter in range (2^22) far outside any path
    constexpr float kMost = 2.0 * kMaxFirstCell;
    const T qf = vclamp(fma(x.ps, T(in.inv_ds), qf0), -kMost, kMost);
    const T tt = (qf + T(-0.5f)) + T(12582912.0f);
    const T fl = tt + T(-12582912.0f);
    // ff = qf - fl, with the cancelling parts in one fused operation and the
    // reciprocal's and the progress's low parts: rounded at the size of ff
    T ff = (fma(x.ps, T(in.inv_ds), -fl) + qf0) + fma(x.psl, T(in.inv_ds), x.ps * T(in.inv_ds_l));
    T x0r, y0r, t0r, x1r, y1r, t1r, x0l, y0l, x1l, y1l;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const int cell = i0 + (__float_as_int(tt.get(i)) - 0x4b400000);
      const int ii = max(min(cell, n_pts - 2), 0);
      ff.set(i, cell == ii ? ff.get(i) : (cell < ii ? 0.f : 1.f));  // beyond an end: that end
      const float4 a = *reinterpret_cast<const float4*>(S.path + 4 * ii);
      const float4 b = *reinterpret_cast<const float4*>(S.path + 4 * ii + 4);
      x0r.set(i, a.x);
      y0r.set(i, a.y);
      t0r.set(i, a.z);
      x1r.set(i, b.x);
      y1r.set(i, b.y);
      t1r.set(i, b.z);
      x0l.set(i, __uint_as_float(__float_as_uint(a.w) << 16));
      y0l.set(i, __uint_as_float(__float_as_uint(a.w) & 0xffff0000u));
      x1l.set(i, __uint_as_float(__float_as_uint(b.w) << 16));
      y1l.set(i, __uint_as_float(__float_as_uint(b.w) & 0xffff0000u));
    }
    // offsets from the row, less the part along the segment: sums of small
    // terms, whatever the distance from the origin
    const T nf = -ff;
    const T dxr = fma(nf, x1r - x0r, x.px - x0r) + fma(nf, x1l - x0l, x.pxl - x0l);
    const T dyr = fma(nf, y1r - y0r, x.py - y0r) + fma(nf, y1l - y0l, x.pyl - y0l);
    const T seg = t1r - t0r;
    T rc;
    if (k.iso) {
      rc = T(k.Ql) * fma(dxr, dxr, dyr * dyr);
    } else {
      T sth, cth;  // the path's heading in the frame
      state_sincos(fma(ff, seg, t0r), &sth, &cth);
      const T ec = fma(sth, dxr, -(cth * dyr)), el = fma(cth, dxr, sth * dyr);
      rc = fma(T(k.Ql) * el, el, T(k.Qc) * ec * ec);
    }
    const T e1 = wrap_pi(fma(nf, seg, x.t1 - t0r)), e2 = wrap_pi(fma(nf, seg, x.t2 - t0r));
    const T dn = T(k.nu_bar) - x.un;
    rc = fma(T(k.Qth), fma(e1, e1, e2 * e2), rc);
    rc = fma(T(k.R0) * x.ua, x.ua, rc);
    rc = fma(T(k.R1) * x.uw, x.uw, rc);
    rc = fma(T(k.R2) * x.un, x.un, rc);
    return fma(T(k.mu) * dn, dn, rc);
  };
  auto visit = [&]() { return Visit{px, pxl, py, pyl, t1, t2, ps, psl, ua, uw, un}; };
  // The cost of a sample is summed over its team: in teams lane
  // (tau - 1) mod TPS keeps the state after step tau, and once every TPS
  // steps each lane evaluates the cost of the state it kept -- one cost
  // sequence in the warp's stream in place of TPS copies of it.
  // The producer variants (one compute warp a scheduler) evaluate it every
  // step on every lane instead: a branch in their step costs more than the
  // copies do (control solve of 4096 samples, H = 50: 40.0 us without the
  // branch, 43.0 us with it).
  constexpr bool SHARE = TPS > 1 && !kNoiseWarps<TPS, BPT, NS>;
  Visit kept = visit();
  auto cost_after = [&](int tau) {  // the state reached by step tau - 1
    if constexpr (!SHARE) {
      const T rc = stage_cost(visit());  // none before the first step: zero is added
      acc2(Jh, Jl, tau > 0 ? rc : T(0.f));
    } else {
      if (lt == ((tau - 1) & (TPS - 1))) kept = visit();
      if (tau > 0 && (tau & (TPS - 1)) == 0) acc2(Jh, Jl, stage_cost(kept));
    }
  };
  // parts of the cost that every lane has its share of, summed over the team
  // at the end
  T Xh = 0.f, Xl = 0.f;
  auto add_share = [&](T c) { acc2(Xh, Xl, c); };
  // the comparison method's collision penalty at the current state (time
  // t): depth of every obstacle it is inside (obstacles spread over the team)
  auto collision_cost = [&](float t, T ce1, T se1, T ce2, T se2) {
    T c = 0.f;
    auto depth = [&](int j) {
      c = c + vmap(row_h(j, t, ce1, se1, ce2, se2), [](float h) { return fmaxf(-h, 0.f); });
    };
    if constexpr (ROWS > 0) {
#pragma unroll
      for (int q = 0; q < ROWS; ++q)
        if (lt + TPS * q < n_rows) depth(lt + TPS * q);
    } else {
      for (int j = lt; j < n_rows; j += TPS) depth(j);
    }
    add_share(T(k.q_coll) * c);
  };

  // stored-trajectory variant: the states of the team's samples after step
  // tau, in world coordinates (written by the team's first lane)
  const bool writer = !producer && lt == 0;
  const bool st_out = writer && in.states_out, in_out = writer && in.inputs_out;
  auto store_state = [&](int tau) {
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      if (s + i >= in.S) break;
      float* o = in.states_out + (static_cast<size_t>(s + i) * static_cast<size_t>(H + 1) + tau) * 7;
      o[0] = fr.ox_h + (fmaf(fr.c0, px.get(i), -(fr.s0 * py.get(i))) +
                        (fr.ox_l + fmaf(fr.c0, pxl.get(i), -(fr.s0 * pyl.get(i)))));
      o[1] = fr.oy_h + (fmaf(fr.s0, px.get(i), fr.c0 * py.get(i)) +
                        (fr.oy_l + fmaf(fr.s0, pxl.get(i), fr.c0 * pyl.get(i))));
      o[2] = (fr.oth_h + t1.get(i)) + fr.oth_l;
      o[3] = (fr.oth_h + t2.get(i)) + fr.oth_l;
      o[4] = v.get(i) + vl.get(i);
      o[5] = dl.get(i);
      o[6] = (fr.psi_h + ps.get(i)) + (fr.psi_l + psl.get(i));
    }
  };
  const bool per_sample_out = in.states_out || in.inputs_out;
  if (st_out) store_state(0);

  // Noise.  Teams of at most two Philox blocks per lane, one sample each (the
  // latency shapes): the producer warps write what the P blocks of every
  // team's step tau + 1 sample (inputs and rates) into a per-team double buffer in shared memory while the
  // compute warps run step tau; one CTA barrier per step hands the buffers
  // over (at barrier tau the producers have written step tau and the compute
  // warps have finished step tau - 1, whose buffer is filled next).
  // Constraint i is built by lane i % TPS, so rows spread evenly over the team.
  //
  // Other shapes draw in registers, where the normals are used: lane lt owns
  // Philox blocks 1 + lt, 1 + lt + TPS, ... and builds their rows.  Block 0
  // (inputs and hitch) is needed by the whole team: lane lt draws it for step
  // tau + lt once every TPS steps, and each step takes it from its lane.
  float* nz = S.noise + team * S.noise_per_team;  // [2][P][4] (producer variants)
  T z0[4];  // in-register noise: this lane's sampled (a, omega, nu) and hitch rate
  // trigonometry of the current state, carried from step to step: the state
  // angles theta1 and phi = theta1 - theta2 of step tau + 1 follow from step
  // tau's state alone (the input enters only the speed, steer angle and
  // progress), so their sin / cos are taken before step tau's projection
  // and stay off its dependency chain; only the steer angle's trigonometry
  // waits for the projection.
  T c1, s1, sp, cp;
  state_sincos(t1, &s1, &c1);
  state_sincos(t1 - t2, &sp, &cp);
  // One step; PROJ is fixed for the whole loop (no branch on the flag
  // inside the step).
  auto step = [&](int tau, auto proj_c) {
    constexpr bool PROJ = decltype(proj_c)::value;
    // the sampled input in the projection's coordinates (M_u^-1 p_u with
    // the projection, else the sampled input itself) and the hitch's rate
    T q0, q1, zn, pam_h;
    const float* cur = nz + (tau & 1) * 4 * in.P;
    if constexpr (kNoiseWarps<TPS, BPT, NS>) {
      step_barrier();  // this step's normals are staged
      const float4 n4 = *reinterpret_cast<const float4*>(cur);
      q0 = n4.x;
      q1 = n4.y;
      zn = n4.z;
      pam_h = n4.w;
    } else {
      if ((tau & (TPS - 1)) == 0) {
        const int td = TPS == 1 ? tau : min(tau + lt, H - 1);
        T n4[4];
        draw_block(0, step_words(td), n4);
#pragma unroll
        for (int j = 0; j < 3; ++j) z0[j] = sampled_input(k, j, S.unom[3 * td + j], n4[j]);
        z0[3] = sampled_rate(k, n4[3]);
      }
      q0 = team_take<TPS>(z0[0], tau);
      q1 = team_take<TPS>(z0[1], tau);
      zn = team_take<TPS>(z0[2], tau);
      pam_h = team_take<TPS>(z0[3], tau);
    }

    // trigonometry of the steer angle (the one state angle the previous
    // projection moved)
    T sd, cd;
    state_sincos(dl, &sd, &cd);
    const T tn = sd * vrcp(cd);  // |cos| >= 4e-9 below 2^16: MUFU reciprocal (~2 ulp)
    const T vv = v + vl;
    const T tl = tn * T(k.inv_l1);
    const T th1dot = vv * tl;

    // cost of the previous step, at this state (independent of the rows)
    T c2 = 0.f, s2 = 0.f;  // the trailer's heading, where a term needs it
    if (DISCS && k.discs) {
      c2 = fma(c1, cp, s1 * sp);
      s2 = fma(s1, cp, -(c1 * sp));
    }
    cost_after(tau);
    if (EXT && k.coll && tau > 0) collision_cost(static_cast<float>(tau) * k.Ts, c1, s1, c2, s2);

    // trailer's heading rate and its parts
    const T kt = T(k.k_hitch) * tn;
    const T G = fma(-cp, kt, sp);
    const T vl2 = vv * T(k.inv_l2);
    const T th2dot = vl2 * G;

    // explicit Euler, the state-only part (right-hand sides at the current
    // state), and the next state's theta1 / phi trigonometry.  Latency
    // shapes (teams) form it before the projection, off its dependency
    // chain; one-lane shapes (issue-bound, many warps) after it, so that the
    // current and next values need not be live at once (no register copies
    // at the end of the step)
    T px_n, pxl_n, py_n, pyl_n, t1_n, t2_n, c1_n, s1_n, sp_n, cp_n;
    auto state_part = [&]() {
      const T Tv = T(k.Ts) * vv;
      px_n = px;
      pxl_n = pxl;
      py_n = py;
      pyl_n = pyl;
      acc2(px_n, pxl_n, Tv * c1);
      acc2(py_n, pyl_n, Tv * s1);
      t1_n = fma(T(k.Ts), th1dot, t1);
      t2_n = fma(T(k.Ts), th2dot, t2);
      if constexpr (TPS > 1) {
        // even lanes take theta1, odd lanes phi, and each pair trades the
        // results: one sin / cos sequence in the warp's stream instead of two
        const bool odd = lt & 1;
        T sa, ca;
        state_sincos(odd ? t1_n - t2_n : t1_n, &sa, &ca);
        const T sb = vshfl_xor(sa, 1), cb = vshfl_xor(ca, 1);
        s1_n = odd ? sb : sa;
        c1_n = odd ? cb : ca;
        sp_n = odd ? sa : sb;
        cp_n = odd ? ca : cb;
      } else {
        state_sincos(t1_n, &s1_n, &c1_n);
        state_sincos(t1_n - t2_n, &sp_n, &cp_n);
      }
    };
    if constexpr (TPS > 1) state_part();

    T za = q0, zw = q1;
    if constexpr (PROJ) {
      // hitch row (Eq. hitch_angle_barrier through the second-order
      // expansion, as hitch_row states it): every lane of the team computes
      // it (same state, same normal); its terms enter the sums once, after
      // the team reduction
      T u_h, w_h, rho_h, cc_h;
      const T sec2 = fma(tn, tn, T(1.f));
      const T phidot = th1dot - th2dot;
      const T kcl = fma(cp, T(k.khl2), T(k.inv_l1));  // k cos(phi) / l2 + 1 / l1
      const T bend = fma(kt, sp, cp);                 // cos(phi) + k tan(delta) sin(phi)
      {
        const T Delta = t2 - t1;
        const T sgT = vmap(Delta, [&](float d) { return copysignf(k.hTs2, d); });
        const T sgTs = vmap(Delta, [&](float d) { return copysignf(k.Ts, d); });
        const T h = fma(T(-k.kappa), vv, T(k.dtheta_max)) - vmap(Delta, [](float d) { return fabsf(d); });
        T Aa = fma(-sgT, fma(G, T(k.inv_l2), -tl), T(-k.Ts * k.kappa));
        const T Aw = (sgT * vv) * (sec2 * kcl);
        T c = phidot * fma(-(sgT * vl2), bend, sgTs);
        if (TERMS && k.jerk) {  // a is a state: its terms join the constant; the jerk enters via -kappa
          c = fma(acc, Aa, c);
          Aa = T(-k.hTs2 * k.kappa);
        }
        // h's sign (h = -0 does not arise: an exact zero rounds to +0)
        const T ht = vmap(h, [&](float x) { return copysignf(fmaxf(fabsf(x), k.h_floor), x); });
        const T r = fma(Aa, q0, fma(Aw, q1, fma(ht, pam_h, fma(alpha_h, h, c))));
        const T iht = vrcp(ht);
        u_h = Aa * iht;
        w_h = Aw * iht;
        rho_h = r * iht;
        cc_h = pam_h - rho_h;
      }

      // obstacle rows; the steer rate does not enter at second order.  Parked
      // ellipses (e = 2): hdot shares dh/da's direction term.  Moving or
      // e = 4 rows (uniform branch): barrier of the relative position at this
      // step's time, relative velocity.  Padding slots read the table's null
      // row (j = n_rows).
      T Saa = 0.f, ga = 0.f, Saw = 0.f, Sww = 0.f, gw = 0.f;
      T ca[OBS_SLOTS];
      T cw[TERMS ? OBS_SLOTS : 1];  // steer-rate column (footprint discs off the rear axle)
      // every slot that the alpha update reads is written below (padding
      // rows as zeros)
      const float tnow = static_cast<float>(tau) * k.Ts;
      T cbuf = 0.f;  // buffer cost of this lane's rows
      // heading accelerations of the bodies with the input held (footprint
      // discs): th1ddot = a1a a + a1w omega, th2ddot = a20 + a2a a + a2w omega
      T a1w = 0.f, a20 = 0.f, a2a = 0.f, a2w = 0.f;
      if (DISCS && k.discs) {
        a1w = vv * sec2 * T(k.inv_l1);
        a2a = G * T(k.inv_l2);
        a2w = -(vv * T(k.khl2) * cp * sec2);
        a20 = vl2 * bend * phidot;
      }
      // per-step factors of the parked-ellipse rows.  With (gx, gy) =
      // grad h / 2 = Q d and the heading e1 = (c1, s1): the a-column is
      // Ts^2/2 dh/da = Ts^2 (gx, gy) . e1 and the rest term
      // -(Ts hdot + Ts^2/2 hddot0) = -2 Ts v g - Ts^2 (v th1dot turn + v^2
      // e1^T Q e1), g and turn the products of (gx, gy) with e1 and n1:
      // linear in (gx, gy, Qxx, Qxy, Qyy) with factors of the state alone
      const T ax_row = T(k.Ts2) * c1, ay_row = T(k.Ts2) * s1;
      const T cg_row = T(-2.f * k.Ts) * vv, vth_row = T(-k.Ts2) * (vv * th1dot), vq_row = T(-k.Ts2) * (vv * vv);
      const T bx_row = fma(cg_row, c1, -(vth_row * s1)), by_row = fma(cg_row, s1, vth_row * c1);
      const T qxx_row = vq_row * (c1 * c1), qyy_row = vq_row * (s1 * s1), qxy_row = (vq_row + vq_row) * (c1 * s1);
      auto obstacle_row = [&](int j, int slot, T pam, T& al, T& u, T& w) {  // pam: p_alpha / m_alpha
        T h, Aa, Aw = 0.f, brest;
        if constexpr (!EXT) {
          // staged as (cx, cy, Qxx, Qxy, Qyy): h = d^T Q d - 1 in the frame
          const float4 o0 = ROWS > 0 ? row_a[slot] : *reinterpret_cast<const float4*>(S.obs + 8 * j);
          const T qxx = o0.z, qxy = o0.w, qyy = ROWS > 0 ? row_b[slot].x : S.obs[8 * j + 4];
          const T dx = (px - T(o0.x)) + pxl, dy = (py - T(o0.y)) + pyl;
          const T gx = fma(qxx, dx, qxy * dy), gy = fma(qxy, dx, qyy * dy);
          h = fma(gx, dx, fma(gy, dy, T(-1.f)));
          Aa = fma(gx, ax_row, gy * ay_row);
          brest = fma(gx, bx_row, fma(gy, by_row, fma(qxx_row, qxx, fma(qxy_row, qxy, qyy_row * qyy))));
        } else {
          // row j: obstacle o, seen from the rear axle or (kDiscs) from
          // footprint disc m (obstacle-major).  Unit headings in the obstacle
          // frame: e1' = (dirx, diry), n1' = (-diry, dirx), e2' = (d2x, d2y),
          // n2' = (-d2y, d2x); e = 4 flagged by a negated kx; with
          // X = xp^(e-2) / Ax^e: h = xp^2 X + ..., h_x = e xp X,
          // h_xx = e (e-1) X
          int o = j;
          if constexpr (DISCS) o = (k.nd == 1) ? j : __float2int_rz((static_cast<float>(j) + 0.5f) * k.inv_nd);
          const bool kept_row = ROWS > 0 && !DISCS;
          const float4 o0 = kept_row ? row_a[ROWS > 0 ? slot : 0] : *reinterpret_cast<const float4*>(S.obs + 8 * o);
          const float4 o1 = kept_row ? row_b[ROWS > 0 ? slot : 0] : *reinterpret_cast<const float4*>(S.obs + 8 * o + 4);
          const T co = o0.z, so = o0.w;
          const T dirx = fma(co, c1, so * s1), diry = fma(co, s1, -(so * c1));
          const T dx = (px - T(o0.x)) + pxl, dy = (py - T(o0.y)) + pyl;
          // position relative to the (moving) obstacle centre at tnow
          T xp = fma(co, dx, fma(so, dy, T(-tnow * o1.z)));
          T yp = fma(co, dy, fma(-so, dx, T(-tnow * o1.w)));
          T lx = 0.f, ly = 0.f, d2x = 0.f, d2y = 0.f;
          if constexpr (DISCS) {
            const float2 lvp = *reinterpret_cast<const float2*>(S.disc + 2 * (j - o * k.nd));  // lever arms on e1, e2
            lx = lvp.x;
            ly = lvp.y;
            d2x = fma(co, c2, so * s2);
            d2y = fma(co, s2, -(so * c2));
            xp = fma(lx, dirx, fma(ly, d2x, xp));
            yp = fma(lx, diry, fma(ly, d2y, yp));
          }
          const bool e4 = o1.x < 0.f;
          const T kx = fabsf(o1.x), ky = o1.y;
          const T x2 = xp * xp, y2 = yp * yp;
          const T X = e4 ? x2 * kx : kx, Y = e4 ? y2 * ky : ky;
          const T ce = e4 ? 4.f : 2.f, cee = e4 ? 12.f : 2.f;
          h = fma(x2, X, fma(y2, Y, T(-1.f)));
          const T hx = ce * xp * X, hy = ce * yp * Y;
          const T ge = fma(hx, dirx, hy * diry);     // grad h . e1'
          const T gn = fma(hy, dirx, -(hx * diry));  // grad h . n1'
          // velocity relative to the obstacle; acceleration = acc0 + a acc_a
          // + omega acc_w, at the rear axle v th1dot n1 and a e1
          T velx = fma(vv, dirx, T(-o1.z)), vely = fma(vv, diry, T(-o1.w));
          const T vw = vv * th1dot;
          T ga0 = vw * gn;  // grad h . acc0
          Aa = T(k.hTs2) * ge;
          if constexpr (DISCS) {
            const T lt1 = lx * th1dot, lt2 = ly * th2dot;
            velx = velx - fma(lt1, diry, lt2 * d2y);
            vely = vely + fma(lt1, dirx, lt2 * d2x);
            const T g2 = fma(hx, d2x, hy * d2y), n2 = fma(hy, d2x, -(hx * d2y));  // grad h . e2', n2'
            Aa = T(k.hTs2) * (ge + fma(lx * tl, gn, ly * a2a * n2));
            Aw = T(k.hTs2) * fma(lx * a1w, gn, ly * a2w * n2);
            ga0 = ga0 + fma(-(lt1 * th1dot), ge, fma(ly * a20, n2, -(lt2 * th2dot * g2)));
          }
          const T hdot = fma(hx, velx, hy * vely);
          const T wHx = cee * X * velx, wHy = cee * Y * vely;  // Hess h w
          const T hdd0 = ga0 + fma(wHx, velx, wHy * vely);
          brest = fma(T(-k.Ts), hdot, T(-k.hTs2) * hdd0);
          if (TERMS && k.third) {
            // Ts^3/6 hdddot at the rear axle (lever arms zero), affine in
            // (a, omega): pdddot = 2 a th1dot n1 + v th1ddot n1 - v th1dot^2 e1,
            // hdddot = grad h . pdddot + 3 w^T Hess h pddot + D3 h [w, w, w]
            const T ca3 = fma(fma(T(2.f), th1dot, vv * tl), gn, T(3.f) * fma(wHx, dirx, wHy * diry));
            const T cw3 = vv * vv * sec2 * T(k.inv_l1) * gn;
            T c03 = fma(-(vw * th1dot), ge, T(3.f) * vw * fma(wHy, dirx, -(wHx * diry)));
            const T k3x = e4 ? 24.f * fabsf(o1.x) : 0.f, k3y = e4 ? 24.f * o1.y : 0.f;
            c03 = fma(xp * k3x * velx * velx, velx, fma(yp * k3y * vely * vely, vely, c03));
            Aa = fma(T(k.Ts3_6), ca3, Aa);
            Aw = fma(T(k.Ts3_6), cw3, Aw);
            brest = fma(T(-k.Ts3_6), c03, brest);
          }
          if (TERMS && k.jerk) {
            // a is a state (rear-axle point): its terms join the constant;
            // the jerk enters only at third order, through grad h . e1'
            brest = fma(-acc, Aa, brest);
            Aa = k.third ? T(k.Ts3_6) * ge : T(0.f);
          }
        }
        const T ht = vmap(h, [&](float x) { return copysignf(fmaxf(fabsf(x), k.h_floor), x); });
        T r = fma(Aa, q0, fma(ht, pam, fma(al, h, -brest)));
        if constexpr (TERMS) r = fma(Aw, q1, r);
        const T iht = vrcp(ht);  // MUFU reciprocal (~1 ulp)
        u = Aa * iht;
        const T rho = r * iht;
        Saa = fma(u, u, Saa);
        ga = fma(u, rho, ga);
        if (TERMS && k.abuf) {
          // buffer zone: positive rates charged with weight clip(1 - h/h_buf)
          const T wz = vclamp(fma(h, T(-k.inv_hbuf), T(1.f)), 0.f, 1.f);
          const T ap = vmap(al, [](float x) { return fmaxf(x, 0.f); });
          cbuf = fma(T(j < n_rows ? k.q_abuf : 0.f) * wz, ap * ap, cbuf);
        }
        // the rate's update without its part in y, added after the 2x2 solve
        al = al + (pam - rho);
        if constexpr (TERMS) {
          w = Aw * iht;
          Saw = fma(u, w, Saw);
          Sww = fma(w, w, Sww);
          gw = fma(w, rho, gw);
        }
      };

      if constexpr (!kNoiseWarps<TPS, BPT, NS>) {
        // row j uses normal 4 + j: block 1 + j/4, drawn here, a pass over the
        // team's lanes at a time
        const StepWords now = step_words(tau);
#pragma unroll 1
        for (int g = 0; g < passes; ++g) {
          const int b = 1 + g * TPS + lt;
          T nb[4];
          draw_block(TPS == 1 ? b : min(b, in.P - 1), now, nb);
          float* row = rows + 4 * g * row_stride;
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int j = 4 * (b - 1) + m;
            if (TPS > 1 || j < n_rows) {
              T al, u, w = 0.f;
              load_row<TERMS, NS>(row + m * row_stride, al, u, w);
              al = fma(u, ya_p, al);
              if constexpr (TERMS) al = fma(w, yw_p, al);
              obstacle_row(min(j, n_rows), 0, sampled_rate(k, nb[m]), al, u, w);
              store_row<TERMS, NS>(row + m * row_stride, al, u, w);
            }
          }
        }
      } else {
        // row j on lane j % TPS.  ROWS > 0: exactly ROWS slots a lane, all
        // of them run, no branch in the step; else the team's slot count
        const int per_lane = (n_rows + TPS - 1) / TPS;
#pragma unroll
        for (int slot = 0; slot < OBS_SLOTS; ++slot) {
          if (ROWS == 0) {
            ca[slot] = 0.f;
            if constexpr (TERMS) cw[slot] = 0.f;
          }
          if (ROWS > 0 || slot < per_lane) {
            const int j = lt + TPS * slot;
            T w = 0.f;
            obstacle_row(min(j, n_rows), slot, T(cur[4 + min(j, n_rows - 1)]), alpha[slot], ca[slot], w);
            if constexpr (TERMS) cw[slot] = w;
          }
        }
      }
      if (TERMS && k.abuf) add_share(cbuf);
      const T m_a = k.m_a;
      Saa = fma(m_a, fma(u_h, u_h, team_sum<TPS>(Saa)), T(k.m_u0));
      ga = m_a * fma(u_h, rho_h, team_sum<TPS>(ga));
      if constexpr (TERMS) {
        Saw = m_a * fma(u_h, w_h, team_sum<TPS>(Saw));
        Sww = fma(m_a, fma(w_h, w_h, team_sum<TPS>(Sww)), T(k.m_u1));
        gw = m_a * fma(w_h, rho_h, team_sum<TPS>(gw));
      } else {
        // the plain family's ellipse rows have no steer-rate column
        Saw = m_a * (u_h * w_h);
        Sww = fma(m_a, w_h * w_h, T(k.m_u1));
        gw = m_a * (w_h * rho_h);
      }
      const T idet = vrcp(fma(Saa, Sww, -(Saw * Saw)));  // SPD: det > 0
      const T ya = fma(Sww, ga, -(Saw * gw)) * idet;
      const T yw = fma(Saa, gw, -(Saw * ga)) * idet;
      za = q0 - ya;
      zw = q1 - yw;
      alpha_h = alpha_h + fma(w_h, yw, fma(u_h, ya, cc_h));
      auto alpha_update = [&](int slot) {
        alpha[slot] = fma(ca[slot], ya, alpha[slot]);
        if constexpr (TERMS) alpha[slot] = fma(cw[slot], yw, alpha[slot]);
      };
      if constexpr (!PRODUCED) {
        ya_p = ya;
        yw_p = yw;
      } else {
#pragma unroll
        for (int slot = 0; slot < OBS_SLOTS; ++slot) alpha_update(slot);
      }
    }
    ua = vclamp(za, k.zlo0, k.zhi0);
    uw = vclamp(zw, k.zlo1, k.zhi1);
    un = vclamp(zn, k.zlo2, k.zhi2);
    if constexpr (TPS == 1) state_part();

    // explicit Euler, the input-driven part; the state-only part was formed
    // from the same right-hand sides
    px = px_n;
    pxl = pxl_n;
    py = py_n;
    pyl = pyl_n;
    t1 = t1_n;
    t2 = t2_n;
    if (TERMS && k.jerk) {  // input 0 is the jerk; the acceleration state drives the speed
      acc2(v, vl, T(k.Ts) * acc);
      acc = fma(T(k.Ts), ua, acc);
    } else {
      acc2(v, vl, T(k.Ts) * ua);
    }
    dl = fma(T(k.Ts), uw, dl);
    acc2(ps, psl, T(k.Ts) * un);
    c1 = c1_n;
    s1 = s1_n;
    sp = sp_n;
    cp = cp_n;

    if (lt == 0) {
      store_pair(uh + (3 * tau + 0) * spb + team * NS, ua);
      store_pair(uh + (3 * tau + 1) * spb + team * NS, uw);
      store_pair(uh + (3 * tau + 2) * spb + team * NS, un);
    }
    if (!per_sample_out) return;  // the same for every thread
    if (st_out) store_state(tau + 1);
    if (in_out) {
#pragma unroll
      for (int i = 0; i < NS; ++i) {
        if (s + i >= in.S) break;
        float* o = in.inputs_out + (static_cast<size_t>(s + i) * static_cast<size_t>(H) + tau) * 3;
        o[0] = ua.get(i);
        o[1] = uw.get(i);
        o[2] = un.get(i);
      }
    }
  };
  if (!producer) {
    if (k.proj) {
      for (int tau = 0; tau < H; ++tau) step(tau, std::true_type{});
    } else {
      for (int tau = 0; tau < H; ++tau) step(tau, std::false_type{});
    }
  }
  if (!producer) {  // cost of the last step, and the team's sum
    if constexpr (!SHARE) {
      cost_after(H);
    } else {
      if (lt == ((H - 1) & (TPS - 1))) kept = visit();
      const T last = stage_cost(kept);  // lanes past the last step were summed already
      acc2(Jh, Jl, lt <= ((H - 1) & (TPS - 1)) ? last : T(0.f));
    }
    if (EXT && k.coll)
      collision_cost(static_cast<float>(H) * k.Ts, c1, s1, fma(c1, cp, s1 * sp), fma(s1, cp, -(c1 * sp)));
    auto team_pair = [&](T& h, T& l) {
#pragma unroll
      for (int m = 1; m < TPS; m <<= 1) {
        const T oh = vshfl_xor(h, m), ol = vshfl_xor(l, m);
        acc2(h, l, oh);
        l = l + ol;
      }
    };
    if constexpr (SHARE) team_pair(Jh, Jl);
    if constexpr (EXT) {
      if (k.coll || k.abuf) {
        team_pair(Xh, Xl);
        acc2(Jh, Jl, Xh);
        Jl = Jl + Xl;
      }
    }
  }

  // --- per-sample cost: normalise the pair
  if (writer) {
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const float jh = Jh.get(i) + Jl.get(i);
      const float jl = Jl.get(i) - (jh - Jh.get(i));
      const bool valid = s + i < in.S;
      const bool fin = valid && isfinite(jh) && isfinite(jl);
      S.jh[team * NS + i] = fin ? jh : CUDART_INF_F;
      S.jl[team * NS + i] = fin ? jl : 0.f;
      if (valid && in.J_out) in.J_out[s + i] = jh;  // the normalised pair's high part
      if (valid && in.J_lo_out) in.J_lo_out[s + i] = jl;
    }
  }
  __syncthreads();

  // --- tile softmin partial: min pair, weights, weight sum, weighted inputs
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {
    float mh = CUDART_INF_F, ml = 0.f;
    for (int t = lane; t < spb; t += 32) {
      const float h = S.jh[t], l = S.jl[t];
      if (pair_less(h, l, mh, ml)) { mh = h; ml = l; }
    }
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, mh, m);
      const float ol = __shfl_xor_sync(0xffffffffu, ml, m);
      if (pair_less(oh, ol, mh, ml)) { mh = oh; ml = ol; }
    }
    if (lane == 0) { sh.red_h[0] = mh; sh.red_l[0] = ml; }
  }
  __syncthreads();
  const float bmh = sh.red_h[0], bml = sh.red_l[0];
  const bool any_finite = bmh < CUDART_INF_F;
  for (int t = threadIdx.x; t < spb; t += blockDim.x) {
    const float h = S.jh[t];
    float w = 0.f;
    if (any_finite && h < CUDART_INF_F) w = expf(-((h - bmh) + (S.jl[t] - bml)) * k.inv_lambda);
    S.w[t] = w;
  }
  __syncthreads();
  float* part = in.part + static_cast<size_t>(tile - in.tile_base) * in.part_stride;
  const int nrows = 3 * H + 1;  // row 3H: the weight sum
  // one thread per row: its spb weighted inputs in sample order, four
  // chains (samples t mod 4) combined in a fixed order; the row's loads are
  // issued together (one L2 round trip per row instead of one per warp pass)
  const bool vec = (spb & 3) == 0 && (reinterpret_cast<uintptr_t>(uh) & 15) == 0;
  for (int row = threadIdx.x; row < nrows; row += blockDim.x) {
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    const float* src = uh + static_cast<size_t>(row) * spb;
    const bool wsum = row == 3 * H;
    int t = 0;
    if (vec) {
#pragma unroll 8
      for (; t < spb; t += 4) {
        const float4 w4 = *reinterpret_cast<const float4*>(S.w + t);
        const float4 v4 = wsum ? make_float4(1.f, 1.f, 1.f, 1.f) : *reinterpret_cast<const float4*>(src + t);
        a0 += w4.x * v4.x;
        a1 += w4.y * v4.y;
        a2 += w4.z * v4.z;
        a3 += w4.w * v4.w;
      }
    }
    for (; t < spb; ++t) a0 += S.w[t] * (wsum ? 1.f : src[t]);
    part[3 + row] = (a0 + a1) + (a2 + a3);
  }
  if (threadIdx.x == 0) {
    part[0] = bmh;
    part[1] = bml;
    part[2] = 0.f;
  }
}

// Exclusive prefix sum over the 32 lanes of a warp (lane order), offset by
// `carry`; `carry` advances by the warp's total (chunked scans).
static __device__ __forceinline__ float warp_exclusive_scan(float x, float& carry) {
  const int lane = threadIdx.x & 31;
  float s = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float y = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += y;
  }
  const float total = __shfl_sync(0xffffffffu, s, 31);
  float e = __shfl_up_sync(0xffffffffu, s, 1);
  if (lane == 0) e = 0.f;
  const float r = carry + e;
  carry += total;
  return r;
}

// --------------------------------------- merge of an instance's partials
// Run by the CTA that finished the instance's last tile: global minimum
// pair, rescaled sums in tile order, U*, warm start, status and the optimal
// trajectory (x0 integrated with U*).
// Optimal trajectory: x0 integrated with U* in the relative frame (explicit
// Euler, as the rollouts).  Speed, steer angle, progress, the acceleration
// of the jerk-input model and the tractor heading are prefix sums, scanned
// by warp 0 32 steps at a time; the trailer angle is the one nonlinear
// recurrence (thread 0, serial) while warp 1 scans the positions.  Per-step
// values go to `scratch` (8 (H+1) floats: the CTA's table regions when they
// can hold them, else the instance's consumed tile partials).  The
// elementary functions are the SFU approximations (absolute error ~2^-21
// per call, far inside the trajectory tolerance).
static __device__ void optimal_trajectory(const KConst& k, const Inst& in, const Smem& S, Shared& sh,
                                          float* __restrict__ scratch) {
  const int H = in.H, n = H + 1;
  const Frame& fr = sh.fr;
  float* V = scratch;          // speed
  float* D = scratch + n;      // steer angle
  float* Q = scratch + 2 * n;  // progress
  float* T = scratch + 3 * n;  // tan(steer angle)
  float* A = scratch + 4 * n;  // tractor heading
  float* B = scratch + 5 * n;  // trailer heading
  float* X = scratch + 6 * n;  // x
  float* Y = scratch + 7 * n;  // y
  const float* __restrict__ ustar = S.ustar;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float Ts = k.Ts;
  __syncthreads();
  if (warp == 0) {
    float cv = fr.v_h + fr.v_l, cd = fr.dl, cq = 0.f, ca = fr.a0, c1 = 0.f;
    for (int base = 0; base < n; base += 32) {
      const int tau = base + lane;
      const bool step = tau < H;  // an input acts at tau < H; states run to H
      const float u0 = step ? ustar[3 * tau + 0] : 0.f;
      const float u1 = step ? ustar[3 * tau + 1] : 0.f;
      const float u2 = step ? ustar[3 * tau + 2] : 0.f;
      float iv = Ts * u0;
      if (k.jerk) {  // the speed integrates the acceleration state
        const float acc = warp_exclusive_scan(Ts * u0, ca);
        iv = step ? Ts * acc : 0.f;
      }
      const float v = warp_exclusive_scan(iv, cv);
      const float d = warp_exclusive_scan(Ts * u1, cd);
      const float q = warp_exclusive_scan(Ts * u2, cq);
      float sd, cs;
      __sincosf(d, &sd, &cs);
      const float t = __fdividef(sd, cs);
      const float a = warp_exclusive_scan(step ? (Ts * v) * t * k.inv_l1 : 0.f, c1);
      if (tau < n) {
        V[tau] = v;
        D[tau] = d;
        Q[tau] = q;
        T[tau] = t;
        A[tau] = a;
      }
    }
  }
  __syncthreads();
  const float c0 = fr.c0, s0 = fr.s0;
  auto positions = [&]() {  // one warp
    float cx = 0.f, cy = 0.f;
    for (int base = 0; base < n; base += 32) {
      const int tau = base + lane;
      float ix = 0.f, iy = 0.f;
      if (tau < H) {
        float a1, b1;
        __sincosf(A[tau], &a1, &b1);
        const float Tv = Ts * V[tau];
        ix = Tv * (c0 * b1 - s0 * a1);
        iy = Tv * (s0 * b1 + c0 * a1);
      }
      const float x = warp_exclusive_scan(ix, cx);
      const float y = warp_exclusive_scan(iy, cy);
      if (tau < n) {
        X[tau] = x;
        Y[tau] = y;
      }
    }
  };
  if (threadIdx.x == 0) {  // trailer angle
    // step tau + 1's coefficients are loaded before step tau's store, so
    // the loads overlap the chain (A, V, T and B share one scratch array)
    float q2 = fr.t2;
    float an = A[0], cn = (Ts * V[0]) * k.inv_l2, en = k.k_hitch * T[0];
    for (int tau = 0; tau < H; ++tau) {
      const float a = an, c = cn, e = en;
      if (tau + 1 < H) {
        an = A[tau + 1];
        cn = (Ts * V[tau + 1]) * k.inv_l2;
        en = k.k_hitch * T[tau + 1];
      }
      B[tau] = q2;
      float a2, b2;
      __sincosf(a - q2, &a2, &b2);
      q2 = fmaf(c, fmaf(-e, b2, a2), q2);
    }
    B[H] = q2;
  }
  if (warp == 1) positions();
  __syncthreads();
  if (blockDim.x < 64 && warp == 0) {  // no second warp: positions after the headings
    positions();
    __syncwarp();
  }
  float* tr = in.traj_out;
  for (int tau = threadIdx.x; tau <= H; tau += blockDim.x) {
    tr[7 * tau + 0] = (fr.ox_h + X[tau]) + fr.ox_l;
    tr[7 * tau + 1] = (fr.oy_h + Y[tau]) + fr.oy_l;
    tr[7 * tau + 2] = (fr.oth_h + A[tau]) + fr.oth_l;
    tr[7 * tau + 3] = (fr.oth_h + B[tau]) + fr.oth_l;
    tr[7 * tau + 4] = V[tau];
    tr[7 * tau + 5] = D[tau];
    tr[7 * tau + 6] = (fr.psi_h + Q[tau]) + fr.psi_l;
  }
}

// The same, one thread, no scratch (when neither scratch region can hold
// 8 (H+1) floats).
static __device__ void serial_trajectory(const KConst& k, const Inst& in, const Smem& S, Shared& sh) {
  const Frame& fr = sh.fr;
  const float c0 = fr.c0, s0 = fr.s0;
  const float* ustar = S.ustar;
  const int H = in.H;
  float qx = 0.f, qy = 0.f, q1 = 0.f, q2 = fr.t2, qv = fr.v_h + fr.v_l, qd = fr.dl, qp = 0.f, qa = fr.a0;
  float* tr = in.traj_out;
  for (int tau = 0; tau <= H; ++tau) {
    tr[7 * tau + 0] = (fr.ox_h + qx) + fr.ox_l;
    tr[7 * tau + 1] = (fr.oy_h + qy) + fr.oy_l;
    tr[7 * tau + 2] = (fr.oth_h + q1) + fr.oth_l;
    tr[7 * tau + 3] = (fr.oth_h + q2) + fr.oth_l;
    tr[7 * tau + 4] = qv;
    tr[7 * tau + 5] = qd;
    tr[7 * tau + 6] = (fr.psi_h + qp) + fr.psi_l;
    if (tau == H) break;
    float a1, b1, a2, b2, ad, bd;
    __sincosf(q1, &a1, &b1);
    __sincosf(q1 - q2, &a2, &b2);
    __sincosf(qd, &ad, &bd);
    const float tq = __fdividef(ad, bd);
    const float Tv = k.Ts * qv;
    qx += Tv * (c0 * b1 - s0 * a1);
    qy += Tv * (s0 * b1 + c0 * a1);
    q2 += Tv * k.inv_l2 * (a2 - k.k_hitch * b2 * tq);
    q1 += Tv * tq * k.inv_l1;
    if (k.jerk) {
      qv += k.Ts * qa;
      qa += k.Ts * ustar[3 * tau + 0];
    } else {
      qv += k.Ts * ustar[3 * tau + 0];
    }
    qd += k.Ts * ustar[3 * tau + 1];
    qp += k.Ts * ustar[3 * tau + 2];
  }
}

// Minimum pair over the partials of an instance held in shared memory
// (tile b at mp + b * stride), into sh.red_h[1] / sh.red_l[1].
static __device__ void smem_pair_min(const float* mp, int nb, int stride, Shared& sh) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  float mh = CUDART_INF_F, ml = 0.f;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const float h = mp[static_cast<size_t>(b) * stride + 0], l = mp[static_cast<size_t>(b) * stride + 1];
    if (pair_less(h, l, mh, ml)) { mh = h; ml = l; }
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, mh, m);
    const float ol = __shfl_xor_sync(0xffffffffu, ml, m);
    if (pair_less(oh, ol, mh, ml)) { mh = oh; ml = ol; }
  }
  if (lane == 0) { sh.wred_h[warp] = mh; sh.wred_l[warp] = ml; }
  __syncthreads();
  if (warp == 0) {
    mh = lane < nwarps ? sh.wred_h[lane] : CUDART_INF_F;
    ml = lane < nwarps ? sh.wred_l[lane] : 0.f;
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, mh, m);
      const float ol = __shfl_xor_sync(0xffffffffu, ml, m);
      if (pair_less(oh, ol, mh, ml)) { mh = oh; ml = ol; }
    }
    if (lane == 0) { sh.red_h[1] = mh; sh.red_l[1] = ml; }
  }
  __syncthreads();
}

// SMEM_PARTS: the instance's tile partials are copied into the CTA's shared
// memory at once (one L2 round trip; the launch reserved the room) and
// merged from there; else they are read from L2 in passes.  Both sum each
// row in the same order (four chains, tiles t mod 4, the tail on the first),
// so they give the same bits.
template <bool SMEM_PARTS>
static __device__ void merge_instance(const KConst& k, const Inst& in, const Smem& S, Shared& sh) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const int nb = in.tiles;
  const int stride = in.part_stride;
  const int H = in.H;
  const int nrows = 3 * H + 1;
  float* ustar = S.ustar;
  bool ok;
  if constexpr (SMEM_PARTS) {
    // the partials region (nb * stride floats, a multiple of 4, 16-byte
    // aligned) into the regions after the disc table (noise, history: no
    // longer read); the error bits' atomic round trip overlaps the copy
    float* mp = S.noise;
    const int nf = nb * stride;
    for (int i = 4 * static_cast<int>(threadIdx.x); i < nf; i += 4 * static_cast<int>(blockDim.x))
      cp_async16(mp + i, in.part + i);
    if (threadIdx.x == 0) sh.err = atomicAdd(in.sync + 1, 0u);
    cp_async_wait_all();
    __syncthreads();
    smem_pair_min(mp, nb, stride, sh);
    const float gmh = sh.red_h[1], gml = sh.red_l[1];
    ok = gmh < CUDART_INF_F;
    for (int q = threadIdx.x; q < nrows; q += blockDim.x) ustar[q] = 0.f;
    for (int b0 = 0; b0 < nb; b0 += 256) {
      __syncthreads();
      for (int t = threadIdx.x; t < 256 && b0 + t < nb; t += blockDim.x) {
        const float* pt = mp + static_cast<size_t>(b0 + t) * stride;
        const float h = pt[0], l = pt[1];
        S.chunk[t] = (ok && h < CUDART_INF_F) ? expf(-((h - gmh) + (l - gml)) * k.inv_lambda) : 0.f;
      }
      __syncthreads();
      const int bend = min(256, nb - b0);
      for (int q = threadIdx.x; q < nrows; q += blockDim.x) {
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
        const float* col = mp + static_cast<size_t>(b0) * stride + 3 + q;
        int t = 0;
        for (; t + 4 <= bend; t += 4) {
          a0 += S.chunk[t + 0] * col[static_cast<size_t>(t + 0) * stride];
          a1 += S.chunk[t + 1] * col[static_cast<size_t>(t + 1) * stride];
          a2 += S.chunk[t + 2] * col[static_cast<size_t>(t + 2) * stride];
          a3 += S.chunk[t + 3] * col[static_cast<size_t>(t + 3) * stride];
        }
        for (; t < bend; ++t) a0 += S.chunk[t] * col[static_cast<size_t>(t) * stride];
        ustar[q] += (a0 + a1) + (a2 + a3);
      }
    }
  } else {
    // global pair minimum: every thread its tiles (b = tid, tid + blockDim,
    // ...), then warps, then warp 0; the pair of tile tid stays in registers
    // for the weights below (one L2 round trip for both)
    float h0 = CUDART_INF_F, l0 = 0.f;
    // the solve's error bits, read now (an atomic round trip) and used after the sums
    if (threadIdx.x == 0) sh.err = atomicAdd(in.sync + 1, 0u);
    // the first 64 tiles' entries of this thread's first row, loaded now: their
    // round trip overlaps the minimum's (instances of at least 64 tiles)
    const bool pre_ok = static_cast<int>(threadIdx.x) < nrows && nb >= 64;
    float pre[64];
#pragma unroll
    for (int m = 0; m < 64; ++m)
      pre[m] = pre_ok ? __ldcg(in.part + static_cast<size_t>(m) * stride + 3 + threadIdx.x) : 0.f;
    {
      float mh = CUDART_INF_F, ml = 0.f;
      for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        const float h = __ldcg(in.part + static_cast<size_t>(b) * stride + 0);
        const float l = __ldcg(in.part + static_cast<size_t>(b) * stride + 1);
        if (b == static_cast<int>(threadIdx.x)) {
          h0 = h;
          l0 = l;
        }
        if (pair_less(h, l, mh, ml)) { mh = h; ml = l; }
      }
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, mh, m);
        const float ol = __shfl_xor_sync(0xffffffffu, ml, m);
        if (pair_less(oh, ol, mh, ml)) { mh = oh; ml = ol; }
      }
      if (lane == 0) { sh.wred_h[warp] = mh; sh.wred_l[warp] = ml; }
      __syncthreads();
      if (warp == 0) {
        mh = lane < nwarps ? sh.wred_h[lane] : CUDART_INF_F;
        ml = lane < nwarps ? sh.wred_l[lane] : 0.f;
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) {
          const float oh = __shfl_xor_sync(0xffffffffu, mh, m);
          const float ol = __shfl_xor_sync(0xffffffffu, ml, m);
          if (pair_less(oh, ol, mh, ml)) { mh = oh; ml = ol; }
        }
        if (lane == 0) { sh.red_h[1] = mh; sh.red_l[1] = ml; }
      }
    }
    __syncthreads();
    const float gmh = sh.red_h[1], gml = sh.red_l[1];
    ok = gmh < CUDART_INF_F;
    for (int q = threadIdx.x; q < nrows; q += blockDim.x) ustar[q] = 0.f;
    for (int b0 = 0; b0 < nb; b0 += 256) {
      __syncthreads();
      for (int t = threadIdx.x; t < 256 && b0 + t < nb; t += blockDim.x) {
        const size_t base = static_cast<size_t>(b0 + t) * stride;
        const bool held = b0 == 0 && t == static_cast<int>(threadIdx.x);
        const float h = held ? h0 : __ldcg(in.part + base + 0), l = held ? l0 : __ldcg(in.part + base + 1);
        S.chunk[t] = (ok && h < CUDART_INF_F) ? expf(-((h - gmh) + (l - gml)) * k.inv_lambda) : 0.f;
      }
      __syncthreads();
      const int bend = min(256, nb - b0);
      for (int q = threadIdx.x; q < nrows; q += blockDim.x) {
        // four independent chains (tiles t mod 4), combined in a fixed order;
        // 64 (then 16) L2 loads in flight per pass
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
        const float* col = in.part + static_cast<size_t>(b0) * stride + 3 + q;
        int t = 0;
        for (; t + 64 <= bend; t += 64) {
          // `pre` is the pass buffer: it already holds the first pass of the
          // thread's first row
          if (!(pre_ok && b0 == 0 && t == 0 && q == static_cast<int>(threadIdx.x))) {
#pragma unroll
            for (int m = 0; m < 64; ++m) pre[m] = __ldcg(col + static_cast<size_t>(t + m) * stride);
          }
#pragma unroll
          for (int m = 0; m < 64; m += 4) {
            a0 += S.chunk[t + m + 0] * pre[m + 0];
            a1 += S.chunk[t + m + 1] * pre[m + 1];
            a2 += S.chunk[t + m + 2] * pre[m + 2];
            a3 += S.chunk[t + m + 3] * pre[m + 3];
          }
        }
        for (; t + 16 <= bend; t += 16) {
          float v[16];
#pragma unroll
          for (int m = 0; m < 16; ++m) v[m] = __ldcg(col + static_cast<size_t>(t + m) * stride);
#pragma unroll
          for (int m = 0; m < 16; m += 4) {
            a0 += S.chunk[t + m + 0] * v[m + 0];
            a1 += S.chunk[t + m + 1] * v[m + 1];
            a2 += S.chunk[t + m + 2] * v[m + 2];
            a3 += S.chunk[t + m + 3] * v[m + 3];
          }
        }
        for (; t + 4 <= bend; t += 4) {
          a0 += S.chunk[t + 0] * __ldcg(col + static_cast<size_t>(t + 0) * stride);
          a1 += S.chunk[t + 1] * __ldcg(col + static_cast<size_t>(t + 1) * stride);
          a2 += S.chunk[t + 2] * __ldcg(col + static_cast<size_t>(t + 2) * stride);
          a3 += S.chunk[t + 3] * __ldcg(col + static_cast<size_t>(t + 3) * stride);
        }
        for (; t < bend; ++t) a0 += S.chunk[t] * __ldcg(col + static_cast<size_t>(t) * stride);
        ustar[q] += (a0 + a1) + (a2 + a3);
      }
    }
  }
  // path turns between consecutive rows (this CTA's frame-shifted table;
  // 1e-4 rad over pi/4 covers the shift's rounding): an out-of-range turn
  // rejects the solve
  int turn_bad = 0;
  for (int j = threadIdx.x; j + 1 < in.n_pts; j += blockDim.x)
    turn_bad |= !(fabsf(S.path[4 * j + 6] - S.path[4 * j + 2]) <= kMaxPathTurn + 1e-4f);
  const bool turns_bad = __syncthreads_or(turn_bad);
  const float lsum = ustar[3 * H];
  const unsigned err = sh.err | (turns_bad ? ERR_PATH_TURN : 0u);
  for (int q = threadIdx.x; q < 3 * H; q += blockDim.x) {
    const float u = ok ? ustar[q] / lsum : in.U_nom[q];
    ustar[q] = u;
    in.U_out[q] = u;
  }
  __syncthreads();
  if (in.U_next) {
    for (int q = threadIdx.x; q < 3 * H; q += blockDim.x) {
      const int tau = q / 3, j = q % 3;
      in.U_next[q] = ustar[3 * min(tau + 1, H - 1) + j];
    }
  }
  if (threadIdx.x == 0) {
    if (in.status) {
      int32_t st = 0;
      if (err & (ERR_EXPONENT | ERR_PATH_TURN)) st = -1;
      else if ((err & ERR_NONFINITE_X0) || !ok) st = -5;
      *in.status = st;
    }
    in.sync[1] = 0u;
    in.sync[0] = 0u;
  }
  if (in.traj_out) {
    // scratch: the obstacle, path and nominal-input tables (contiguous, no
    // longer read by this CTA's merge), else the consumed partials
    if (static_cast<long long>(S.ustar - S.obs) >= 8LL * (H + 1)) {
      optimal_trajectory(k, in, S, sh, S.obs);
    } else if (static_cast<long long>(in.tiles) * in.part_stride >= 8LL * (H + 1)) {
      optimal_trajectory(k, in, S, sh, in.part);
    } else if (threadIdx.x == 0) {
      serial_trajectory(k, in, S, sh);
    }
  }
  __syncthreads();
}

// The tile's applied-input history in global memory is dead once the tile's
// weighted sums have read it: its L2 lines are dropped without being written
// back to DRAM (discard.global.L2, whole 128-byte lines only, so a line
// shared with the neighbouring CTA's slot is left alone).  Every read of the
// history must be complete (after a CTA barrier); the next tile writes
// before it reads.
__device__ __forceinline__ void discard_history(const float* uh, int n_floats) {
  const unsigned long long b0 = reinterpret_cast<unsigned long long>(uh);
  const unsigned long long b1 = b0 + 4ull * static_cast<unsigned long long>(n_floats);
  const unsigned long long first = (b0 + 127ull) & ~127ull, last = b1 & ~127ull;
  for (unsigned long long a = first + 128ull * threadIdx.x; a < last; a += 128ull * blockDim.x) {
    unsigned long long g;
    asm volatile("cvta.to.global.u64 %0, %1;" : "=l"(g) : "l"(a));
    asm volatile("discard.global.L2 [%0], 128;" ::"l"(g) : "memory");
  }
}

// -------------------------------------------------------------- the kernel
// EXT: the family (Family, above run_tile).
// Launch bound of the two-sample variants: 384 threads an SM (168 registers),
// in CTAs of up to 192.  One lane a sample without optional terms keeps nearly
// all of its step in 128 registers (36 B spilled), and a fourth warp a
// scheduler is worth more: on GB300 48 solves of S = 4096, H = 50, 8 rows
// 410 -> 386 us, 256 uneven ones 1820 -> 1800.  Moving rows lose by it (32
// solves of S = 4096 338 -> 354 us), and so do third-order rows (422 -> 434).
constexpr int kPairCtas = 2;
constexpr int pair_threads(int tps, int family) { return tps == 1 && family == kPlain ? 256 : 192; }
template <int TPS, int BPT, int EXT, int ROWS = 0, int NS = 1, bool LOCAL = false>
// Launch bound: 512 threads (128 registers a thread); the exact-rows
// single-solve instantiations 384 (up to 170 registers: one CTA per SM on
// the latency shapes, where registers buy a longer schedule)
__global__ void __launch_bounds__(ROWS > 0 ? 384 : (NS > 1 ? pair_threads(TPS, EXT) : 512), NS > 1 ? kPairCtas : 1) solve_kernel(const KConst k, const LaunchDesc L) {
  extern __shared__ __align__(16) float dyn[];
  __shared__ Shared sh;
  const int spb = compute_threads<TPS>(L.noise_warps) / TPS * NS;
  const Smem S(dyn, L.caps, spb);
  // applied-input history of the CTA's tile: shared memory in the exact-rows
  // variants (the launch reserved it), else the CTA's global slot
  float* uh;
  if constexpr (ROWS > 0) {
    uh = S.noise + L.caps.noise_per_team * spb;
  } else {
    uh = L.uh + static_cast<size_t>(blockIdx.x) * L.uh_stride;
  }

  // Programmatic dependent launch: the CTAs of a solve may start while the
  // kernel before it on the stream drains, and stage what belongs to no solve;
  // the wait returns once that kernel has completed and its writes are
  // visible, so everything after it is as in a plain launch.  The next solve
  // may be started at once for the same reason.  Back to back, S = 256, H = 30
  // 20.5 -> 17.8 us, S = 4096, H = 50 34.8 -> 31.7 us; a solve behind a copy or on
  // an idle stream gains nothing by it.
  stage_tables(S);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  for (int iter = 0;; ++iter) {
    int inst_id = 0, tile;
    if (L.work) {
      if (threadIdx.x == 0) sh.item = static_cast<int>(atomicAdd(L.work_ctr, 1u));
      __syncthreads();
      const int item = sh.item;
      __syncthreads();
      if (item >= L.n_work) break;
      const int2 w = L.work[item];
      inst_id = w.x;
      tile = w.y;
    } else {
      if (iter > 0) break;
      tile = L.single.tile_base + static_cast<int>(blockIdx.x);
    }
    Inst in;
    if (L.work) in = L.inst[inst_id];
    else in = L.single;
    run_tile<TPS, BPT, EXT, ROWS, NS, LOCAL>(k, in, tile, uh, S, sh, L.noise_warps);

    // the CTA that completes an instance's last tile merges its partials
    __threadfence();
    __syncthreads();
    if constexpr (ROWS == 0) discard_history(uh, 3 * in.H * spb);
    if (in.no_merge) continue;  // a share of the tiles: merged elsewhere (single launches only)
    if (threadIdx.x == 0) sh.last = (atomicAdd(in.sync, 1u) == static_cast<unsigned>(in.tiles - 1));
    __syncthreads();
    if (sh.last) {
      __threadfence();
      merge_instance<(ROWS > 0)>(k, in, S, sh);
    }
    __syncthreads();
  }
  if (L.work) {
    // the last CTA to run out of work resets the work counters for the
    // next launch (no CTA reads them after its final fetch)
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(L.work_ctr + 1, 1u) == gridDim.x - 1) {
        L.work_ctr[0] = 0u;
        L.work_ctr[1] = 0u;
      }
    }
  }
}

// ------------------------------------------------ merge of gathered tiles
// One CTA merges an instance's complete set of tile partials, produced by
// no-merge launches (one per rank of a sample-partitioned solve) and
// gathered in tile order: the same frame, tables and merge as the CTA that
// finishes a single launch's last tile, so the results are the same bits.
template <bool EXT>
__global__ void __launch_bounds__(256) merge_tiles_kernel(const KConst k, const Inst in, const SmemCaps caps) {
  extern __shared__ __align__(16) float dyn[];
  __shared__ Shared sh;
  const Smem S(dyn, caps, 1);
  stage_path(in, S);
  if (threadIdx.x < 32) make_frame_warp(in.x0, in.inv_ds_d, in.sync + 1, sh.fr, EXT && k.jerk);
  const bool obs8 = EXT && k.obs8;
  for (int o = threadIdx.x; o < in.n_obs; o += blockDim.x) {
    const float e = in.obs[(obs8 ? 8 : 6) * o + 5];
    if (e != 2.0f && !(obs8 && e == 4.0f)) atomicOr(in.sync + 1, ERR_EXPONENT);
  }
  cp_async_wait_all();
  __syncthreads();
  const Frame& fr = sh.fr;
  shift_path(in, S, fr, blockDim.x);  // as the tiles stage it
  __syncthreads();
  merge_instance<false>(k, in, S, sh);
}

}  // namespace brmppi
