// Trajectory planning (Sec. IV-A, Eq. mp_length_only with the tendon speed / acceleration limits by
// finite differences) and kinematic calibration.
//
// One CTA per trajectory, one thread per timestep t. Each thread runs the forward phase of its own
// state (chain, clearance, penalty rows), shares its tip position and tendon state through shared
// memory, evaluates the coupling rows it owns (length, speed, acceleration between t and its
// predecessors), shares their derivatives, and runs the reverse phase of its state with the tip
// force of the length rows (and of the goal pose at the last state). Sums over the trajectory are
// deterministic block reductions.
#pragma once

#include "cr_solve_impl.cuh"

namespace crk {

template <typename T> struct TrajW {
  T dt, vmax, amax, w_len, rho_v, rho_a;
};

// Deterministic block sum: butterfly inside each warp, then every thread adds the warp totals in
// warp order. red[] holds 32 values; blockDim.x is a multiple of 32.
template <typename T> __device__ T block_sum(T v, T* red) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  T s = T(0);
  for (int k = 0; k < nw; ++k) s += red[k];
  return s;
}
template <typename T> __device__ T block_max(T v, T* red) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = c_max(v, __shfl_xor_sync(0xffffffffu, v, off));
  const int nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  T s = red[0];
  for (int k = 1; k < nw; ++k) s = c_max(s, red[k]);
  return s;
}

// Shared buffers of one trajectory: tip positions [Tn][3], states [Tn][D], speed and acceleration
// row derivatives [Tn][D] each, reduction scratch [32]; for the split evaluation (two threads per
// state, see traj_state_eval) the second thread's clearance aggregates [Tn][8 N] and the gradient
// handed back to it [Tn][D].
template <typename T> struct TrajSmem {
  T* p;
  T* u;
  T* sv;
  T* sa;
  T* red;
  T* xag;
  T* xg;
  __host__ __device__ static size_t bytes(int Tn, int D) {
    return sizeof(T) * ((size_t)Tn * (3 + 3 * D) + 32 + (size_t)Tn * (8 * (D / 3) + D));
  }
  __device__ void carve(unsigned char* base, int Tn, int D) {
    T* q = reinterpret_cast<T*>(base);
    p = q;
    u = p + (size_t)Tn * 3;
    sv = u + (size_t)Tn * D;
    sa = sv + (size_t)Tn * D;
    red = sa + (size_t)Tn * D;
    xag = red + 32;
    xg = xag + (size_t)Tn * 8 * (D / 3);
  }
};

// Thread t's share of the trajectory cost; with GRAD, gu = dF/du_t (zero for t = 0 and t >= Tn).
// Every thread of the block must call it (it synchronises). Split evaluation (split = true): two
// threads per state, each with its own part of the spheres (sph, no); the helper (aux = true) adds
// only the clearance rows of its spheres to F and passes their force / moment aggregates to the
// owner through shared memory, the owner runs everything else and hands the gradient back.
template <typename T, int N, bool OBST, bool GRAD, bool QUICK = (N <= 4)>
__device__ T traj_state_eval(const RobotK<T>& rb, const WeightsK<T>& w, const TrajW<T>& tw, int t, int Tn,
                             const T (&u)[3 * N], const TargetK<T>& goal, ObsK<T> sph, int no,
                             TrajSmem<T>& sm, T (&gu)[3 * N], bool split = false, bool aux = false) {
  constexpr int D = 3 * N;
  const bool active = t < Tn;
  Chain<T, N> ch;
  StateAgg<T, N> ag;
  T F = T(0);
  T Ftip[3] = {T(0), T(0), T(0)}, Rtip[3] = {T(0), T(0), T(0)};
  if (aux) {
    if (active && t >= 1) {
      T coll = T(0);
      state_forward<T, N, OBST, GRAD, false, true, CR_MODEL_TENDON, false, QUICK>(
          rb, w, sph, no, u, ch, ag, &coll, false);  // the owner has the self rows
      F = coll;
      if (GRAD) {
        T* x = sm.xag + (size_t)t * 8 * N;
#pragma unroll
        for (int i = 0; i < N; ++i) {
#pragma unroll
          for (int a = 0; a < 3; ++a) { x[6 * i + a] = ag.G[i][a]; x[6 * i + 3 + a] = ag.M[i][a]; }
          x[6 * N + 2 * i] = ag.Dx[i];
          x[6 * N + 2 * i + 1] = ag.Dy[i];
        }
      }
    }
    __syncthreads();
    if (!GRAD) return F;
    __syncthreads();
    __syncthreads();
#pragma unroll
    for (int q = 0; q < D; ++q) gu[q] = (active && t >= 1) ? sm.xg[(size_t)t * D + q] : T(0);
    return F;
  }
  if (active) {
    if (t == 0) {
      chain_forward(rb, u, ch);  // the start state is fixed: only its tip enters the length rows
    } else {
      F = state_forward<T, N, OBST, GRAD, false, true, CR_MODEL_TENDON, false, QUICK>(rb, w, sph, no, u, ch, ag, nullptr);
    }
    if (t == Tn - 1) {
      T r[6], e[3], ang, sn, cs;
      pose_rows(CR_TASK_IK6, w, goal, ch.R, ch.p, r, e, ang, sn, cs);
      F += T(0.5) * (r[0] * r[0] + r[1] * r[1] + r[2] * r[2] + r[3] * r[3] + r[4] * r[4] + r[5] * r[5]);
      if (GRAD) pose_tip_force(CR_TASK_IK6, w, goal, ch.R, r, e, Ftip, Rtip);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) sm.p[t * 3 + a] = ch.p[a];
#pragma unroll
    for (int q = 0; q < D; ++q) sm.u[t * D + q] = u[q];
  }
  __syncthreads();
  T sv[D], sa[D];
#pragma unroll
  for (int q = 0; q < D; ++q) { sv[q] = T(0); sa[q] = T(0); }
  if (active && t >= 1) {
    T dp0 = ch.p[0] - sm.p[(t - 1) * 3], dp1 = ch.p[1] - sm.p[(t - 1) * 3 + 1], dp2 = ch.p[2] - sm.p[(t - 1) * 3 + 2];
    F += T(0.5) * tw.w_len * (dp0 * dp0 + dp1 * dp1 + dp2 * dp2);
    const T idt = T(1) / tw.dt, idt2 = idt * idt;
#pragma unroll
    for (int q = 0; q < D; ++q) {
      T v = (u[q] - sm.u[(t - 1) * D + q]) * idt;
      T hu = v - tw.vmax, hl = -tw.vmax - v;
      hu = hu > T(0) ? hu : T(0);
      hl = hl > T(0) ? hl : T(0);
      F += T(0.5) * tw.rho_v * (hu * hu + hl * hl);
      sv[q] = tw.rho_v * (hu - hl) * idt;
      if (t >= 2) {
        T acc = (u[q] - T(2) * sm.u[(t - 1) * D + q] + sm.u[(t - 2) * D + q]) * idt2;
        T au = acc - tw.amax, al = -tw.amax - acc;
        au = au > T(0) ? au : T(0);
        al = al > T(0) ? al : T(0);
        F += T(0.5) * tw.rho_a * (au * au + al * al);
        sa[q] = tw.rho_a * (au - al) * idt2;
      }
    }
  }
  if (!GRAD) return F;
  if (active) {
#pragma unroll
    for (int q = 0; q < D; ++q) { sm.sv[t * D + q] = sv[q]; sm.sa[t * D + q] = sa[q]; }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < D; ++q) gu[q] = T(0);
  if (split && active && t >= 1) {  // add the helper's clearance aggregates
    const T* x = sm.xag + (size_t)t * 8 * N;
#pragma unroll
    for (int i = 0; i < N; ++i) {
#pragma unroll
      for (int a = 0; a < 3; ++a) { ag.G[i][a] += x[6 * i + a]; ag.M[i][a] += x[6 * i + 3 + a]; }
      ag.Dx[i] += x[6 * N + 2 * i];
      ag.Dy[i] += x[6 * N + 2 * i + 1];
    }
  }
  if (active && t >= 1) {
    // length rows (t-1, t) and (t, t+1) act on the tip of state t
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      T f = tw.w_len * (ch.p[a] - sm.p[(t - 1) * 3 + a]);
      if (t + 1 < Tn) f -= tw.w_len * (sm.p[(t + 1) * 3 + a] - ch.p[a]);
      Ftip[a] += f;
    }
    state_reverse<T, N, false>(rb, w, u, ch, ag, Ftip, Rtip, gu, nullptr, nullptr);
    // speed rows of t and t+1, acceleration rows of t, t+1 and t+2 act on u_t directly
#pragma unroll
    for (int q = 0; q < D; ++q) {
      T g = sv[q] + sa[q];
      if (t + 1 < Tn) g += -sm.sv[(t + 1) * D + q] - T(2) * sm.sa[(t + 1) * D + q];
      if (t + 2 < Tn) g += sm.sa[(t + 2) * D + q];
      gu[q] += g;
    }
  }
  if (split) {  // hand the gradient to the helper thread of the same state
    if (active) {
#pragma unroll
      for (int q = 0; q < D; ++q) sm.xg[(size_t)t * D + q] = gu[q];
    }
    __syncthreads();
  }
  return F;
}

template <typename T> struct TrajArgs {
  const double* u_start;  // [D][P]
  const double* goal;     // [7][P]
  int64_t P;
  int Tn;
  const double* spheres;
  int no;
  const double* prims;
  int np;
  int sph_pp;
  // cost / gradient
  const T* x;             // [D][P*(Tn-1)]
  T* cost;
  T* grad;
  const T* upstream;
  // solve
  const double* u_goal;   // [D][P]
  const double* x_init;   // [D][P*Tn] initial states (nullable: linear interpolation to u_goal)
  int k_traj;
  T alpha0;
  double lim_tol;
  double dt_d, vmax_d, amax_d;
  double* X_out;          // [D][P*Tn]
  double* F_out;
  double* goal_pos;
  double* goal_rot;
  double* speed;
  double* accel;
  unsigned char* lim_ok;
  unsigned char* col_ok;
};

// Stage problem p's obstacle set (the shared one without per-problem scenes) at base (PRIMS:
// stage_obstacles_as).
template <bool PRIMS = true, typename T, typename A>
__device__ ObsK<T> stage_traj_obstacles(const A& a, int64_t p, const RobotK<T>& rb, T delta, unsigned char* base) {
  const int64_t q = a.sph_pp ? p : 0;
  return stage_obstacles_as<PRIMS>(a.spheres + q * a.no * 4, a.no,
                                   a.np > 0 ? a.prims + q * a.np * CR_PRIM_DOUBLES : nullptr, a.np, rb, delta, base);
}

template <typename T, int N, bool OBST, bool GRAD>
__global__ void __launch_bounds__(256) k_traj_cost(RobotK<T> rb, WeightsK<T> w, TrajW<T> tw, TrajArgs<T> a) {
  constexpr int D = 3 * N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int64_t p = blockIdx.x;
  const int t = threadIdx.x, Tn = a.Tn;
  size_t off = (obstacles_smem<T>(a.no, a.np) + 15) & ~size_t(15);
  TrajSmem<T> sm;
  sm.carve(smem_raw + off, Tn, D);
  ObsK<T> sph(nullptr);
  if (OBST) {
    sph = stage_traj_obstacles(a, p, rb, w.delta, smem_raw);
    __syncthreads();
  }
  const int64_t ld = a.P * (Tn - 1);
  T u[D];
#pragma unroll
  for (int q = 0; q < D; ++q) {
    if (t == 0) u[q] = T(a.u_start[q * a.P + p]);
    else if (t < Tn) u[q] = a.x[q * ld + p * (Tn - 1) + (t - 1)];
    else u[q] = T(0);
  }
  TargetK<T> goal = load_target<T>(a.goal, a.P, p, CR_TASK_IK6);
  T gu[D];
  T F = traj_state_eval<T, N, OBST, GRAD>(rb, w, tw, t, Tn, u, goal, sph, a.no + a.np, sm, gu);
  T Ft = block_sum(F, sm.red);
  if (t == 0) a.cost[p] = Ft;
  if (GRAD && t >= 1 && t < Tn) {
    T s = a.upstream ? a.upstream[p] : T(1);
#pragma unroll
    for (int q = 0; q < D; ++q) a.grad[q * ld + p * (Tn - 1) + (t - 1)] = s * gu[q];
  }
}

// Trajectory planning after the goal IK: linear initialisation (or the given initial states x_init), k_traj
// projected-gradient steps of all free states, FP64 metrics of the result.
template <typename T, int N, bool OBST, bool PRIMS = true>
__global__ void __launch_bounds__(256, 1) k_traj_solve(RobotK<T> rb, WeightsK<T> w, TrajW<T> tw, RobotK<double> rbd,
                                                     WeightsK<double> wd, TrajArgs<T> a) {
  constexpr int D = 3 * N;
  constexpr bool QUICK = N <= 3 || (N == 4 && !PRIMS);  // see segment_masks
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int64_t p = blockIdx.x;
  const int Tn = a.Tn, Wt = ((Tn + 31) / 32) * 32;
  // split evaluation (blockDim = 2 Wt): thread t and t + Wt share state t, each with half the obstacles
  const bool split = (int)blockDim.x == 2 * Wt;
  const bool aux = split && (int)threadIdx.x >= Wt;
  const int t = aux ? (int)threadIdx.x - Wt : (int)threadIdx.x;
  const int nob = a.no + a.np;
  const size_t offd = (obstacles_smem<T>(a.no, a.np) + 15) & ~size_t(15);
  size_t off = offd + ((obstacles_smem<double>(a.no, a.np) + 15) & ~size_t(15));
  TrajSmem<T> sm;
  sm.carve(smem_raw + off, Tn, D);
  ObsK<T> sph(nullptr);
  ObsK<double> sphd(nullptr);
  if (OBST) {
    sph = stage_traj_obstacles<PRIMS>(a, p, rb, w.delta, smem_raw);
    sphd = stage_traj_obstacles<PRIMS>(a, p, rbd, wd.delta, smem_raw + offd);
    __syncthreads();
  }
  const bool active = t < Tn;
  const int nh = split ? (nob + 1) / 2 : nob;
  const ObsK<T> sph_m = aux ? sph.from(nh) : sph;
  const int no_m = aux ? nob - nh : nh;
  T u[D];
#pragma unroll
  for (int q = 0; q < D; ++q) {
    if (a.x_init) {
      u[q] = active ? T(a.x_init[q * a.P * Tn + p * Tn + t]) : T(0);
      continue;
    }
    double u0 = a.u_start[q * a.P + p], ug = a.u_goal[q * a.P + p];
    u[q] = active ? T(u0 + (double)t / (Tn - 1) * (ug - u0)) : T(0);
  }
  TargetK<T> goal = load_target<T>(a.goal, a.P, p, CR_TASK_IK6);
  T g[D];
  T F = block_sum(traj_state_eval<T, N, OBST, true, QUICK>(rb, w, tw, t, Tn, u, goal, sph_m, no_m, sm, g, split, aux),
                  sm.red);
  T alpha = a.alpha0;
  const bool free_state = active && t >= 1;
  for (int it = 0; it < a.k_traj; ++it) {
    T gn2l = T(0);
#pragma unroll
    for (int q = 0; q < D; ++q) gn2l += aux ? T(0) : g[q] * g[q];  // the helper holds a copy
    T gn2 = block_sum(gn2l, sm.red);
    T scale = gn2 > T(0) ? alpha * c_rsqrt(gn2) : T(0);
    T u1[D];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (free_state)
        project3(u[3 * i] - scale * g[3 * i], u[3 * i + 1] - scale * g[3 * i + 1], u[3 * i + 2] - scale * g[3 * i + 2],
                 rb.umax[i], u1[3 * i], u1[3 * i + 1], u1[3 * i + 2]);
      else {
        u1[3 * i] = u[3 * i]; u1[3 * i + 1] = u[3 * i + 1]; u1[3 * i + 2] = u[3 * i + 2];
      }
    }
    T g1[D];
    T F1 = block_sum(traj_state_eval<T, N, OBST, true, QUICK>(rb, w, tw, t, Tn, u1, goal, sph_m, no_m, sm, g1, split, aux),
                     sm.red);
    if (F1 < F) {
#pragma unroll
      for (int q = 0; q < D; ++q) { u[q] = u1[q]; g[q] = g1[q]; }
      F = F1;
      alpha *= T(1.25);
    } else {
      alpha *= T(0.5);
    }
  }
  // outputs and FP64 metrics
  double ud[D];
#pragma unroll
  for (int q = 0; q < D; ++q) ud[q] = double(u[q]);
  const bool owner = active && !aux;  // outputs and FP64 metrics from one thread per state
  if (owner) {
#pragma unroll
    for (int q = 0; q < D; ++q) a.X_out[q * (a.P * Tn) + p * Tn + t] = ud[q];
  }
  double pos = 0, rot = 0;
  unsigned char flags = 3;
  if (owner) {
    TargetK<double> gd = load_target<double>(a.goal, a.P, p, CR_TASK_IK6);
    accept_fp64<N, OBST>(rbd, wd, CR_TASK_IK6, gd, sphd, nob, ud, a.lim_tol, pos, rot, flags);
  }
  // speed / acceleration ratios in FP64 over the states shared in a double buffer
  double* sd = reinterpret_cast<double*>(smem_raw + off + ((TrajSmem<T>::bytes(Tn, D) + 15) & ~size_t(15)));
  double* redd = sd + (size_t)Tn * D;
  if (owner)
#pragma unroll
    for (int q = 0; q < D; ++q) sd[t * D + q] = ud[q];
  __syncthreads();
  double vmax_r = 0, amax_r = 0;
  if (owner && t >= 1) {
#pragma unroll
    for (int q = 0; q < D; ++q) {
      vmax_r = fmax(vmax_r, fabs(ud[q] - sd[(t - 1) * D + q]) / a.dt_d / a.vmax_d);
      if (t >= 2)
        amax_r = fmax(amax_r, fabs(ud[q] - 2.0 * sd[(t - 1) * D + q] + sd[(t - 2) * D + q]) / (a.dt_d * a.dt_d) / a.amax_d);
    }
  }
  double vr = block_max(vmax_r, redd);
  double ar = block_max(amax_r, redd);
  double lim = block_max(double((flags & 1) ? 0 : 1), redd);
  double col = block_max(double((flags & 2) ? 0 : 1), redd);
  if (!aux && t == Tn - 1) {
    a.goal_pos[p] = pos;
    a.goal_rot[p] = rot;
  }
  if (!aux && t == 0) {
    a.F_out[p] = double(F);
    a.speed[p] = vr;
    a.accel[p] = ar;
    a.lim_ok[p] = lim == 0.0;
    a.col_ok[p] = col == 0.0;
  }
}

// ------------------------------------------------------------------------------------------------
// Calibration: theta = (L_1..n, r_c,1..n); residual p(u_k; theta) - p_k.
// ------------------------------------------------------------------------------------------------
// dp/dL_i = Rb_i d_i / L_i (everything after segment i translates); dp/dr_c,i = -(ax dp/dax +
// ay dp/day) / r_c with dp/da_k = v + w x p from the segment twists.
template <typename T, int N>
__device__ void calib_rows(const RobotK<T>& rb, const T (&u)[3 * N], const double* pm, T (&r)[3], T (&J)[3][2 * N]) {
  Chain<T, N> ch;
  chain_forward(rb, u, ch);
  T tv[N][2][3], tw[N][2][3];
  segment_twists(rb, ch, tv, tw);
#pragma unroll
  for (int a = 0; a < 3; ++a) r[a] = ch.p[a] - T(pm[a]);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    T di[3], Rd[3];
    di[0] = rb.L[i] * ch.c[i] * ch.ax[i];
    di[1] = rb.L[i] * ch.c[i] * ch.ay[i];
    di[2] = rb.L[i] * ch.s[i];
    matvec(ch.Rb[i], di, Rd);
    T wp0[3], wp1[3];
    cross(tw[i][0], ch.p, wp0);
    cross(tw[i][1], ch.p, wp1);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      J[a][i] = Rd[a] / rb.L[i];
      T dpx = tv[i][0][a] + wp0[a], dpy = tv[i][1][a] + wp1[a];
      J[a][N + i] = -(ch.ax[i] * dpx + ch.ay[i] * dpy) / rb.rc[i];
    }
  }
}

// FP64 form of calib_rows with what the radius column does not need left out: theta scales with 1 / r_c,
// so that column is the derivative along the bend's own direction, a turn about the bend's fixed axis
// w = (-ay, ax, 0) (J_l(w) w = w) and L d(c ax, c ay, s)/dscale = L (ax (c + 2x c'), ay (c + 2x c'), 2x s').
// The four coefficients are Taylor polynomials up to theta = 3.1417 (seg_coef_poly), the library's sine and
// cosine beyond. About 600 FP64 instructions a pose and three segments against 1000 through
// segment_twists; each holds a sub-partition's FP64 unit 64 cycles.
constexpr double inv_fact(int n) {
  double f = 1.0;
  for (int k = 2; k <= n; ++k) f *= double(k);
  return 1.0 / f;
}
// sum_{k < M} (-1)^k c_k z^k with c_k = 1 / (2k + A)! (times k + 1 with LIN), by Horner's rule. 12 terms in
// y = x / 4 <= 2.468 and 14 in x <= 9.87 leave less than 1e-17 of the leading term.
template <int M, int A, bool LIN> CR_HD double taylor_alt(double z) {
  double v = 0.0;
#pragma unroll
  for (int k = M - 1; k >= 0; --k) {
    const double c = (k % 2 ? -1.0 : 1.0) * (LIN ? double(k + 1) : 1.0) * inv_fact(2 * k + A);
    v = k == M - 1 ? c : fma(v, z, c);
  }
  return v;
}
CR_HD void seg_coef_poly(double x, double& s, double& c, double& s3, double& cp) {
  if (x <= double(kPolyMaxX)) {
    const double y = 0.25 * x;
    const double sc = taylor_alt<12, 1, false>(y);  // sinc(theta / 2)
    s = sc * taylor_alt<12, 0, false>(y);
    c = 0.5 * sc * sc;
    s3 = taylor_alt<14, 3, false>(x);
    cp = -taylor_alt<14, 4, true>(x);
  } else {
    seg_sc_lib(x, s, c);
    seg_deriv_lib(x, s, c, s3, cp);
  }
}
template <int N>
__device__ void calib_pose_f64(const RobotK<double>& rb, const double (&u)[3 * N], const double* pm, double (&r)[3],
                               double (&J)[3][2 * N]) {
  double R[9] = {1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0}, p[3] = {0.0, 0.0, 0.0};
  double v[N][3], wv[N][3], pe[N][3];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double ax, ay, s, c, s3, cp;
    bend_of(rb.K[i], u[3 * i], u[3 * i + 1], u[3 * i + 2], ax, ay);
    const double x = ax * ax + ay * ay, L = rb.L[i];
    seg_coef_poly(x, s, c, s3, cp);
    const double d[3] = {c * ax, c * ay, s};
    const double q = L * fma(2.0 * x, cp, c);
    const double dd[3] = {q * ax, q * ay, L * x * (s3 - c)};  // 2x s' = x (s3 - c)
    if (i == 0) {  // base frame = identity
#pragma unroll
      for (int a = 0; a < 3; ++a) { J[a][i] = d[a]; v[i][a] = dd[a]; }
      wv[i][0] = -ay; wv[i][1] = ax; wv[i][2] = 0.0;
    } else {
      double t[3];
      matvec(R, d, t);
#pragma unroll
      for (int a = 0; a < 3; ++a) J[a][i] = t[a];
      matvec(R, dd, v[i]);
#pragma unroll
      for (int a = 0; a < 3; ++a) wv[i][a] = R[3 * a + 1] * ax - R[3 * a] * ay;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      p[a] = fma(L, J[a][i], p[a]);
      pe[i][a] = p[a];
    }
    if (i + 1 < N) {
      double Ri[9], di[3];
      seg_transform(ax, ay, x, s, c, L, Ri, di);
      if (i == 0) {
#pragma unroll
        for (int a = 0; a < 9; ++a) R[a] = Ri[a];
      } else {
        double Rn[9];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) Rn[3 * a + b] = R[3 * a] * Ri[b] + R[3 * a + 1] * Ri[3 + b] + R[3 * a + 2] * Ri[6 + b];
#pragma unroll
        for (int a = 0; a < 9; ++a) R[a] = Rn[a];
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) r[a] = p[a] - pm[a];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double t[3], wx[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) t[a] = p[a] - pe[i][a];
    cross(wv[i], t, wx);
#pragma unroll
    for (int a = 0; a < 3; ++a) J[a][N + i] = -(v[i][a] + wx[a]) * rb.rc[i];  // rc holds 1 / r_c here (calib_robot_f64)
  }
}

// The LM iteration as one launch, 32 poses (a tile) to a warp. Launch j (1, 2, ...) adds the partial sums
// that launch j - 1 left at its point, applies the LM rule to it, solves for the next trial point and
// evaluates residuals, J^T J, J^T r and F there; so a step costs one evaluation and one launch, and an
// accepted trial's normal equations are at hand. Every block repeats the (short) sums and the solve, which
// spares a grid barrier; block 0 keeps the state. Partial sums and states alternate between two buffers,
// because blocks of one launch still read what the last one wrote. A trial point equal to theta needs no
// evaluation (its cost is F). All sums have a fixed order: a lane adds one entry over its warp's poses in
// order, the block its warps, every block the blocks' partials in four runs; F adds tile totals t, t + 32,
// ... on lane t and then the lanes, which the single-block cost kernel repeats.
// Bound: the FP64 pipe and its latency; 1024 poses are 32 warps in 8 blocks, on 32 of 608 sub-partitions, each busy with
// its own poses' instructions. 20 iterations of 1024 poses in FP64: 0.50 ms; as two launches an iteration, the
// second one block that evaluated the trial cost of all poses on one SM, 2.57 ms.
constexpr int kCalibThreads = 128, kCalibWarps = kCalibThreads / 32;
constexpr int kCalibMaxBlocks = 304;  // two per SM; more tiles are looped over
template <int N> constexpr int calib_nv() { return (2 * N) * (2 * N + 1) / 2 + 2 * N + 1; }
inline __host__ __device__ int64_t calib_tiles(int64_t K) { return (K + 31) / 32; }
inline __host__ __device__ int calib_blocks(int64_t K) {
  const int64_t b = (calib_tiles(K) + kCalibWarps - 1) / kCalibWarps;
  return (int)(b < kCalibMaxBlocks ? b : kCalibMaxBlocks);
}

template <typename T, int N> __device__ RobotK<T> calib_robot(RobotK<T> rb, const double* theta) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    rb.L[i] = T(theta[i]);
    // FP64 rows take 1 / r_c (calib_pose_f64)
    rb.rc[i] = sizeof(T) == 8 ? T(1.0 / theta[N + i]) : T(theta[N + i]);
    rb.K[i] = T(-2.0 / (3.0 * theta[N + i]));
  }
  return rb;
}

__device__ inline double warp_sum_d(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Residual (and Jacobian) of pose k; zero rows past the last pose.
template <typename T, int N>
__device__ void calib_load_pose(const RobotK<T>& rb, const T* __restrict__ U, const double* __restrict__ Pm, int64_t K,
                                int64_t k, T (&r)[3], T (&J)[3][2 * N]) {
  constexpr int D = 3 * N, NP = 2 * N;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r[a] = T(0);
#pragma unroll
    for (int x = 0; x < NP; ++x) J[a][x] = T(0);
  }
  if (k >= K) return;
  T u[D];
#pragma unroll
  for (int q = 0; q < D; ++q) u[q] = U[q * K + k];
  const double pm[3] = {Pm[k], Pm[K + k], Pm[2 * K + k]};
  if constexpr (sizeof(T) == 8) calib_pose_f64<N>(rb, u, pm, r, J);
  else calib_rows<T, N>(rb, u, pm, r, J);
}
// 1/2 |r|^2 of a tile, the same in every lane.
template <typename T> __device__ double calib_tile_cost(const T (&r)[3]) {
  const double r0 = double(r[0]), r1 = double(r[1]), r2 = double(r[2]);
  return warp_sum_d(0.5 * __fma_rn(r2, r2, __fma_rn(r1, r1, __dmul_rn(r0, r0))));
}

// Shared scratch of an evaluation: the poses' rows, column-major with an odd stride, one set per warp.
template <int N> struct CalibSmem {
  static constexpr int NC = 2 * N + 1;  // columns: J, then r
  double row[kCalibWarps][3 * NC][33];
  double red[kCalibWarps][calib_nv<N>()];
};

// This block's share of the sums at theta (robot rb): part [NV - 1] of the block, tileF of its tiles.
template <typename T, int N>
__device__ void calib_eval(const RobotK<T>& rb, const T* __restrict__ U, const double* __restrict__ Pm, int64_t K,
                           double* part, double* tileF, CalibSmem<N>& sm) {
  constexpr int NP = 2 * N, NV = calib_nv<N>(), NE = NV - 1, PER = (NE + 31) / 32, NC = CalibSmem<N>::NC;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int ex[PER], ey[PER];  // this lane's entries: products of columns ex and ey (NP: the residual)
#pragma unroll
  for (int m = 0; m < PER; ++m) {
    int e = lane + 32 * m;
    e = e < NE ? e : NE - 1;
    if (e >= NE - NP) {
      ex[m] = e - (NE - NP);
      ey[m] = NP;
    } else {
      int x = 0;
      while ((x + 1) * (x + 2) / 2 <= e) ++x;
      ex[m] = x;
      ey[m] = e - x * (x + 1) / 2;
    }
  }
  double acc[PER];
#pragma unroll
  for (int m = 0; m < PER; ++m) acc[m] = 0.0;
  const int64_t nt = calib_tiles(K);
  for (int64_t t = (int64_t)blockIdx.x * kCalibWarps + wid; t < nt; t += (int64_t)gridDim.x * kCalibWarps) {
    T r[3], J[3][NP];
    calib_load_pose<T, N>(rb, U, Pm, K, t * 32 + lane, r, J);
    const double Ft = calib_tile_cost(r);
    if (lane == 0) tileF[t] = Ft;
    __syncwarp();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
      for (int x = 0; x < NP; ++x) sm.row[wid][a * NC + x][lane] = double(J[a][x]);
      sm.row[wid][a * NC + NP][lane] = double(r[a]);
    }
    __syncwarp();
#pragma unroll
    for (int m = 0; m < PER; ++m) {
      double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll 8
      for (int j = 0; j < 32; ++j) {
        s0 = fma(sm.row[wid][ex[m]][j], sm.row[wid][ey[m]][j], s0);
        s1 = fma(sm.row[wid][NC + ex[m]][j], sm.row[wid][NC + ey[m]][j], s1);
        s2 = fma(sm.row[wid][2 * NC + ex[m]][j], sm.row[wid][2 * NC + ey[m]][j], s2);
      }
      acc[m] += s0 + s1 + s2;
    }
  }
#pragma unroll
  for (int m = 0; m < PER; ++m)
    if (lane + 32 * m < NE) sm.red[wid][lane + 32 * m] = acc[m];
  __syncthreads();
  for (int e = threadIdx.x; e < NE; e += kCalibThreads) {
    double s = sm.red[0][e];
    for (int w = 1; w < kCalibWarps; ++w) s += sm.red[w][e];
    part[(int64_t)blockIdx.x * NE + e] = s;
  }
}

// The partial sums of nblk blocks and nt tiles added up into tot [NV] (shared), by a block of kCalibThreads.
template <int N>
__device__ void calib_total(const double* part, int nblk, const double* tileF, int64_t nt, double* tot,
                            CalibSmem<N>& sm) {
  constexpr int NV = calib_nv<N>(), NE = NV - 1;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int per = (nblk + kCalibWarps - 1) / kCalibWarps;
  const int b0 = wid * per, b1 = b0 + per < nblk ? b0 + per : nblk;
  for (int e = lane; e < NE; e += 32) {
    double s = 0.0;
#pragma unroll 4
    for (int b = b0; b < b1; ++b) s += part[(int64_t)b * NE + e];
    sm.red[wid][e] = s;
  }
  if (wid == kCalibWarps - 1) {
    double f = 0.0;
#pragma unroll 4
    for (int64_t t = lane; t < nt; t += 32) f += tileF[t];
    f = warp_sum_d(f);
    if (lane == 0) tot[NV - 1] = f;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < NE; e += kCalibThreads) {
    double s = sm.red[0][e];
    for (int w = 1; w < kCalibWarps; ++w) s += sm.red[w][e];
    tot[e] = s;
  }
  __syncthreads();
}

// One warp: the damped step from the sums tot [NV] at theta: trial [NP] (theta where the factorisation
// fails) and the predicted decrease, the same in every lane; returns whether every pivot was positive.
template <int N>
__device__ bool calib_solve(const double* tot, const double* theta, double lam, double* trial, double& pred,
                            double* col, double* colr) {
  constexpr int NP = 2 * N, NA = NP * (NP + 1) / 2, SL = AugSlots<NP>::SL;
  const int lane = threadIdx.x & 31;
  const AugSlots<NP> sl = aug_slots<NP>(lane);
  double v[SL];
#pragma unroll
  for (int s = 0; s < SL; ++s) {
    v[s] = 0.0;
    if (!sl.on[s]) continue;
    const int i = sl.r[s], j = sl.c[s];
    if (i < NP) {
      v[s] = tot[tri(i, j)];
      if (i == j) v[s] += lam * fmax(v[s], 1e-12);
    } else if (j < NP) {
      v[s] = -tot[NA + j];
    }
  }
  const bool ok = sweep_aug<double, NP>(v, sl, col, colr);
#pragma unroll
  for (int s = 0; s < SL; ++s)
    if (sl.on[s] && sl.r[s] == NP && sl.c[s] < NP) col[sl.c[s]] = v[s];
  __syncwarp();
  double pl = 0.0;
  if (lane < NP) {
    const double x = col[lane];
    trial[lane] = ok ? theta[lane] + x : theta[lane];
    pl = x * (lam * fmax(tot[tri(lane, lane)], 1e-12) * x - tot[NA + lane]);
  }
  pred = 0.5 * warp_sum_d(pl);
  __syncwarp();
  return ok;
}

// The LM rule for a trial of cost Fn (taken = whether theta moves to it).
__device__ inline bool calib_rule(bool ok, double F, double Fn, double pred, double& lam, double& nu) {
  if (ok && Fn < F) {
    const double rho = (F - Fn) / pred, tt = 2.0 * rho - 1.0;
    lam *= fmax(1.0 / 3.0, 1.0 - tt * tt * tt);
    nu = 2.0;
    return true;
  }
  lam *= nu;
  nu *= 2.0;
  return false;
}

// Workspace of cr_calibrate, in doubles: two states [4 + 2 NP + NV] (lambda, nu, predicted decrease, 0 =
// evaluated / 1 = trial equal to theta / 2 = failed factorisation, theta, trial, sums at theta), then two
// sets of partial sums [nblk][NV - 1] and tile costs [tiles].
template <int N> constexpr int calib_state_len() { return 4 + 4 * N + calib_nv<N>(); }
inline size_t calibrate_ws_bytes(int n, int64_t K) {
  const int NP = 2 * n, NV = NP * (NP + 1) / 2 + NP + 1;
  return (size_t)(2 * ((4 + 2 * NP + NV) + (int64_t)calib_blocks(K) * (NV - 1) + calib_tiles(K))) * sizeof(double);
}

template <typename T, int N>
__global__ void __launch_bounds__(kCalibThreads) k_calib_eval(RobotK<T> rb0, const T* __restrict__ U,
                                                             const double* __restrict__ Pm, int64_t K,
                                                             const double* theta, double* part, double* tileF) {
  __shared__ CalibSmem<N> sm;
  __shared__ RobotK<T> rbs;
  if (threadIdx.x == 0) rbs = calib_robot<T, N>(rb0, theta);
  __syncthreads();
  calib_eval<T, N>(rbs, U, Pm, K, part, tileF, sm);
}

// Launch j of the calibration (see above); j = iters + 1 only applies the rule and writes the results.
template <typename T, int N>
__global__ void __launch_bounds__(kCalibThreads) k_calib_iter(RobotK<T> rb0, const T* __restrict__ U,
                                                             const double* __restrict__ Pm, int64_t K, int nblk, int j,
                                                             int iters, double lambda0, double* theta, double* ws,
                                                             double* F_out, double* hist) {
  constexpr int NP = 2 * N, NV = calib_nv<N>(), ST = calib_state_len<N>();
  __shared__ CalibSmem<N> sm;
  __shared__ RobotK<T> rbs;
  __shared__ double tot[NV], cur[NV], th[NP], tr[NP], col[32], colr[32];
  __shared__ int skip;
  const int64_t nt = calib_tiles(K);
  const int64_t pset = (int64_t)nblk * (NV - 1) + nt;
  const double* old = ws + (j & 1 ? 0 : ST);  // the state that launch j - 1 wrote
  double* neu = ws + (j & 1 ? ST : 0);
  const double* part = ws + 2 * ST + (j & 1 ? 0 : pset);
  double* partn = ws + 2 * ST + (j & 1 ? pset : 0);
  const int was = j > 1 ? (int)old[3] : 0;  // how the last trial ended
  if (was == 0) calib_total<N>(part, nblk, part + (int64_t)nblk * (NV - 1), nt, tot, sm);
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    double lam = lambda0, nu = 2.0;
    bool taken = true;
    if (j > 1) {
      lam = old[0];
      nu = old[1];
      const double F = old[4 + 2 * NP + NV - 1];
      taken = calib_rule(was != 2, F, was == 0 ? tot[NV - 1] : F, old[2], lam, nu);
    }
    if (lane < NP) th[lane] = j == 1 ? theta[lane] : old[4 + (taken ? NP : 0) + lane];
    for (int e = lane; e < NV; e += 32) cur[e] = taken ? tot[e] : old[4 + 2 * NP + e];
    __syncwarp();
    if (blockIdx.x == 0 && hist && j > 1 && lane < NP) hist[(int64_t)(j - 2) * NP + lane] = th[lane];
    if (j == iters + 1) {
      if (blockIdx.x == 0) {
        if (lane < NP) theta[lane] = th[lane];
        if (lane == 0) *F_out = cur[NV - 1];
      }
      if (lane == 0) skip = 1;
    } else {
      double pred;
      const bool ok = calib_solve<N>(cur, th, lam, tr, pred, col, colr);
      const bool still = __all_sync(0xffffffffu, lane >= NP || tr[lane < NP ? lane : 0] == th[lane < NP ? lane : 0]);
      if (lane == 0) skip = !ok ? 2 : (still ? 1 : 0);
      if (blockIdx.x == 0) {
        if (lane == 0) {
          neu[0] = lam;
          neu[1] = nu;
          neu[2] = pred;
          neu[3] = double(!ok ? 2 : (still ? 1 : 0));
        }
        if (lane < NP) {
          neu[4 + lane] = th[lane];
          neu[4 + NP + lane] = tr[lane];
        }
        for (int e = lane; e < NV; e += 32) neu[4 + 2 * NP + e] = cur[e];
      }
    }
  }
  __syncthreads();
  if (skip) return;
  if (threadIdx.x == 0) rbs = calib_robot<T, N>(rb0, tr);
  __syncthreads();
  calib_eval<T, N>(rbs, U, Pm, K, partn, partn + (int64_t)nblk * (NV - 1), sm);
}

// Sharded calibration: the pieces of k_calib_iter as separate launches, so that processes holding
// shares of the poses can add their partial sums (an all-reduce) in between. Each piece runs the same
// routines in the same order, so one process running them equals cr_calibrate.
// sums [NV]: the share's packed J^T J, J^T r and F; state [4]: lambda, nu, ok, pred.
template <int N>
__global__ void __launch_bounds__(kCalibThreads) k_calib_sum_parts(int nblk, int64_t nt, const double* part,
                                                                  const double* tileF, double* sums) {
  constexpr int NV = calib_nv<N>();
  __shared__ CalibSmem<N> sm;
  __shared__ double tot[NV];
  calib_total<N>(part, nblk, tileF, nt, tot, sm);
  for (int e = threadIdx.x; e < NV; e += blockDim.x) sums[e] = tot[e];
}

template <int N>
__global__ void __launch_bounds__(32) k_calib_trial(const double* sums, const double* theta, double* state,
                                                    double* theta_trial) {
  constexpr int NP = 2 * N, NV = calib_nv<N>();
  __shared__ double tot[NV], th[NP], tr[NP], col[32], colr[32];
  for (int e = threadIdx.x; e < NV; e += 32) tot[e] = sums[e];
  if (threadIdx.x < NP) th[threadIdx.x] = theta[threadIdx.x];
  __syncwarp();
  double pred;
  const bool ok = calib_solve<N>(tot, th, state[0], tr, pred, col, colr);
  if (threadIdx.x < NP) theta_trial[threadIdx.x] = tr[threadIdx.x];
  if (threadIdx.x == 0) {
    state[2] = ok ? 1.0 : 0.0;
    state[3] = ok ? pred : 0.0;
  }
}

// F at theta over all poses by one block of 32 warps' worth of tile runs (run l: tiles l, l + 32, ...), added
// in calib_total's order.
constexpr int kCalibCostThreads = 256;
template <typename T, int N>
__global__ void __launch_bounds__(kCalibCostThreads) k_calib_cost(RobotK<T> rb0, const T* __restrict__ U,
                                                                 const double* __restrict__ Pm, int64_t K,
                                                                 const double* theta, double* F_out) {
  __shared__ RobotK<T> rbs;
  __shared__ double run[32];
  if (threadIdx.x == 0) rbs = calib_robot<T, N>(rb0, theta);
  __syncthreads();
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t nt = calib_tiles(K);
  for (int l = wid; l < 32; l += kCalibCostThreads / 32) {
    double f = 0.0;
    for (int64_t t = l; t < nt; t += 32) {
      T r[3], J[3][2 * N];
      calib_load_pose<T, N>(rbs, U, Pm, K, t * 32 + lane, r, J);
      f += calib_tile_cost(r);
    }
    if (lane == 0) run[l] = f;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const double F = warp_sum_d(run[lane]);
    if (lane == 0) *F_out = F;
  }
}

template <int N>
__global__ void k_calib_accept(const double* sums, const double* F_trial, const double* theta_trial, double* theta,
                               double* state) {
  constexpr int NP = 2 * N, NV = calib_nv<N>();
  if (threadIdx.x != 0) return;
  double lam = state[0], nu = state[1];
  if (calib_rule(state[2] != 0.0, sums[NV - 1], *F_trial, state[3], lam, nu)) {
#pragma unroll
    for (int q = 0; q < NP; ++q) theta[q] = theta_trial[q];
  }
  state[0] = lam;
  state[1] = nu;
}

// ------------------------------------------------------------------------------------------------
// Host launchers
// ------------------------------------------------------------------------------------------------
struct TrajLaunch {
  cr_robot robot;
  cr_scene scene;
  cr_traj_task task;
  const void* x;
  void *cost, *grad;
  const void* upstream;
  // solve
  const double* u_goal;
  const double* x_init;  // nullable
  int k_traj;
  double alpha0, lim_tol;
  double *X_out, *F_out, *goal_pos, *goal_rot, *speed, *accel;
  unsigned char *lim_ok, *col_ok;
  // calibration
  const void* U;
  const double* Pm;
  int64_t K;
  int iters;
  double lambda0;
  double *theta_dev, *F_dev, *hist_dev;
  void* calib_ws;
  // sharded calibration: which piece (0 sums, 1 trial, 2 cost, 3 accept) and its arrays
  int calib_piece;
  double *sums, *state, *theta_trial;
  const double* F_trial;
  cudaStream_t stream;
};

template <typename T> cr_status launch_traj_cost(const TrajLaunch& l);
template <typename T> cr_status launch_traj_solve(const TrajLaunch& l);
template <typename T> cr_status launch_calibrate(const TrajLaunch& l);
template <typename T> cr_status launch_calib_piece(const TrajLaunch& l);

template <typename T> TrajW<T> traj_w(const cr_weights& w) {
  TrajW<T> t;
  t.dt = T(w.dt);
  t.vmax = T(w.v_max);
  t.amax = T(w.a_max);
  t.w_len = T(w.w_len);
  t.rho_v = T(w.rho_v);
  t.rho_a = T(w.rho_a);
  return t;
}

template <typename T> TrajArgs<T> traj_args(const TrajLaunch& l) {
  TrajArgs<T> a{};
  a.u_start = l.task.u_start;
  a.goal = l.task.goal;
  a.P = l.task.P;
  a.Tn = l.task.T;
  a.spheres = l.scene.spheres;
  a.no = l.scene.n_o;
  a.prims = l.scene.prims;
  a.np = l.scene.n_p;
  a.sph_pp = (l.scene.per_problem && l.scene.n_o + l.scene.n_p > 0) ? 1 : 0;
  a.x = (const T*)l.x;
  a.cost = (T*)l.cost;
  a.grad = (T*)l.grad;
  a.upstream = (const T*)l.upstream;
  a.u_goal = l.u_goal;
  a.x_init = l.x_init;
  a.k_traj = l.k_traj;
  a.alpha0 = T(l.alpha0);
  a.lim_tol = l.lim_tol;
  a.dt_d = l.task.w.dt;
  a.vmax_d = l.task.w.v_max;
  a.amax_d = l.task.w.a_max;
  a.X_out = l.X_out;
  a.F_out = l.F_out;
  a.goal_pos = l.goal_pos;
  a.goal_rot = l.goal_rot;
  a.speed = l.speed;
  a.accel = l.accel;
  a.lim_ok = l.lim_ok;
  a.col_ok = l.col_ok;
  return a;
}

template <typename T, int N> cr_status traj_cost_n(const TrajLaunch& l) {
  constexpr int D = 3 * N;
  RobotK<T> rb = crh::robot_k<T>(l.robot);
  WeightsK<T> w = crh::weights_k<T>(l.task.w);
  TrajW<T> tw = traj_w<T>(l.task.w);
  TrajArgs<T> a = traj_args<T>(l);
  const int threads = ((a.Tn + 31) / 32) * 32;
  size_t sm = ((obstacles_smem<T>(a.no, a.np) + 15) & ~size_t(15)) + TrajSmem<T>::bytes(a.Tn, D);
  cr_status st;
  if (a.no + a.np > 0 || w.rho_s > T(0)) {  // collision rows: obstacles and / or self-contact
    if (l.grad) { if ((st = set_smem(k_traj_cost<T, N, true, true>, sm))) return st;
      k_traj_cost<T, N, true, true><<<(unsigned)a.P, threads, sm, l.stream>>>(rb, w, tw, a); }
    else { if ((st = set_smem(k_traj_cost<T, N, true, false>, sm))) return st;
      k_traj_cost<T, N, true, false><<<(unsigned)a.P, threads, sm, l.stream>>>(rb, w, tw, a); }
  } else {
    if (l.grad) { if ((st = set_smem(k_traj_cost<T, N, false, true>, sm))) return st;
      k_traj_cost<T, N, false, true><<<(unsigned)a.P, threads, sm, l.stream>>>(rb, w, tw, a); }
    else { if ((st = set_smem(k_traj_cost<T, N, false, false>, sm))) return st;
      k_traj_cost<T, N, false, false><<<(unsigned)a.P, threads, sm, l.stream>>>(rb, w, tw, a); }
  }
  return crh::check_launch("cr_traj_cost");
}

template <typename T, int N> cr_status traj_solve_n(const TrajLaunch& l) {
  constexpr int D = 3 * N;
  RobotK<T> rb = crh::robot_k<T>(l.robot);
  WeightsK<T> w = crh::weights_k<T>(l.task.w);
  RobotK<double> rbd = crh::robot_k<double>(l.robot);
  WeightsK<double> wd = crh::weights_k<double>(l.task.w);
  TrajW<T> tw = traj_w<T>(l.task.w);
  TrajArgs<T> a = traj_args<T>(l);
  // FP32 with obstacles: two threads per state share the clearance rows (the FP64 form keeps one, its
  // sums in the oracle's order)
  const int Wt = ((a.Tn + 31) / 32) * 32;
  const int threads = (sizeof(T) == 4 && a.no + a.np >= 2 && 2 * Wt <= 256) ? 2 * Wt : Wt;
  size_t sm = ((obstacles_smem<T>(a.no, a.np) + 15) & ~size_t(15)) +
              ((obstacles_smem<double>(a.no, a.np) + 15) & ~size_t(15)) +
              ((TrajSmem<T>::bytes(a.Tn, D) + 15) & ~size_t(15)) + ((size_t)a.Tn * D + 32) * sizeof(double);
  cr_status st;
  if (a.np > 0) {
    if ((st = set_smem(k_traj_solve<T, N, true>, sm))) return st;
    k_traj_solve<T, N, true><<<(unsigned)a.P, threads, sm, l.stream>>>(rb, w, tw, rbd, wd, a);
  } else if (a.no > 0 || w.rho_s > T(0)) {  // spheres and / or self-contact: the form without primitive code
    if ((st = set_smem(k_traj_solve<T, N, true, false>, sm))) return st;
    k_traj_solve<T, N, true, false><<<(unsigned)a.P, threads, sm, l.stream>>>(rb, w, tw, rbd, wd, a);
  } else {
    if ((st = set_smem(k_traj_solve<T, N, false>, sm))) return st;
    k_traj_solve<T, N, false><<<(unsigned)a.P, threads, sm, l.stream>>>(rb, w, tw, rbd, wd, a);
  }
  return crh::check_launch("cr_solve_traj");
}

template <typename T, int N> cr_status calibrate_n(const TrajLaunch& l) {
  const RobotK<T> rb = crh::robot_k<T>(l.robot);
  const int nblk = calib_blocks(l.K);
  double* ws = (double*)l.calib_ws;
  const T* U = (const T*)l.U;
  double* part = ws + 2 * calib_state_len<N>();
  k_calib_eval<T, N><<<nblk, kCalibThreads, 0, l.stream>>>(rb, U, l.Pm, l.K, l.theta_dev, part,
                                                          part + (int64_t)nblk * (calib_nv<N>() - 1));
  for (int j = 1; j <= l.iters + 1; ++j)
    k_calib_iter<T, N><<<j <= l.iters ? nblk : 1, kCalibThreads, 0, l.stream>>>(
        rb, U, l.Pm, l.K, nblk, j, l.iters, l.lambda0, l.theta_dev, ws, l.F_dev, l.hist_dev);
  return crh::check_launch("cr_calibrate");
}

template <typename T, int N> cr_status calib_piece_n(const TrajLaunch& l) {
  RobotK<T> rb = crh::robot_k<T>(l.robot);
  const T* U = (const T*)l.U;
  switch (l.calib_piece) {
    case 0: {  // partial sums of this share: per-block partials, then their total
      const int nblk = calib_blocks(l.K);
      double* part = (double*)l.calib_ws + 2 * calib_state_len<N>();
      double* tileF = part + (int64_t)nblk * (calib_nv<N>() - 1);
      k_calib_eval<T, N><<<nblk, kCalibThreads, 0, l.stream>>>(rb, U, l.Pm, l.K, l.theta_dev, part, tileF);
      k_calib_sum_parts<N><<<1, kCalibThreads, 0, l.stream>>>(nblk, calib_tiles(l.K), part, tileF, l.sums);
      break;
    }
    case 1: k_calib_trial<N><<<1, 32, 0, l.stream>>>(l.sums, l.theta_dev, l.state, l.theta_trial); break;
    case 2:
      k_calib_cost<T, N><<<1, kCalibCostThreads, 0, l.stream>>>(rb, U, l.Pm, l.K, l.theta_dev, l.F_dev);
      break;
    default: k_calib_accept<N><<<1, 32, 0, l.stream>>>(l.sums, l.F_trial, l.theta_trial, l.theta_dev, l.state);
  }
  return crh::check_launch("sharded calibration");
}

#define CR_TRAJ_DISPATCH(FN, T, l)         \
  switch ((l).robot.n) {                   \
    case 1: return FN<T, 1>(l);            \
    case 2: return FN<T, 2>(l);            \
    case 3: return FN<T, 3>(l);            \
    case 4: return FN<T, 4>(l);            \
    case 5: return FN<T, 5>(l);            \
    default: return FN<T, 6>(l);           \
  }

template <typename T> cr_status launch_traj_cost(const TrajLaunch& l) { CR_TRAJ_DISPATCH(traj_cost_n, T, l) }
template <typename T> cr_status launch_traj_solve(const TrajLaunch& l) { CR_TRAJ_DISPATCH(traj_solve_n, T, l) }
template <typename T> cr_status launch_calibrate(const TrajLaunch& l) { CR_TRAJ_DISPATCH(calibrate_n, T, l) }
template <typename T> cr_status launch_calib_piece(const TrajLaunch& l) { CR_TRAJ_DISPATCH(calib_piece_n, T, l) }

#define CR_TRAJ_INSTANTIATE(EXT, T)                                  \
  EXT template cr_status launch_traj_cost<T>(const TrajLaunch&);     \
  EXT template cr_status launch_traj_solve<T>(const TrajLaunch&);    \
  EXT template cr_status launch_calibrate<T>(const TrajLaunch&);    \
  EXT template cr_status launch_calib_piece<T>(const TrajLaunch&);

}  // namespace crk
