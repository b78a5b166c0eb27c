// Tangent-linear (forward-mode) derivative of the substep along a direction
// of the rates (d k_off, d v_walk, d k_on), carried alongside the state
// (mm_set_tangent): every substep advances the state and its tangent
// (dpsi, dMb, dMf, dn_b) together, in one launch, so the derivative of an
// observable with respect to one scalar parameter costs one pass of about
// twice the forward's memory traffic and needs no checkpoints -- the reverse
// sweep (mm_adjoint_step) is the tool for many parameters at once (the
// velocity field, the initial psi).
//
// The map differentiated is the discrete substep exactly as the forward
// computes it, at a fixed dt, on the branches the forward takes (donor-cell
// upwinding, the Superbee limiter, the Alg. 2 scale-down), the float32 form's
// mass-correction factor a constant of the map: the same readings as the
// reverse sweep and the oracle's tangent substep. The forward part of the
// kernel is the plain substep's arithmetic (psi_point; the flux of walk_dflux), so the
// state advances as in the plain path up to the rounding of the row loads.
#include <algorithm>

#include "mm_cell.cuh"
#include "mm_rows.cuh"
#include "mm_host.h"

namespace mm {

template <typename T>
struct TanArgs {
  StepArgs<T> a;
  const T* dpsi_in;
  T* dpsi_out;
  const T* dnb_in;
  T* dnb_out;
  T* dmb;       // [cells][nth][ns] in place
  T* dmf;       // [cells] in place
  double dkoff, dvw, dkon;
};

// Per-warp shared memory of the tangent substep: the new psi and dpsi of the
// cell, and the new rows' n_b and dn_b.
__host__ __device__ inline size_t tan_warp_smem(int nth, int tsz) {
  return (size_t)4 * nth * tsz;
}

// d of the donor-cell flux max(A, 0) pl + min(A, 0) pr on the branch taken
// (the right state when A = 0).
template <typename T>
__device__ __forceinline__ T donor_tl(T A, T pl, T pr, T dA, T dpl, T dpr) {
  return fma_t(tmax(A, T(0)), dpl, tmin(A, T(0)) * dpr) + dA * (A > T(0) ? pl : pr);
}

// dpsi^{n+1} of one (cell, theta), with no velocity perturbation: the face
// velocities change through dn_b (the gliding speed), the fluxes through them
// and through dpsi. The face speeds are psi_point's, so that the two inlined
// side by side compute them once.
template <typename T>
__device__ __forceinline__ T psi_point_tl(const PsiConst<T>& q, const CellVel<T>& u,
                                          const LaneTrig<T>& t, const PsiIn<T>& in,
                                          const PsiIn<T>& di) {
  const T g = q.g;
  const T Pc = g * in.pc, Pe = g * in.pe, Pw = g * in.pw, Pn = g * in.pn, Ps = g * in.ps;
  const T dPc = g * di.pc, dPe = g * di.pe, dPw = g * di.pw, dPn = g * di.pn, dPs = g * di.ps;
  const T ck = t.ck, sk = t.sk;
  const T Vc = fma_t(q.glide, in.nc, q.vsp), Ve = fma_t(q.glide, in.ne, q.vsp);
  const T Vw = fma_t(q.glide, in.nw, q.vsp);
  const T Vn = fma_t(q.glide, in.nn, q.vsp);
  const T Vs = fma_t(q.glide, in.ns, q.vsp);
  const T axc = fma_t(-Vc, ck, u.uxc), axe = fma_t(-Ve, ck, u.uxe), axw = fma_t(-Vw, ck, u.uxw);
  const T ayc = fma_t(-Vc, sk, u.uyc), ayn = fma_t(-Vn, sk, u.uyn), ays = fma_t(-Vs, sk, u.uys);
  const T Ae = half_t(axc + axe), Aw = half_t(axw + axc);
  const T An = half_t(ayc + ayn), As = half_t(ays + ayc);
  // d(u - (v_sp + glide n_b) p) = -glide dn_b p
  const T gc = -q.glide * ck, gs = -q.glide * sk;
  const T daxc = gc * di.nc, daxe = gc * di.ne, daxw = gc * di.nw;
  const T dayc = gs * di.nc, dayn = gs * di.nn, days = gs * di.ns;
  const T dAe = T(0.5) * (daxc + daxe), dAw = T(0.5) * (daxw + daxc);
  const T dAn = T(0.5) * (dayc + dayn), dAs = T(0.5) * (days + dayc);
  const T cp = t.cp, sp = t.sp, cm = t.cm, sm = t.sm;
  const T wp = fma_t(-sp, fma_t(u.Gxx, cp, u.Gxy * sp), cp * fma_t(u.Gyx, cp, u.Gyy * sp));
  const T wm = fma_t(-sm, fma_t(u.Gxx, cm, u.Gxy * sm), cm * fma_t(u.Gyx, cm, u.Gyy * sm));
  const T dFe = donor_tl(Ae, Pc, Pe, dAe, dPc, dPe), dFw = donor_tl(Aw, Pw, Pc, dAw, dPw, dPc);
  const T dFn = donor_tl(An, Pc, Pn, dAn, dPc, dPn), dFs = donor_tl(As, Ps, Pc, dAs, dPs, dPc);
  const T dFp = donor_tl(wp, Pc, g * in.pp, T(0), dPc, g * di.pp);
  const T dFm = donor_tl(wm, g * in.pm, Pc, T(0), g * di.pm, dPc);
  return dPc - q.dt * ((dFe - dFw) * q.inv_dx + (dFn - dFs) * q.inv_dy + (dFp - dFm) * q.inv_dth);
}

// Orientation k of a cell and its neighbours from the columns at p and n (the
// cell's and its neighbours' offsets in o), without the theta neighbours.
template <typename T>
__device__ __forceinline__ PsiIn<T> psi_in(const T* p, const T* n, const size_t (&o)[5], int k) {
  return PsiIn<T>{p[o[0] + k], p[o[1] + k], p[o[2] + k], p[o[3] + k], p[o[4] + k], T(0),
                  T(0),        n[o[0] + k], n[o[1] + k], n[o[2] + k], n[o[3] + k], n[o[4] + k]};
}

// The walking term and its tangent on a lane's V nodes: D as walk_dflux, and
// dD = dF_{j-1} - dF_j with dF = dM + ga da + gb db on the Superbee branch
// the forward takes (ga, gb from walk_dflux).
//
// The branch is chosen with the comparisons of walk_dflux<..., true> and its
// term taken at once: sigma/2 is one of a, b/2, a/2, b or 0, so its
// derivative is the same one of da, db/2, da/2, db or 0 (each exact), and
// dF = dM + that term rounds once, as dM + ga da + gb db does.
template <typename T, int V>
__device__ __forceinline__ void walk_tl(const T (&M)[V], const T (&dM)[V], T (&D)[V], T (&dD)[V],
                                        bool first, bool last, int seg) {
  T ml = __shfl_up_sync(0xffffffffu, M[V - 1], 1, seg);
  const T mr = __shfl_down_sync(0xffffffffu, M[0], 1, seg);
  T dml = __shfl_up_sync(0xffffffffu, dM[V - 1], 1, seg);
  const T dmr = __shfl_down_sync(0xffffffffu, dM[0], 1, seg);
  if (first) {
    ml = T(0);
    dml = T(0);
  }
  // d[i] = M_i - M_{i-1} and dd[i] = dM_i - dM_{i-1}, i = 0..V
  T d[V + 1], hd[V + 1], dd[V + 1];
  d[0] = M[0] - ml;
  dd[0] = dM[0] - dml;
#pragma unroll
  for (int v = 1; v < V; ++v) {
    d[v] = M[v] - M[v - 1];
    dd[v] = dM[v] - dM[v - 1];
  }
  d[V] = mr - M[V - 1];
  dd[V] = dmr - dM[V - 1];
#pragma unroll
  for (int i = 0; i <= V; ++i) hd[i] = T(0.5) * d[i];
  T F[V], dF[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    bool pos, p1, x1a, x2a;
    if constexpr (sizeof(T) == 8) {
      // the flux and decisions of walk_dflux<double, V, true> (bit patterns)
      const Lim64 q = superbee64(d[v], hd[v], d[v + 1], hd[v + 1], v == V - 1 && last, M[v]);
      F[v] = q.F;
      pos = q.pos;
      p1 = q.p1;
      x1a = q.x1a;
      x2a = q.x2a;
    } else {
      T sgn = copysign(T(1), d[v + 1]);
      if (v == V - 1 && last) sgn = T(0);  // plus end: F = M, no slope
      const T A = d[v] * sgn, hA = hd[v] * sgn;
      const T hB = fabs(hd[v + 1]), B = fabs(d[v + 1]);
      const T t1 = tmin(A, hB), t2 = tmin(hA, B);
      const T r = max3_t(t1, t2, T(0));
      F[v] = fma_t(r, sgn, M[v]);
      pos = r > T(0);
      p1 = t1 > t2;
      x1a = A < hB;
      x2a = hA < B;
    }
    const T e1 = x1a ? dd[v] : T(0.5) * dd[v + 1];   // t1 = a (sigma/2 = a) or |b|/2
    const T e2 = x2a ? T(0.5) * dd[v] : dd[v + 1];   // t2 = a/2 or |b|
    const T g = pos ? (p1 ? e1 : e2) : T(0);
    dF[v] = dM[v] + g;
  }
  T fl = __shfl_up_sync(0xffffffffu, F[V - 1], 1, seg);
  T dfl = __shfl_up_sync(0xffffffffu, dF[V - 1], 1, seg);
  if (first) {
    fl = T(0);
    dfl = T(0);
  }
  D[0] = fl - F[0];
  dD[0] = dfl - dF[0];
#pragma unroll
  for (int v = 1; v < V; ++v) {
    D[v] = F[v - 1] - F[v];
    dD[v] = dF[v - 1] - dF[v];
  }
}

// walk_tl for float32 on register pairs (nodes 2k, 2k + 1): the branch as
// coefficients (branch_x2), dF = dM + ga da + gb db. One of ga, gb is 0, so
// the sum rounds once, as above.
template <int V>
__device__ __forceinline__ void walk_tl_x2(const float2 (&M)[V / 2], const float2 (&dM)[V / 2],
                                           float2 (&D)[V / 2], float2 (&dD)[V / 2], bool first,
                                           bool last, int seg) {
  constexpr int H = V / 2;
  float ml = __shfl_up_sync(0xffffffffu, M[H - 1].y, 1, seg);
  const float mr = __shfl_down_sync(0xffffffffu, M[0].x, 1, seg);
  float dml = __shfl_up_sync(0xffffffffu, dM[H - 1].y, 1, seg);
  const float dmr = __shfl_down_sync(0xffffffffu, dM[0].x, 1, seg);
  if (first) {
    ml = 0.0f;
    dml = 0.0f;
  }
  // backward differences of the nodes and, last, the forward one of node V - 1
  float2 d[H], dd[H], hd[H];
#pragma unroll
  for (int k = 0; k < H; ++k) {
    d[k] = make_float2(M[k].x - (k ? M[k ? k - 1 : 0].y : ml), M[k].y - M[k].x);
    dd[k] = make_float2(dM[k].x - (k ? dM[k ? k - 1 : 0].y : dml), dM[k].y - dM[k].x);
  }
  const float dV = mr - M[H - 1].y, hdV = 0.5f * dV, ddV = dmr - dM[H - 1].y;
  const float2 half2 = make_float2(0.5f, 0.5f);
#pragma unroll
  for (int k = 0; k < H; ++k) hd[k] = __fmul2_rn(half2, d[k]);
  float2 F[H], dF[H];
#pragma unroll
  for (int k = 0; k < H; ++k) {
    const int n = k + 1 < H ? k + 1 : k;
    const float b1 = k + 1 < H ? d[n].x : dV, hb1 = k + 1 < H ? hd[n].x : hdV;
    const float db1 = k + 1 < H ? dd[n].x : ddV;
    float2 sg = make_float2(copysignf(1.0f, d[k].y), copysignf(1.0f, b1));
    if (k == H - 1 && last) sg.y = 0.0f;  // plus end: F = M, no slope
    float2 r, ga, gb;
    branch_x2(__fmul2_rn(d[k], sg), __fmul2_rn(hd[k], sg),
              make_float2(fabsf(hd[k].y), fabsf(hb1)), make_float2(fabsf(d[k].y), fabsf(b1)), r, ga,
              gb);
    F[k] = __ffma2_rn(r, sg, M[k]);
    dF[k] = __ffma2_rn(gb, make_float2(dd[k].y, db1), __ffma2_rn(ga, dd[k], dM[k]));
  }
  float fl = __shfl_up_sync(0xffffffffu, F[H - 1].y, 1, seg);
  float dfl = __shfl_up_sync(0xffffffffu, dF[H - 1].y, 1, seg);
  if (first) {
    fl = 0.0f;
    dfl = 0.0f;
  }
#pragma unroll
  for (int k = 0; k < H; ++k) {
    D[k] = make_float2((k ? F[k ? k - 1 : 0].y : fl) - F[k].x, F[k].x - F[k].y);
    dD[k] = make_float2((k ? dF[k ? k - 1 : 0].y : dfl) - dF[k].x, dF[k].x - dF[k].y);
  }
}

// The scalars of the rows' equations: the substep's and their tangents, and
// the cell's sources.
template <typename T>
struct TlRow {
  T cw, koff, dt, hdt, dcw, dkoff;
  T c3, e3, dsrc;  // dt/2 k_on Mf, dt k_on Mf, d(k_on Mf)
};

// The RK2 of Eq. 4 and its tangent on a lane's V nodes, in place:
// Ms = M + dt/2 R(M), dMs = dM + dt/2 dR(M, dM), then M + dt R(Ms) and
// dM + dt dR(Ms, dMs); snb and sdnb are the sums of the new nodes, of eight as
// two fours (slot 1 is 0 for fewer).
template <typename T, int V>
__device__ __forceinline__ void rows_tl(T (&M)[V], T (&dM)[V], const TlRow<T>& q, bool first,
                                        bool last, int seg, T (&snb)[2], T (&sdnb)[2]) {
  snb[0] = snb[1] = T(0);
  sdnb[0] = sdnb[1] = T(0);
  if constexpr (sizeof(T) == 4 && V % 2 == 0) {
    constexpr int H = V / 2;
    const auto b2 = [](float x) { return make_float2(x, x); };
    float2 m[H], dm[H], D[H], dD[H], s[H], ds[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
      m[k] = make_float2(M[2 * k], M[2 * k + 1]);
      dm[k] = make_float2(dM[2 * k], dM[2 * k + 1]);
    }
    walk_tl_x2<V>(m, dm, D, dD, first, last, seg);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      s[k] = __ffma2_rn(b2(q.hdt * q.cw), D[k],
                        __ffma2_rn(b2(1.0f - q.hdt * q.koff), m[k], b2(q.c3)));
      const float2 dR = __ffma2_rn(
          b2(q.cw), dD[k],
          __ffma2_rn(b2(q.dcw), D[k],
                     __ffma2_rn(b2(-q.koff), dm[k], __ffma2_rn(b2(-q.dkoff), m[k], b2(q.dsrc)))));
      ds[k] = __ffma2_rn(b2(q.hdt), dR, dm[k]);
    }
    walk_tl_x2<V>(s, ds, D, dD, first, last, seg);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const float2 dR = __ffma2_rn(
          b2(q.cw), dD[k],
          __ffma2_rn(b2(q.dcw), D[k],
                     __ffma2_rn(b2(-q.koff), ds[k], __ffma2_rn(b2(-q.dkoff), s[k], b2(q.dsrc)))));
      const float2 y = __ffma2_rn(b2(q.dt * q.cw), D[k],
                                  __ffma2_rn(b2(-q.dt * q.koff), s[k], __fadd2_rn(m[k], b2(q.e3))));
      const float2 dy = __ffma2_rn(b2(q.dt), dR, dm[k]);
      M[2 * k] = y.x;
      M[2 * k + 1] = y.y;
      dM[2 * k] = dy.x;
      dM[2 * k + 1] = dy.y;
      snb[k / 2] = (snb[k / 2] + y.x) + y.y;
      sdnb[k / 2] = (sdnb[k / 2] + dy.x) + dy.y;
    }
  } else {
    T D[V], dD[V], Ms[V], dMs[V];
    walk_tl<T, V>(M, dM, D, dD, first, last, seg);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      Ms[v] = fma_t(q.hdt * q.cw, D[v], fma_t(T(1) - q.hdt * q.koff, M[v], q.c3));
      const T dR = fma_t(q.cw, dD[v], fma_t(q.dcw, D[v], fma_t(-q.koff, dM[v],
                                                               fma_t(-q.dkoff, M[v], q.dsrc))));
      dMs[v] = fma_t(q.hdt, dR, dM[v]);
    }
    walk_tl<T, V>(Ms, dMs, D, dD, first, last, seg);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const T dR = fma_t(q.cw, dD[v], fma_t(q.dcw, D[v], fma_t(-q.koff, dMs[v],
                                                               fma_t(-q.dkoff, Ms[v], q.dsrc))));
      M[v] = fma_t(q.dt * q.cw, D[v], fma_t(-q.dt * q.koff, Ms[v], M[v] + q.e3));
      dM[v] = fma_t(q.dt, dR, dM[v]);
      snb[0] += M[v];
      sdnb[0] += dM[v];
    }
  }
}

// Blocks an SM of the tangent substep. The kernel is bound by instruction
// issue (68% of the cycles issue; the half-rate pipe of minima and comparisons
// 48%, FMA 42%) with the rest waits on the dependent chain of a row pass, so
// the registers are held to what five or six blocks leave in float32. Float64
// is bound by its own pipe, which two blocks keep as busy as four without
// spills (64^2 cells of 32 x 32: 419 against 494 us a substep).
template <typename T, int V>
constexpr int tan_min_blocks() {
  return sizeof(T) == 8 ? 2 : V == 8 ? 5 : 6;
}

// One substep of the state and its tangent (warp per cell, persistent grid).
// Per cell: psi^{n+1} by Eq. 1 (the plain substep's code) and dpsi^{n+1};
// every s-row by the RK2 of Eq. 4 and its tangent,
//   dR = (v/ds) dD + (dv/ds) D - k_off dM - dk_off M + k_on dMf + dk_on Mf,
// n_b and dn_b of the new rows; C = sum psi n_b dtheta and dC; where the
// scale-down acts, Mb' = f Mb and dMb' = f dMb + df Mb with df = -f dC / C
// (then C = M, dMf = 0), else dMf = -dC. Rows are read with plain vector
// loads, the next pass's rows while the current one is computed. Up to 32
// orientations the columns of Eq. 1 stay in registers and psi and dpsi share
// their face speeds (staged in shared memory five columns at a time and
// computed one after the other before: twenty loads in five rounds of
// latency). 128^2 cells of 32 x 32, float32, a substep of a pass of 50: 97 us
// with selects along the branches and staged columns, 94 with the branch as
// coefficients on register pairs, 88 with the columns in registers, 80 with
// eight nodes to a lane.
template <typename T, int V, bool MASSCORR>
__global__ void __launch_bounds__(128, tan_min_blocks<T, V>()) k_substep_tl(const TanArgs<T> t) {
  extern __shared__ __align__(16) unsigned char tl_smem[];
  const StepArgs<T>& a = t.a;
  const int nth = a.nth, ns = a.ns, seg = a.seg, nx = a.nx, ny = a.ny;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  T* pnew = reinterpret_cast<T*>(tl_smem + (size_t)wib * tan_warp_smem(nth, sizeof(T)));
  T* dpnew = pnew + nth;
  T* s_nb = dpnew + nth;
  T* s_dnb = s_nb + nth;
  const int gw = blockIdx.x * (blockDim.x >> 5) + wib;
  const int W = gridDim.x * (blockDim.x >> 5);
  const int nc = (int)a.ncells;
  const StepScalars<T> sc = step_scalars<T, MASSCORR>(a.prm, a, lane);
  const PsiConst<T> pq{sc.dt, sc.g, sc.glide, sc.vsp, sc.inv_dx, sc.inv_dy, sc.inv_dth, sc.dth,
                       a.trig};
  const T dkoff = (T)t.dkoff, dkon = (T)t.dkon, dcw = (T)(t.dvw / a.ds);
  const LaneGeom lg = lane_geom(lane, seg, ns, V);
  const LaneTrig<T> lt = lane_trig(a.trig, nth, lane);
  T mass_hi = T(0), mass_lo = T(0);
  for (int cell = gw; cell < nc; cell += W) {
    const int iy = cell / nx, ix = cell - iy * nx;
    const int xp = ix + 1 == nx ? 0 : ix + 1, xm = ix == 0 ? nx - 1 : ix - 1;
    const int yp = iy + 1 == ny ? 0 : iy + 1, ym = iy == 0 ? ny - 1 : iy - 1;
    const size_t nbr[5] = {(size_t)cell * nth, (size_t)(iy * nx + xp) * nth,
                           (size_t)(iy * nx + xm) * nth, (size_t)(yp * nx + ix) * nth,
                           (size_t)(ym * nx + ix) * nth};
    const CellVel<T> uv = load_cell_vel(a.ucell, cell);
    T cell_mass = T(0);
    if (nth <= 32) {
      // one orientation to a lane, its columns in registers: the twenty loads
      // in flight together, theta +- 1 by shuffles
      const int kl = lane < nth ? lane : nth - 1;
      PsiIn<T> in = psi_in(a.psi_in, a.nb_in, nbr, kl), di = psi_in(t.dpsi_in, t.dnb_in, nbr, kl);
      const int kp = kl + 1 == nth ? 0 : kl + 1, km = kl == 0 ? nth - 1 : kl - 1;
      in.pp = __shfl_sync(0xffffffffu, in.pc, kp);
      in.pm = __shfl_sync(0xffffffffu, in.pc, km);
      di.pp = __shfl_sync(0xffffffffu, di.pc, kp);
      di.pm = __shfl_sync(0xffffffffu, di.pc, km);
      const T pv = psi_point(pq, uv, lt, in), dv = psi_point_tl(pq, uv, lt, in, di);
      if (lane < nth) {
        pnew[lane] = pv;
        dpnew[lane] = dv;
        a.psi_out[nbr[0] + lane] = pv;
        t.dpsi_out[nbr[0] + lane] = dv;
        cell_mass = pv;
      }
    } else {
      for (int k = lane; k < nth; k += 32) {
        PsiIn<T> in = psi_in(a.psi_in, a.nb_in, nbr, k), di = psi_in(t.dpsi_in, t.dnb_in, nbr, k);
        const int kp = k + 1 == nth ? 0 : k + 1, km = k == 0 ? nth - 1 : k - 1;
        in.pp = a.psi_in[nbr[0] + kp];
        in.pm = a.psi_in[nbr[0] + km];
        di.pp = t.dpsi_in[nbr[0] + kp];
        di.pm = t.dpsi_in[nbr[0] + km];
        const LaneTrig<T> tr = trig_at(a.trig, nth, k);
        const T pv = psi_point(pq, uv, tr, in), dv = psi_point_tl(pq, uv, tr, in, di);
        pnew[k] = pv;
        dpnew[k] = dv;
        a.psi_out[nbr[0] + k] = pv;
        t.dpsi_out[nbr[0] + k] = dv;
        cell_mass += pv;
      }
    }
    two_sum_acc(mass_hi, mass_lo, cell_mass);
    const T mf = a.mf_in[cell], dmf = t.dmf[cell];
    // the rows: Mf frozen over both stages
    const TlRow<T> rq{sc.cw, sc.koff, sc.dt, sc.hdt, dcw, dkoff, sc.hdt * sc.kon * mf,
                      sc.dt * sc.kon * mf, fma_t(sc.kon, dmf, dkon * mf)};
    Pack<T, V> qn, dqn;
    auto load_pass = [&](int r0) {
      const int k = r0 + lg.rslot;
      if (k < nth && lg.lane_ok) {
        const size_t off = ((size_t)cell * nth + k) * ns + lg.sl * V;
        qn = *reinterpret_cast<const Pack<T, V>*>(a.mb_in + off);
        dqn = *reinterpret_cast<const Pack<T, V>*>(t.dmb + off);
      }
    };
    load_pass(0);
    for (int r0 = 0; r0 < nth; r0 += lg.rpp) {
      const int k = r0 + lg.rslot;
      const bool row_ok = k < nth, act = row_ok && lg.lane_ok;
      const size_t roff = ((size_t)cell * nth + (row_ok ? k : 0)) * ns + lg.sl * V;
      T M[V], dM[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        M[v] = act ? qn.v[v] : T(0);
        dM[v] = act ? dqn.v[v] : T(0);
      }
      if (r0 + lg.rpp < nth) load_pass(r0 + lg.rpp);
      T snb[2], sdnb[2];
      rows_tl<T, V>(M, dM, rq, lg.first, lg.last, seg, snb, sdnb);
      if (act) {
        Pack<T, V> q, dq;
#pragma unroll
        for (int v = 0; v < V; ++v) {
          q.v[v] = M[v];
          dq.v[v] = dM[v];
        }
        *reinterpret_cast<Pack<T, V>*>(a.mb_out + roff) = q;
        *reinterpret_cast<Pack<T, V>*>(t.dmb + roff) = dq;
      } else {
        snb[0] = snb[1] = T(0);
        sdnb[0] = sdnb[1] = T(0);
      }
      // (the sums' order is that of four nodes to a lane)
      T nb = seg_sum(snb[0], seg), dnb = seg_sum(sdnb[0], seg);
      if constexpr (V == 8) {
        nb += seg_sum(snb[1], seg);
        dnb += seg_sum(sdnb[1], seg);
      }
      if (lg.first && row_ok) {
        s_nb[k] = nb * sc.ds;
        s_dnb[k] = dnb * sc.ds;
      }
    }
    __syncwarp();
    // Eq. 5, the scale-down of Alg. 2, Eq. 6 and their tangents
    T acc = T(0), dacc = T(0);
    for (int k = lane; k < nth; k += 32) {
      acc = fma_t(pnew[k] * s_nb[k], sc.dth, acc);
      dacc = fma_t(fma_t(dpnew[k], s_nb[k], pnew[k] * s_dnb[k]), sc.dth, dacc);
    }
    const T Cpre = warp_sum_t(acc), dC = warp_sum_t(dacc);
    const T mtot = a.mtot[cell];
    const size_t cb = (size_t)cell * nth;
    if (mtot < Cpre) {
      const T f = mtot / Cpre, df = -f * dC / Cpre;
      T* base = a.mb_out + cb * ns;
      T* dbase = t.dmb + cb * ns;
      for (int e = lane; e < nth * ns; e += 32) {
        const T m = __ldcg(base + e);
        dbase[e] = fma_t(f, __ldcg(dbase + e), df * m);
        base[e] = m * f;
      }
      for (int k = lane; k < nth; k += 32) {
        a.nb_out[cb + k] = s_nb[k] * f;
        t.dnb_out[cb + k] = fma_t(f, s_dnb[k], df * s_nb[k]);
      }
      if (lane == 0) {
        a.c[cell] = mtot;
        a.mf_out[cell] = T(0);
        t.dmf[cell] = T(0);
      }
    } else {
      for (int k = lane; k < nth; k += 32) {
        a.nb_out[cb + k] = s_nb[k];
        t.dnb_out[cb + k] = s_dnb[k];
      }
      if (lane == 0) {
        a.c[cell] = Cpre;
        a.mf_out[cell] = mtot - Cpre;
        t.dmf[cell] = -dC;
      }
    }
    __syncwarp();
  }
  // sum psi^{n+1} (fixed order) and the float32 form's correction factor, as
  // in the plain substep
  __shared__ double s_red[32];
  __shared__ unsigned int s_last;
  const double m = warp_sum_ff(mass_hi, mass_lo);
  if (lane == 0) s_red[wib] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = s_red[0];
    for (int q = 1; q < (int)(blockDim.x >> 5); ++q) b += s_red[q];
    a.partial[blockIdx.x] = b;
    __threadfence();
    const unsigned int prev = atomicInc(&a.prm->counter, gridDim.x - 1);
    s_last = prev == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last && wib == 0) {
    __threadfence();
    const double tot = warp_sum_ldcg(a.partial, (int)gridDim.x, 1, lane);
    if (lane == 0) {
      a.prm->mass = tot;
      if (MASSCORR && a.mass_correct) a.prm->psi_scale = a.prm->mass0 / tot;
    }
  }
}

// The sums a built-in observable and its derivative need: sum psi cos, sum psi
// sin, sum psi, sum psi m1, and the same of the tangent (psi taken with the
// pending correction factor g, dpsi with g as a constant), over all cells into
// tot[8], in float64 for either state precision. A warp per cell: the rows' m1
// of Mb and dMb (packed rows, eight nodes per lane), then lanes over theta.
// Partial sums per warp, block and last block in a fixed order. Bound by the
// float64 pipe, two operations a node (a thread per row and one warp for the
// total took 620 us at 128^2 x 32^2, float-float sums on the float32 pipe 70,
// with errors of 2^-48 in place of 2^-53).
template <typename T, int VW>
__global__ void __launch_bounds__(128)
    k_tan_sums(const T* psi, const T* mb, const T* dpsi, const T* dmb, const double* trig64,
               DevParams* prm, long long ncells, int nth, int ns, double ds, double* partial,
               double* tot) {
  extern __shared__ __align__(16) unsigned char tan_raw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const PackedGeom pg = packed_geom(lane, ns);
  double2* s_d = reinterpret_cast<double2*>(tan_raw) + (size_t)wib * nth;  // 2 m1 / ds^2, of Mb and dMb
  const double g = prm->psi_scale;
  double sj[8];
#pragma unroll
  for (int v = 0; v < 8; ++v) sj[v] = (double)(2 * (pg.sl * 8 + v) + 1 - ns);  // 2 s_j / ds
  double s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (long long cell = blockIdx.x * 4LL + wib; cell < ncells; cell += (long long)gridDim.x * 4) {
    for (int r0 = 0; r0 < nth; r0 += 2 * pg.rpp) {
      T m[4][8];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int k = r0 + u * pg.rpp + pg.rslot;
        const size_t off = ((size_t)cell * nth + (k < nth ? k : 0)) * ns + pg.sl * 8;
        load_row8<T, VW>(mb + off, k < nth ? pg.nv : 0, m[2 * u]);
        load_row8<T, VW>(dmb + off, k < nth ? pg.nv : 0, m[2 * u + 1]);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (r0 + u * pg.rpp >= nth) break;  // (every lane)
        const int k = r0 + u * pg.rpp + pg.rslot;
        double a = 0.0, b = 0.0;
#pragma unroll
        for (int v = 0; v < 8; ++v) {
          a = fma(sj[v], widen(m[2 * u][v]), a);
          b = fma(sj[v], widen(m[2 * u + 1][v]), b);
        }
        a = packed_sum(a, pg.nl, pg.sl);
        b = packed_sum(b, pg.nl, pg.sl);
        if (pg.sl == 0 && pg.rslot < pg.rpp && k < nth) s_d[k] = make_double2(a, b);
      }
    }
    __syncwarp();
    for (int k = lane; k < nth; k += 32) {
      const size_t r = (size_t)cell * nth + k;
      const double p = widen(psi[r]), dp = widen(dpsi[r]);
      const double c = trig64[k], sn = trig64[nth + k];
      const double2 m = s_d[k];
      s[0] = fma(p, c, s[0]);
      s[1] = fma(p, sn, s[1]);
      s[2] += p;
      s[3] = fma(p, m.x, s[3]);
      s[4] = fma(dp, c, s[4]);
      s[5] = fma(dp, sn, s[5]);
      s[6] += dp;
      s[7] = fma(p, m.y, fma(dp, m.x, s[7]));
    }
    __syncwarp();
  }
  __shared__ double s_part[4][8];
  __shared__ unsigned int s_last;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    s[q] = warp_sum(s[q]);
    if (lane == 0) s_part[wib][q] = s[q];
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    double b = s_part[0][threadIdx.x];
    for (int w = 1; w < 4; ++w) b += s_part[w][threadIdx.x];
    partial[(size_t)blockIdx.x * 8 + threadIdx.x] = b;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicInc(&prm->counter2, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int q = wib; q < 8; q += 4) {
    const double t = warp_sum_ldcg(partial + q, (int)gridDim.x, 8, lane);
    if (lane == 0) tot[q] = g * (q == 3 || q == 7 ? 0.5 * ds * ds * t : t);
  }
}

}  // namespace mm

using namespace mmh;

namespace {

template <typename T, int V>
cudaError_t tan_launch_t(mm_handle* h, int parity, cudaStream_t s) {
  mm::TanArgs<T> t;
  t.a = step_args<T>(h, parity);
  t.a.seg = h->tan_seg;
  t.dpsi_in = (const T*)h->tan_psi[parity];
  t.dpsi_out = (T*)h->tan_psi[parity ^ 1];
  t.dnb_in = (const T*)h->tan_nb[parity];
  t.dnb_out = (T*)h->tan_nb[parity ^ 1];
  t.dmb = (T*)h->tan_mb;
  t.dmf = (T*)h->tan_mf;
  t.dkoff = h->tan_dp[0];
  t.dvw = h->tan_dp[1];
  t.dkon = h->tan_dp[2];
  const size_t smem = 4 * mm::tan_warp_smem(h->g.ntheta, sizeof(T));
  if (t.a.mass_correct)
    mm::k_substep_tl<T, V, true><<<h->tan_grid, 128, smem, s>>>(t);
  else
    mm::k_substep_tl<T, V, false><<<h->tan_grid, 128, smem, s>>>(t);
  return cudaGetLastError();
}

template <typename T, int V>
cudaError_t tan_prepare_t(mm_handle* h, int* per_sm) {
  const size_t smem = 4 * mm::tan_warp_smem(h->g.ntheta, sizeof(T));
  const void* fns[2] = {(const void*)mm::k_substep_tl<T, V, true>,
                        (const void*)mm::k_substep_tl<T, V, false>};
  for (const void* f : fns) {
    cudaError_t e = mm::raise_smem_limit(f, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, mm::k_substep_tl<T, V, true>, 128,
                                                       smem);
}

// Row passes of a cell times the nodes a lane holds: the work of a lane with
// its idle slots, for rows of ns nodes, V to a lane.
int tan_lane_nodes(int nth, int ns, int V) {
  int seg = 1;
  while (seg < ns / V) seg <<= 1;
  const int rpp = 32 / seg;
  return (nth + rpp - 1) / rpp * V;
}

// Vector width of the tangent kernel: the registers hold the row and its
// tangent, so at most 8 float32 (2 float64) values per lane. Eight rather
// than four halve the shuffles and the row sums of a pass (128^2 cells of
// 32 x 32: 80 against 88 us a substep), unless the few orientations of a cell
// would leave lanes of the wider pass idle.
int tan_width(const mm_handle* h) {
  const int ns = h->g.ns, nth = h->g.ntheta;
  if (h->prec == MM_FP64) return (ns % 2 == 0 && ns / 2 <= 32) ? 2 : 1;
  if (ns % 4 == 0 && ns / 4 <= 32)
    return ns % 8 == 0 && tan_lane_nodes(nth, ns, 8) <= tan_lane_nodes(nth, ns, 4) ? 8 : 4;
  if (ns % 2 == 0 && ns / 2 <= 32) return 2;
  return 1;
}

template <template <typename, int> class F, typename... A>
cudaError_t tan_by_width(mm_handle* h, A... args) {
  const int V = tan_width(h);
  if (h->prec == MM_FP64) return V == 2 ? F<double, 2>::run(h, args...) : F<double, 1>::run(h, args...);
  if (V == 8) return F<float, 8>::run(h, args...);
  if (V == 4) return F<float, 4>::run(h, args...);
  return V == 2 ? F<float, 2>::run(h, args...) : F<float, 1>::run(h, args...);
}
template <typename T, int V>
struct TanLaunchF {
  static cudaError_t run(mm_handle* h, int parity, cudaStream_t s) {
    return tan_launch_t<T, V>(h, parity, s);
  }
};
template <typename T, int V>
struct TanPrepareF {
  static cudaError_t run(mm_handle* h, int* per_sm) { return tan_prepare_t<T, V>(h, per_sm); }
};

}  // namespace

namespace mmh {

void tangent_free(mm_handle* h) {
  void* p[6] = {h->tan_mb, h->tan_psi[0], h->tan_psi[1], h->tan_nb[0], h->tan_nb[1], h->tan_mf};
  for (void* q : p)
    if (q) cudaFree(q);
  h->tan_mb = h->tan_psi[0] = h->tan_psi[1] = h->tan_nb[0] = h->tan_nb[1] = h->tan_mf = nullptr;
  h->tangent = false;
}

cudaError_t launch_tangent_substep(mm_handle* h, int parity, cudaStream_t s) {
  return tan_by_width<TanLaunchF>(h, parity, s);
}

// A new state starts the tangent from zero (the direction is in the rates).
mm_status tangent_zero(mm_handle* h) {
  const size_t t = h->tsz;
  CK(cudaMemsetAsync(h->tan_mb, 0, h->mbn * t, h->stream));
  for (int p = 0; p < 2; ++p) {
    CK(cudaMemsetAsync(h->tan_psi[p], 0, h->rows * t, h->stream));
    CK(cudaMemsetAsync(h->tan_nb[p], 0, h->rows * t, h->stream));
  }
  CK(cudaMemsetAsync(h->tan_mf, 0, (size_t)h->ncells * t, h->stream));
  return MM_OK;
}

}  // namespace mmh

extern "C" {

mm_status mm_set_tangent(mm_handle* h, const double* dparams) {
  MM_TRACE("mm_set_tangent");
  if (!h) return MM_ERR_INVALID;
  if (h->batch || h->owner) return fail(h, MM_ERR_UNSUPPORTED, "the tangent is not available in a batch");
  if (h->rec.active)
    return fail(h, MM_ERR_STATE, "an adjoint recording is active: end it first");
  if (dparams && (h->anchors || h->capture))
    return fail(h, MM_ERR_UNSUPPORTED,
                "the tangent is not available with non-local anchors or a capture radius");
  DeviceGuard dg(h->device);
  CK(cudaStreamSynchronize(h->stream));
  for (auto& kv : h->graphs) cudaGraphExecDestroy(kv.second);
  h->graphs.clear();
  if (!dparams) {
    tangent_free(h);
    return MM_OK;
  }
  for (int q = 0; q < 3; ++q)
    if (!std::isfinite(dparams[q])) return fail(h, MM_ERR_INVALID, "dparams must be finite");
  if (!h->tan_mb) {
    const size_t t = h->tsz;
    size_t freeb = 0, totalb = 0;
    CK(cudaMemGetInfo(&freeb, &totalb));
    const size_t need = h->mbn * t + 4 * h->rows * t + (size_t)h->ncells * t;
    if (need + (64u << 20) > freeb) return fail(h, MM_ERR_OOM, "the tangent state does not fit");
    CK(cudaMalloc(&h->tan_mb, h->mbn * t));
    for (int p = 0; p < 2; ++p) {
      CK(cudaMalloc(&h->tan_psi[p], h->rows * t));
      CK(cudaMalloc(&h->tan_nb[p], h->rows * t));
    }
    CK(cudaMalloc(&h->tan_mf, (size_t)h->ncells * t));
  }
  const int V = tan_width(h);
  int seg = 1;
  while (seg < h->g.ns / V) seg <<= 1;
  if (seg > 32) return fail(h, MM_ERR_UNSUPPORTED, "ns too large for the tangent kernel");
  h->tan_seg = seg;
  // (the limit of a kernel that staged five cells' columns, kept as it was:
  // six times what the columns take now)
  if (6 * 4 * mm::tan_warp_smem(h->g.ntheta, (int)h->tsz) > kSmemBudget)
    return fail(h, MM_ERR_UNSUPPORTED, "ntheta too large for the tangent kernel");
  int per_sm = 0;
  CK(tan_by_width<TanPrepareF>(h, &per_sm));
  if (per_sm < 1) return fail(h, MM_ERR_UNSUPPORTED, "the tangent kernel cannot be resident");
  h->tan_grid = (int)std::max<long long>(
      1, std::min<long long>((h->ncells + 3) / 4, (long long)per_sm * h->sms));
  // the per-block partial sums of psi share the plain substep's buffer
  h->tan_grid = std::min(h->tan_grid, h->npartial);
  h->tan_dp[0] = dparams[0];
  h->tan_dp[1] = dparams[1];
  h->tan_dp[2] = dparams[2];
  h->tangent = true;
  return tangent_zero(h);
}

mm_status mm_get_tangent(mm_handle* h, double* dpsi, double* dmb, double* dmf, int on_device) {
  MM_TRACE("mm_get_tangent");
  if (!h) return MM_ERR_INVALID;
  if (!h->tangent) return fail(h, MM_ERR_STATE, "no tangent (mm_set_tangent)");
  DeviceGuard dg(h->device);
  mm_status st;
  const double* scale = h->prec == MM_FP32_MIXED ? &h->prm->psi_scale : nullptr;
  if (dpsi && (st = get_array(h, dpsi, h->tan_psi[h->parity], h->rows, on_device, scale)) != MM_OK)
    return st;
  if (dmb && (st = get_array(h, dmb, h->tan_mb, h->mbn, on_device, nullptr)) != MM_OK) return st;
  if (dmf && (st = get_array(h, dmf, h->tan_mf, (size_t)h->ncells, on_device, nullptr)) != MM_OK)
    return st;
  CK(cudaStreamSynchronize(h->stream));
  return check_status(h);
}

mm_status mm_tangent_observable(mm_handle* h, int observable, double* value, double* dvalue) {
  MM_TRACE("mm_tangent_observable");
  if (!h || !value || !dvalue) return MM_ERR_INVALID;
  if (!h->tangent) return fail(h, MM_ERR_STATE, "no tangent (mm_set_tangent)");
  if (observable != MM_OBS_POLAR_ORDER && observable != MM_OBS_MEAN_STRESS)
    return fail(h, MM_ERR_INVALID, "observable must be MM_OBS_POLAR_ORDER or MM_OBS_MEAN_STRESS");
  DeviceGuard dg(h->device);
  const long long nc = h->ncells;
  const double ds = h->g.L / h->g.ns, dth = 2.0 * kPi / h->g.ntheta;
  // per-cell sums in the moments' field buffer (12 doubles per cell available)
  double* cells = h->fields;
  double* tot = h->partial;  // 8 doubles; the partial sums are free between substeps
  const int nth = h->g.ntheta, ns = h->g.ns;
  const int grid = (int)std::max<long long>(1, std::min<long long>((nc + 3) / 4, 8LL * h->sms));
  const size_t smem = 4 * (size_t)nth * 16;
  auto go = [&](auto kern, auto t) -> cudaError_t {
    using T = decltype(t);
    if (smem > 48 * 1024) {
      const cudaError_t e = mm::raise_smem_limit(kern, smem);
      if (e != cudaSuccess) return e;
    }
    kern<<<grid, 128, smem, h->stream>>>((const T*)h->psi[h->parity], (const T*)h->mb,
                                         (const T*)h->tan_psi[h->parity], (const T*)h->tan_mb,
                                         h->trig64, h->prm, nc, nth, ns, ds, cells, tot);
    return cudaGetLastError();
  };
  if (h->prec == MM_FP64)
    CK(ns % 2 == 0 ? go(mm::k_tan_sums<double, 2>, 0.0) : go(mm::k_tan_sums<double, 1>, 0.0));
  else
    CK(ns % 4 == 0   ? go(mm::k_tan_sums<float, 4>, 0.f)
       : ns % 2 == 0 ? go(mm::k_tan_sums<float, 2>, 0.f)
                     : go(mm::k_tan_sums<float, 1>, 0.f));
  double s[8];
  CK(cudaMemcpyAsync(s, tot, sizeof s, cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  if (observable == MM_OBS_POLAR_ORDER) {
    // L = |S| / N with S = sum psi e^{i theta}, N = sum psi
    const double S = std::sqrt(s[0] * s[0] + s[1] * s[1]), N = s[2];
    *value = S / N;
    const double dS = S > 0.0 ? (s[0] * s[4] + s[1] * s[5]) / S : 0.0;
    *dvalue = dS / N - S * s[6] / (N * N);
  } else {
    // L = mean over cells of tr sigma_a = F_m ell dth sum psi m1 / cells
    const double c = h->r.force_scale * h->r.ell * dth / (double)nc;
    *value = c * s[3];
    *dvalue = c * s[7];
  }
  return check_status(h);
}

}  // extern "C"
