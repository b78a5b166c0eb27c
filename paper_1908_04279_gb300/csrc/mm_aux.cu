// Auxiliary kernels: precision conversion, state set-up (Eq. 5-6 with the
// Alg. 2 scale-down), the maxima of the adaptive-substep rule, and the
// macroscale moments (Alg. 1 after the inner loop; Eq. 10's force and force
// dipole with anchors in the filament's own cell).
#include "mm_rows.cuh"

namespace mm {

namespace {


// The copies of a CopySegs: 16-byte vectors where both addresses are 16-byte
// aligned, then the remaining bytes one by one; every thread of the grid takes
// its share of each segment in turn.
__global__ void k_copy_multi(const CopySegs c) {
  const size_t tid = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (int q = 0; q < c.n; ++q) {
    const unsigned char* s = static_cast<const unsigned char*>(c.src[q]);
    unsigned char* d = static_cast<unsigned char*>(c.dst[q]);
    const size_t b = c.bytes[q];
    const bool vec = ((reinterpret_cast<uintptr_t>(s) | reinterpret_cast<uintptr_t>(d)) & 15) == 0;
    const size_t nv = vec ? b / 16 : 0;
    const uint4* s4 = reinterpret_cast<const uint4*>(s);
    uint4* d4 = reinterpret_cast<uint4*>(d);
    for (size_t i = tid; i < nv; i += stride) d4[i] = s4[i];
    for (size_t i = nv * 16 + tid; i < b; i += stride) d[i] = s[i];
  }
}

template <typename TO, typename TI>
__device__ __forceinline__ TO converted(TI x) {
  if constexpr (sizeof(TO) == 8 && sizeof(TI) == 4)
    return widen(x);
  else
    return (TO)x;
}

// out = in (times *scale); without a scale in pairs, 8 bytes on one side and 16 on
// the other, where the addresses allow it (512^2 x 64^2 exports 0.69 -> 0.52 ms
// per 268 M values).
template <typename TO, typename TI>
__global__ void k_convert(TO* out, const TI* in, size_t n, const double* scale) {
  const size_t tid = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  if (scale) {
    const double sc = *scale;
    for (size_t i = tid; i < n; i += stride) out[i] = (TO)((double)in[i] * sc);
    return;
  }
  struct alignas(2 * sizeof(TI)) In {
    TI a, b;
  };
  struct alignas(2 * sizeof(TO)) Out {
    TO a, b;
  };
  const bool vec = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
  const size_t nv = vec ? n / 2 : 0;
  for (size_t i = tid; i < nv; i += stride) {
    const In v = reinterpret_cast<const In*>(in)[i];
    reinterpret_cast<Out*>(out)[i] = Out{converted<TO, TI>(v.a), converted<TO, TI>(v.b)};
  }
  for (size_t i = 2 * nv + tid; i < n; i += stride) out[i] = converted<TO, TI>(in[i]);
}

__device__ __forceinline__ void atomic_max_nonneg(double* addr, double v) {
  // Non-negative doubles order like their bit patterns as unsigned integers.
  atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}

// Maxima of the adaptive-substep rule: max(|ax|/dx + |ay|/dy),
// max |omega(theta_{k+1/2})| / dtheta, and max_cell sum_k psi dtheta, in the
// state precision (float64 in the float64 form, whose dt must agree with a
// float64 evaluation; float32 in the float32 form, whose state is float32
// anyway); the maxima are exact. A cell takes `seg` lanes (nth rounded up to a
// power of two, 32 at most), so that a warp holds 32 / seg cells. Bound by
// latency: full occupancy hides it, and a block reduces its maxima before the
// three atomics (one set per warp kept the atomics of one address in a queue:
// 128^2 x 32 15 us).
// The greater of two non-negative values, none of them NaN (float64: on the bit
// patterns, off the narrow float64 pipe).
__device__ __forceinline__ float max_nonneg(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double max_nonneg(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return __longlong_as_double(x > y ? x : y);
}
template <typename T>
__device__ __forceinline__ T warp_max_nonneg(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = max_nonneg(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

constexpr int kDtBlock = 512;

template <typename T>
__global__ void __launch_bounds__(kDtBlock)
    k_dt_max(const T* psi, const T* nb, const T* u, const T* trig, int ncells, int nx, int ny,
             int nth, int seg, double inv_dx64, double inv_dy64, double inv_dth64, double dth64,
             double glide64, double vsp64, DevParams* prm) {
  const int lane = threadIdx.x & 31;
  const int cps = 32 / seg, sub = lane / seg, kl = lane - sub * seg;
  const long long gw = blockIdx.x * (long long)(kDtBlock / 32) + (threadIdx.x >> 5);
  const long long W = (long long)gridDim.x * (kDtBlock / 32);
  const T g = (T)prm->psi_scale;
  const T inv_dx = (T)inv_dx64, inv_dy = (T)inv_dy64, inv_dth = (T)inv_dth64, dth = (T)dth64;
  const T glide = (T)glide64, vsp = (T)vsp64, h = T(0.5);
  T adv = T(0), rot = T(0), rhomax = T(0);
  const T* ux = u;
  const T* uy = u + ncells;
  for (long long c0 = gw * cps; c0 < ncells; c0 += W * cps) {
    const bool on = c0 + sub < ncells;
    const int cell = on ? (int)c0 + sub : 0;
    const int iy = cell / nx, ix = cell - iy * nx;
    const size_t ce = (size_t)iy * nx + (ix + 1 == nx ? 0 : ix + 1);
    const size_t cw = (size_t)iy * nx + (ix == 0 ? nx - 1 : ix - 1);
    const size_t cn = (size_t)(iy + 1 == ny ? 0 : iy + 1) * nx + ix;
    const size_t cs = (size_t)(iy == 0 ? ny - 1 : iy - 1) * nx + ix;
    const T Gxx = (ux[ce] - ux[cw]) * h * inv_dx, Gxy = (ux[cn] - ux[cs]) * h * inv_dy;
    const T Gyx = (uy[ce] - uy[cw]) * h * inv_dx, Gyy = (uy[cn] - uy[cs]) * h * inv_dy;
    const T uxc = ux[cell], uyc = uy[cell];
    T rho = T(0);
    for (int k = kl; on && k < nth; k += seg) {
      const size_t e = (size_t)cell * nth + k;
      const T V = vsp + glide * nb[e];
      const T ax = uxc - V * trig[k], ay = uyc - V * trig[nth + k];
      adv = tmax(adv, fabs(ax) * inv_dx + fabs(ay) * inv_dy);
      const T cp = trig[2 * nth + k], sp = trig[3 * nth + k];
      const T w = -sp * (Gxx * cp + Gxy * sp) + cp * (Gyx * cp + Gyy * sp);
      rot = tmax(rot, fabs(w) * inv_dth);
      rho += psi[e] * g * dth;
    }
    rhomax = tmax(rhomax, seg_sum(rho, seg));
  }
  __shared__ T red[3][kDtBlock / 32];
  adv = warp_max_nonneg(adv);
  rot = warp_max_nonneg(rot);
  rhomax = warp_max_nonneg(rhomax);
  if (lane == 0) {
    red[0][threadIdx.x >> 5] = adv;
    red[1][threadIdx.x >> 5] = rot;
    red[2][threadIdx.x >> 5] = rhomax;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    T m = red[threadIdx.x][0];
    for (int q = 1; q < kDtBlock / 32; ++q) m = max_nonneg(m, red[threadIdx.x][q]);
    atomic_max_nonneg(&prm->dtmax[threadIdx.x], (double)m);
  }
}

constexpr int kMomPasses = 4;  // passes of rows in flight before they are reduced

// Set-up of a state, a warp per cell, in float64 for either state precision: n_b
// of every row, C = sum_k psi n_b dtheta, the Alg. 2 scale-down where C > M, Mf =
// M - C (which may cancel: float-float sums left 2^-47 of C in it). Bound by the
// float64 pipe, one operation a node: every lane loads 32 (64) consecutive
// bytes, four passes of rows in flight per warp (a thread per row, one node per
// load and a serial sum took 90 us at 128^2 x 32^2 where the bytes need 10).
template <typename T, int VW>
__global__ void __launch_bounds__(128)
    k_init_cells(T* mb, const T* psi, T* nb, T* mf, T* c, const T* mtot, int ncells, int nth,
                 int ns, double ds, double dth) {
  const int lane = threadIdx.x & 31;
  const PackedGeom g = packed_geom(lane, ns);
  const int gw = blockIdx.x * 4 + (threadIdx.x >> 5), W = gridDim.x * 4;
  for (long long cl = gw; cl < ncells; cl += W) {
    const int cell = (int)cl;
    T* rows = mb + (size_t)cell * nth * ns + g.sl * 8;
    const T* pc = psi + (size_t)cell * nth;
    T* nbc = nb + (size_t)cell * nth;
    double acc = 0.0;
    for (int r0 = 0; r0 < nth; r0 += kMomPasses * g.rpp) {
      T m[kMomPasses][8];
#pragma unroll
      for (int u = 0; u < kMomPasses; ++u) {
        const int k = r0 + u * g.rpp + g.rslot;
        load_row8<T, VW>(rows + (size_t)(k < nth ? k : 0) * ns, k < nth ? g.nv : 0, m[u]);
      }
#pragma unroll
      for (int u = 0; u < kMomPasses; ++u) {
        if (r0 + u * g.rpp >= nth) break;  // (every lane)
        const int k = r0 + u * g.rpp + g.rslot;
        double x[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) x[v] = widen(m[u][v]);
        const double s = packed_sum(((x[0] + x[1]) + (x[2] + x[3])) +
                                        ((x[4] + x[5]) + (x[6] + x[7])),
                                    g.nl, g.sl) *
                         ds;
        if (g.sl == 0 && g.rslot < g.rpp && k < nth) {
          nbc[k] = (T)s;
          acc = fma(widen(pc[k]), s, acc);
        }
      }
    }
    // C, and the scale-down where it exceeds the total motors
    const double M = widen(mtot[cell]), C = warp_sum(acc) * dth;
    const bool over = M < C;
    if (lane == 0) {
      c[cell] = (T)(over ? M : C);
      mf[cell] = (T)(over ? 0.0 : M - C);
    }
    if (over) {
      const double f = M / C;
      __syncwarp();
      T* all = mb + (size_t)cell * nth * ns;
      for (int e = lane; e < nth * ns; e += 32) all[e] = (T)((double)all[e] * f);
      for (int k = lane; k < nth; k += 32) nbc[k] = (T)((double)nbc[k] * f);
    }
  }
}

// The sum of psi over all cells and angles into prm->sum_psi (the reference of
// the float32 form's mass correction): per thread, block and last block in a
// fixed order, float-float in the float32 form.
template <typename T>
__global__ void __launch_bounds__(512) k_sum_psi(const T* psi, size_t n, double* partial,
                                                 DevParams* prm) {
  __shared__ double s_red[16];
  __shared__ unsigned int s_last;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if constexpr (sizeof(T) == 4) {
    float2* red = reinterpret_cast<float2*>(s_red);
    float2* part = reinterpret_cast<float2*>(partial);
    float2 a = make_float2(0.f, 0.f), b = a;
    for (; i + stride < n; i += 2 * stride) {
      const float x = psi[i], y = psi[i + stride];
      two_sum_acc2(a, x);
      two_sum_acc2(b, y);
    }
    if (i < n) two_sum_acc2(a, psi[i]);
    a = warp_sum_ff2(ff2_add(a, b));
    if (lane == 0) red[w] = a;
    __syncthreads();
    if (w == 0) {
      a = warp_sum_ff2(lane < 16 ? red[lane] : make_float2(0.f, 0.f));
      if (lane == 0) part[blockIdx.x] = a;
    }
  } else {
    double a = 0.0, b = 0.0;
    for (; i + stride < n; i += 2 * stride) {
      a += psi[i];
      b += psi[i + stride];
    }
    if (i < n) a += psi[i];
    a = warp_sum(a + b);
    if (lane == 0) s_red[w] = a;
    __syncthreads();
    if (w == 0) {
      a = warp_sum(lane < 16 ? s_red[lane] : 0.0);
      if (lane == 0) partial[blockIdx.x] = a;
    }
  }
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicInc(&prm->counter2, gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last || w != 0) return;
  __threadfence();
  if constexpr (sizeof(T) == 4) {
    const float2 t = warp_sum_ldcg_ff2(reinterpret_cast<const float2*>(partial), (int)gridDim.x, lane);
    if (lane == 0) prm->sum_psi = (double)t.x + (double)t.y;
  } else {
    const double t = warp_sum_ldcg(partial, (int)gridDim.x, 1, lane);
    if (lane == 0) prm->sum_psi = t;
  }
}

// Sums over the warp of 16 values per lane by reduce-scatter (16 float64
// additions instead of 16 x 5): at each step a lane keeps half of its values
// and adds its partner's copies of them. Returns the total of value
// f(lane) = 8 b4 + 4 b3 + 2 b2 + b1 (b_i the bits of the lane index), which
// lanes 2 f and 2 f + 1 both hold.
__device__ __forceinline__ double warp_sum16_scatter(double (&v)[16], int lane) {
#pragma unroll
  for (int step = 0; step < 4; ++step) {
    const int o = 16 >> step, half = 8 >> step;
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const double keep = up ? v[half + i] : v[i];
      const double give = up ? v[i] : v[half + i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}
// The same reduce-scatter in float-float.
__device__ __forceinline__ FF warp_sum16_scatter_ff(FF (&v)[16], int lane) {
#pragma unroll
  for (int step = 0; step < 4; ++step) {
    const int o = 16 >> step, half = 8 >> step;
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const FF keep = up ? v[half + i] : v[i];
      const FF give = up ? v[i] : v[half + i];
      const FF got{__shfl_xor_sync(0xffffffffu, give.hi, o), __shfl_xor_sync(0xffffffffu, give.lo, o)};
      v[i] = ff_sum(keep, got);
    }
  }
  const FF got{__shfl_xor_sync(0xffffffffu, v[0].hi, 1), __shfl_xor_sync(0xffffffffu, v[0].lo, 1)};
  return ff_sum(v[0], got);
}
__device__ __forceinline__ int scatter_field(int lane) {
  return ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
}

// Moments, one warp per cell, no block barriers before the final sums. The s-rows of the cell are
// read as packed rows (eight consecutive nodes per lane, vector loads) and
// reduced to n_b and m1: in float64 in the float64 form (the float64 pipe bounds
// it: eight nodes per lane leave 2.5 additions a node with the cross-lane sums,
// two per lane 6: 128^2 x 32^2 343 -> 161 us), float-float in the float32 form
// (the float32 pipe: 17 operations a node, the two sums as one pair; a node per
// lane where ns is not a multiple of 4 had the cross-lane sums at every node: 85 x
// 61 x 24 x 30 42 -> 24 us; 256^2 x 64^2 352 -> 315 us) -- these are the
// s-reductions feeding the force and the force dipole. Then lanes over theta form the 12 fields.
// Each warp keeps partial global sums, added per block at the end; the last
// block to finish adds the block partials in a fixed order.
template <typename T, int VW, int NL>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 4 : 1) k_moments(const T* psi, const T* mb, const T* mf, const T* c,
                          const double* trig, long long ncells, int nth, int ns, double dth, double ds, double L, double dA, float hds, double* fields,
                          double* partial, DevParams* prm) {
  extern __shared__ double msm[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  double* s_nb = msm + (size_t)wib * 2 * nth;
  double* s_m1 = s_nb + nth;
  // float32 form: the rows' float-float sums, converted once per row below
  float4* s_ff = reinterpret_cast<float4*>(msm + (size_t)(blockDim.x >> 5) * 2 * nth) +
                 (size_t)wib * nth;
  const long long gw = blockIdx.x * (long long)(blockDim.x >> 5) + wib;
  const long long W = (long long)gridDim.x * (blockDim.x >> 5);
  const double g = prm->psi_scale;
  const double Fm = prm->force_scale, ell = prm->ell;
  const PackedGeom pg = packed_geom(lane, ns);
  const int sl = pg.sl, rslot = pg.rslot, rpp = pg.rpp;
  T sj[8];
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    // s_j = (2j + 1 - ns) ds / 2; the float32 form in float32 (one rounding)
    if constexpr (sizeof(T) == 4)
      sj[v] = (float)(2 * (sl * 8 + v) + 1 - ns) * hds;
    else
      sj[v] = -0.5 * L + ((double)(sl * 8 + v) + 0.5) * ds;
  }
  // global accumulators: N_psi, bound, free, sum psi cos, sum psi sin, sum psi, sum tr
  double gs[7] = {0, 0, 0, 0, 0, 0, 0};
  const int fq = scatter_field(lane);
  // float32 form: every float64 warp instruction costs the float64 pipe as
  // much as a full warp's, so the per-cell bookkeeping stays in float-float:
  // acc is the lane's field total summed over its cells, acc2 (lanes 1, 3) the
  // sum of C and of Mf; each field total is scaled by its constant (psi_scale,
  // ds F, ds F ell) split into a float pair
  FF acc{0.f, 0.f}, acc2{0.f, 0.f};
  FF scf{0.f, 0.f};
  if constexpr (sizeof(T) == 4) {
    const double sc = fq < 5 ? g : (fq < 7 ? g * (ds * Fm) : g * (ds * Fm * ell));
    scf.hi = (float)sc;
    scf.lo = (float)(sc - (double)scf.hi);
  }
  for (long long cell = gw; cell < ncells; cell += W) {
    // kMomPasses passes of rows loaded before they are reduced (more bytes in
    // flight per warp)
    for (int r0 = 0; r0 < nth; r0 += kMomPasses * rpp) {
      T m[kMomPasses][8];
#pragma unroll
      for (int u = 0; u < kMomPasses; ++u) {
        const int k = r0 + u * rpp + rslot;
        load_row8<T, VW>(mb + ((size_t)cell * nth + (k < nth ? k : 0)) * ns + sl * 8,
                         k < nth ? pg.nv : 0, m[u]);
      }
#pragma unroll
      for (int u = 0; u < kMomPasses; ++u) {
        if (r0 + u * rpp >= nth) break;  // (every lane)
        const int k = r0 + u * rpp + rslot;
        const bool own = sl == 0 && rslot < rpp && k < nth;
        if constexpr (sizeof(T) == 4) {
          const FF2x a = packed_sum_ff2x<NL>(row_sums8(m[u], sj), pg.nl, sl);
          if (own) s_ff[k] = make_float4(a.hi.x, a.lo.x, a.hi.y, a.lo.y);
        } else {
          double a = 0.0, b = 0.0;
#pragma unroll
          for (int v = 0; v < 8; ++v) {
            a += m[u][v];
            b = fma(sj[v], m[u][v], b);
          }
          a = packed_sum(a, pg.nl, sl);
          b = packed_sum(b, pg.nl, sl);
          if (own) {
            s_nb[k] = a * ds;
            s_m1[k] = b * ds;
          }
        }
      }
    }
    __syncwarp();
    // ten field sums over theta (weights w[q][k] built on the host: dth,
    // cos dth, sin dth, (cos^2 - 1/2) dth, cos sin dth, cos, sin, cos^2 dth,
    // cos sin dth, sin^2 dth); slots 10..15 stay zero. Lane pair (2q, 2q + 1)
    // gets the total of field q.
    if constexpr (sizeof(T) == 4) {
      // Float32 form: the sums in float-float on the float32 pipe (each product
      // exact to about 2^-48 of itself, the weights split into float pairs on
      // the host); psi_scale and the constant factors ds F, ds F ell multiply
      // each total once, in float64.
      const float2* wf = reinterpret_cast<const float2*>(trig + 14 * (size_t)nth);
      FF f[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) f[q] = FF{0.f, 0.f};
      for (int k = lane; k < nth; k += 32) {
        const float4 q4 = s_ff[k];
        const float p = (float)psi[cell * nth + k];
        const FF pn = ff_scale(p, FF{q4.x, q4.y}), pm = ff_scale(p, FF{q4.z, q4.w});
        FF wq[10];
#pragma unroll
        for (int q = 0; q < 10; ++q) {
          const float2 t = wf[(size_t)q * nth + k];
          wq[q] = FF{t.x, t.y};
        }
#pragma unroll
        for (int q = 0; q < 5; ++q) f[q] = ff_sum(f[q], ff_scale(p, wq[q]));
        f[5] = ff_sum(f[5], ff_prod(pn, wq[1]));
        f[6] = ff_sum(f[6], ff_prod(pn, wq[2]));
#pragma unroll
        for (int q = 7; q < 10; ++q) f[q] = ff_sum(f[q], ff_prod(pm, wq[q]));
      }
      __syncwarp();
      const FF t = warp_sum16_scatter_ff(f, lane);
      acc = ff_sum(acc, t);
      const FF ts = ff_prod(t, scf);
      const double tot = (double)ts.hi + (double)ts.lo;
      if ((lane & 1) == 0 && fq < 10) fields[(size_t)(fq < 5 ? fq : fq + 2) * ncells + cell] = tot;
      // C and Mf as they are (lanes 1 and 3: one conversion for both)
      if (lane == 1 || lane == 3) {
        const float v = lane == 1 ? (float)c[cell] : (float)mf[cell];
        fields[(size_t)(lane == 1 ? 5 : 6) * ncells + cell] = (double)v;
        ff_add(acc2, v);
      }
    } else {
      double f[16] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
      const double* w = trig + 4 * (size_t)nth;
      for (int k = lane; k < nth; k += 32) {
        const double nbk = s_nb[k], m1k = s_m1[k];
        const double p = (double)psi[cell * nth + k] * g;
        const double pn = p * nbk * Fm, pm = p * m1k * (Fm * ell);
        f[0] = fma(p, w[k], f[0]);
        f[1] = fma(p, w[nth + k], f[1]);
        f[2] = fma(p, w[2 * nth + k], f[2]);
        f[3] = fma(p, w[3 * nth + k], f[3]);
        f[4] = fma(p, w[4 * nth + k], f[4]);
        f[5] = fma(pn, w[nth + k], f[5]);
        f[6] = fma(pn, w[2 * nth + k], f[6]);
        f[7] = fma(pm, w[7 * nth + k], f[7]);
        f[8] = fma(pm, w[8 * nth + k], f[8]);
        f[9] = fma(pm, w[9 * nth + k], f[9]);
        gs[3] = fma(p, w[5 * nth + k], gs[3]);
        gs[4] = fma(p, w[6 * nth + k], gs[4]);
        gs[5] += p;
      }
      __syncwarp();
      const double tot = warp_sum16_scatter(f, lane);
      // output slot of field q: 0-4 as is, 5-9 to 7-11 (5 and 6 are C and Mf)
      if ((lane & 1) == 0 && fq < 10) fields[(size_t)(fq < 5 ? fq : fq + 2) * ncells + cell] = tot;
      const double f0 = __shfl_sync(0xffffffffu, tot, 0);   // field 0 (lane 0)
      const double f7 = __shfl_sync(0xffffffffu, tot, 14);  // field 7: bits 3, 2, 1 set
      if (lane == 0) {
        const double cc = (double)c[cell], ff = (double)mf[cell];
        fields[5 * ncells + cell] = cc;
        fields[6 * ncells + cell] = ff;
        gs[0] += f0 * dA;
        gs[1] += cc * dA;
        gs[2] += ff * dA;
      }
      // tr sigma_a = f7 + f9
      const double f9 = __shfl_sync(0xffffffffu, tot, 18);  // field 9: bits 4, 1 set
      if (lane == 0) gs[6] += f7 + f9;
    }
  }
  __shared__ double s_g[32 * 8];
  __shared__ unsigned int s_last;
  const int nw = (int)(blockDim.x >> 5);
  if constexpr (sizeof(T) == 4) {
    // The warp's quantities in float-float, lane q holding quantity q:
    // 0 N_psi (field 0), 1 C, 2 Mf, 3 sum psi cos (field 1), 4 sum psi sin
    // (field 2), 5 sum psi (field 0), 6 tr sigma_a (fields 7 + 9); unscaled.
    const int sa = lane == 3 ? 2 : lane == 4 ? 4 : lane == 6 ? 14 : 0;
    const int sb = lane == 2 ? 3 : 1;
    FF v{__shfl_sync(0xffffffffu, acc.hi, sa), __shfl_sync(0xffffffffu, acc.lo, sa)};
    const FF w2{__shfl_sync(0xffffffffu, acc2.hi, sb), __shfl_sync(0xffffffffu, acc2.lo, sb)};
    const FF a9{__shfl_sync(0xffffffffu, acc.hi, 18), __shfl_sync(0xffffffffu, acc.lo, 18)};
    if (lane == 1 || lane == 2) v = w2;
    if (lane == 6) v = ff_sum(v, a9);
    // per block in warp order, then the last block adds the block partials
    // (float pairs in the 8-byte slots) in a fixed order
    float2* s_ff2 = reinterpret_cast<float2*>(s_g);
    if (lane < 7) s_ff2[wib * 8 + lane] = make_float2(v.hi, v.lo);
    __syncthreads();
    float2* pf = reinterpret_cast<float2*>(partial);
    if (wib == 0 && lane < 7) {
      FF b{s_ff2[lane].x, s_ff2[lane].y};
      for (int w2i = 1; w2i < nw; ++w2i) b = ff_sum(b, FF{s_ff2[w2i * 8 + lane].x, s_ff2[w2i * 8 + lane].y});
      pf[(size_t)blockIdx.x * 8 + lane] = make_float2(b.hi, b.lo);
      __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned int prev = atomicInc(&prm->counter2, gridDim.x - 1);
      s_last = prev == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // scales: psi_scale dA, dA, dA, psi_scale / dth (x3), psi_scale ds F ell
    for (int q = wib; q < 7; q += nw) {
      FF b{0.f, 0.f};
      for (int i = lane; i < (int)gridDim.x; i += 32) {
        const float2 t = __ldcg(pf + (size_t)i * 8 + q);
        b = ff_sum(b, FF{t.x, t.y});
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        b = ff_sum(b, FF{__shfl_xor_sync(0xffffffffu, b.hi, o), __shfl_xor_sync(0xffffffffu, b.lo, o)});
      if (lane == 0) {
        const double sq = q == 0 ? g * dA : q < 3 ? dA : q < 6 ? g / dth : g * (ds * Fm * ell);
        s_g[8 * 8 + q] = ((double)b.hi + (double)b.lo) * sq;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double t[7];
      for (int q = 0; q < 7; ++q) t[q] = s_g[8 * 8 + q];
      prm->scalars[0] = t[0];
      prm->scalars[1] = t[1];
      prm->scalars[2] = t[2];
      prm->scalars[3] = t[1] + t[2];
      prm->scalars[4] = sqrt(t[3] * t[3] + t[4] * t[4]) / t[5];
      prm->scalars[5] = t[6] / (double)ncells;
      prm->scalars[6] = t[3];
      prm->scalars[7] = t[4];
      prm->sum_psi = t[5];
    }
  } else {
#pragma unroll
    for (int q = 0; q < 7; ++q) gs[q] = warp_sum(gs[q]);
    // per block in warp order, then the last block adds the block partials in a
    // fixed order (warp q of that block sums quantities q, q + nw, ...)
    if (lane == 0)
      for (int q = 0; q < 7; ++q) s_g[wib * 8 + q] = gs[q];
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int q = 0; q < 7; ++q) {
        double b = s_g[q];
        for (int w2 = 1; w2 < nw; ++w2) b += s_g[w2 * 8 + q];
        partial[(size_t)blockIdx.x * 8 + q] = b;
      }
      __threadfence();
      const unsigned int prev = atomicInc(&prm->counter2, gridDim.x - 1);
      s_last = prev == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
      __threadfence();
      for (int q = wib; q < 7; q += nw) {
        const double tq = warp_sum_ldcg(partial + q, (int)gridDim.x, 8, lane);
        if (lane == 0) s_g[q] = tq;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        double t[7];
        for (int q = 0; q < 7; ++q) t[q] = s_g[q];
        prm->scalars[0] = t[0];
        prm->scalars[1] = t[1];
        prm->scalars[2] = t[2];
        prm->scalars[3] = t[1] + t[2];
        prm->scalars[4] = sqrt(t[3] * t[3] + t[4] * t[4]) / t[5];
        prm->scalars[5] = t[6] / (double)ncells;
        prm->scalars[6] = t[3];
        prm->scalars[7] = t[4];
        prm->sum_psi = t[5];
      }
    }
  }
}

// The adaptive-substep rule, evaluated on the device in float64 from the
// maxima of k_dt_max: dt = cfl / max(v/ds, adv, rot, k_off + k_on L rho_max).
// A non-finite or non-positive rate leaves dt unchanged and sets status bit 1.
__global__ void k_dt_finalize(DevParams* prm, double ds, double L, double cfl) {
  const double rate = fmax(fmax(prm->v_walk / ds, prm->dtmax[0]),
                           fmax(prm->dtmax[1], prm->k_off + prm->k_on * L * prm->dtmax[2]));
  if (rate > 0.0 && isfinite(rate))
    prm->dt = cfl / rate;
  else
    atomicOr(&prm->status, 2);
}

// Per-cell velocity data of the psi transport: the cell's own u, the x
// component at the east/west neighbours, the y component at the north/south
// neighbours, and the central-difference velocity gradient G_ab = du_a/dx_b.
template <typename T>
__global__ void k_prep_ucell(T* ucell, const double* u64, long long ncells, int nx, int ny,
                             double inv_dx, double inv_dy) {
  const double* ux = u64;
  const double* uy = u64 + ncells;
  for (long long cell = blockIdx.x * (long long)blockDim.x + threadIdx.x; cell < ncells;
       cell += (long long)gridDim.x * blockDim.x) {
    const int ix = (int)(cell % nx), iy = (int)(cell / nx);
    const int xp = ix + 1 == nx ? 0 : ix + 1, xm = ix == 0 ? nx - 1 : ix - 1;
    const int yp = iy + 1 == ny ? 0 : iy + 1, ym = iy == 0 ? ny - 1 : iy - 1;
    const long long ce = (long long)iy * nx + xp, cw = (long long)iy * nx + xm;
    const long long cn = (long long)yp * nx + ix, cs = (long long)ym * nx + ix;
    T* o = ucell + cell * 12;
    o[0] = (T)ux[cell];
    o[1] = (T)uy[cell];
    o[2] = (T)ux[ce];
    o[3] = (T)ux[cw];
    o[4] = (T)uy[cn];
    o[5] = (T)uy[cs];
    // differences of the stored (precision T) velocities, as the oracle
    // differences its own velocity array
    o[6] = ((T)ux[ce] - (T)ux[cw]) * (T)(0.5 * inv_dx);
    o[7] = ((T)ux[cn] - (T)ux[cs]) * (T)(0.5 * inv_dy);
    o[8] = ((T)uy[ce] - (T)uy[cw]) * (T)(0.5 * inv_dx);
    o[9] = ((T)uy[cn] - (T)uy[cs]) * (T)(0.5 * inv_dy);
    o[10] = T(0);
    o[11] = T(0);
  }
}

int grid_for(long long n, int block) {
  long long g = (n + block - 1) / block;
  if (g > 152 * 16) g = 152 * 16;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

cudaError_t launch_copy_multi(const CopySegs& c, cudaStream_t s) {
  size_t most = 0;
  for (int q = 0; q < c.n; ++q) most = c.bytes[q] > most ? c.bytes[q] : most;
  if (most == 0) return cudaSuccess;
  k_copy_multi<<<grid_for((long long)((most + 15) / 16), 256), 256, 0, s>>>(c);
  return cudaGetLastError();
}

template <typename TO, typename TI>
cudaError_t launch_convert(TO* out, const TI* in, size_t n, const double* scale, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_convert<TO, TI><<<grid_for((long long)((n + 1) / 2), 256), 256, 0, s>>>(out, in, n, scale);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_prep_ucell(T* ucell, const double* u64, long long ncells, int nx, int ny,
                              double inv_dx, double inv_dy, cudaStream_t s) {
  k_prep_ucell<T><<<grid_for(ncells, 256), 256, 0, s>>>(ucell, u64, ncells, nx, ny, inv_dx, inv_dy);
  return cudaGetLastError();
}

// Widest vector of 16 bytes at most whose values divide ns.
template <typename T>
int row_vector(int ns) {
  for (int v = 16 / (int)sizeof(T); v > 1; v /= 2)
    if (ns % v == 0) return v;
  return 1;
}

template <typename T>
cudaError_t launch_init_cells(T* mb, const T* psi, T* nb, T* mf, T* c, const T* mtot,
                              long long ncells, int nth, int ns, double ds, double dth,
                              cudaStream_t s) {
  const int g = grid_for(ncells * 32, 128);
  auto go = [&](auto kern) {
    kern<<<g, 128, 0, s>>>(mb, psi, nb, mf, c, mtot, (int)ncells, nth, ns, ds, dth);
    return cudaGetLastError();
  };
  const int vw = row_vector<T>(ns);
  if constexpr (sizeof(T) == 4)
    if (vw == 4) return go(k_init_cells<T, 4>);
  return vw == 2 ? go(k_init_cells<T, 2>) : go(k_init_cells<T, 1>);
}

template <typename T>
cudaError_t launch_sum_psi(const T* psi, size_t n, double* partial, int max_partial,
                           DevParams* prm, cudaStream_t s) {
  int g = grid_for((long long)((n + 7) / 8), 512);
  if (g > max_partial) g = max_partial;
  k_sum_psi<T><<<g, 512, 0, s>>>(psi, n, partial, prm);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_dt_max(const T* psi, const T* nb, const T* u, const T* trig, long long ncells,
                          int nx, int ny, int nth, double inv_dx, double inv_dy, double inv_dth,
                          double dth, double glide, double vsp, DevParams* prm, cudaStream_t s) {
  int seg = 1;
  while (seg < 32 && seg < nth) seg <<= 1;
  int g = grid_for((ncells + 32 / seg - 1) / (32 / seg) * 32, kDtBlock);
  // at most the blocks that run at once, in float64 half of them: a block's end
  // costs more than a shorter share of the cells saves (mm_set_velocity in us at one,
  // two and four blocks an SM: float64 88^2 x 32 orientations 45, 49, 54, float32
  // 528^2 x 8 60, 53, 53)
  const int most = 152 * (sizeof(T) == 8 ? 1 : 2);
  if (g > most) g = most;
  k_dt_max<T><<<g, kDtBlock, 0, s>>>(psi, nb, u, trig, (int)ncells, nx, ny, nth, seg, inv_dx,
                                     inv_dy, inv_dth, dth, glide, vsp, prm);
  return cudaGetLastError();
}

cudaError_t launch_dt_finalize(DevParams* prm, double ds, double L, double cfl, cudaStream_t s) {
  k_dt_finalize<<<1, 1, 0, s>>>(prm, ds, L, cfl);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_moments(const T* psi, const T* mb, const T* mf, const T* c,
                           const double* trig, long long ncells, int nth, int ns, double dth,
                           double ds, double L, double dA, double* fields, double* partial,
                           int nblocks, DevParams* prm, cudaStream_t s) {
  // nblocks blocks of 4 warps; the partial buffer holds 8 doubles per warp
  const int block = 128;
  // per warp: n_b and m1 of the rows (float64), and their float-float sums
  const size_t smem = (size_t)4 * 2 * nth * sizeof(double) + (size_t)4 * nth * 16;
  auto go = [&](auto kern) -> cudaError_t {
    if (smem > 48 * 1024) {
      cudaError_t e = mm::raise_smem_limit(kern, (int)smem);
      if (e != cudaSuccess) return e;
    }
    kern<<<nblocks, block, smem, s>>>(psi, mb, mf, c, trig, ncells, nth, ns, dth, ds, L, dA,
                                      (float)(0.5 * ds), fields, partial, prm);
    return cudaGetLastError();
  };
  const int vw = row_vector<T>(ns);
  if constexpr (sizeof(T) == 4) {
    // rows of a power of two of full lanes: the cross-lane sums unrolled
    switch (ns % 8 == 0 ? ns / 8 : 0) {
      case 1: return go(k_moments<T, 4, 1>);
      case 2: return go(k_moments<T, 4, 2>);
      case 4: return go(k_moments<T, 4, 4>);
      case 8: return go(k_moments<T, 4, 8>);
      case 16: return go(k_moments<T, 4, 16>);
    }
    if (vw == 4) return go(k_moments<T, 4, 0>);
  }
  return vw == 2 ? go(k_moments<T, 2, 0>) : go(k_moments<T, 1, 0>);
}

template cudaError_t launch_sum_psi<float>(const float*, size_t, double*, int, DevParams*,
                                           cudaStream_t);
template cudaError_t launch_sum_psi<double>(const double*, size_t, double*, int, DevParams*,
                                            cudaStream_t);
template cudaError_t launch_convert<float, double>(float*, const double*, size_t, const double*,
                                                   cudaStream_t);
template cudaError_t launch_convert<double, float>(double*, const float*, size_t, const double*,
                                                   cudaStream_t);
template cudaError_t launch_convert<double, double>(double*, const double*, size_t,
                                                    const double*, cudaStream_t);
template cudaError_t launch_prep_ucell<float>(float*, const double*, long long, int, int, double,
                                              double, cudaStream_t);
template cudaError_t launch_prep_ucell<double>(double*, const double*, long long, int, int,
                                               double, double, cudaStream_t);
template cudaError_t launch_init_cells<float>(float*, const float*, float*, float*, float*,
                                              const float*, long long, int, int, double, double,
                                              cudaStream_t);
template cudaError_t launch_init_cells<double>(double*, const double*, double*, double*, double*,
                                               const double*, long long, int, int, double, double,
                                               cudaStream_t);
template cudaError_t launch_dt_max<float>(const float*, const float*, const float*, const float*,
                                          long long, int, int, int, double, double, double,
                                          double, double, double, DevParams*, cudaStream_t);
template cudaError_t launch_dt_max<double>(const double*, const double*, const double*,
                                           const double*, long long, int, int, int, double, double,
                                           double, double, double, double, DevParams*, cudaStream_t);
template cudaError_t launch_moments<float>(const float*, const float*, const float*,
                                           const float*, const double*, long long, int, int,
                                           double, double, double, double, double*, double*, int,
                                           DevParams*, cudaStream_t);
template cudaError_t launch_moments<double>(const double*, const double*, const double*,
                                            const double*, const double*, long long, int, int,
                                            double, double, double, double, double*, double*, int,
                                            DevParams*, cudaStream_t);

}  // namespace mm
