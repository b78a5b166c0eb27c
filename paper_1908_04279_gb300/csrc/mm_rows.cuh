// Row sums outside the substep (state set-up, moments, observables): s-rows
// read eight nodes per lane, and the float-float arithmetic of the float32
// form's sums.
#pragma once

#include "mm_walk.cuh"

namespace mm {

// float32 to float64 on the integer and float32 pipes (exact; the conversion
// instruction runs on the narrow float64 pipe, which held the exports at 4.7 TB/s
// of the 6.8 a copy reaches, and which bounds the float64 sums): the exponent
// rebiased, subnormal values brought into the normal range first.
__device__ __forceinline__ double widen(float x) {
  const unsigned u0 = __float_as_uint(x), mag = u0 & 0x7fffffffu;
  const bool sub = mag < 0x00800000u;
  const unsigned u = __float_as_uint(x * (sub ? 16777216.0f : 1.0f));
  const unsigned bias = sub ? 0x36800000u : mag < 0x7f800000u ? 0x38000000u : 0x70000000u;
  const unsigned hi = mag == 0u ? 0u : ((u & 0x7fffffffu) >> 3) + bias;
  return __hiloint2double((int)(hi | (u0 & 0x80000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

// Compensated float32 accumulator (hi + lo), error-free transformations of
// Knuth (TwoSum) and of the fused multiply-add (TwoProduct).
struct FF {
  float hi, lo;
};
__device__ __forceinline__ void ff_add(FF& a, float x) {
  const float s = a.hi + x;
  const float bb = s - a.hi;
  const float e = (a.hi - (s - bb)) + (x - bb);
  a.hi = s;
  a.lo += e;
}
// a + b (TwoSum of the high parts, low parts added)
__device__ __forceinline__ FF ff_sum(const FF& a, const FF& b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
  return FF{s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
}
// p w for a float p and a float-float w (TwoProduct of the high part)
__device__ __forceinline__ FF ff_scale(float p, const FF& w) {
  const float h = __fmul_rn(p, w.hi);
  return FF{h, __fmaf_rn(p, w.lo, __fmaf_rn(p, w.hi, -h))};
}
// a w for float-float a and w (the lo * lo term dropped)
__device__ __forceinline__ FF ff_prod(const FF& a, const FF& w) {
  const float h = __fmul_rn(a.hi, w.hi);
  return FF{h, __fmaf_rn(a.hi, w.lo, __fmaf_rn(a.lo, w.hi, __fmaf_rn(a.hi, w.hi, -h)))};
}

// The eight nodes of an s-row that a lane holds (8 sl ..., nv of them; the rest
// zero), in vectors of VW values: VW divides ns, so that every row, and every
// slot of eight, starts on a vector.
template <typename T, int VW>
struct alignas(sizeof(T) * VW) VPack {
  T v[VW];
};
template <typename T, int VW>
__device__ __forceinline__ void load_row8(const T* src, int nv, T (&m)[8]) {
#pragma unroll
  for (int q = 0; q < 8 / VW; ++q) {
    if (q * VW < nv) {
      const VPack<T, VW> x = reinterpret_cast<const VPack<T, VW>*>(src)[q];
#pragma unroll
      for (int v = 0; v < VW; ++v) m[q * VW + v] = x.v[v];
    } else {
#pragma unroll
      for (int v = 0; v < VW; ++v) m[q * VW + v] = T(0);
    }
  }
}
// Where a lane sits in packed rows: nl = ceil(ns / 8) lanes of eight nodes per
// row, floor(32 / nl) rows per pass.
struct PackedGeom {
  int nl, rpp, rslot, sl, nv;
};
__device__ __forceinline__ PackedGeom packed_geom(int lane, int ns) {
  PackedGeom g;
  g.nl = (ns + 7) / 8;
  g.rpp = 32 / g.nl;
  g.rslot = lane / g.nl;
  g.sl = lane - g.rslot * g.nl;
  g.nv = g.rslot < g.rpp ? min(8, ns - 8 * g.sl) : 0;
  return g;
}

// Two float-float accumulators in one register pair each (packed two-value
// instructions): a += x by TwoSum, differences as products with -1.
struct FF2x {
  float2 hi, lo;
};
__device__ __forceinline__ void ff2x_add(FF2x& a, float2 x) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 s = __fadd2_rn(a.hi, x);
  const float2 bb = __ffma2_rn(a.hi, m1, s);
  const float2 e1 = __ffma2_rn(__ffma2_rn(bb, m1, s), m1, a.hi);
  const float2 e2 = __ffma2_rn(bb, m1, x);
  a.lo = __fadd2_rn(a.lo, __fadd2_rn(e1, e2));
  a.hi = s;
}
// Sums over the nl lanes of a packed row, valid in its first lane. NL: nl where
// it is a power of two known at compile time (what the other lanes pick up
// from the next row is not used), else 0.
template <int NL>
__device__ __forceinline__ FF2x packed_sum_ff2x(FF2x x, int nl, int sl) {
  const float2 m1 = make_float2(-1.f, -1.f);
#pragma unroll
  for (int o = NL ? NL / 2 : 16; o > 0; o >>= 1) {
    if (NL || o < nl) {
      float2 h, l;
      h.x = __shfl_down_sync(0xffffffffu, x.hi.x, o);
      h.y = __shfl_down_sync(0xffffffffu, x.hi.y, o);
      l.x = __shfl_down_sync(0xffffffffu, x.lo.x, o);
      l.y = __shfl_down_sync(0xffffffffu, x.lo.y, o);
      if (NL || sl + o < nl) {
        ff2x_add(x, h);
        x.lo = __fadd2_rn(x.lo, l);
      }
    }
  }
  // high parts normalised
  const float2 s = __fadd2_rn(x.hi, x.lo);
  x.lo = __ffma2_rn(__ffma2_rn(x.hi, m1, s), m1, x.lo);
  x.hi = s;
  return x;
}

// n_b / ds (first) and m1 / ds (second) of a lane's nodes, one pair of
// accumulators: 17 float32 operations a node, and it is the float32 pipe that
// bounds these sums (packing the nodes in pairs instead needs the pairs added).
__device__ __forceinline__ FF2x row_sums8(const float (&m)[8], const float (&sj)[8]) {
  FF2x a{{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    const float p = __fmul_rn(m[v], sj[v]);
    const float pe = __fmaf_rn(m[v], sj[v], -p);
    ff2x_add(a, make_float2(m[v], p));
    a.lo.y = __fadd_rn(a.lo.y, pe);
  }
  return a;
}

}  // namespace mm
