// Many substeps in one launch with the motor density resident on the chip
// (float32 form): the substeps of k_substep for instances whose Mb fits the
// shared memory of all SMs together (up to about 30 MB).
//
// One block per SM owns a run of consecutive cells for the whole call and
// keeps their s-rows in shared memory: Mb crosses HBM once per call instead
// of once per substep, and the launch, the ring set-up, the scalar loads and
// the last-block sum that every k_substep launch pays are paid once. Between
// two substeps the blocks exchange only psi and n_b (through L2) and the
// filament number that fixes the float32 mass-correction factor, and no block
// waits for it idly: the motor rows of a cell need nothing but the cell's own
// Mf, so a warp goes on with the rows of substep n + 1 as soon as it has closed
// its cells of substep n, while one more warp of the block (the exchange warp)
// publishes the block's psi sum, waits for those of all the others and
// forms the factor. A warp waits (on an mbarrier in shared memory) only when it
// comes to psi of substep n + 1.
//
// Exchange: block b publishes the float pair of its psi sum in two 8-byte words,
// each with the substep's tag in its other half, so that a word is either old
// or whole; the word sets of two substeps alternate (a block can publish
// substep n + 2 only after every block published n + 1, hence read n). One
// counter of all arrivals is what is polled -- one sector, where polling the 152
// pairs of words kept L2 busy enough to delay them -- and the sums are read
// once it is complete, while the workers already load the neighbours' psi. The
// counter and the tags grow over the life of the handle, so no reset is needed
// between launches. The launch is cooperative (all blocks resident); every wait is
// bounded (DevParams::wait_limit polls): a block that gives up sets the status
// word and leaves, and the others then give up too.
//
// A worker warp owns `own` consecutive cells. Their rows go through the RK2 as
// one run: a row takes nl = ceil(ns / 8) lanes of eight nodes each and a pass
// takes the next floor(32 / nl) rows, of one cell or of several, so that neither
// short rows, nor odd ones, nor a row count that is no multiple of a pass
// leaves lanes idle (the streaming kernel gives a lane one node where ns is not
// a multiple of 4). With RAG the nodes past a row's end are kept at zero and
// the last node's slope is dropped by a factor. Rows in shared memory are
// lane-major: a pass is two arrays of 32 float4, lane l's eight nodes at [0][l]
// and [1][l], four conflict-free 16-byte accesses per lane whatever ns is. Psi
// takes one lane per orientation, 32 / seg cells at once where nth <= 16 (seg:
// nth rounded up to a power of two).
//
// Bound by instruction issue at the larger sizes (27 cells of 32 x 32 values per
// SM) and by the chain rows -> close -> arrival -> neighbours' psi at the
// smallest. Measured on a GB300, us per substep against k_substep in a CUDA
// graph: 32^2 x 16^2 8.0 -> 4.5, 64^2 x 32^2 13.2 -> 6.6, 85 x 61 x 24 x 30
// 57 -> 7.9, 128^2 x 16^2 (108 cells per SM) 24 -> 10.2.
#include <map>
#include <mutex>

#include "mm_async.cuh"
#include "mm_cell.cuh"
#include "mm_host.h"

namespace mm {

constexpr int kResXch = 5;        // published sums a lane of the exchange warp reads: 160 blocks
constexpr int kResMaxWarps = 15;  // workers of a block, beside the exchange warp

struct ResidentArgs {
  StepArgs<float> s;        // psi_in / nb_in: the state; psi_out / nb_out: the other buffers
  int n;                    // substeps
  int nl, rpp;              // lanes per row, rows per pass
  int vl;                   // nodes of a row's last lane
  int own;                  // most cells of a worker
  int passes;               // passes of a worker's rows at most
  int seg;                  // lanes per cell of the psi phase
  unsigned epoch;           // tags of this launch: epoch + 1 .. epoch + n
  unsigned arrivals;        // the arrival counter at this launch's start
  unsigned long long* xch;  // the arrival counter (16 bytes), then [2][gridDim][2] psi sums
};

struct ResidentSmem {
  size_t mass, cell, nb, tiles, total;
};
constexpr int kResCell = 20;  // 32-bit words per cell: u[10], Mf, M, five cell indices, spare
__host__ __device__ inline ResidentSmem resident_smem(int workers, int own, int nth, int passes) {
  ResidentSmem L;
  size_t off = 64;  // three mbarriers, the factor and the abort flag
  L.mass = off;
  off += 128;  // one float pair per worker
  L.cell = off;
  off += (size_t)workers * own * kResCell * 4;
  L.nb = off;
  off += (size_t)workers * own * nth * 4;
  off = (off + 15) & ~(size_t)15;
  L.tiles = off;
  off += (size_t)workers * passes * 1024;
  L.total = off;
  return L;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// The two words of a published sum: {value bits, tag}.
__device__ __forceinline__ unsigned long long tagged(float v, unsigned tag) {
  return ((unsigned long long)tag << 32) | __float_as_uint(v);
}

// The exchange warp: per substep, the block's psi sum out, all blocks' sums in.
// Returns early (abort flag set, workers released) when a wait gives up.
__device__ void exchange(const ResidentArgs& a, uint64_t* bars, const float2* s_mass,
                         volatile float* s_scale, volatile int* s_abort, int workers, int lane) {
  const unsigned G = gridDim.x;
  DevParams* P = a.s.prm;
  const uint32_t limit = P->wait_limit;
  const bool never = (P->debug_flags & 1u) != 0;  // test knob: every wait runs out
  const double mass0 = P->mass0;
  for (int t = 0; t < a.n; ++t) {
    // the workers' psi and n_b of this substep are written
    bool ok = mbar_wait(&bars[0], (uint32_t)(t & 1), kDrainLimit);
    const float2 own = warp_sum_ff2(lane < workers ? s_mass[lane] : make_float2(0.f, 0.f));
    unsigned long long* words = a.xch + 2 + (size_t)(t & 1) * 2 * G;
    const unsigned tag = a.epoch + 1u + (unsigned)t;
    if (lane == 0) {
      __threadfence();
      asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(
                       words + 2 * (size_t)blockIdx.x),
                   "l"(tagged(own.x, tag)), "l"(tagged(own.y, tag))
                   : "memory");
      asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(a.xch) : "memory");
    }
    const bool done = t + 1 == a.n;
    if (done && blockIdx.x != 0) break;  // block 0 stores the final sum
    if (lane == 0 && ok) {
      const unsigned target = a.arrivals + (unsigned)(t + 1) * G;
      for (uint32_t i = 0;; ++i) {
        unsigned c;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(a.xch) : "memory");
        if (!never && (int)(c - target) >= 0) break;
        if (i >= limit) {
          ok = false;
          break;
        }
      }
      __threadfence();
    }
    ok = __all_sync(0xffffffffu, ok);
    if (ok && lane == 0) mbar_arrive(&bars[1]);  // the neighbours' psi and n_b may be read
    // the sums, all of a lane's words in flight at once (a word may still be on
    // its way when its block's arrival has been counted: the tag tells)
    unsigned long long w0[kResXch], w1[kResXch];
    for (uint32_t i = 0; ok; ++i) {
      bool all = true;
#pragma unroll
      for (int q = 0; q < kResXch; ++q)  // (past the end: the last block's again, not added)
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
                     : "=l"(w0[q]), "=l"(w1[q])
                     : "l"(words + 2 * (size_t)min(lane + 32u * q, G - 1u))
                     : "memory");
#pragma unroll
      for (int q = 0; q < kResXch; ++q)
        all = all && (unsigned)(w0[q] >> 32) == tag && (unsigned)(w1[q] >> 32) == tag;
      if (__all_sync(0xffffffffu, all)) break;
      if (i >= limit) ok = false;
    }
    if (!ok) {
      if (lane == 0) {
        atomicOr(&P->status, 1);
        *s_abort = 1;
        __threadfence_block();
        mbar_arrive(&bars[1]);  // (where the arrivals were counted, the next phase: none waits)
        mbar_arrive(&bars[2]);
      }
      return;
    }
    float2 sum = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kResXch; ++q)
      if (lane + 32u * q < G)
        sum = ff2_add(sum, make_float2(__uint_as_float((unsigned)w0[q]),
                                       __uint_as_float((unsigned)w1[q])));
    const float2 m2 = warp_sum_ff2(sum);
    if (lane == 0) {
      const double m = (double)m2.x + (double)m2.y;
      const double scale = a.s.mass_correct ? mass0 / m : P->psi_scale;
      if (done) {
        P->mass = m;
        P->psi_scale = scale;
      } else {
        *s_scale = (float)scale;
        __threadfence_block();
        mbar_arrive(&bars[2]);
      }
    }
    __syncwarp();
  }
}

// NL: lanes per row when ns = 8 NL fills its lanes (2, 4 or 8); 0: any row.
template <int NL>
__global__ void __launch_bounds__(32 * (kResMaxWarps + 1), 1)
    k_substep_resident(const ResidentArgs a) {
  constexpr bool RAG = NL == 0;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int nth = a.s.nth, ns = a.s.ns, nx = a.s.nx, ny = a.s.ny;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int NW = (int)(blockDim.x >> 5) - 1;
  const ResidentSmem L = resident_smem(NW, a.own, nth, a.passes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_raw);  // written, readable, factor
  volatile float* s_scale = reinterpret_cast<float*>(smem_raw + 24);
  volatile int* s_abort = reinterpret_cast<int*>(smem_raw + 28);
  float2* s_mass = reinterpret_cast<float2*>(smem_raw + L.mass);
  if (threadIdx.x == 0) {
    mbar_init(&bars[0], (uint32_t)NW);
    mbar_init(&bars[1], 1);
    mbar_init(&bars[2], 1);
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (w == NW) {
    exchange(a, bars, s_mass, s_scale, s_abort, NW, lane);
    return;
  }

  // this warp's cells cw .. cw + ncw - 1 of the block's run
  const long long nc = a.s.ncells;
  const int c0 = (int)(nc * blockIdx.x / gridDim.x);
  const int ncl = (int)(nc * (blockIdx.x + 1) / gridDim.x) - c0;
  const int cw = c0 + w * a.own;
  const int ncw = max(0, min(a.own, ncl - w * a.own));
  const int nrows = ncw * nth;
  const int nl = NL ? NL : a.nl;
  const int rpp = NL ? 32 / (NL ? NL : 1) : a.rpp;
  const int passes = (nrows + rpp - 1) / rpp;
  const int rslot = lane / nl, sl = lane - rslot * nl;
  const bool first = sl == 0, last = sl == nl - 1;
  const bool lane_ok = rslot < rpp;
  const int nv = RAG && last ? a.vl : 8;  // nodes this lane holds
  float2 keep[4], valid[4];
  if constexpr (RAG) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      keep[h] = make_float2(last && 2 * h == nv - 1 ? 0.f : 1.f,
                            last && 2 * h + 1 == nv - 1 ? 0.f : 1.f);
      valid[h] = make_float2(2 * h < nv ? 1.f : 0.f, 2 * h + 1 < nv ? 1.f : 0.f);
    }
  }
  float* s_cell = reinterpret_cast<float*>(smem_raw + L.cell) + (size_t)w * a.own * kResCell;
  float* s_nb = reinterpret_cast<float*>(smem_raw + L.nb) + (size_t)w * a.own * nth;
  float4* tile = reinterpret_cast<float4*>(smem_raw + L.tiles) + (size_t)w * a.passes * 64 + lane;

  // load: the rows (row R of the warp's run is row cw nth + R of Mb), the
  // per-cell scalars and the neighbour indices
  for (int p = 0; p < passes; ++p) {
    const int R = p * rpp + rslot;
    float v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = 0.f;
    if (lane_ok && R < nrows) {
      const float* src = a.s.mb_in + ((size_t)cw * nth + R) * ns + sl * 8;
      if constexpr (RAG) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q < nv) v[q] = src[q];
      } else {
        const float4 x = reinterpret_cast<const float4*>(src)[0];
        const float4 y = reinterpret_cast<const float4*>(src)[1];
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
      }
    }
    tile[p * 64] = make_float4(v[0], v[1], v[2], v[3]);
    tile[p * 64 + 32] = make_float4(v[4], v[5], v[6], v[7]);
  }
  for (int j = 0; j < ncw; ++j) {
    const int cell = cw + j;
    float* sc = s_cell + j * kResCell;
    if (lane < 10) sc[lane] = a.s.ucell[(size_t)cell * 12 + lane];
    if (lane == 10) sc[10] = a.s.mf_in[cell];
    if (lane == 11) sc[11] = a.s.mtot[cell];
    if (lane == 12) {
      const int iy = cell / nx, ix = cell - iy * nx;
      int* id = reinterpret_cast<int*>(sc + 12);
      id[0] = cell;
      id[1] = iy * nx + (ix + 1 == nx ? 0 : ix + 1);
      id[2] = iy * nx + (ix == 0 ? nx - 1 : ix - 1);
      id[3] = (iy + 1 == ny ? 0 : iy + 1) * nx + ix;
      id[4] = (iy == 0 ? ny - 1 : iy - 1) * nx + ix;
    }
  }
  __syncwarp();

  const StepScalars<float> sc = step_scalars<float, true>(a.s.prm, a.s, lane);
  const float ds = sc.ds;
  const float c1 = sc.hdt * sc.cw, c2 = 1.0f - sc.hdt * sc.koff;
  const float e1 = sc.dt * sc.cw, e2 = -sc.dt * sc.koff;
  const float hk = sc.hdt * sc.kon, fk = sc.dt * sc.kon;
  const float2 c1_ = make_float2(c1, c1), c2_ = make_float2(c2, c2);
  const float2 e1_ = make_float2(e1, e1), e2_ = make_float2(e2, e2);
  PsiConst<float> pq{sc.dt,     sc.g,       sc.glide, sc.vsp, sc.inv_dx,
                     sc.inv_dy, sc.inv_dth, sc.dth,   a.s.trig};
  // psi phase: lane (sub, kl) takes orientations kl, kl + seg, ... of every
  // cps-th cell of the warp from its sub-th on
  const int seg = a.seg, cps = 32 / seg;
  const int sub = lane / seg, kl = lane - sub * seg;
  const int nk = (nth + seg - 1) / seg;  // 1 unless nth > 32
  const LaneTrig<float> lt = lane_trig(a.s.trig, nth, kl);
  float* pbuf[2] = {const_cast<float*>(a.s.psi_in), a.s.psi_out};
  float* nbuf[2] = {const_cast<float*>(a.s.nb_in), a.s.nb_out};
  const int jq = rpp / nth, jr = rpp - jq * nth;  // rows of a pass in cells and rows
  const int j0 = rslot / nth, r0 = rslot - j0 * nth;

  bool aborted = false;
  for (int t = 0; t < a.n; ++t) {
    // ---- the motor rows of this warp's cells by Eq. 4
    {
      int j = j0, r = r0;  // cell and orientation of the lane's row
#pragma unroll kStepUnroll
      for (int p = 0; p < passes; ++p) {
        const float mf = s_cell[min(j, ncw - 1) * kResCell + 10];
        const float c3 = hk * mf, e3 = fk * mf;
        const float2 c3_ = make_float2(c3, c3), e3_ = make_float2(e3, e3);
        const float4 x = tile[p * 64], y = tile[p * 64 + 32];
        float2 M[4] = {make_float2(x.x, x.y), make_float2(x.z, x.w), make_float2(y.x, y.y),
                       make_float2(y.z, y.w)};
        float2 D[4], Ms[4];
        walk_dflux_x2<8, RAG>(M, D, first, last, 32, keep);
#pragma unroll
        for (int h = 0; h < 4; ++h) Ms[h] = __ffma2_rn(c1_, D[h], __ffma2_rn(c2_, M[h], c3_));
        walk_dflux_x2<8, RAG>(Ms, D, first, last, 32, keep);
#pragma unroll
        for (int h = 0; h < 4; ++h)
          M[h] = __ffma2_rn(e1_, D[h], __ffma2_rn(e2_, Ms[h], __fadd2_rn(M[h], e3_)));
        if constexpr (RAG) {
#pragma unroll
          for (int h = 0; h < 4; ++h) M[h] = __fmul2_rn(M[h], valid[h]);
        }
        tile[p * 64] = make_float4(M[0].x, M[0].y, M[1].x, M[1].y);
        tile[p * 64 + 32] = make_float4(M[2].x, M[2].y, M[3].x, M[3].y);
        float2 acc = M[0];
#pragma unroll
        for (int h = 1; h < 4; ++h) acc = __fadd2_rn(acc, M[h]);
        const float snb = packed_sum(acc.x + acc.y, nl, sl);
        const int R = p * rpp + rslot;
        if (first && lane_ok && R < nrows) s_nb[R] = snb * ds;
        j += jq;
        r += jr;
        if (r >= nth) {
          r -= nth;
          ++j;
        }
      }
    }
    __syncwarp();

    // ---- psi of the substep before is everywhere written; its factor is known
    if (t > 0) {
      const bool ok = mbar_wait(&bars[1], (uint32_t)((t - 1) & 1), kDrainLimit);
      if (!__all_sync(0xffffffffu, ok) || *s_abort) {
        aborted = true;
        break;
      }
    }
    const float* psi_in = pbuf[t & 1];
    const float* nb_in = nbuf[t & 1];
    float* psi_out = pbuf[(t & 1) ^ 1];
    float* nb_out = nbuf[(t & 1) ^ 1];
    // (cell, theta) values are read through L2: other SMs wrote them
    auto load = [&](int j, int kk) {
      PsiIn<float> in{};
      const int k = kk * seg + kl;
      if (j < ncw && k < nth) {
        const int* id = reinterpret_cast<const int*>(s_cell + j * kResCell + 12);
        const int kp = k + 1 == nth ? 0 : k + 1, km = k == 0 ? nth - 1 : k - 1;
        const size_t o0 = (size_t)id[0] * nth, o1 = (size_t)id[1] * nth, o2 = (size_t)id[2] * nth;
        const size_t o3 = (size_t)id[3] * nth, o4 = (size_t)id[4] * nth;
        in.pc = __ldcg(psi_in + o0 + k);
        in.pe = __ldcg(psi_in + o1 + k);
        in.pw = __ldcg(psi_in + o2 + k);
        in.pn = __ldcg(psi_in + o3 + k);
        in.ps = __ldcg(psi_in + o4 + k);
        in.pp = __ldcg(psi_in + o0 + kp);
        in.pm = __ldcg(psi_in + o0 + km);
        in.nc = __ldcg(nb_in + o0 + k);
        in.ne = __ldcg(nb_in + o1 + k);
        in.nw = __ldcg(nb_in + o2 + k);
        in.nn = __ldcg(nb_in + o3 + k);
        in.ns = __ldcg(nb_in + o4 + k);
      }
      return in;
    };
    PsiIn<float> next = load(sub, 0);
    if (t > 0) {
      const bool ok = mbar_wait(&bars[2], (uint32_t)((t - 1) & 1), kDrainLimit);
      if (!__all_sync(0xffffffffu, ok) || *s_abort) {
        aborted = true;
        break;
      }
      pq.g = *s_scale;
    }

    // ---- Eq. 1 for psi, then Eq. 5, Alg. 2 and Eq. 6 (the next cells' values
    // loaded while one set is computed)
    float mass_hi = 0.f, mass_lo = 0.f;
    for (int jb = 0; jb < ncw; jb += cps) {
      const int j = jb + sub;
      const bool on = j < ncw;
      float* scl = s_cell + (on ? j : 0) * kResCell;
      const CellVel<float> uv{scl[0], scl[1], scl[2], scl[3], scl[4],
                              scl[5], scl[6], scl[7], scl[8], scl[9]};
      const float* nbc = s_nb + (on ? j : 0) * nth;
      const size_t cbase = (size_t)(cw + j) * nth;
      float acc = 0.f, cell_mass = 0.f;
      for (int kk = 0; kk < nk; ++kk) {
        const PsiIn<float> in = next;
        next = kk + 1 < nk ? load(j, kk + 1) : load(j + cps, 0);
        const int k = kk * seg + kl;
        if (on && k < nth) {
          const float pnew = psi_point(pq, uv, nk == 1 ? lt : trig_at(a.s.trig, nth, k), in);
          __stcg(psi_out + cbase + k, pnew);
          cell_mass += pnew;
          acc = fma_t(pnew * nbc[k], pq.dth, acc);
        }
      }
      two_sum_acc(mass_hi, mass_lo, cell_mass);
      const float Cpre = seg_sum(acc, seg);
      const float mtot = scl[11];
      float f = 1.f, C = Cpre;
      if (on && mtot < Cpre) {
        f = mtot / Cpre;
        C = mtot;
      }
      if (__any_sync(0xffffffffu, f != 1.f)) {  // Alg. 2 scale-down (rare): the cells' rows
        for (int q = 0; q < cps; ++q) {
          const float fq = __shfl_sync(0xffffffffu, f, q * seg);
          const int lo = (jb + q) * nth, hi = lo + nth;
          if (fq != 1.f)
            for (int p = lo / rpp; p <= (hi - 1) / rpp; ++p) {
              const int R = p * rpp + rslot;
              if (R >= lo && R < hi)
                for (int g = 0; g < 64; g += 32) {
                  float4 x = tile[p * 64 + g];
                  x.x *= fq; x.y *= fq; x.z *= fq; x.w *= fq;
                  tile[p * 64 + g] = x;
                }
            }
        }
      }
      for (int k = kl; on && k < nth; k += seg)
        __stcg(nb_out + cbase + k, f != 1.f ? nbc[k] * f : nbc[k]);
      __syncwarp();
      if (on && kl == 0) {
        scl[10] = mtot - C;
        if (t + 1 == a.n) {
          a.s.c[cw + j] = C;
          a.s.mf_out[cw + j] = mtot - C;
        }
      }
    }
    const float2 wsum = warp_sum_ff2(make_float2(mass_hi, mass_lo));
    if (lane == 0) s_mass[w] = wsum;
    __syncwarp();
    if (lane == 0) mbar_arrive(&bars[0]);
  }
  if (aborted) return;

  // store the rows
  for (int p = 0; p < passes; ++p) {
    const int R = p * rpp + rslot;
    if (!(lane_ok && R < nrows)) continue;
    const float4 x = tile[p * 64], y = tile[p * 64 + 32];
    float* dst = a.s.mb_out + ((size_t)cw * nth + R) * ns + sl * 8;
    if constexpr (RAG) {
      const float v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q < nv) dst[q] = v[q];
    } else {
      reinterpret_cast<float4*>(dst)[0] = x;
      reinterpret_cast<float4*>(dst)[1] = y;
    }
  }
}

}  // namespace mm

namespace mmh {

namespace {

constexpr size_t kResidentBudget = 227 * 1024;  // shared memory a block may have

const void* resident_kernel(int NL) {
  return NL == 2   ? (const void*)mm::k_substep_resident<2>
         : NL == 4 ? (const void*)mm::k_substep_resident<4>
         : NL == 8 ? (const void*)mm::k_substep_resident<8>
                   : (const void*)mm::k_substep_resident<0>;
}

// Resident launches of one device run one after the other, on whatever
// streams and from whatever threads they come: each fills every SM, and two of
// them part-way resident would wait for each other's blocks. The event of the
// last one orders the next.
struct DeviceOrder {
  std::mutex m;
  std::map<int, cudaEvent_t> last;
};
DeviceOrder& device_order() {
  static DeviceOrder* d = new DeviceOrder();  // never destroyed: launches may outlive statics
  return *d;
}

}  // namespace

// Plan: one block per SM with ceil(cells / SMs) cells, as many workers as give
// every warp the same number of cells. Off (h->res_grid = 0) in float64 and
// where a block's rows do not fit its shared memory.
mm_status resident_configure(mm_handle* h) {
  h->res_grid = 0;
  if (h->prec != MM_FP32_MIXED) return MM_OK;
  int coop = 0;
  CK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->device));
  if (!coop) return MM_OK;
  const int ns = h->g.ns, nth = h->g.ntheta;
  const int nl = (ns + 7) / 8;
  h->res_NL = ns % 8 == 0 && (nl == 2 || nl == 4 || nl == 8) ? nl : 0;
  const long long grid = std::min<long long>({h->sms, h->ncells, 32 * mm::kResXch});
  const long long cells = (h->ncells + grid - 1) / grid;
  if (cells * nth * nl * 32 > (long long)kResidentBudget) return MM_OK;
  h->res_own = (int)((cells + mm::kResMaxWarps - 1) / mm::kResMaxWarps);
  const int workers = (int)((cells + h->res_own - 1) / h->res_own);
  const int rpp = 32 / nl;
  h->res_passes = (h->res_own * nth + rpp - 1) / rpp;
  const size_t smem = mm::resident_smem(workers, h->res_own, nth, h->res_passes).total;
  if (smem > kResidentBudget) return MM_OK;
  const void* f = resident_kernel(h->res_NL);
  CK(mm::raise_smem_limit(f, smem));
  int bps = 0;
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, f, 32 * (workers + 1), smem));
  if (bps < 1) return MM_OK;
  h->res_block = 32 * (workers + 1);
  h->res_smem = smem;
  h->res_grid = (int)grid;
  return MM_OK;
}

// n substeps on the live state in one launch; *done = false (and nothing
// launched) where the resident kernel does not apply: no plan, a single
// substep, another substep kernel in effect, or a stream being captured (the
// ordering event belongs to no capture).
mm_status resident_substeps(mm_handle* h, int n, bool* done) {
  *done = false;
  if (h->res_grid == 0 || n < 2 || h->anchors || h->capture || h->tangent) return MM_OK;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  CK(cudaStreamIsCapturing(h->stream, &cs));
  if (cs != cudaStreamCaptureStatusNone) return MM_OK;
  mm::ResidentArgs a{};
  a.s = step_args<float>(h, h->parity);
  a.n = n;
  a.nl = (h->g.ns + 7) / 8;
  a.rpp = 32 / a.nl;
  a.vl = h->g.ns - 8 * (a.nl - 1);
  a.own = h->res_own;
  a.passes = h->res_passes;
  a.seg = 1;
  while (a.seg < 32 && a.seg < h->g.ntheta) a.seg <<= 1;
  a.epoch = h->res_epoch;
  a.arrivals = h->res_arrivals;
  a.xch = h->res_xch;
  h->res_epoch += (unsigned)n;
  h->res_arrivals += (unsigned)n * (unsigned)h->res_grid;
  void* args[1] = {&a};
  DeviceOrder& o = device_order();
  std::lock_guard<std::mutex> lock(o.m);
  cudaEvent_t& ev = o.last[h->device];
  if (!ev)
    CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
  else
    CK(cudaStreamWaitEvent(h->stream, ev, 0));
  CK(cudaLaunchCooperativeKernel(resident_kernel(h->res_NL), dim3((unsigned)h->res_grid),
                                 dim3((unsigned)h->res_block), args, h->res_smem, h->stream));
  CK(cudaEventRecord(ev, h->stream));
  h->parity ^= n & 1;
  *done = true;
  return MM_OK;
}

}  // namespace mmh
