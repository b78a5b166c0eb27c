// Many substeps in one launch with the motor density resident on the chip
// (float32 form): the substeps of k_substep for instances up to about twice the
// size of L2 (resident_limit, mm_plan.h). Mb is kept in the shared memory of all SMs
// together (about 33 MB), whole or in part; the row passes that do not fit are
// read and written every substep through each worker's ring.
//
// A block (one per SM; fewer of a small instance) owns a run of cells for the call and
// keeps their s-rows in shared memory: what is kept crosses HBM once per call
// instead of once per substep, and the launch, the ring set-up, the scalar loads and
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
// leaves lanes idle. With RAG the nodes past a row's end are kept at zero and
// the last node's slope is dropped by a factor. Rows in shared memory are
// lane-major: a pass is two arrays of 32 float4, lane l's eight nodes at [0][l]
// and [1][l], four conflict-free 16-byte accesses per lane whatever ns is. Psi
// takes one lane per orientation, 32 / seg cells at once where nth <= 16 (seg:
// nth rounded up to a power of two).
//
// Where Mb is larger than the shared memory of all SMs, a worker keeps the first
// `tiles` passes of its rows and reads and writes the others every substep, each
// lane copying its own values to its own slots two passes ahead (cp.async) and
// storing the new ones straight back; they stay in the L2 up to about twice its
// size (resident_limit says where k_substep takes over).
//
// A batch's members are independent, so several go into one launch
// (k_substep_resident_group), each over its own share of the SMs with its own
// exchange.
//
// Bound by instruction issue at the larger sizes (about 58 % of the slots; the
// rest goes to fixed latencies, psi loads and the half-rate minima) and by the
// chain rows -> close -> arrival -> neighbours' psi at the smallest. 15 workers of
// 128 registers: 19 of 96 are within 3 %, 11 or 23 slower. Measured on a GB300,
// us per substep against k_substep in a CUDA graph: 32^2 x 16^2 7.2 -> 4.1, 64^2 x
// 32^2 13.4 -> 6.4, 128^2 x 16^2 23 -> 9.7, 128^2 x 32^2 35.2 -> 25.4, 256^2 x 16^2
// 77 -> 35; against one launch a call 85 x 61 x 24 x 30 20 -> 8.0, 200 x 150 x 24 x 30 69 ->
// 45, 400^2 x 24 x 30 331 -> 243; the 64-member ensemble 594 (tuned) -> 424.
#include <map>
#include <mutex>

#include "mm_async.cuh"
#include "mm_cell.cuh"
#include "mm_host.h"

namespace mm {

constexpr int kResXch = 5;        // published sums a lane of the exchange warp reads: 160 blocks
constexpr int kResRing = 2;       // ring stages of a worker
constexpr int kResMaxWarps = 15;  // workers of a block, beside the exchange warp

struct ResidentArgs {
  StepArgs<float> s;        // psi_in / nb_in: the state; psi_out / nb_out: the other buffers
  int n;                    // substeps
  int nl, rpp;              // lanes per row, rows per pass
  int vl;                   // nodes of a row's last lane
  int own;                  // most cells of a worker
  int tiles;                // passes of a worker kept in shared memory at most
  int ring;                 // stages of a worker for the passes read every substep (0: none)
  int vw;                   // values of a vector that divides ns: 4, 2 or 1
  int workers;              // worker warps of a block
  int grid;                 // blocks of the instance
  int NL;                   // lanes per row when ns = 8 NL fills them (2, 4 or 8), else 0
  int seg;                  // lanes per cell of the psi phase
  unsigned epoch;           // tags of this launch: epoch + 1 .. epoch + n
  unsigned arrivals;        // the arrival counter at this launch's start
  unsigned long long* xch;  // the arrival counter (16 bytes), then [2][gridDim][2] psi sums
};

struct ResidentSmem {
  size_t mass, cell, nb, tiles, total;
};
constexpr int kResCell = 20;  // 32-bit words per cell: u[10], Mf, M, offsets of the five
                              // cells' columns, whether its west neighbour is the cell before
__host__ __device__ inline ResidentSmem resident_smem(int workers, int own, int nth, int tiles) {
  ResidentSmem L;
  size_t off = 64;  // three mbarriers, the factor and the abort flag
  L.mass = off;
  off += 256;  // one float pair per worker
  L.cell = off;
  off += (size_t)workers * own * kResCell * 4;
  L.nb = off;
  off += (size_t)workers * own * nth * 4;
  off = (off + 15) & ~(size_t)15;
  L.tiles = off;
  off += (size_t)workers * tiles * 1024;  // kept passes, then ring stages
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
                         volatile float* s_scale, volatile int* s_abort, int block, int lane) {
  const unsigned G = (unsigned)a.grid;
  const int workers = a.workers;
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
                       words + 2 * (size_t)block),
                   "l"(tagged(own.x, tag)), "l"(tagged(own.y, tag))
                   : "memory");
      asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(a.xch) : "memory");
    }
    const bool done = t + 1 == a.n;
    if (done && block != 0) break;  // block 0 stores the final sum
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
    const bool readable = ok;
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
        // (once a phase: a second arrival would complete the next one, and a worker that
        // comes late would take this one, two back by then, for not yet completed)
        if (!readable) mbar_arrive(&bars[1]);
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

// A lane's nv values of a row from global memory (src) into its slots of a
// ring stage, in vectors of vw values.
template <bool RAG>
__device__ __forceinline__ void stage_row8(float* slot, const float* src, int nv, int vw) {
  if (!RAG || vw == 4) {
    cp_async16(slot, src);
    if (!RAG || nv > 4) cp_async16(slot + 128, src + 4);
  } else if (vw == 2) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (2 * q < nv) cp_async8(slot + (q & 1) * 2 + (q >> 1) * 128, src + 2 * q);
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (q < nv) cp_async_t(slot + (q & 3) + (q >> 2) * 128, src + q);
  }
}
template <bool RAG>
__device__ __forceinline__ void store_row8(float* dst, const float2 (&M)[4], int nv, int vw) {
  if (!RAG || vw == 4) {
    reinterpret_cast<float4*>(dst)[0] = make_float4(M[0].x, M[0].y, M[1].x, M[1].y);
    if (!RAG || nv > 4)
      reinterpret_cast<float4*>(dst)[1] = make_float4(M[2].x, M[2].y, M[3].x, M[3].y);
  } else if (vw == 2) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (2 * q < nv) reinterpret_cast<float2*>(dst)[q] = M[q];
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (2 * q < nv) dst[2 * q] = M[q].x;
      if (2 * q + 1 < nv) dst[2 * q + 1] = M[q].y;
    }
  }
}

// The whole of one block: block `block` of the a.grid blocks of an instance.
// NL: lanes per row when ns = 8 NL fills its lanes (2, 4 or 8); 0: any row.
template <int NL>
__device__ __forceinline__ void resident_block(const ResidentArgs& a, int block) {
  constexpr bool RAG = NL == 0;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int nth = a.s.nth, ns = a.s.ns, nx = a.s.nx, ny = a.s.ny;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int NW = a.workers;
  const ResidentSmem L = resident_smem(NW, a.own, nth, a.tiles + a.ring);
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
  if (w == NW) exchange(a, bars, s_mass, s_scale, s_abort, block, lane);
  if (w >= NW) return;

  // this warp's cells cw .. cw + ncw - 1 of the block's run
  const long long nc = a.s.ncells;
  const int c0 = (int)(nc * block / a.grid);
  const int ncl = (int)(nc * (block + 1) / a.grid) - c0;
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
  float4* tile =
      reinterpret_cast<float4*>(smem_raw + L.tiles) + (size_t)w * (a.tiles + a.ring) * 64 + lane;
  float4* ring = tile + a.tiles * 64;
  const int kept = min(passes, a.tiles), streamed = passes - kept;
  // the lane's slot of pass p: row R = p rpp + rslot of the run, which is row
  // cw nth + R of Mb
  float* rows = a.s.mb_out + ((size_t)cw * nth + rslot) * ns + sl * 8;
  const size_t pass_vals = (size_t)rpp * ns;

  // load: the kept rows, the per-cell scalars and the neighbour indices
  for (int p = 0; p < kept + a.ring; ++p) {
    tile[p * 64] = make_float4(0.f, 0.f, 0.f, 0.f);
    tile[p * 64 + 32] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncwarp();
  for (int p = 0; p < kept; ++p)
    if (lane_ok && p * rpp + rslot < nrows)
      stage_row8<RAG>(reinterpret_cast<float*>(tile + p * 64), rows + p * pass_vals, nv, a.vw);
  cp_async_commit();
  cp_async_wait<0>();
  for (int j = 0; j < ncw; ++j) {
    const int cell = cw + j;
    float* sc = s_cell + j * kResCell;
    if (lane < 10) sc[lane] = a.s.ucell[(size_t)cell * 12 + lane];
    if (lane == 10) sc[10] = a.s.mf_in[cell];
    if (lane == 11) sc[11] = a.s.mtot[cell];
    if (lane == 12) {
      const int iy = cell / nx, ix = cell - iy * nx;
      unsigned* id = reinterpret_cast<unsigned*>(sc + 12);
      id[0] = (unsigned)cell * nth;
      id[1] = (unsigned)(iy * nx + (ix + 1 == nx ? 0 : ix + 1)) * nth;
      id[2] = (unsigned)(iy * nx + (ix == 0 ? nx - 1 : ix - 1)) * nth;
      id[3] = (unsigned)((iy + 1 == ny ? 0 : iy + 1) * nx + ix) * nth;
      id[4] = (unsigned)((iy == 0 ? ny - 1 : iy - 1) * nx + ix) * nth;
      id[5] = ix != 0;
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
  // psi phase: lane (sub, kl) takes orientations kl, kl + seg, ... of the cells
  // of the sub-th part of the warp's run, `half` cells
  const int seg = a.seg, cps = 32 / seg;
  const int sub = lane / seg, kl = lane - sub * seg;
  const int half = (ncw + cps - 1) / cps;
  const int nk = (nth + seg - 1) / seg;  // 1 unless nth > 32
  const LaneTrig<float> lt = lane_trig(a.s.trig, nth, kl);
  const int up = sub * seg + (kl + 1 >= nth ? 0 : kl + 1);    // lanes of theta + 1 and
  const int down = sub * seg + (kl == 0 ? nth - 1 : kl - 1);  // theta - 1 (nth <= 32)
  float* pbuf[2] = {const_cast<float*>(a.s.psi_in), a.s.psi_out};
  float* nbuf[2] = {const_cast<float*>(a.s.nb_in), a.s.nb_out};
  const int jq = rpp / nth, jr = rpp - jq * nth;  // rows of a pass in cells and rows
  const int j0 = rslot / nth, r0 = rslot - j0 * nth;

  bool aborted = false;
  for (int t = 0; t < a.n; ++t) {
    // ---- the motor rows of this warp's cells by Eq. 4
    {
      int j = j0, r = r0;  // cell and orientation of the lane's row
      auto rk2 = [&](const float4* t, int p, float2 (&M)[4]) {
        const float mf = s_cell[min(j, ncw - 1) * kResCell + 10];
        const float c3 = hk * mf, e3 = fk * mf;
        const float2 c3_ = make_float2(c3, c3), e3_ = make_float2(e3, e3);
        const float4 x = t[0], y = t[32];
        M[0] = make_float2(x.x, x.y);
        M[1] = make_float2(x.z, x.w);
        M[2] = make_float2(y.x, y.y);
        M[3] = make_float2(y.z, y.w);
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
        const float snb = row_sum_x2(M, RAG ? a.vl : 8, nl, sl);
        const int R = p * rpp + rslot;
        if (first && lane_ok && R < nrows) s_nb[R] = snb * ds;
        j += jq;
        r += jr;
        if (r >= nth) {
          r -= nth;
          ++j;
        }
      };
      // streamed passes: a lane copies its own values to its own slots `ring`
      // passes ahead (the first of them under the kept passes) and stores the
      // new ones straight back
      auto issue = [&](int q) {
        const int p = kept + q;
        if (q < streamed && lane_ok && p * rpp + rslot < nrows)
          stage_row8<RAG>(reinterpret_cast<float*>(ring + (q % kResRing) * 64),
                          rows + p * pass_vals, nv, a.vw);
        cp_async_commit();
      };
      if (streamed > 0) {
        __threadfence_block();  // after this lane's stores of the substep before
        for (int q = 0; q < kResRing; ++q) issue(q);
      }
#pragma unroll 1
      for (int p = 0; p < kept; ++p) {
        float2 M[4];
        rk2(tile + p * 64, p, M);
        tile[p * 64] = make_float4(M[0].x, M[0].y, M[1].x, M[1].y);
        tile[p * 64 + 32] = make_float4(M[2].x, M[2].y, M[3].x, M[3].y);
      }
#pragma unroll 1
      for (int q = 0; q < streamed; ++q) {
        cp_async_wait<kResRing - 1>();
        const int p = kept + q;
        float2 M[4];
        rk2(ring + (q % kResRing) * 64, p, M);
        if (lane_ok && p * rpp + rslot < nrows)
          store_row8<RAG>(rows + p * pass_vals, M, nv, a.vw);
        issue(q + kResRing);
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
    float mass_hi = 0.f, mass_lo = 0.f;
    // Eq. 5, Alg. 2 and Eq. 6 of cell j (of each sub's cell at once), from the
    // lanes' parts of the coarse density
    auto close = [&](int it, int j, bool on, float cell_mass, float acc, float mtot) {
      float* scl = s_cell + j * kResCell;
      const float* nbc = s_nb + j * nth;
      two_sum_acc(mass_hi, mass_lo, cell_mass);
      const float Cpre = seg_sum(acc, seg);
      float f = 1.f, C = Cpre;
      if (on && mtot < Cpre) {
        f = mtot / Cpre;
        C = mtot;
      }
      if (__any_sync(0xffffffffu, f != 1.f)) {  // Alg. 2 scale-down (rare): the cells' rows
        for (int q = 0; q < cps; ++q) {
          const float fq = __shfl_sync(0xffffffffu, f, q * seg);
          const int lo = (q * half + it) * nth, hi = lo + nth;
          if (fq != 1.f)
            for (int p = lo / rpp; p <= (hi - 1) / rpp; ++p) {
              const int R = p * rpp + rslot;
              if (!lane_ok || R < lo || R >= hi) continue;
              if (p < kept) {
                for (int g = 0; g < 64; g += 32) {
                  float4 x = tile[p * 64 + g];
                  x.x *= fq; x.y *= fq; x.z *= fq; x.w *= fq;
                  tile[p * 64 + g] = x;
                }
              } else {
                for (int v = 0; v < nv; ++v) rows[p * pass_vals + v] *= fq;
              }
            }
        }
      }
      float* nbo = nb_out + (size_t)(cw + j) * nth;
      for (int k = kl; on && k < nth; k += seg) __stcg(nbo + k, f != 1.f ? nbc[k] * f : nbc[k]);
      __syncwarp();
      if (on && kl == 0) {
        scl[10] = mtot - C;
        if (t + 1 == a.n) {
          a.s.c[cw + j] = C;
          a.s.mf_out[cw + j] = mtot - C;
        }
      }
    };
    auto factor = [&]() {  // the pending correction factor; false: a wait gave up
      if (t > 0) {
        const bool ok = mbar_wait(&bars[2], (uint32_t)((t - 1) & 1), kDrainLimit);
        if (!__all_sync(0xffffffffu, ok) || *s_abort) return false;
        pq.g = *s_scale;
      }
      return true;
    };

    // ---- Eq. 1 for psi, then Eq. 5, Alg. 2 and Eq. 6, a cell (one per sub) at a
    // time with the next one's values loaded ahead; psi and n_b are read
    // through L2, other SMs wrote them
    if (nk == 1) {
      // The cells of a run follow one another in x: the cell before is the west
      // neighbour, and its east face, its own centre and its east neighbour are
      // this cell's west face, west neighbour and centre, the same bits. The
      // theta neighbours come by shuffle, as does the flux of the face theta - 1/2.
      struct In {
        float pe, pn, ps, ne, nn, ns, pc, pw, nc, nw;
      };
      const float* pk = psi_in + kl;
      const float* nbk = nb_in + kl;
      const bool kon = kl < nth;
      auto load = [&](int it) {
        In in{};
        const int j = sub * half + it;
        if (kon && it < half && j < ncw) {
          const uint4 o = *reinterpret_cast<const uint4*>(s_cell + j * kResCell + 12);
          const uint2 o2 = *reinterpret_cast<const uint2*>(s_cell + j * kResCell + 16);
          in.pe = __ldcg(pk + o.y);
          in.pn = __ldcg(pk + o.w);
          in.ps = __ldcg(pk + o2.x);
          in.ne = __ldcg(nbk + o.y);
          in.nn = __ldcg(nbk + o.w);
          in.ns = __ldcg(nbk + o2.x);
          if (it == 0 || !o2.y) {
            in.pc = __ldcg(pk + o.x);
            in.pw = __ldcg(pk + o.z);
            in.nc = __ldcg(nbk + o.x);
            in.nw = __ldcg(nbk + o.z);
          }
        }
        return in;
      };
      In next = load(0);
      if (!factor()) {
        aborted = true;
        break;
      }
      const float g = pq.g;
      const float ck = lt.ck, sk = lt.sk, cp = lt.cp, sp = lt.sp;
      float Pe = 0.f, Ve = 0.f, axe = 0.f, Fe = 0.f;  // the cell before's
      for (int it = 0; it < half; ++it) {
        const In in = next;
        next = load(it + 1);
        const bool on = sub * half + it < ncw;
        const int j = on ? sub * half + it : 0;
        const float4* q4 = reinterpret_cast<const float4*>(s_cell + j * kResCell);
        const float4 ua = q4[0], ub = q4[1], uc = q4[2];  // u at c, e, w (x) and n, s (y); grad u
        float Pc = Pe, Vc = Ve, axc = axe, Fw = Fe;
        if (it == 0 || !reinterpret_cast<const unsigned*>(q4)[17]) {
          const float Pw = g * in.pw, Vw = fma_t(pq.glide, in.nw, pq.vsp);
          Pc = g * in.pc;
          Vc = fma_t(pq.glide, in.nc, pq.vsp);
          axc = fma_t(-Vc, ck, ua.x);
          const float axw = fma_t(-Vw, ck, ua.w);
          Fw = donor(0.5f * (axw + axc), Pw, Pc);
        }
        Pe = g * in.pe;
        const float Pn = g * in.pn, Ps = g * in.ps;
        Ve = fma_t(pq.glide, in.ne, pq.vsp);
        const float Vn = fma_t(pq.glide, in.nn, pq.vsp), Vs = fma_t(pq.glide, in.ns, pq.vsp);
        axe = fma_t(-Ve, ck, ua.z);
        const float ayc = fma_t(-Vc, sk, ua.y);
        const float ayn = fma_t(-Vn, sk, ub.x), ays = fma_t(-Vs, sk, ub.y);
        const float wp = fma_t(-sp, fma_t(ub.z, cp, ub.w * sp), cp * fma_t(uc.x, cp, uc.y * sp));
        Fe = donor(0.5f * (axc + axe), Pc, Pe);
        const float Fn = donor(0.5f * (ayc + ayn), Pc, Pn);
        const float Fs = donor(0.5f * (ays + ayc), Ps, Pc);
        const float Fp = donor(wp, Pc, __shfl_sync(0xffffffffu, Pc, up));
        const float Fm = __shfl_sync(0xffffffffu, Fp, down);
        const float div =
            fma_t(Fp - Fm, pq.inv_dth, fma_t(Fn - Fs, pq.inv_dy, (Fe - Fw) * pq.inv_dx));
        const float pnew = fma_t(-pq.dt, div, Pc);
        float acc = 0.f;
        if (on && kon) {
          __stcg(psi_out + (size_t)(cw + j) * nth + kl, pnew);
          acc = fma_t(pnew * s_nb[j * nth + kl], pq.dth, 0.f);
        }
        close(it, j, on, on && kon ? pnew : 0.f, acc, uc.w);
      }
    } else {
      // more than 32 orientations: a lane takes several of every cell
      auto load = [&](int j, int kk) {
        PsiIn<float> in{};
        const int k = kk * 32 + lane;
        if (j < ncw && k < nth) {
          const unsigned* id = reinterpret_cast<const unsigned*>(s_cell + j * kResCell + 12);
          const int kp = k + 1 == nth ? 0 : k + 1, km = k == 0 ? nth - 1 : k - 1;
          const float *p0 = psi_in + id[0], *n0 = nb_in + k;
          in.pc = __ldcg(p0 + k);
          in.pp = __ldcg(p0 + kp);
          in.pm = __ldcg(p0 + km);
          in.pe = __ldcg(psi_in + id[1] + k);
          in.pw = __ldcg(psi_in + id[2] + k);
          in.pn = __ldcg(psi_in + id[3] + k);
          in.ps = __ldcg(psi_in + id[4] + k);
          in.nc = __ldcg(n0 + id[0]);
          in.ne = __ldcg(n0 + id[1]);
          in.nw = __ldcg(n0 + id[2]);
          in.nn = __ldcg(n0 + id[3]);
          in.ns = __ldcg(n0 + id[4]);
        }
        return in;
      };
      PsiIn<float> next = load(0, 0);
      if (!factor()) {
        aborted = true;
        break;
      }
      for (int j = 0; j < ncw; ++j) {
        const float* scl = s_cell + j * kResCell;
        const CellVel<float> uv{scl[0], scl[1], scl[2], scl[3], scl[4],
                                scl[5], scl[6], scl[7], scl[8], scl[9]};
        const float* nbc = s_nb + j * nth;
        float acc = 0.f, cell_mass = 0.f;
        for (int kk = 0; kk < nk; ++kk) {
          const PsiIn<float> in = next;
          next = kk + 1 < nk ? load(j, kk + 1) : load(j + 1, 0);
          const int k = kk * 32 + lane;
          if (k < nth) {
            const float pnew = psi_point(pq, uv, trig_at(a.s.trig, nth, k), in);
            __stcg(psi_out + (size_t)(cw + j) * nth + k, pnew);
            cell_mass += pnew;
            acc = fma_t(pnew * nbc[k], pq.dth, acc);
          }
        }
        close(j, j, true, cell_mass, acc, scl[11]);
      }
    }
    const float2 wsum = warp_sum_ff2(make_float2(mass_hi, mass_lo));
    if (lane == 0) s_mass[w] = wsum;
    __syncwarp();
    if (lane == 0) mbar_arrive(&bars[0]);
  }
  if (aborted) return;

  // store the kept rows
  for (int p = 0; p < kept; ++p) {
    if (!(lane_ok && p * rpp + rslot < nrows)) continue;
    const float4 x = tile[p * 64], y = tile[p * 64 + 32];
    const float2 M[4] = {make_float2(x.x, x.y), make_float2(x.z, x.w), make_float2(y.x, y.y),
                         make_float2(y.z, y.w)};
    store_row8<RAG>(rows + p * pass_vals, M, nv, a.vw);
  }
}

template <int NL>
__global__ void __launch_bounds__(32 * (kResMaxWarps + 1), 1)
    k_substep_resident(const ResidentArgs a) {
  resident_block<NL>(a, blockIdx.x);
}

// (its own function per row form: the register allocation of one is not that of
// all four together)
template <int NL>
__device__ __noinline__ void resident_block_of_group(const ResidentArgs& a, int block) {
  resident_block<NL>(a, block);
}

// Several independent instances in one launch: map[blockIdx.x] = (entry of tab,
// block of that instance). Each instance has its own exchange.
__global__ void __launch_bounds__(32 * (kResMaxWarps + 1), 1)
    k_substep_resident_group(const ResidentArgs* __restrict__ tab, const int2* __restrict__ map) {
  __shared__ ResidentArgs s_a;
  const int2 m = map[blockIdx.x];
  static_assert(sizeof(ResidentArgs) % 4 == 0, "copied by words");
  for (unsigned i = threadIdx.x; i < sizeof(ResidentArgs) / 4; i += blockDim.x)
    reinterpret_cast<unsigned*>(&s_a)[i] = reinterpret_cast<const unsigned*>(tab + m.x)[i];
  __syncthreads();
  switch (s_a.NL) {
    case 2: resident_block_of_group<2>(s_a, m.y); break;
    case 4: resident_block_of_group<4>(s_a, m.y); break;
    case 8: resident_block_of_group<8>(s_a, m.y); break;
    default: resident_block_of_group<0>(s_a, m.y); break;
  }
}

}  // namespace mm

namespace mmh {

namespace {

constexpr size_t kResidentBudget = 226 * 1024;  // dynamic shared memory of a block

const void* resident_kernel(int NL) {
  return NL == 2   ? (const void*)mm::k_substep_resident<2>
         : NL == 4 ? (const void*)mm::k_substep_resident<4>
         : NL == 8 ? (const void*)mm::k_substep_resident<8>
                   : (const void*)mm::k_substep_resident<0>;
}

// How an instance goes over `grid` blocks of one SM each: ceil(cells / grid) cells
// to a block, the same number `own` to each worker, `tiles` passes of a worker's
// rows kept in shared memory and, where that is not all of them, a ring for the
// others, which are read and written every substep. False where it does not fit
// (resident_limit says where it pays).
struct ResidentPlan {
  int own, workers, tiles, ring;
  size_t smem;
};
bool resident_plan(const mm_handle* h, int grid, ResidentPlan* p) {
  const int nth = h->g.ntheta, nl = (h->g.ns + 7) / 8, rpp = 32 / nl;
  const long long cells = (h->ncells + grid - 1) / grid;
  if (cells > 1 << 16 || h->rows > 0x7fffffffULL) return false;  // (column offsets are 32-bit)
  p->own = (int)((cells + mm::kResMaxWarps - 1) / mm::kResMaxWarps);
  p->workers = (int)((cells + p->own - 1) / p->own);
  const long long passes = ((long long)p->own * nth + rpp - 1) / rpp;
  const size_t fixed = mm::resident_smem(p->workers, p->own, nth, 0).total;
  if (fixed >= kResidentBudget) return false;
  const long long room = (long long)((kResidentBudget - fixed) / ((size_t)p->workers * 1024));
  p->ring = passes <= room ? 0 : mm::kResRing;
  p->tiles = (int)(passes <= room ? passes : room - p->ring);
  if (p->tiles < 0) return false;
  p->smem = mm::resident_smem(p->workers, p->own, nth, p->tiles + p->ring).total;
  return true;
}

// Whether the resident kernel is the faster one for n substeps of an instance it
// can hold.
bool resident_pays(const mm_handle* h, int n) {
  return h->mbn * h->tsz <= resident_limit(h->g.ntheta, h->g.ns, n);
}

// Kernel arguments of n substeps of h's live state. Nothing of h changes until the
// launch has been made (resident_advance).
mm::ResidentArgs resident_args(mm_handle* h, int grid, const ResidentPlan& p, int n) {
  mm::ResidentArgs a{};
  a.s = step_args<float>(h, h->parity);
  a.n = n;
  a.nl = (h->g.ns + 7) / 8;
  a.rpp = 32 / a.nl;
  a.vl = h->g.ns - 8 * (a.nl - 1);
  a.vw = h->g.ns % 4 == 0 ? 4 : h->g.ns % 2 == 0 ? 2 : 1;
  a.own = p.own;
  a.tiles = p.tiles;
  a.ring = p.ring;
  a.workers = p.workers;
  a.grid = grid;
  a.NL = h->res_NL;
  a.seg = 1;
  while (a.seg < 32 && a.seg < h->g.ntheta) a.seg <<= 1;
  a.epoch = h->res_epoch;
  a.arrivals = h->res_arrivals;
  a.xch = h->res_xch;
  return a;
}
// After the launch: the tags and arrivals of its substeps are used, and the state is
// theirs. (Taken before a launch that then fails, they would have every later one
// wait for arrivals that nothing makes.)
void resident_advance(mm_handle* h, int grid, int n) {
  h->res_epoch += (unsigned)n;
  h->res_arrivals += (unsigned)n * (unsigned)grid;
  h->parity ^= n & 1;
}

// Resident launches of one device, on whatever streams and from whatever threads
// they come, may run together as long as their blocks have an SM each: two of them
// part-way resident would wait for each other's blocks. The SMs are shared out as
// kSlots equal slots; a launch takes as many as its blocks need, the least recently
// used, and waits for the launches that had them last. (One after the other
// throughout, 16 handles of 16^2 x 16^2 on as many streams took 63 us a substep of all
// of them, one launch a substep 9.)
struct Slots {
  static constexpr int kSlots = 8;
  std::vector<cudaEvent_t> ev;  // of launches
  std::vector<int> uses;        // slots that hold each event
  int last[kSlots];             // event of the slot's last launch, -1: none
  unsigned long long used[kSlots] = {}, clock = 0;
  Slots() { std::fill(last, last + kSlots, -1); }
};
struct DeviceOrder {
  std::mutex m;
  std::map<int, Slots> dev;
};
DeviceOrder& device_order() {
  static DeviceOrder* d = new DeviceOrder();  // never destroyed: launches may outlive statics
  return *d;
}

}  // namespace

namespace {

mm_status launch_ordered(mm_handle* h, const void* f, int grid, int block, size_t smem,
                         void** args) {
  if (h->fail_launches > 0 && --h->fail_launches == 0)  // (tests: mm_debug_set)
    return cuda_fail(h, "resident launch", cudaErrorLaunchOutOfResources);
  DeviceOrder& o = device_order();
  std::lock_guard<std::mutex> lock(o.m);
  Slots& S = o.dev[h->device];
  const int per = std::max(1, h->sms / Slots::kSlots);
  const int need = std::min(Slots::kSlots, (grid + per - 1) / per);
  int order[Slots::kSlots];
  for (int q = 0; q < Slots::kSlots; ++q) order[q] = q;
  std::stable_sort(order, order + Slots::kSlots,
                   [&](int a, int b) { return S.used[a] < S.used[b]; });
  size_t e = 0;  // an event that no slot holds
  while (e < S.ev.size() && S.uses[e] > 0) ++e;
  if (e == S.ev.size()) {
    cudaEvent_t ev;
    CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    S.ev.push_back(ev);
    S.uses.push_back(0);
  }
  for (size_t w = 0; w < S.ev.size(); ++w)
    if (std::any_of(order, order + need, [&](int q) { return S.last[q] == (int)w; }))
      CK(cudaStreamWaitEvent(h->stream, S.ev[w], 0));
  CK(cudaLaunchCooperativeKernel(f, dim3((unsigned)grid), dim3((unsigned)block), args, smem,
                                 h->stream));
  CK(cudaEventRecord(S.ev[e], h->stream));
  ++S.clock;
  for (int q = 0; q < need; ++q) {
    const int s = order[q];
    if (S.last[s] >= 0) --S.uses[S.last[s]];
    S.last[s] = (int)e;
    S.used[s] = S.clock;
  }
  S.uses[e] = need;
  return MM_OK;
}

// Blocks of a small instance's longer calls (32 substeps and more): the fewest that
// leave a worker no more than a few passes, so that several instances run side by
// side. The chain between the substeps bounds those: 32^2 x 16^2 takes 3.8 us a
// substep on 35 blocks and on 152, 32^2 x 32^2 4.1 on 69 and 152, 24^2 x 32^2 4.1 on 39
// and 3.7. A launch's start and end take up to 4 us more on fewer SMs (shorter
// calls keep all of them), and beyond 32 orientations a substep 1.1 times as long.
constexpr int kSmallCalls = 32;
int resident_small_grid(const mm_handle* h, int most) {
  for (int g = 1; g < most && h->g.ntheta <= 32; ++g) {
    ResidentPlan p;
    if (resident_plan(h, g, &p) && p.ring == 0 && p.own <= 2 && p.tiles <= 4 &&
        p.workers * p.tiles <= 60)
      return g;
  }
  return most;
}

}  // namespace

// Off (h->res_grid = 0) in float64 and where no plan fits.
mm_status resident_configure(mm_handle* h) {
  h->res_grid = 0;
  if (h->prec != MM_FP32_MIXED) return MM_OK;
  int coop = 0;
  CK(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->device));
  if (!coop) return MM_OK;
  const int ns = h->g.ns, nl = (ns + 7) / 8;
  h->res_NL = ns % 8 == 0 && (nl == 2 || nl == 4 || nl == 8) ? nl : 0;
  const int grid = (int)std::min<long long>({h->sms, h->ncells, 32 * mm::kResXch});
  ResidentPlan p;
  if (!resident_pays(h, 3) || !resident_plan(h, grid, &p)) return MM_OK;
  const void* f = resident_kernel(h->res_NL);
  CK(mm::raise_smem_limit(f, kResidentBudget));
  int bps = 0;
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, f, 32 * (p.workers + 1), p.smem));
  if (bps < 1) return MM_OK;
  h->res_grid = grid;
  h->res_small = resident_small_grid(h, grid);
  return MM_OK;
}

// Whether n substeps of h go through the resident kernel: not without a plan
// that pays, for a single substep, with another substep kernel in effect, or on
// a stream being captured (the ordering event belongs to no capture).
static bool resident_applies(mm_handle* h, int n) {
  if (h->res_grid == 0 || n < 2 || h->anchors || h->capture || h->tangent || !resident_pays(h, n))
    return false;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(h->stream, &cs) == cudaSuccess &&
         cs == cudaStreamCaptureStatusNone;
}

// n substeps on the live state in one launch; *done = false (and nothing
// launched) where the resident kernel does not apply.
mm_status resident_substeps(mm_handle* h, int n, bool* done) {
  *done = false;
  if (!resident_applies(h, n)) return MM_OK;
  const int grid = n >= kSmallCalls ? h->res_small : h->res_grid;
  ResidentPlan p;
  if (!resident_plan(h, grid, &p)) return MM_OK;
  mm::ResidentArgs a = resident_args(h, grid, p, n);
  void* args[1] = {&a};
  const mm_status st = launch_ordered(h, resident_kernel(h->res_NL), grid, 32 * (p.workers + 1),
                                      p.smem, args);
  if (st != MM_OK) return st;
  resident_advance(h, grid, n);
  *done = true;
  return MM_OK;
}

// ---- groups of batch members

namespace {

// Relative work of one cell in a substep: a pass of rows and, for psi and the
// close, about 0.8 of one (half where two cells share a warp).
double cell_work(const mm_handle* h) {
  const int nth = h->g.ntheta, nl = (h->g.ns + 7) / 8;
  int seg = 1;
  while (seg < 32 && seg < nth) seg <<= 1;
  return nth * nl / 32.0 + 0.8 * (seg / 32.0) * ((nth + seg - 1) / seg);
}
double block_work(const mm_handle* h, int grid) {
  ResidentPlan p;
  if (!resident_plan(h, grid, &p)) return 1e30;
  return p.workers * p.own * cell_work(h);
}

}  // namespace

// Splits the members that the resident kernel holds into groups that run one
// after the other, each over all SMs: as many members as shared memory takes
// and as the L2 holds what is not kept there (about 110 MB of Mb), the largest
// first; within a group every member gets the fewest SMs it fits on and the
// others go to whichever has the most work per SM. in[i] = 1 for the members
// taken.
mm_status resident_group_plan(mm_handle* h, const std::vector<mm_handle*>& members,
                              std::vector<ResidentGroup>* groups, std::vector<char>* in) {
  constexpr size_t kGroupBytes = (size_t)110 << 20;
  groups->clear();
  in->assign(members.size(), 0);
  if (h->prec != MM_FP32_MIXED) return MM_OK;
  std::vector<int> order;
  for (size_t i = 0; i < members.size(); ++i)
    if (members[i]->res_grid > 0) order.push_back((int)i);
  std::stable_sort(order.begin(), order.end(),
                   [&](int a, int b) { return members[a]->mbn > members[b]->mbn; });
  struct Load {
    int sms = 0;
    size_t bytes = 0;
  };
  std::vector<Load> loads;
  for (int i : order) {
    const mm_handle* m = members[i];
    ResidentPlan p;
    int g = 1;
    while (g < m->res_grid && !resident_plan(m, g, &p)) ++g;
    if (!resident_plan(m, g, &p)) continue;
    const size_t bytes = m->mbn * m->tsz;
    size_t q = 0;
    while (q < groups->size() && (loads[q].sms + g > h->sms ||
                                  (loads[q].bytes > 0 && loads[q].bytes + bytes > kGroupBytes)))
      ++q;
    if (q == groups->size()) {
      groups->push_back({});
      loads.push_back({});
    }
    (*groups)[q].member.push_back(i);
    (*groups)[q].blocks.push_back(g);
    loads[q].sms += g;
    loads[q].bytes += bytes;
    (*in)[i] = 1;
  }
  for (size_t q = 0; q < groups->size(); ++q) {
    ResidentGroup& G = (*groups)[q];
    std::vector<double> work;
    for (size_t k = 0; k < G.member.size(); ++k)
      work.push_back(block_work(members[G.member[k]], G.blocks[k]));
    for (int left = h->sms - loads[q].sms; left > 0; --left) {
      int best = -1;
      for (size_t k = 0; k < work.size(); ++k)
        if (G.blocks[k] < members[G.member[k]]->res_grid && (best < 0 || work[k] > work[best]))
          best = (int)k;
      if (best < 0) break;
      ++G.blocks[best];
      work[best] = block_work(members[G.member[best]], G.blocks[best]);
    }
    G.grid = G.block = 0;
    G.smem = 0;
    std::vector<int2> map;
    for (size_t k = 0; k < G.member.size(); ++k) {
      ResidentPlan p;
      resident_plan(members[G.member[k]], G.blocks[k], &p);
      G.block = std::max(G.block, 32 * (p.workers + 1));
      G.smem = std::max(G.smem, p.smem);
      for (int b = 0; b < G.blocks[k]; ++b) map.push_back(make_int2((int)k, b));
    }
    G.grid = (int)map.size();
    CK(cudaMalloc(&G.map, map.size() * sizeof(int2)));
    CK(cudaMemcpy(G.map, map.data(), map.size() * sizeof(int2), cudaMemcpyHostToDevice));
    CK(cudaMalloc(&G.tab, G.member.size() * sizeof(mm::ResidentArgs)));
  }
  if (!groups->empty())
    CK(mm::raise_smem_limit((const void*)mm::k_substep_resident_group, kResidentBudget));
  return MM_OK;
}

void resident_group_free(std::vector<ResidentGroup>* groups) {
  for (ResidentGroup& G : *groups) {
    if (G.map) cudaFree(G.map);
    if (G.tab) cudaFree(G.tab);
  }
  groups->clear();
}

// n substeps of a group's members; their parities advance.
mm_status resident_group_step(mm_handle* h, const std::vector<mm_handle*>& members,
                              ResidentGroup& G, int n) {
  std::vector<mm::ResidentArgs> tab;
  for (size_t k = 0; k < G.member.size(); ++k) {
    mm_handle* m = members[G.member[k]];
    ResidentPlan p;
    resident_plan(m, G.blocks[k], &p);
    tab.push_back(resident_args(m, G.blocks[k], p, n));
  }
  // stream-ordered after the launch that read the table before; the pageable
  // source is staged before the call returns
  CK(cudaMemcpyAsync(G.tab, tab.data(), tab.size() * sizeof(mm::ResidentArgs),
                     cudaMemcpyHostToDevice, h->stream));
  const mm::ResidentArgs* dt = (const mm::ResidentArgs*)G.tab;
  const int2* dm = (const int2*)G.map;
  void* args[2] = {&dt, &dm};
  const mm_status st = launch_ordered(h, (const void*)mm::k_substep_resident_group, G.grid,
                                      G.block, G.smem, args);
  if (st != MM_OK) return st;
  for (size_t k = 0; k < G.member.size(); ++k)
    resident_advance(members[G.member[k]], G.blocks[k], n);
  return MM_OK;
}

// Whether n substeps of a batch may go through its groups: not a single one, not on
// a stream being captured, and, as for a handle, not two where the members together
// are more than the L2 holds (a group's rows are loaded and stored for them: 256 x
// 32^2 x 16^2, 268 MB, 283 us a substep against 260 over all tiles; 64 of them 63
// against 75).
bool resident_group_applies(mm_handle* h, const std::vector<mm_handle*>& members, int n) {
  if (n < 2) return false;
  size_t bytes = 0;
  for (const mm_handle* m : members) bytes += m->mbn * m->tsz;
  if (n == 2 && bytes > (size_t)125 << 20) return false;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(h->stream, &cs) == cudaSuccess &&
         cs == cudaStreamCaptureStatusNone;
}

}  // namespace mmh
