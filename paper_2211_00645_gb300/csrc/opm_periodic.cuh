// Live view for plans whose plane coordinate advances by a rational p/q
// planes per output column (pixel/step = p/q, p <= q): the periodic path.
//
// Along one camera row, the lower interpolation plane of column j is
// floor((j - J0) p/q - beta_k).  Relative to the first column of a 32-column
// tile it is floor((t p + ph) / q), t = 0..31, for one phase ph in [0, q):
// a tile row steps through its staged planes in one of only q patterns (the
// plan checks every tile and row with the kernels' own IEEE arithmetic and
// records the phase).  Each pattern is compiled into straight-line code:
// the planes a row needs are loaded and converted once, each column's plane
// pair is a fixed register, and a column costs one packed FMA per row, one
// 3-input max per voxel pair into the z-max and, for the y-max, only the
// first and last column of each plane interval (along a row the voxels of
// one interval are a + w (b - a) with w increasing in j, and a correctly
// rounded FMA is monotone in w; the plan checks that the weights increase
// inside every interval).  Where pixel / step is p/q up to rounding every q-th
// column has the same weight, bit for bit (the plan builds its tables from the
// exact ratio), and a row's q weights stay in registers (REP); other plans that
// step alike read every column's (131 us against 129 below).  The arithmetic is
// that of every other kernel of the library (the plan's weights, FMA on the exact
// plane difference), so the outputs are the same bit for bit.
//
// The two rows of a stage have the same phase: the plan pairs every tile's
// rows by phase (RowPair), and a unit is a run of such pairs.  That leaves q
// bodies of code instead of q^2, 18 KB for q = 3.  Straight-line code starves
// the schedulers once the bodies in use outgrow the instruction caches (a
// probe of independent maxima: three bodies of 4 KB run at full rate, six at a
// quarter to two thirds of it), and with rows paired in order six of nine 6 KB
// bodies were in use.  What bounds it now is dispatch: packed FMAs, adds and
// 3-input maxima take two to three cycles each, and more warps do not help (5
// CTAs per SM were slower).  Device time, us, rows in order with a weight pair per
// column -> this: 200 x 512 x 2048 (35 deg, step 0.3, pixel 0.1) 142 -> 129, 1024 of
// its columns 79 -> 73, 256 columns 32 -> 30; step 0.2 (1/2) 151 -> 150, 80 -> 78,
// 25 -> 24.
//
// CTA: one producer warp (TMA ring of two camera rows per stage, as in
// opm_tma.cuh) and two compute warps.  Each compute warp owns all 32 columns
// j of the tile for 64 columns x (2 per lane), so a row's y-max over the tile
// is complete in one lane and goes to the global y-MIP with one atomic max;
// the compute warps never wait for each other, only for staged slabs.
#pragma once

#include "opm_tma.cuh"

namespace opm {
namespace {

namespace per {

constexpr int kXL = 2;                  // columns x per lane
constexpr int kXW = 32 * kXL;           // columns x per compute warp
constexpr int kXH = kX / kXW;           // x-halves of the 128-column x-tile
constexpr int kMaxCW = 4;               // compute warps per CTA at most

// A compute warp owns a run of RUN columns j (16 or 32) for kXW columns x.
template <int RUN>
struct Cfg {
  static_assert(RUN == 16 || RUN == 32, "runs of 16 or 32 columns");
  static constexpr int kRuns = kTileJ / RUN;       // column runs per tile
  static constexpr int kCW = kRuns * kXH;          // compute warps per CTA
  static constexpr int kThreads = 32 * (kCW + 1);
};

// Shared memory for S stages of slab depth P.
__host__ __device__ inline size_t off_tab(int S, int P) { return S * fast::stage_slab_bytes(P); }  // FastRow [S][2]
__host__ __device__ inline size_t off_bar(int S, int P) { return off_tab(S, P) + S * 2 * sizeof(FastRow); }
__host__ __device__ inline size_t off_jobs(int S, int P) { return off_bar(S, P) + 2 * S * 8; }  // JobP [kMaxCW]
__host__ __device__ inline size_t off_rows(int S, int P) { return off_jobs(S, P) + kMaxCW * 48; }  // int2 [S]: camera rows
__host__ __device__ inline size_t total(int S, int P) { return off_rows(S, P) + S * 8; }

struct JobP {  // a compute warp's job fields, parked in shared memory
  float* zmip;
  float* ymip;
  int nx, j0, xbase;
  int gend;  // stage count at the end of the job
  int pad[4];
};
static_assert(sizeof(JobP) == 48, "JobP layout");

// Plane of column t of a tile row, relative to the tile's first column, for
// pixel/step = p/q at phase ph.
__host__ __device__ constexpr int pofs(int p, int q, int ph, int t) { return per_ofs(p, q, ph, t); }
// Column t is the first or the last of its plane interval within a run of
// `run` columns.
__host__ __device__ constexpr bool pcand(int p, int q, int ph, int t, int run) {
  return t == 0 || t == run - 1 || pofs(p, q, ph, t) != pofs(p, q, ph, t - 1) ||
         pofs(p, q, ph, t + 1) != pofs(p, q, ph, t);
}
// Number of y-max candidates before column t.
__host__ __device__ constexpr int pcount(int p, int q, int ph, int t, int run) {
  int n = 0;
  for (int i = 0; i < t; ++i) n += pcand(p, q, ph, i, run) ? 1 : 0;
  return n;
}

}  // namespace per

// The ring in shared memory: S stages for slab depth Pl.
struct PerRing {
  unsigned char* base;
  int S, Pl;
  __device__ __forceinline__ FastRow* tab() const { return reinterpret_cast<FastRow*>(base + per::off_tab(S, Pl)); }
  // producer -> consumers: slabs and tables of a stage landed
  __device__ __forceinline__ uint64_t* full() const {
    return reinterpret_cast<uint64_t*>(base + per::off_bar(S, Pl));
  }
  // consumers -> producer: slot read by every compute warp
  __device__ __forceinline__ uint64_t* sfree() const { return full() + S; }
  __device__ __forceinline__ per::JobP* jobs() const {
    return reinterpret_cast<per::JobP*>(base + per::off_jobs(S, Pl));
  }
  // camera rows of each stage
  __device__ __forceinline__ int2* rows() const { return reinterpret_cast<int2*>(base + per::off_rows(S, Pl)); }
};

__device__ __forceinline__ PerRing per_ring(unsigned char* smem, int S, int Pl) {
  PerRing r;
  r.base = smem;
  r.S = S;
  r.Pl = Pl;
  return r;
}

// Whole CTA: barrier init, then a CTA barrier.
__device__ __forceinline__ void per_ring_init(const PerRing& r, int ncw) {
  if (threadIdx.x == 0) {
    for (int s = 0; s < r.S; ++s) {
      mbar_init(&r.full()[s], 1);
      mbar_init(&r.sfree()[s], ncw);
    }
    fence_barrier_init();
  }
  __syncthreads();
}

// Producer warp: stage the job's row pairs once the slot is free.  `g` is the
// CTA's running stage count, advanced by the job's stage count.
__device__ __forceinline__ bool per_produce(const FastJob& jb, const PerRing& r, int& g, unsigned* err, int lane) {
  const uint32_t pitch = kX * 2;
  const int S = r.S;
  const RowPair* pairs = jb.pairs + jb.ks / 2;
  const int nst = (jb.ke - jb.ks) / 2;
  RowPair cur = pairs[min(lane, nst - 1)];  // 32 pairs per load, one group ahead
  RowPair next = pairs[min(32 + lane, nst - 1)];
#pragma unroll 1
  for (int it = 0; it < nst; ++it, ++g) {
    const int s = g % S;
    if (g >= S && !mbar_wait(&r.sfree()[s], ((g - S) / S) & 1, err)) return false;
    if (it > 0 && it % 32 == 0) {
      cur = next;
      next = pairs[min(it + 32 + lane, nst - 1)];
    }
    const int k0 = __shfl_sync(0xffffffffu, cur.k0, it % 32), k1 = __shfl_sync(0xffffffffu, cur.k1, it % 32);
    const int n0 = __shfl_sync(0xffffffffu, cur.n0, it % 32), n1 = __shfl_sync(0xffffffffu, cur.n1, it % 32);
    if (lane == 0) {
      unsigned char* slab = r.base + s * fast::stage_slab_bytes(r.Pl);
      r.rows()[s] = make_int2(k0, k1);
      mbar_arrive_tx(&r.full()[s], (unsigned)(2 * jb.P * pitch + 2 * sizeof(FastRow)));
      tma_load_3d(slab, jb.tmap, &r.full()[s], jb.xbase, k0, n0);
      tma_load_3d(slab + fast::slab_row_bytes(r.Pl), jb.tmap, &r.full()[s], jb.xbase, k1, n1);
      bulk_load(&r.tab()[s * 2 + 0], jb.rows + k0, sizeof(FastRow), &r.full()[s]);
      bulk_load(&r.tab()[s * 2 + 1], jb.rows + k1, sizeof(FastRow), &r.full()[s]);
    }
    __syncwarp();
  }
  return true;
}

// Producer warp, after its last job: the CTA's shared memory must outlive
// every copy it issued (bounded wait on the last S stages).
__device__ __forceinline__ void per_drain(const PerRing& r, int g, bool ok, unsigned* err) {
  for (int q = max(0, g - r.S); q < g; ++q)
    if (!mbar_wait(&r.full()[q % r.S], (q / r.S) & 1, err, ok ? kWaitLimitNs : 50000000ull)) break;
}

// Two uint16 counts of a staged plane (this lane's 2 columns x) as FP32x2.
__device__ __forceinline__ f2 lds_x2(const unsigned char* smem, uint32_t off) {
  return u16x2_to_f2(*reinterpret_cast<const uint32_t*>(smem + off));
}

// Both camera rows of a stage for one compute warp: a run of RUN columns, both
// rows at phase PH.  off0 / off1: shared-memory offset of this lane's 2
// columns x in the tile's first plane of each row; wof0 / wof1: the run's (w,
// w) weight pairs of each row, of which the first Qq repeat (REP) or not.
template <int RUN, int Pp, int Qq, bool YMIP, bool REP, int PH>
__device__ __forceinline__ void per_pair(const unsigned char* __restrict__ smem, uint32_t off0, uint32_t off1,
                                         uint32_t wof0, uint32_t wof1, float (&zmax)[RUN][per::kXL],
                                         float (&ym0)[per::kXL], float (&ym1)[per::kXL]) {
  using namespace per;
  constexpr uint32_t pitch = kX * 2;
  f2 a0 = lds_x2(smem, off0), b0 = lds_x2(smem, off0 + pitch);
  f2 a1 = lds_x2(smem, off1), b1 = lds_x2(smem, off1 + pitch);
  f2 d0 = sub2(b0, a0), d1 = sub2(b1, a1);
  float p0[kXL], p1[kXL];
  constexpr int kW = REP ? Qq : 2;  // weights held per row: the run's, or two columns'
  f2 w0[kW], w1[kW];
  if constexpr (REP) {
#pragma unroll
    for (int t = 0; t < Qq; ++t) {
      w0[t] = *reinterpret_cast<const f2*>(smem + wof0 + 8 * t);
      w1[t] = *reinterpret_cast<const f2*>(smem + wof1 + 8 * t);
    }
  }
#pragma unroll
  for (int t = 0; t < RUN; ++t) {
    // next plane of the rows: integers below 2^24, so the new lower plane is
    // exactly the old upper one
    if (t > 0 && pofs(Pp, Qq, PH, t) != pofs(Pp, Qq, PH, t - 1)) {
      a0 = b0;
      a1 = b1;
      b0 = lds_x2(smem, off0 + (uint32_t)(pofs(Pp, Qq, PH, t) + 1) * pitch);
      b1 = lds_x2(smem, off1 + (uint32_t)(pofs(Pp, Qq, PH, t) + 1) * pitch);
      d0 = sub2(b0, a0);
      d1 = sub2(b1, a1);
    }
    if (!REP && t % 2 == 0) {
      const ulonglong2 q0 = *reinterpret_cast<const ulonglong2*>(smem + wof0 + 8 * t);
      const ulonglong2 q1 = *reinterpret_cast<const ulonglong2*>(smem + wof1 + 8 * t);
      w0[0] = q0.x, w0[1] = q0.y, w1[0] = q1.x, w1[1] = q1.y;
    }
    float v0[kXL], v1[kXL];
    upk(fma2(w0[t % kW], d0, a0), v0[0], v0[1]);
    upk(fma2(w1[t % kW], d1, a1), v1[0], v1[1]);
#pragma unroll
    for (int c = 0; c < kXL; ++c) zmax[t][c] = max3(zmax[t][c], v0[c], v1[c]);
    if (YMIP && pcand(Pp, Qq, PH, t, RUN)) {
      if (pcount(Pp, Qq, PH, t, RUN) % 2 == 0) {
#pragma unroll
        for (int c = 0; c < kXL; ++c) p0[c] = v0[c], p1[c] = v1[c];
      } else {
#pragma unroll
        for (int c = 0; c < kXL; ++c) {
          ym0[c] = max3(ym0[c], p0[c], v0[c]);
          ym1[c] = max3(ym1[c], p1[c], v1[c]);
        }
      }
    }
  }
  if (YMIP && pcount(Pp, Qq, PH, RUN, RUN) % 2 == 1) {
#pragma unroll
    for (int c = 0; c < kXL; ++c) {
      ym0[c] = fmaxf(ym0[c], p0[c]);
      ym1[c] = fmaxf(ym1[c], p1[c]);
    }
  }
}

// Phase ph in [LO, HI), by a balanced branch tree.
template <int RUN, int Pp, int Qq, bool YMIP, bool REP, int LO, int HI>
__device__ __forceinline__ void per_tree(int ph, const unsigned char* __restrict__ smem, uint32_t off0, uint32_t off1,
                                         uint32_t wof0, uint32_t wof1, float (&zmax)[RUN][per::kXL],
                                         float (&ym0)[per::kXL], float (&ym1)[per::kXL]) {
  if constexpr (HI - LO == 1) {
    per_pair<RUN, Pp, Qq, YMIP, REP, LO>(smem, off0, off1, wof0, wof1, zmax, ym0, ym1);
  } else {
    constexpr int MID = (LO + HI) / 2;
    if (ph < MID)
      per_tree<RUN, Pp, Qq, YMIP, REP, LO, MID>(ph, smem, off0, off1, wof0, wof1, zmax, ym0, ym1);
    else
      per_tree<RUN, Pp, Qq, YMIP, REP, MID, HI>(ph, smem, off0, off1, wof0, wof1, zmax, ym0, ym1);
  }
}

// The phase of each 8-column chunk (its first column's position within the
// period) is kept in bits 16..23 of its step word; a run's is that of its
// first chunk.
constexpr int kPhaseShift = 16;

// Compute warp i: run h = i % kRuns of the job's tile (columns
// j0 + RUN h .. + RUN - 1) for columns x xbase + 64 (i / kRuns) .. + 63,
// both rows of every stage.  z-maxima stay in registers and are folded into
// zmip at the end of the job; each row's y-max over the run goes to ymip
// right away.  Returns false when a bounded wait gave up.
template <int RUN, int Pp, int Qq, bool YMIP, bool REP>
__device__ __forceinline__ bool per_consume(const FastJob& jb, const PerRing& r, int& g, unsigned* err, int i,
                                            int lane) {
  using namespace per;
  constexpr int kRuns = Cfg<RUN>::kRuns;
  const int h = i % kRuns, xh = i / kRuns;
  const uint32_t pitch = kX * 2;
  const int S = r.S;
  const unsigned char* smem = r.base;
  JobP* js = r.jobs() + i;
  if (lane == 0) {
    js->zmip = jb.zmip;
    js->ymip = jb.ymip;
    js->nx = jb.nx;
    js->j0 = jb.j0;
    js->xbase = jb.xbase;
    js->gend = g + (jb.ke - jb.ks) / 2;
  }
  __syncwarp();
  float zmax[RUN][kXL];
#pragma unroll
  for (int t = 0; t < RUN; ++t)
#pragma unroll
    for (int c = 0; c < kXL; ++c) zmax[t][c] = 0.0f;  // uint16 voxels are >= 0
  bool ok = true;
  const uint32_t xoff = (uint32_t)(xh * kXW + lane * kXL) * 2;  // this lane's bytes within a staged plane

#pragma unroll 1
  for (; g < lds_volatile_s32(&js->gend); ++g) {
    const int s = g % S;
    if (!mbar_wait(&r.full()[s], (g / S) & 1, err)) {
      ok = false;
      break;
    }
    const uint32_t tab0 = (uint32_t)(per::off_tab(S, r.Pl) + (size_t)(s * 2) * sizeof(FastRow));
    const uint32_t rec = (uint32_t)(offsetof(FastRow, rec) + (h * RUN / 8) * sizeof(FastRec));
    const uint2 rr0 = *reinterpret_cast<const uint2*>(smem + tab0 + rec);
    const uint2 rr1 = *reinterpret_cast<const uint2*>(smem + tab0 + (uint32_t)sizeof(FastRow) + rec);
    const int2 rows = r.rows()[s];
    const uint32_t row0 = (uint32_t)(s * fast::stage_slab_bytes(r.Pl)) + xoff;
    const uint32_t row1 = row0 + (uint32_t)fast::slab_row_bytes(r.Pl);
    float ym0[kXL], ym1[kXL];
#pragma unroll
    for (int c = 0; c < kXL; ++c) ym0[c] = ym1[c] = 0.0f;
    const uint32_t wof0 = tab0 + (uint32_t)(h * RUN * 8);
    per_tree<RUN, Pp, Qq, YMIP, REP, 0, Qq>((int)((rr0.x >> kPhaseShift) & 255u), smem, row0 + rr0.y * pitch,
                                            row1 + rr1.y * pitch, wof0, wof0 + (uint32_t)sizeof(FastRow), zmax, ym0,
                                            ym1);
    __syncwarp();
    if (lane == 0) mbar_arrive(&r.sfree()[s]);
    if constexpr (!YMIP) continue;
    float* ymip = lds_volatile_ptr(&js->ymip);
    if (ymip) {
      const int nx = lds_volatile_s32(&js->nx);
      const int x = lds_volatile_s32(&js->xbase) + xh * kXW + lane * kXL;
#pragma unroll
      for (int c = 0; c < kXL; ++c) {
        if (x + c < nx) {
          atomicMax(reinterpret_cast<int*>(ymip + (size_t)rows.x * nx + x + c), __float_as_int(ym0[c]));
          atomicMax(reinterpret_cast<int*>(ymip + (size_t)rows.y * nx + x + c), __float_as_int(ym1[c]));
        }
      }
    }
  }

  float* zmip = lds_volatile_ptr(&js->zmip);
  if (zmip) {
    const int nx = lds_volatile_s32(&js->nx);
    const int x = lds_volatile_s32(&js->xbase) + xh * kXW + lane * kXL;
    const int j0 = lds_volatile_s32(&js->j0) + h * RUN;
#pragma unroll
    for (int t = 0; t < RUN; ++t) {
      float* row = zmip + (size_t)(j0 + t) * nx;
#pragma unroll
      for (int c = 0; c < kXL; ++c)
        if (x + c < nx) atomicMax(reinterpret_cast<int*>(row + x + c), __float_as_int(zmax[t][c]));
    }
  }
  return ok;
}

}  // namespace
}  // namespace opm
