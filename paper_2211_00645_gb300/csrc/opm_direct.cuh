// Projection straight from the raw stack in global memory (Fig. 2d): every
// output (z-MIP, z-sum, first arg-max, y-MIP), uint16 or FP32, any width,
// alignment and geometry.  The one-plan kernel and the batched kernel share
// it.
//
// One warp owns a tile of kJ output columns j x kXW columns x and walks
// camera rows k; z-maxima, z-sums and arg-max rows stay in its registers.
// While it works on one row, the planes of its next row are on their way into
// the warp's own shared memory (cp.async, two rows, no other warp involved).
// Along a row it keeps the current plane pair (a, b - a) and steps to the
// next plane where the column's lower plane changes, so a raw value is
// converted once per plane.  The row's planes and weights are worked out by
// the lanes side by side, one column each.
//
// A CTA of kWarps warps covers kWarps / wr neighbouring tiles along j, with
// the rows of each dealt to wr warps in turn (rows ks + r, ks + r + wr, ...).
// wr grows where the tiles alone would leave the GPU idle; for z-sums it depends
// on the output grid only (row_groups), so that one plan always sums in one
// order.  The wr partial results meet in shared memory, where every warp joins a
// share of the columns in the order of r: sums are reproducible bit for bit.
// Rows' y-maxima meet in shared memory over the CTA's tiles and go to the y-MIP
// once per kRows rows.
//
// What bounds it: instruction issue (66 % of the schedulers' cycles, with two-
// and three-cycle packed FMAs, 3-input maxima and byte permutes among them);
// DRAM runs at 10-15 %.  8 columns x 4 x keep the accumulators, the plane pair
// and the walk's state in 128 registers, 16 warps per SM; 24 warps at 80
// registers spill and are slower, and so are 8 warps with all they ask for (all
// outputs of the live-view stack 550 us against 413-422 with the arg-max rows packed
// into half the registers).  Device time, us, against the kernels it replaced
// (one thread per output pixel for rows off 16 bytes, a TMA ring with one row per
// stage otherwise):
//   151 x 333 x 1001 uint16, 45 deg, step 0.2, pixel 0.115, z + y:  447 -> 74
//   200 x 512 x 2048 uint16, 35 deg, 0.3, 0.1, z + sum + y:         436 -> 332
//   the same with arg-max:                                          439 -> 413-422
//   50 x 87 x 1304 uint16, 30 deg, 0.4, 0.115, z + sum + y:          65 -> 22
//   100 x 256 x 512 FP32, 45 deg, 0.2, 0.115, z + y:                180 -> 37
//   100 x 256 x 512 uint16, 35 deg, step 0.05, pixel 0.1, z + y:     98 -> 29
// All outputs of FP32 stacks that fill the GPU are the one form that is slower
// (200 x 512 x 2048 433 -> 442, at 90 degrees 405 -> 425).
#pragma once

#include "opm_tma.cuh"

namespace opm {
namespace {
namespace direct {

constexpr int kJ = 8;            // columns j per warp
constexpr int kXL = 4;           // columns x per lane
constexpr int kXW = 32 * kXL;    // columns x per warp
constexpr int kWarps = 8;        // warps per CTA
constexpr int kCtaThreads = 32 * kWarps;
constexpr int kRows = 32;        // camera rows between two folds of the y-maxima
constexpr int kPart = kWarps * kJ * kXW;  // the warps' partial results, one value per column
// Shared memory: the CTA's y-maxima, the warps' weight tables ((w, w) pairs of
// two rows) and the warps' staged rows (two of `slots` planes).  After the last
// row, the warps' partial results (maxima, arg-max rows and sums) take its
// place.
constexpr int kYBytes = kRows * kXW * 4;
constexpr int kWBytes = kWarps * 2 * kJ * 8;
template <typename T>
__host__ __device__ constexpr int slot_bytes() { return kXW * (int)sizeof(T) + 16; }  // room for a shift
template <typename T>
__host__ __device__ constexpr int warp_bytes(int slots) { return 2 * slots * slot_bytes<T>(); }
template <typename T>
__host__ __device__ constexpr int smem_bytes(int slots, bool sum, bool arg) {
  const int rows = kYBytes + kWBytes + kWarps * warp_bytes<T>(slots), parts = (1 + sum + arg) * kPart * 4;
  return rows > parts ? rows : parts;
}
// Planes staged per row: those of kJ columns that step by rho <= 1 planes
// each (at most floor((kJ - 1) rho) + 1 steps; the 1e-3 allows for the rounding
// of planes next to a tie), or two for every column.
constexpr int kJumpSlots = 2 * kJ;
inline int row_slots(bool jump, double rho) { return jump ? kJumpSlots : (int)((kJ - 1) * rho + 1e-3) + 3; }
constexpr int kEnough = 16 * 152;       // warps that keep every SM busy

// Warps that share a tile's rows: the fewest of 2, 4, 8 that give `enough`
// warps over the output grid's tiles.  2 at least keeps a CTA within a 32-column
// tile.
inline int64_t grid_tiles(int64_t ny, int64_t nx) { return ((ny + kJ - 1) / kJ) * ((nx + kXW - 1) / kXW); }
inline int row_groups(int64_t tiles, int64_t enough = kEnough) {
  int wr = 2;
  while (wr < kWarps && tiles * wr < enough) wr *= 2;
  return wr;
}
// Columns j of one CTA, a divisor of kTileJ.
__host__ __device__ inline int cta_cols(int wr) { return kWarps / wr * kJ; }
static_assert(kWarps / 2 * kJ == kTileJ, "a CTA never spans two 32-column tiles");
static_assert(kXW == kX, "yidx covers a tile's columns x");

struct Job {
  const void* raw;             // sample (0, 0, 0)
  int slots;                   // staged planes per row
  size_t row_pitch, plane_pitch;  // elements
  const Split* A;              // [ny] column split table
  const Split* B;              // [nz] row split table
  Band band;                   // row band of the 32-column tile the job lies in
  int linear, nscan, ny, nz, nx;
  int wr;                      // row groups
  int jc, xb;                  // first output column j of the CTA, first x
  float* zmip;                 // [ny][nx] or NULL
  float* zsum;                 // [ny][nx] or NULL
  float* ymip;                 // [nz][nx] or NULL (pre-set, combined by atomic max)
  int32_t* argz;               // [ny][nx] or NULL
};

// BYTES from global to shared memory, asynchronously; only the first `have`
// are read, the rest is zero.
template <int BYTES>
__device__ __forceinline__ void copy_async(uint32_t dst, const void* src, int have) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(BYTES), "r"(have) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The aligned 16-byte chunks that hold a tile row's columns wherever it begins.
template <typename T>
__host__ __device__ constexpr int row_chunks() { return slot_bytes<T>() / 16; }

// Chunk c of the tile's columns of one camera row of one plane (p: the tile's
// first column; `in`: the plane lies inside the stack, else zeros) into its
// slot: the row's first column ends up p mod 16 bytes into it.  Bytes past
// the stack's ends are not touched, columns past the grid's edge hold
// whatever lies there.
template <typename T>
__device__ __forceinline__ void stage_chunk(uint32_t slot, const T* p, int c, bool in, const T* begin, const T* end) {
  const char* q = reinterpret_cast<const char*>((uintptr_t)p & ~(uintptr_t)15) + 16 * c;
  const uint32_t dst = slot + 16 * c;
  if (!in) {
    copy_async<16>(dst, reinterpret_cast<const void*>((uintptr_t)begin & ~(uintptr_t)15), 0);  // reads nothing
  } else if (q >= reinterpret_cast<const char*>(begin)) {
    const ptrdiff_t left = reinterpret_cast<const char*>(end) - q;
    if (left > 0) copy_async<16>(dst, q, left < 16 ? (int)left : 16);
  } else {  // the chunk the stack begins in
    for (int o = (int)(reinterpret_cast<const char*>(begin) - q); o < 16; o += (int)sizeof(T)) {
      const T* e = reinterpret_cast<const T*>(q + o);
      if (e >= end) break;
      if constexpr (sizeof(T) == 2)
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(dst + o), "h"(__ldg(e)) : "memory");
      else
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(dst + o), "f"(__ldg(e)) : "memory");
    }
  }
}

// `planes` planes from the one p lies in (plane n), one slot after another.
// VEC: every row starts on a vector of kXL elements, one copy per lane and
// plane.  Else chunk by chunk, the planes' chunks dealt to the lanes in turn.
template <typename T, bool VEC>
__device__ __forceinline__ void stage(uint32_t slot, const T* p, int n, int planes, int nscan, ptrdiff_t pp, int lim,
                                      int lane, const T* begin, const T* end) {
  if constexpr (VEC) {
    const int x = lane * kXL;
#pragma unroll 1
    for (int i = 0; i < planes; ++i, p += pp) {
      const bool in = (unsigned)(n + i) < (unsigned)nscan;
      if (x < lim)
        copy_async<kXL * sizeof(T)>(slot + i * slot_bytes<T>() + x * (int)sizeof(T), in ? p + x : begin,
                                    in ? kXL * (int)sizeof(T) : 0);
    }
  } else {
    constexpr int C = row_chunks<T>();
#pragma unroll 1
    for (int u = lane; u < planes * C; u += 32) {
      const int i = u / C;
      stage_chunk<T>(slot + i * slot_bytes<T>(), p + i * pp, u - i * C, (unsigned)(n + i) < (unsigned)nscan, begin, end);
    }
  }
}

// The lane's kXL values of a staged plane: neighbours (VEC), or columns 32
// apart.
template <typename T, bool VEC>
__device__ __forceinline__ void fetch(const unsigned char* slot, int shift, int lane, f2 (&v)[2]) {
  if constexpr (sizeof(T) == 4) {
    const float* f = reinterpret_cast<const float*>(slot);
    if constexpr (VEC) {
      const float4 q = reinterpret_cast<const float4*>(f)[lane];
      v[0] = pk(q.x, q.y);
      v[1] = pk(q.z, q.w);
    } else {
      f = reinterpret_cast<const float*>(slot + shift) + lane;
      v[0] = pk(f[0], f[32]);
      v[1] = pk(f[64], f[96]);
    }
  } else if constexpr (VEC) {
    const uint2 q = reinterpret_cast<const uint2*>(slot)[lane];
    v[0] = u16x2_to_f2(q.x);
    v[1] = u16x2_to_f2(q.y);
  } else {
    const uint16_t* u = reinterpret_cast<const uint16_t*>(slot + shift) + lane;
    const f2 m = pk(8388608.0f, 8388608.0f);
    v[0] = sub2(pk(__uint_as_float(u[0] | 0x4B000000u), __uint_as_float(u[32] | 0x4B000000u)), m);
    v[1] = sub2(pk(__uint_as_float(u[64] | 0x4B000000u), __uint_as_float(u[96] | 0x4B000000u)), m);
  }
}

__device__ __forceinline__ float half(f2 v, int i) {
  float lo, hi;
  upk(v, lo, hi);
  return i ? hi : lo;
}

// What a tile keeps of the arg-max: nothing, the row in 32 bits, or in 16 (two
// columns to a register: beside z-sums the registers that keep two CTAs on an
// SM; needs nz <= kMaxRow16).
enum Arg { kNoArg = 0, kArg32 = 1, kArg16 = 2 };
constexpr int kMaxRow16 = 65535;
inline Arg arg_form(bool arg, bool sum, int64_t nz) { return !arg ? kNoArg : sum && nz <= kMaxRow16 ? kArg16 : kArg32; }

// z = v and half HI of the packed rows = k where v > z.
template <bool HI>
__device__ __forceinline__ void max_row16(float& z, uint32_t& rows, float v, uint32_t k) {
  if constexpr (HI)
    asm("{ .reg .pred p; setp.gt.f32 p, %2, %0; @p mov.f32 %0, %2; @p prmt.b32 %1, %1, %3, 0x5410; }"
        : "+f"(z), "+r"(rows) : "f"(v), "r"(k));
  else
    asm("{ .reg .pred p; setp.gt.f32 p, %2, %0; @p mov.f32 %0, %2; @p prmt.b32 %1, %1, %3, 0x3254; }"
        : "+f"(z), "+r"(rows) : "f"(v), "r"(k));
}

// The job of one CTA; every thread of it takes part.  smem: smem_bytes<T>.
// JUMP: a tile's neighbouring columns may lie more than one plane apart
// (pixel > step, or a plan whose rounded plane table says so).  LEAN: the plane
// difference is worked out for every column instead of held.
template <typename T, bool VEC, bool SUM, int ARG, bool JUMP, bool LEAN = false>
__device__ __forceinline__ void tile(const Job& jb, unsigned char* smem_raw) {
  float* smem = reinterpret_cast<float*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wr = jb.wr, wj = kWarps / wr;
  const int r = warp / wj;                         // row group
  const int j0 = jb.jc + (warp % wj) * kJ;         // first column of the warp's tile
  const int cols = min(kJ, jb.ny - j0);            // <= 0: a tile past the grid
  const int xl = VEC ? lane * kXL : lane;          // the lane's first column x in the tile
  const int lim = jb.nx - jb.xb - xl;              // columns from there to the grid's edge
  const T* base = static_cast<const T*>(jb.raw) + jb.xb;
  const T* begin = static_cast<const T*>(jb.raw);
  const T* end = begin + (jb.nscan - 1) * jb.plane_pitch + (jb.nz - 1) * jb.row_pitch + jb.nx;
  const ptrdiff_t pp = (ptrdiff_t)jb.plane_pitch;
  const int pshift = VEC ? 0 : (int)(jb.plane_pitch * sizeof(T) & 15);  // shift from plane to plane
  constexpr bool kCounts = sizeof(T) == 2;         // uint16: every voxel is >= 0
  const float yzero = kCounts ? 0.0f : -INFINITY;  // what an empty y-maximum holds
  auto xof = [&](int c) { return VEC ? c : 32 * c; };  // of the lane's c-th column
  const Band bd = jb.band;

  float zmax[kJ][kXL];
  f2 zsum[SUM ? kJ : 1][kXL / 2];
  int az[ARG == kArg32 ? kJ : 1][kXL];
  uint32_t az16[ARG == kArg16 ? kJ : 1][kXL / 2];
  // rows before the band are zero: the maximum starts at 0, attained in row 0
  const float zinit = r == 0 && bd.lo > 0 ? 0.0f : -INFINITY;
#pragma unroll
  for (int j = 0; j < kJ; ++j)
#pragma unroll
    for (int c = 0; c < kXL; ++c) {
      zmax[j][c] = zinit;
      if constexpr (SUM) zsum[j][c / 2] = pk(0.0f, 0.0f);
      if constexpr (ARG == kArg32) az[j][c] = r == 0 ? 0 : INT32_MAX;
      if constexpr (ARG == kArg16) az16[j][c / 2] = r == 0 ? 0u : ~0u;
    }
  const bool meet = jb.ymip && wj > 1;  // y-maxima of several tiles meet in shared memory
  if (meet) {
    for (int i = threadIdx.x; i < kRows * kXW; i += kCtaThreads) smem[i] = yzero;
    __syncthreads();
  }

  // a row's planes and weights: lane l works out those of column j0 + l
  const Split aj = jb.A[min(j0 + min(lane, max(cols, 1) - 1), jb.ny - 1)];
  float2* wtab = reinterpret_cast<float2*>(smem_raw + kYBytes) + warp * 2 * kJ;
  unsigned char* slabs = smem_raw + kYBytes + kWBytes + warp * warp_bytes<T>(jb.slots);
  const int tlim = jb.nx - jb.xb;  // columns of the tile before the grid's edge
  int nl = 0, nf = 0;      // lower plane of the lane's column, of the first column
  unsigned step = 0;       // columns whose lower plane differs from the one before
  int shift = 0;           // where the row's first plane begins in its slot
  int buf = 0;             // which of the two rows was prepared last
  constexpr bool kRowAhead = !SUM || (JUMP && !ARG);  // elsewhere the sums leave no registers for it
  Split bk{};              // of the row to prepare next
  if constexpr (kRowAhead) bk = jb.B[min(bd.lo + r, jb.nz - 1)];
  auto prepare = [&](int k) {
    float w;
    if constexpr (kRowAhead) {
      plane_weight(aj, bk, jb.linear, nl, w);
      bk = jb.B[min(k + wr, jb.nz - 1)];
    } else {
      plane_weight(aj, jb.B[k], jb.linear, nl, w);
    }
    buf ^= 1;
    if (lane < kJ) wtab[buf * kJ + lane] = make_float2(w, w);
    const int np = __shfl_up_sync(0xffffffffu, nl, 1);
    step = __ballot_sync(0xffffffffu, lane < kJ && (lane == 0 || nl != np));
    nf = __shfl_sync(0xffffffffu, nl, 0);
    const T* row = base + (size_t)k * jb.row_pitch;
    const uint32_t slab = smem_u32(slabs + buf * jb.slots * slot_bytes<T>());
    if constexpr (JUMP) {  // two planes for every column that changes planes
      for (unsigned todo = step; todo; todo &= todo - 1) {
        const int j = __ffs(todo) - 1;
        const int n = __shfl_sync(0xffffffffu, nl, j);
        stage<T, VEC>(slab + 2 * j * slot_bytes<T>(), row + n * pp, n, 2, jb.nscan, pp, tlim, lane, begin, end);
      }
    } else {  // the planes of all columns, one after another
      const T* q = row + nf * pp;
      shift = VEC ? 0 : (int)((uintptr_t)q & 15);
      stage<T, VEC>(slab, q, nf, __popc(step) + 1, jb.nscan, pp, tlim, lane, begin, end);
    }
    copy_commit();
  };
  // the group's rows inside the band
  const int kend = cols > 0 ? bd.hi : bd.lo;
  int k = bd.lo + r;
  if (k < kend) prepare(k);

#pragma unroll 1
  for (int c0 = bd.lo; c0 < bd.hi; c0 += kRows) {
#pragma unroll 1
    for (; k < min(c0 + kRows, kend); k += wr) {
      const unsigned stepk = step;
      const float2* wk = wtab + buf * kJ;
      const unsigned char* const slot0 = slabs + buf * jb.slots * slot_bytes<T>();
      const unsigned char* slot = slot0;
      int sh = shift;
      const int nlk = nl;
      if (k + wr < kend) {
        prepare(k + wr);
        copy_wait<1>();
      } else {
        copy_wait<0>();
      }
      __syncwarp();
      auto shift_of = [&](int n) {  // JUMP: every plane has its own
        return VEC ? 0 : (int)((uintptr_t)(base + (size_t)k * jb.row_pitch + n * pp) & 15);
      };
      f2 a[2], b[2], d[2];
      if constexpr (JUMP) sh = shift_of(__shfl_sync(0xffffffffu, nlk, 0));
      fetch<T, VEC>(slot, sh, lane, a);
      sh = (sh + pshift) & 15;
      slot += slot_bytes<T>();
      fetch<T, VEC>(slot, sh, lane, b);
      d[0] = sub2(b[0], a[0]);
      d[1] = sub2(b[1], a[1]);
      float ym[kXL], vp[kXL];
#pragma unroll
      for (int c = 0; c < kXL; ++c) ym[c] = yzero;
      ulonglong2 wq;
#pragma unroll
      for (int j = 0; j < kJ; ++j) {
        if (j > 0 && (stepk & (1u << j))) {  // warp-uniform
          if constexpr (JUMP) {
            const unsigned char* sj = slot0 + 2 * j * slot_bytes<T>();
            sh = shift_of(__shfl_sync(0xffffffffu, nlk, j));
            fetch<T, VEC>(sj, sh, lane, a);
            fetch<T, VEC>(sj + slot_bytes<T>(), (sh + pshift) & 15, lane, b);
          } else {
            a[0] = b[0], a[1] = b[1];
            sh = (sh + pshift) & 15;
            slot += slot_bytes<T>();
            fetch<T, VEC>(slot, sh, lane, b);
          }
          d[0] = sub2(b[0], a[0]);
          d[1] = sub2(b[1], a[1]);
        }
        if (j % 2 == 0) wq = *reinterpret_cast<const ulonglong2*>(wk + j);
        f2 v2[2];
        float v[kXL];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          v2[h] = fma2(j % 2 ? wq.y : wq.x, LEAN ? sub2(b[h], a[h]) : d[h], a[h]);
          upk(v2[h], v[2 * h], v[2 * h + 1]);
          if constexpr (SUM) zsum[j][h] = add2(zsum[j][h], v2[h]);
        }
#pragma unroll
        for (int c = 0; c < kXL; ++c) {
          if constexpr (ARG == kArg32) {
            if (v[c] > zmax[j][c]) {
              zmax[j][c] = v[c];
              az[j][c] = k;
            }
          } else if constexpr (ARG == kArg16) {
            if (c % 2)
              max_row16<true>(zmax[j][c], az16[j][c / 2], v[c], k);
            else
              max_row16<false>(zmax[j][c], az16[j][c / 2], v[c], k);
          } else {
            zmax[j][c] = fmaxf(zmax[j][c], v[c]);
          }
          // columns past the grid repeat the last one's plane and weight
          if (j % 2 == 0)
            vp[c] = v[c];
          else
            ym[c] = max3(ym[c], vp[c], v[c]);
        }
      }
      if (jb.ymip && !meet) {
        float* y = jb.ymip + (size_t)k * jb.nx + jb.xb + xl;
#pragma unroll
        for (int c = 0; c < kXL; ++c)
          if (xof(c) < lim) {
            if constexpr (kCounts)
              atomicMax(reinterpret_cast<int*>(y + xof(c)), __float_as_int(ym[c]));
            else
              atomic_max_f(y + xof(c), ym[c]);
          }
      }
      if (meet) {
        float* yb = smem + (k - c0) * kXW;
#pragma unroll
        for (int c = 0; c < kXL; ++c) {
          float* y = yb + yidx(xl + xof(c));
          if constexpr (kCounts)
            atomicMax(reinterpret_cast<int*>(y), __float_as_int(ym[c]));
          else
            atomic_max_f(y, ym[c]);
        }
      }
      __syncwarp();  // the row's slots are read before they are staged again
    }
    if (meet) {
      __syncthreads();
      for (int i = threadIdx.x; i < kRows * kXW; i += kCtaThreads) {
        const int kk = c0 + i / kXW, x = jb.xb + i % kXW;
        float* yb = smem + (i / kXW) * kXW + yidx(i % kXW);
        const float y = *yb;
        *yb = yzero;
        if (y > yzero && kk < jb.nz && x < jb.nx) atomic_max_f(jb.ymip + (size_t)kk * jb.nx + x, y);
      }
      __syncthreads();
    }
  }

  if (!jb.zmip && !SUM && !ARG) return;
  // Every warp's partial results to shared memory; then every warp joins wj of
  // the CTA's columns, in the order of the row groups, and writes them.
  float* mine = smem + warp * kJ * kXW;
  auto put = [&](float* to, auto&& value) {
#pragma unroll
    for (int j = 0; j < kJ; ++j)
#pragma unroll
      for (int c = 0; c < kXL; ++c) to[j * kXW + 32 * c + lane] = value(j, c);
  };
  auto take = [&](const float* from, float (&v)[kXL]) {
#pragma unroll
    for (int c = 0; c < kXL; ++c) v[c] = from[32 * c + lane];
  };
  auto write = [&](float* to, const float (&v)[kXL]) {
    if constexpr (VEC) {
      if ((uintptr_t)to % 16 == 0) {
        if (lim > 0) *reinterpret_cast<float4*>(to + xl) = make_float4(v[0], v[1], v[2], v[3]);
        return;
      }
    }
#pragma unroll
    for (int c = 0; c < kXL; ++c)
      if (xof(c) < lim) to[xl + xof(c)] = v[c];
  };
  const int group = wj * kJ * kXW;  // from one row group's results to the next
  constexpr int kRowAt = kPart, kSumAt = (1 + (ARG != kNoArg)) * kPart;
  __syncthreads();
  put(mine, [&](int j, int c) { return zmax[j][c]; });
  if constexpr (ARG == kArg32) put(mine + kRowAt, [&](int j, int c) { return __int_as_float(az[j][c]); });
  if constexpr (ARG == kArg16)
    put(mine + kRowAt, [&](int j, int c) { return __uint_as_float(az16[j][c / 2] >> (c % 2 * 16) & 0xffffu); });
  if constexpr (SUM) put(mine + kSumAt, [&](int j, int c) { return half(zsum[j][c / 2], c % 2); });
  __syncthreads();
  constexpr int kJoin = SUM && !ARG ? 2 : 1;  // columns at a time (sums 336 -> 333 us on the live-view stack)
#pragma unroll kJoin
  for (int i = 0; i < wj; ++i) {
    const int col = warp * wj + i, j = jb.jc + col;
    if (j >= jb.ny) break;
    const float* q = smem + col * kXW;
    float z[kXL], row[kXL], sum[kXL];
    take(q, z);
    if constexpr (ARG) take(q + kRowAt, row);
    if constexpr (SUM) take(q + kSumAt, sum);
#pragma unroll 1
    for (int g = 1; g < wr; ++g) {
      q += group;
      float t[kXL], k[kXL], u[kXL];
      take(q, t);
      if constexpr (ARG) take(q + kRowAt, k);
      if constexpr (SUM) take(q + kSumAt, u);
#pragma unroll
      for (int c = 0; c < kXL; ++c) {
        if constexpr (ARG) {  // the larger value, or the earlier row of equal ones
          if (t[c] > z[c] || (t[c] == z[c] && __float_as_int(k[c]) < __float_as_int(row[c]))) z[c] = t[c], row[c] = k[c];
        } else {
          z[c] = fmaxf(z[c], t[c]);
        }
        if constexpr (SUM) sum[c] += u[c];
      }
    }
#pragma unroll
    for (int c = 0; c < kXL; ++c)
      if (bd.hi < jb.nz && z[c] < 0.0f) {  // rows after the band are zero too
        z[c] = 0.0f;
        if constexpr (ARG) row[c] = __int_as_float((int)bd.hi);
      }
    const size_t o = (size_t)j * jb.nx + jb.xb;
    if (jb.zmip) write(jb.zmip + o, z);
    if constexpr (ARG)
      if (jb.argz) write(reinterpret_cast<float*>(jb.argz) + o, row);
    if constexpr (SUM)
      if (jb.zsum) write(jb.zsum + o, sum);
  }
}

// Whether a stack's rows start on vectors of kXL elements.
template <typename T>
inline bool vec_rows(const void* raw, int64_t nx, int64_t row_pitch, int64_t plane_pitch) {
  return nx % kXL == 0 && row_pitch % kXL == 0 && plane_pitch % kXL == 0 && (uintptr_t)raw % (kXL * sizeof(T)) == 0;
}

}  // namespace direct
}  // namespace
}  // namespace opm
