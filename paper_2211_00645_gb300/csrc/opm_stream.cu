// Plane-by-plane live view: the projections of a stack accumulated one scan
// plane pair at a time, as the camera delivers frames (the rolling update of
// Fig. 4a).  The call for the pair (n, n + 1) evaluates exactly the voxels
// whose lower interpolation plane is n, V = (1 - w) R~[n] + w R~[n + 1], and
// folds them into the z-MIP, z-sum and y-MIP.  Every voxel has one lower
// plane, so the calls for n = -1 .. nscan - 1 cover the volume once; the
// per-voxel arithmetic (plane, weight, FMA on the plane difference) is the
// fast projection's, so the z-MIP and y-MIP end bit-identical to it.
//
// Both projections are gathered.  The lower plane falls along k and grows
// along j, so the rows of one column j that belong to pair n are one run
// (1 / (rho cos theta) rows, 3.7 on the live-view geometry, all of them at 90
// degrees), and so are the columns of one row k (1 / rho); each output value is
// written by one thread, once, with no atomics and nothing zeroed beforehand.
// A warp takes one column j (or row k) x 128 columns x and finds its run by 32
// candidates around the place the geometry gives; the 8 warps of a CTA take
// neighbours, whose runs share camera rows.  Where runs are long and columns few
// several warps share a column (column_share).  Consecutive pairs' runs adjoin,
// so the sliding view folds its complete pair and its mixed pair in one walk,
// together with the maxima it combines them with; columns outside both runs are
// passed through unsearched.
//
// What bounds it: the latency of search and walk, and issue (a push at 55 %; L2
// and DRAM at 18 %); the suffix pass runs at 82 % of DRAM.  Device time back to
// back, 512 x 2048 frames, 35 deg, step 0.3, pixel 0.1: a pair 7.2 us, with a z-sum
// 7.6; a push on 200 planes 13.1; 87 x 1304 frames: pair 3.2, push 4.8.  (A scatter
// of shared and global atomic maxima took 10 and 15; a push made of two of them, one
// zeroing and two elementwise maxima 31, and 15 on the small frames.)
// Four rows' loads ahead in a short run cost occupancy and were slower.
#include <algorithm>

#include "opm_tma.cuh"

namespace opm {

namespace {

constexpr int kSXL = 4;            // columns x per lane
constexpr int kSXW = 32 * kSXL;    // columns x per warp
constexpr int kSWarps = 8;         // warps per CTA: neighbouring columns j (or rows k), S warps to a column
__host__ __device__ constexpr int cta_warps(int S) { return S > kSWarps ? S : kSWarps; }
constexpr int kNoPair = -0x40000000;

__global__ void k_stream_zero(float* zmip, float* zsum, long long nj, float* ymip, long long nk) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nj; i += stride) {
    if (zmip) zmip[i] = 0.0f;
    if (zsum) zsum[i] = 0.0f;
  }
  if (ymip)
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nk; i += stride) ymip[i] = 0.0f;
}

// Plane pair n (frames lo = n and hi = n + 1; a frame outside the stack is
// NULL and reads as zero).
struct Pair {
  const uint16_t* lo;
  const uint16_t* hi;
  int n;  // kNoPair: none
};

// First index in [0, count) for which `reached` holds (it holds from there
// on), count if none.  Whole warp: 32 candidates around `guess` first, then
// 32 evenly spaced ones at a time.
template <typename Pred>
__device__ __forceinline__ int first_index(int count, int lane, float guess, const Pred& reached) {
  int lo = 0, hi = count;  // the answer lies in [lo, hi]
  const int i0 = max(0, (int)fminf(guess, (float)count) - 15);
  const unsigned b0 = __ballot_sync(0xffffffffu, i0 + lane >= count || reached(i0 + lane));
  const int f0 = b0 ? __ffs(b0) - 1 : 32;
  if (f0 == 32)
    lo = i0 + 32;
  else if (f0 > 0 || i0 == 0)
    return min(i0 + f0, count);
  else
    hi = min(i0, count);
  while (lo < hi) {
    const int st = (hi - lo + 31) >> 5;
    const int i = lo + lane * st;
    const unsigned b = __ballot_sync(0xffffffffu, i >= hi || reached(i));
    if (b == 0) {
      lo += 31 * st + 1;
    } else {
      const int f = __ffs(b) - 1;
      if (f == 0) return lo;
      hi = min(hi, lo + f * st);
      lo += (f - 1) * st + 1;
    }
  }
  return lo;
}

// First row k of column j whose lower plane is at most n, nz if none (it
// falls along k); rows = 1 / (rho cos theta).
__device__ __forceinline__ int first_row(const PlanView& v, float rows, const Split& aj, int n, int lane) {
  return first_index(v.nz, lane, ((float)(aj.i - n - 1) + aj.f) * rows, [&](int k) {
    const Split b = v.B[k];
    return aj.i - b.i - (aj.f - b.f < 0.0f) <= n;
  });
}

// This lane's kSXL counts of a camera row, two to a word: neighbours (VEC) or
// columns XS apart (zeros past the edge).
template <bool VEC, int XS = 32>
__device__ __forceinline__ uint2 load_words(const uint16_t* __restrict__ p, int lim) {
  if constexpr (VEC) {
    return __ldg(reinterpret_cast<const uint2*>(p));
  } else {
    uint2 w = make_uint2(0, 0);
    if (0 < lim) w.x = __ldg(p);
    if (XS < lim) w.x |= (uint32_t)__ldg(p + XS) << 16;
    if (2 * XS < lim) w.y = __ldg(p + 2 * XS);
    if (3 * XS < lim) w.y |= (uint32_t)__ldg(p + 3 * XS) << 16;
    return w;
  }
}

// The same as FP32 values, of element o of one frame; zeros for a missing frame.
template <bool VEC>
__device__ __forceinline__ void load_counts(const uint16_t* __restrict__ frame, size_t o, int lim, f2 (&out)[2]) {
  uint2 w = make_uint2(0, 0);
  if (frame) w = load_words<VEC>(frame + o, lim);
  out[0] = u16x2_to_f2(w.x);
  out[1] = u16x2_to_f2(w.y);
}

// Maxima (and sums of A's voxels) over one column's or row's voxels in pairs A
// and B.
struct Fold {
  float a[kSXL], b[kSXL], s[kSXL];
  bool any;  // A or B has a voxel here
};

__device__ __forceinline__ void fold_voxel(float w, const f2 (&lo)[2], const f2 (&hi)[2], float (&m)[kSXL],
                                           float (&v)[kSXL]) {
  const f2 w2 = pk(w, w);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    upk(fma2(w2, sub2(hi[h], lo[h]), lo[h]), v[2 * h], v[2 * h + 1]);  // the difference is exact
    m[2 * h] = fmaxf(m[2 * h], v[2 * h]);
    m[2 * h + 1] = fmaxf(m[2 * h + 1], v[2 * h + 1]);
  }
}

// Column j: its rows in pair B (nB = nA + 1, which come first) and pair A.
template <bool VEC, bool SUM>
__device__ __forceinline__ void fold_column(const PlanView& v, float rows, const Pair& A, const Pair& B, int j, int lane,
                                            int x0, int lim, Fold& f) {
  const Split aj = v.A[j];
  const int top = B.n != kNoPair ? B.n : A.n;
  for (int k = first_row(v, rows, aj, top, lane); k < v.nz; ++k) {
    int n0;
    float w;
    plane_weight(aj, v.B[k], v.linear, n0, w);
    if (n0 < A.n) break;
    f.any = true;
    const bool isB = n0 == B.n;
    const size_t o = (size_t)k * v.ncols + x0;
    f2 lo[2], hi[2];
    load_counts<VEC>(isB ? B.lo : A.lo, o, lim, lo);
    load_counts<VEC>(isB ? B.hi : A.hi, o, lim, hi);
    float val[kSXL];
    if (isB) {
      fold_voxel(w, lo, hi, f.b, val);
    } else {
      fold_voxel(w, lo, hi, f.a, val);
      if constexpr (SUM)
#pragma unroll
        for (int c = 0; c < kSXL; ++c) f.s[c] += val[c];
    }
  }
}

// The same for a run of many rows, shared by S warps of G row groups each (32 /
// G lanes to a row): row group g = G s + lane / (32 / G) takes rows g, g + S G,
// ... of the run, kAhead at a time.  Their loads overlap: which pair a row
// belongs to is searched for, not read with the row, and a missing frame is a
// mask, not a branch.  BOTH: pair B is given.  Afterwards the first 32 / G lanes
// of warp s = 0 hold the column's results, joined in the order of the groups.
// Every warp of the CTA takes part (live: it has a column).
template <bool VEC, bool SUM, bool BOTH, int S, int G>
__device__ __forceinline__ void fold_long_column(const PlanView& v, float per_plane, const Pair& A, const Pair& B,
                                                 int j, bool live, int x0, int lim, Fold& f) {
  constexpr int kAhead = 4, XS = 32 / G;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, s = warp % S;
  if (live) {
    const Split aj = v.A[j];
    const int k0 = first_row(v, per_plane, aj, BOTH ? B.n : A.n, lane);
    const int rows = first_row(v, per_plane, aj, A.n - 1, lane) - k0;
    const int rowsB = BOTH ? first_row(v, per_plane, aj, A.n, lane) - k0 : 0;
    f.any = rows > 0;
    const uint16_t* const alo = A.lo ? A.lo : A.hi;
    const uint16_t* const ahi = A.hi ? A.hi : A.lo;
    const uint32_t malo = A.lo ? ~0u : 0u, mahi = A.hi ? ~0u : 0u;
    const uint16_t* const blo = BOTH ? (B.lo ? B.lo : B.hi) : nullptr;
    const uint16_t* const bhi = BOTH ? (B.hi ? B.hi : B.lo) : nullptr;
    const uint32_t mblo = BOTH && B.lo ? ~0u : 0u, mbhi = BOTH && B.hi ? ~0u : 0u;
#pragma unroll 1
    for (int r = s * G; r < rows; r += kAhead * S * G) {
      uint2 lo[kAhead], hi[kAhead];
      Split bk[kAhead];
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int i = min(r + u * S * G + lane / XS, rows - 1);  // the last row again: maxima do not mind
        const bool isB = BOTH && i < rowsB;
        const size_t o = (size_t)(k0 + i) * v.ncols + x0;
        bk[u] = v.B[k0 + i];
        lo[u] = load_words<VEC, XS>((isB ? blo : alo) + o, lim);
        hi[u] = load_words<VEC, XS>((isB ? bhi : ahi) + o, lim);
      }
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int i = r + u * S * G + lane / XS;
        const bool isB = BOTH && min(i, rows - 1) < rowsB;
        const uint32_t ml = isB ? mblo : malo, mh = isB ? mbhi : mahi;
        const f2 l[2] = {u16x2_to_f2(lo[u].x & ml), u16x2_to_f2(lo[u].y & ml)};
        const f2 h[2] = {u16x2_to_f2(hi[u].x & mh), u16x2_to_f2(hi[u].y & mh)};
        int n0;
        float w, val[kSXL];
        plane_weight(aj, bk[u], v.linear, n0, w);
        if (isB) {
          fold_voxel(w, l, h, f.b, val);
        } else {
          fold_voxel(w, l, h, f.a, val);
          if constexpr (SUM)
            if (i < rows) {
#pragma unroll
              for (int c = 0; c < kSXL; ++c) f.s[c] += val[c];
            }
        }
      }
    }
#pragma unroll
    for (int d = XS; d < 32; d *= 2)
#pragma unroll
      for (int c = 0; c < kSXL; ++c) {
        f.a[c] = fmaxf(f.a[c], __shfl_xor_sync(0xffffffffu, f.a[c], d));
        if (BOTH) f.b[c] = fmaxf(f.b[c], __shfl_xor_sync(0xffffffffu, f.b[c], d));
        if (SUM) f.s[c] += __shfl_xor_sync(0xffffffffu, f.s[c], d);
      }
  }
  __shared__ float part[BOTH || SUM ? 2 : 1][cta_warps(S)][kSXW / G];
  if (s > 0 && lane < XS)
#pragma unroll
    for (int c = 0; c < kSXL; ++c) {
      part[0][warp][XS * c + lane] = f.a[c];
      if (BOTH || SUM) part[1][warp][XS * c + lane] = BOTH ? f.b[c] : f.s[c];
    }
  __syncthreads();
  if (s > 0 || lane >= XS) return;
#pragma unroll 1
  for (int q = 1; q < S; ++q)
#pragma unroll
    for (int c = 0; c < kSXL; ++c) {
      f.a[c] = fmaxf(f.a[c], part[0][warp + q][XS * c + lane]);
      if (BOTH) f.b[c] = fmaxf(f.b[c], part[1][warp + q][XS * c + lane]);
      if (SUM) f.s[c] += part[1][warp + q][XS * c + lane];
    }
}

// Row k: its columns in pair A (which come first) and pair B.
template <bool VEC>
__device__ __forceinline__ void fold_row(const PlanView& v, const Pair& A, const Pair& B, int k, int lane, int x0,
                                         int lim, Fold& f) {
  const Split b = v.B[k];
  const int top = B.n != kNoPair ? B.n : A.n;
  const float guess = (float)v.J0 + ((float)(A.n + b.i) + b.f - (v.linear ? 0.0f : 0.5f)) * v.rinv;
  const int first = first_index(v.ny, lane, guess, [&](int j) {
    const Split a = v.A[j];
    return a.i - b.i - (a.f - b.f < 0.0f) >= A.n;
  });
  const size_t o = (size_t)k * v.ncols + x0;
  f2 lo[2], hi[2];
  int held = kNoPair;
  for (int jb = first; jb < v.ny; jb += 32) {
    int nl;
    float wl;
    plane_weight(v.A[min(jb + lane, v.ny - 1)], b, v.linear, nl, wl);  // of 32 columns at once
    const int columns = __popc(__ballot_sync(0xffffffffu, jb + lane < v.ny && nl <= top));
    f.any |= columns > 0;
#pragma unroll 1
    for (int t = 0; t < columns; ++t) {
      const int n0 = __shfl_sync(0xffffffffu, nl, t);
      const float w = __shfl_sync(0xffffffffu, wl, t);
      const bool isB = n0 == B.n;
      if (n0 != held) {
        load_counts<VEC>(isB ? B.lo : A.lo, o, lim, lo);
        load_counts<VEC>(isB ? B.hi : A.hi, o, lim, hi);
        held = n0;
      }
      float val[kSXL];
      if (isB)
        fold_voxel(w, lo, hi, f.b, val);
      else
        fold_voxel(w, lo, hi, f.a, val);
    }
    if (columns < 32) break;
  }
}

template <bool VEC, int XS>
__device__ __forceinline__ void get(const float* p, int lim, float (&out)[kSXL]) {
  if constexpr (VEC) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    out[0] = q.x, out[1] = q.y, out[2] = q.z, out[3] = q.w;
  } else {
#pragma unroll
    for (int c = 0; c < kSXL; ++c) out[c] = XS * c < lim ? p[XS * c] : 0.0f;
  }
}
template <bool VEC, int XS>
__device__ __forceinline__ void put(float* p, int lim, const float (&v)[kSXL]) {
  if constexpr (VEC) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int c = 0; c < kSXL; ++c)
      if (XS * c < lim) p[XS * c] = v[c];
  }
}
__device__ __forceinline__ void max_into(float (&a)[kSXL], const float (&b)[kSXL]) {
#pragma unroll
  for (int c = 0; c < kSXL; ++c) a[c] = fmaxf(a[c], b[c]);
}

// Blocks of a launch, x-tiles fastest in each part: columns [j0, j1), which may
// hold voxels of the pairs, S warps to a column and kSXW / G columns x to a
// tile; the other columns (a push only) and the rows, one warp and kSXW columns
// x each.
struct Parts {
  int xtiles, xtiles_live;
  int j0, j1;
  unsigned live, idle;  // blocks of the first two parts
  float rows;           // rows of a column in one pair, 1 / (rho cos theta)
};

// What a warp works on: column j or row k, and its lane's columns x.
struct Place {
  bool ok;      // there is such a column or row
  int i;        // j or k
  int x0, lim;  // first column x of the lane, columns from there to the edge
};
template <bool VEC, int XS>
__device__ __forceinline__ Place place(const PlanView& v, bool ok, int i, int xt) {
  const int lane = (threadIdx.x & 31) % XS;
  Place p{ok, i, xt * XS * kSXL + (VEC ? lane * kSXL : lane), 0};
  p.lim = v.nx - p.x0;
  if (VEC && p.lim <= 0) p.x0 = 0;  // reads something, writes nothing
  return p;
}
template <bool VEC, int S, int G>
__device__ __forceinline__ Place live_column(const PlanView& v, const Parts& t) {
  constexpr int C = cta_warps(S) / S;
  const int g = blockIdx.x / t.xtiles_live, j = t.j0 + g * C + (int)(threadIdx.x >> 5) / S;
  return place<VEC, 32 / G>(v, j < t.j1, j, blockIdx.x - g * t.xtiles_live);
}
template <bool VEC, int S>
__device__ __forceinline__ Place idle_column(const PlanView& v, const Parts& t) {
  const unsigned b = blockIdx.x - t.live;
  const int g = b / t.xtiles, i = g * cta_warps(S) + (int)(threadIdx.x >> 5);
  const int j = i < t.j0 ? i : i + (t.j1 - t.j0);
  return place<VEC, 32>(v, j < v.ny, j, b - g * t.xtiles);
}
template <bool VEC, int S>
__device__ __forceinline__ Place some_row(const PlanView& v, const Parts& t) {
  const unsigned b = blockIdx.x - t.live - t.idle;
  const int g = b / t.xtiles, k = g * cta_warps(S) + (int)(threadIdx.x >> 5);
  return place<VEC, 32>(v, k < v.nz, k, b - g * t.xtiles);
}

// A column's voxels in the pairs; false for lanes that have nothing to write.
template <bool VEC, bool SUM, bool BOTH, int S, int G>
__device__ __forceinline__ bool fold_live(const PlanView& v, const Parts& t, const Pair& A, const Pair& B, const Place& p,
                                          Fold& f) {
  if constexpr (S == 1) {
    static_assert(G == 1, "one row at a time");
    if (p.ok) fold_column<VEC, SUM>(v, t.rows, A, B, p.i, threadIdx.x & 31, p.x0, p.lim, f);
    return p.ok && p.lim > 0;
  } else {
    fold_long_column<VEC, SUM, BOTH, S, G>(v, t.rows, A, B, p.i, p.ok, p.x0, p.lim, f);
    return p.ok && p.lim > 0 && (threadIdx.x >> 5) % S == 0 && (threadIdx.x & 31) < 32 / G;
  }
}

// Five CTAs per SM where a warp has a column (a push of 512 x 2048 frames 12.8 us
// at the 56 registers it would take, 11.6 at 48); where columns are shared 64
// registers, so that the rows and a push's idle columns beside them find room for
// enough warps.
template <int S>
constexpr int min_ctas() { return S == 1 ? 5 : 32 / cta_warps(S); }

// Pair A into the outputs (any of them NULL): columns [j0, j1) hold its voxels.
template <bool VEC, bool SUM, int S, int G>
__global__ void __launch_bounds__(32 * cta_warps(S), min_ctas<S>())
k_stream_pair(PlanView v, Pair A, Parts t, float* zmip, float* zsum, float* ymip) {
  const Pair none{nullptr, nullptr, kNoPair};
  Fold f{};
  float old[kSXL];
  if (blockIdx.x < t.live) {
    constexpr int XS = 32 / G;
    const Place p = live_column<VEC, S, G>(v, t);
    if (!fold_live<VEC, SUM, false, S, G>(v, t, A, none, p, f) || !f.any) return;
    const size_t o = (size_t)p.i * v.nx + p.x0;
    if (zmip) {
      get<VEC, XS>(zmip + o, p.lim, old);
      max_into(f.a, old);
      put<VEC, XS>(zmip + o, p.lim, f.a);
    }
    if constexpr (SUM) {
      get<VEC, XS>(zsum + o, p.lim, old);
#pragma unroll
      for (int c = 0; c < kSXL; ++c) old[c] += f.s[c];
      put<VEC, XS>(zsum + o, p.lim, old);
    }
  } else {
    const Place p = some_row<VEC, S>(v, t);
    if (!p.ok) return;
    fold_row<VEC>(v, A, none, p.i, threadIdx.x & 31, p.x0, p.lim, f);
    if (!f.any || p.lim <= 0) return;
    float* y = ymip + (size_t)p.i * v.nx + p.x0;
    get<VEC, 32>(y, p.lim, old);
    max_into(f.a, old);
    put<VEC, 32>(y, p.lim, f.a);
  }
}

// One push of the sliding view (launch_sliding_push): pair A is complete, B is
// the mixed pair, or the stack's last (`last`: complete as well).
//   run  = max(run, A[, B])   (fresh: without the old run)
//   slotA = A, slotB = B      (where given)
//   view = max(run, next, B)
struct Slide {
  float* run;
  float* slotA;
  float* slotB;
  const float* next;
  float* view;
  bool fresh, last;
};

template <bool VEC, int XS>
__device__ __forceinline__ void slide_load(const Slide& s, size_t o, int lim, float (&run)[kSXL], float (&next)[kSXL]) {
  if (!s.fresh) get<VEC, XS>(s.run + o, lim, run);
  if (s.next) get<VEC, XS>(s.next + o, lim, next);
}
template <bool VEC, int XS>
__device__ __forceinline__ void slide_store(const Slide& s, size_t o, int lim, const Fold& f, float (&run)[kSXL],
                                            const float (&next)[kSXL]) {
  if (s.slotA) put<VEC, XS>(s.slotA + o, lim, f.a);
  if (s.slotB) put<VEC, XS>(s.slotB + o, lim, f.b);
  max_into(run, f.a);
  if (s.last) max_into(run, f.b);
  if (f.any || s.fresh) put<VEC, XS>(s.run + o, lim, run);
  max_into(run, next);
  max_into(run, f.b);
  put<VEC, XS>(s.view + o, lim, run);
}

template <bool VEC, int S, int G>
__global__ void __launch_bounds__(32 * cta_warps(S), min_ctas<S>())
k_sliding_push(PlanView v, Pair A, Pair B, Slide s, Parts t) {
  float run[kSXL] = {}, next[kSXL] = {};
  Fold f{};
  if (blockIdx.x < t.live) {
    constexpr int XS = 32 / G;
    const Place p = live_column<VEC, S, G>(v, t);
    const size_t o = (size_t)p.i * v.nx + p.x0;
    if (S == 1 && p.ok && p.lim > 0) slide_load<VEC, XS>(s, o, p.lim, run, next);  // on their way during the search
    if (!fold_live<VEC, false, true, S, G>(v, t, A, B, p, f)) return;
    if (S > 1) slide_load<VEC, XS>(s, o, p.lim, run, next);
    slide_store<VEC, XS>(s, o, p.lim, f, run, next);
    return;
  }
  const bool row = blockIdx.x >= t.live + t.idle;
  const Place p = row ? some_row<VEC, S>(v, t) : idle_column<VEC, S>(v, t);
  if (!p.ok) return;
  const size_t o = (row ? (size_t)v.ny * v.nx : (size_t)0) + (size_t)p.i * v.nx + p.x0;
  if (p.lim > 0) slide_load<VEC, 32>(s, o, p.lim, run, next);
  if (row) fold_row<VEC>(v, A, B, p.i, threadIdx.x & 31, p.x0, p.lim, f);
  if (p.lim > 0) slide_store<VEC, 32>(s, o, p.lim, f, run, next);
}

// Suffix maxima of the slots: slot q = max(slot q, .., slot last), q = last - 1
// down to 1, one element (four when vec) per thread.
template <typename V>
__global__ void __launch_bounds__(256)
k_suffix_max(V* slots, size_t per, int last) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= per) return;
  V* p = slots + (size_t)last * per + i;
  V m = *p;
  // a few slots' loads in flight at a time
  constexpr int kAhead = 4;
  int q = last - 1;
  for (; q >= kAhead; q -= kAhead) {
    V t[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) t[u] = __ldcs(p - (size_t)(u + 1) * per);
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      p -= per;
      if constexpr (sizeof(V) == 16)
        m = make_float4(fmaxf(m.x, t[u].x), fmaxf(m.y, t[u].y), fmaxf(m.z, t[u].z), fmaxf(m.w, t[u].w));
      else
        m = fmaxf(m, t[u]);
      *p = m;
    }
  }
  for (; q >= 1; --q) {
    p -= per;
    const V t = *p;
    if constexpr (sizeof(V) == 16)
      m = make_float4(fmaxf(m.x, t.x), fmaxf(m.y, t.y), fmaxf(m.z, t.z), fmaxf(m.w, t.w));
    else
      m = fmaxf(m, t);
    *p = m;
  }
}

// out[i] = max(a[i], b[i]) over n FP32 values (out may alias a or b):
// the combine of the sliding view's partial projections.  Four values per
// thread when all three arrays are 16-byte aligned and n is a multiple of 4.
__global__ void __launch_bounds__(256)
k_max_combine(float* out, const float* a, const float* b, long long n, int vec) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (vec) {
    const long long n4 = n / 4;
    for (; i < n4; i += stride) {
      const float4 x = reinterpret_cast<const float4*>(a)[i];
      const float4 y = reinterpret_cast<const float4*>(b)[i];
      reinterpret_cast<float4*>(out)[i] =
          make_float4(fmaxf(x.x, y.x), fmaxf(x.y, y.y), fmaxf(x.z, y.z), fmaxf(x.w, y.w));
    }
  } else {
    for (; i < n; i += stride) out[i] = fmaxf(a[i], b[i]);
  }
}

}  // namespace

opm_status launch_stream_begin(const opm_plan* p, float* zmip, float* zsum, float* ymip, cudaStream_t s) {
  const PlanView& v = p->view;
  k_stream_zero<<<4 * 152, 256, 0, s>>>(zmip, zsum, (long long)v.ny * v.nx, ymip, (long long)v.nz * v.nx);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? OPM_OK : cuda_fail(e, "launch k_stream_zero");
}

// Vectors of kSXL when frames and outputs start every row on one.
static bool stream_vec(const PlanView& v, const void* f0, const void* f1, const void* f2) {
  return v.nx % kSXL == 0 && (uintptr_t)f0 % 8 == 0 && (uintptr_t)f1 % 8 == 0 && (uintptr_t)f2 % 8 == 0;
}
static bool vec_out(const void* p) { return (uintptr_t)p % 16 == 0; }

// A way to share a column: S warps of G row groups.
template <int S_, int G_>
struct Share {
  static constexpr int S = S_, G = G_;
};

// Rows of a column in one pair (all of them at 90 degrees).
static double run_rows(const opm_plan* p) { return std::min((double)p->nz, 1.0 / std::max(p->rho * p->c, 1e-12)); }

// Warps per column for runs of `run` rows; `warps`: columns x x-tiles, the warps
// that one to a column would make.  One serves while they fill the GPU or the
// runs are short; beyond that a run is walked by 4, 8 or 16 (x 4 row groups).
// The lines lie where both sides cost the same on frames of 87 to 2048 rows.
// us per pair (z + y) with 1 / 4 / 8 / 16 warps, and with the scatter before:
//   512 x 2048, step 0.3, pixel 0.1, 75 deg (run 12, warps 2160)  6.3 / 9.5 / - / -        9.8
//   ..., 85 deg (34, 768)                                       11.7 / 7.6 / 8.2 / 31      9.7
//   ..., 89 deg (172, 192)                                        48 / 7.1 / 7.0 / 12      9.6
//   ..., 90 deg (512, 48)                                        137 / 15 / 9.6 / 7.6      9.5
//   87 x 1304, step 0.4, pixel 0.115, 90 deg (87, 55)              25 / 5.0 / 4.1 / 4.3    5.3
//   1024 x 256, step 0.5, pixel 0.1, 90 deg (1024, 10)            275 / 27 / 15 / 6.0      5.6
// Rows off 8 bytes cost four times the loads, which sharing hides as well:
//   333 x 1001 with a z-sum, step 0.2, pixel 0.115, 75 deg (6.7, 704) 8.4 / 6.3 / - / 35   7.3
static int column_share(double run, long long warps, bool vec) {
  if (warps == 0) return 1;
  if (run >= 64.0 && (double)warps <= (vec ? 0.17 : 1.0) * run) return 16;
  if (run >= 64.0 && (double)warps <= 1.5 * run) return 8;
  return run * 1000.0 > (vec ? 12.0 : 5.0) * (double)warps ? 4 : 1;
}

// Calls go(Share) for the chosen one.
template <typename Go>
static void with_share(int S, const Go& go) {
  if (S == 1)
    go(Share<1, 1>{});
  else if (S == 4)
    go(Share<4, 1>{});
  else if (S == 8)
    go(Share<8, 1>{});
  else
    go(Share<16, 4>{});
}

// The blocks for columns [j0, j1), the others if `idle`, and all rows if `rows`;
// their number, or 0 when there are none or too many.
static unsigned stream_parts(const opm_plan* p, int S, int j0, int j1, bool idle, bool rows, Parts* t) {
  const PlanView& v = p->view;
  const auto up = [](long long a, long long b) { return (a + b - 1) / b; };
  const int G = S == 16 ? Share<16, 4>::G : 1, W = cta_warps(S);
  const long long xt = up(v.nx, kSXW), xl = up(v.nx, kSXW / G);
  const long long live = xl * up(j1 - j0, W / S), off = idle ? xt * up(v.ny - (j1 - j0), W) : 0;
  const long long all = live + off + (rows ? xt * up(v.nz, W) : 0);
  if (all > 0x7fffffffLL) return 0;
  *t = Parts{(int)xt, (int)xl, j0, j1, (unsigned)live, (unsigned)off, (float)run_rows(p)};
  return (unsigned)all;
}

// Columns with a voxel in the pairs n .. last: n0 grows with j and falls with k.
static void pair_columns(const opm_plan* p, int n, int last, int* j0, int* j1) {
  const auto lower = [](const Split& a, const Split& b) { return a.i - b.i - (a.f - b.f < 0.0f ? 1 : 0); };
  const auto first = [&](const Split& b, int least) {
    return (int)(std::partition_point(p->hA.begin(), p->hA.end(), [&](const Split& a) { return lower(a, b) < least; }) -
                 p->hA.begin());
  };
  *j0 = first(p->hB.front(), n);
  *j1 = std::max(*j0, first(p->hB.back(), last + 1));
}

opm_status launch_stream_pair(const opm_plan* p, const uint16_t* lo, const uint16_t* hi, int n, float* zmip,
                              float* zsum, float* ymip, cudaStream_t s) {
  const PlanView& v = p->view;
  if (v.nz > 65535) return fail(OPM_ERR_UNSUPPORTED, "more than 65535 camera rows");
  int j0 = 0, j1 = 0;
  if (zmip || zsum) pair_columns(p, n, n, &j0, &j1);
  if (j1 == j0 && !ymip) return OPM_OK;  // the pair has no voxel
  const bool vec = stream_vec(v, lo, hi, nullptr) && vec_out(zmip) && vec_out(zsum) && vec_out(ymip);
  const int share = column_share(run_rows(p), (j1 - j0) * (long long)((v.nx + kSXW - 1) / kSXW), vec);
  Parts t;
  const unsigned blocks = stream_parts(p, share, j0, j1, false, ymip != nullptr, &t);
  if (blocks == 0) return fail(OPM_ERR_UNSUPPORTED, "plane-pair grid exceeds launch limits");
  with_share(share, [&](auto sh) {
    constexpr int S = decltype(sh)::S, G = decltype(sh)::G;
    const auto kern = zsum ? (vec ? k_stream_pair<true, true, S, G> : k_stream_pair<false, true, S, G>)
                           : (vec ? k_stream_pair<true, false, S, G> : k_stream_pair<false, false, S, G>);
    kern<<<blocks, 32 * cta_warps(S), 0, s>>>(v, Pair{lo, hi, n}, t, zmip, zsum, ymip);
  });
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? OPM_OK : cuda_fail(e, "launch k_stream_pair");
}

}  // namespace opm

namespace opm {
namespace {

opm_status launch_max_combine(float* out, const float* a, const float* b, int64_t n, cudaStream_t s) {
  if (n == 0) return OPM_OK;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_fail(e, "device query (max combine)");
  const int vec = (n % 4 == 0) && ((uintptr_t)out % 16 == 0) && ((uintptr_t)a % 16 == 0) && ((uintptr_t)b % 16 == 0);
  const long long work = vec ? n / 4 : n;
  const long long blocks = std::min<long long>((work + 255) / 256, (long long)std::max(nsm, 1) * 8);
  k_max_combine<<<(unsigned)blocks, 256, 0, s>>>(out, a, b, (long long)n, vec);
  e = cudaGetLastError();
  return e == cudaSuccess ? OPM_OK : cuda_fail(e, "launch k_max_combine");
}

}  // namespace

// The sliding view after frame m of the current stack has been written to
// stack[m] (frames 0..m new, m+1..nscan-1 the previous stack's).  Each
// projection buffer is one z-MIP [ny][nx] followed by one y-MIP [nz][nx];
// `run` holds the maximum of the new stack's complete pairs, slot q of
// `slots` the previous stack's suffix maximum over its pairs q..nscan-1
// until the new stack's pair q replaces it.  The maximum is associative and
// exact, so `view` ends equal to the projection of the whole buffer.
opm_status launch_sliding_push(const opm_plan* p, const uint16_t* stack, int m, float* run, float* slots,
                               float* view, cudaStream_t s) {
  const PlanView& v = p->view;
  if (v.nz > 65535) return fail(OPM_ERR_UNSUPPORTED, "more than 65535 camera rows");
  const int N = v.nscan;
  const size_t per = ((size_t)v.ny + v.nz) * v.nx;
  const size_t frame = (size_t)v.nrows * v.ncols;
  auto F = [&](int n) { return n >= 0 && n < N ? stack + (size_t)n * frame : nullptr; };
  auto slot = [&](int q) { return slots + (size_t)q * per; };
  const bool last = m == N - 1;
  // the pair that frame m completes, and the one it opens (with the previous
  // stack's frame m + 1, or with nothing behind the last frame)
  const Pair A{F(m - 1), F(m), m - 1}, B{F(m), F(m + 1), m};
  Slide sl;
  sl.run = run;
  sl.slotA = m >= 2 ? slot(m - 1) : nullptr;  // pairs -1 and 0 are never read from a slot
  sl.slotB = last ? slot(m) : nullptr;
  sl.next = last ? nullptr : slot(m + 1);
  sl.view = view;
  sl.fresh = m == 0;
  sl.last = last;
  int j0, j1;
  pair_columns(p, A.n, B.n, &j0, &j1);
  const bool vec = stream_vec(v, A.lo, A.hi, B.hi) && per % kSXL == 0 && vec_out(run) && vec_out(slots) && vec_out(view);
  const int share = column_share(run_rows(p), (j1 - j0) * (long long)((v.nx + kSXW - 1) / kSXW), vec);
  Parts t;
  const unsigned blocks = stream_parts(p, share, j0, j1, true, true, &t);
  if (blocks == 0) return fail(OPM_ERR_UNSUPPORTED, "sliding-view grid exceeds launch limits");
  with_share(share, [&](auto sh) {
    constexpr int S = decltype(sh)::S, G = decltype(sh)::G;
    (vec ? k_sliding_push<true, S, G> : k_sliding_push<false, S, G>)<<<blocks, 32 * cta_warps(S), 0, s>>>(v, A, B, sl, t);
  });
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "launch k_sliding_push");
  if (last && N > 2) {  // the next stack's suffixes
    const size_t n = vec ? per / 4 : per;
    const size_t nb = (n + 255) / 256;
    if (nb > 0x7fffffffULL) return fail(OPM_ERR_UNSUPPORTED, "sliding-view grid exceeds launch limits");
    if (vec)
      k_suffix_max<<<(unsigned)nb, 256, 0, s>>>(reinterpret_cast<float4*>(slots), n, N - 1);
    else
      k_suffix_max<<<(unsigned)nb, 256, 0, s>>>(slots, n, N - 1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "launch k_suffix_max");
  }
  return OPM_OK;
}

}  // namespace opm

using namespace opm;

extern "C" opm_status opm_max_combine(float* out, const float* a, const float* b, int64_t n, void* stream) {
  if (!out || !a || !b) return fail(OPM_ERR_INVALID_ARG, "out, a and b must be non-NULL");
  if (n < 0) return fail(OPM_ERR_INVALID_ARG, "n must be >= 0");
  return launch_max_combine(out, a, b, n, static_cast<cudaStream_t>(stream));
}
