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
// (1 / (rho cos theta) rows, 3.7 on the live-view geometry), and so are the
// columns of one row k (1 / rho); each output value is written by one thread,
// once, with no atomics and nothing zeroed beforehand.  A warp takes one
// column j (or row k) x 128 columns x and finds its run with a 32-way search
// of the split table; the 8 warps of a CTA take neighbours, whose runs share
// camera rows.  Consecutive pairs' runs adjoin, so the sliding view folds its
// complete pair and its mixed pair in one walk, together with the maxima it
// combines them with.
//
// What bounds it: L2 traffic (a push reads the run and one slot and writes a
// slot and the view, 45 MB at 200 planes) and the search's latency.  Device
// time back to back, 512 x 2048 frames, 35 deg, step 0.3, pixel 0.1, before
// (a scatter of shared and global atomic maxima; a push was two of them, one
// zeroing and two elementwise maxima) -> now: one pair 9.8 -> 9.2 us, with a
// z-sum 14.9 -> 10.2; a push on 200 planes 30.3 -> 17.7, the last one with the
// next suffixes 1240 -> 773 (5 GB of slots read and written, 6.5 TB/s); 87 x
// 1304 frames of 50 planes: pair 5.0 -> 3.4, push 16.9 -> 5.7, last 135 -> 33.
// Four rows' loads ahead cost occupancy and were slower (18.9 a push).
#include <algorithm>

#include "opm_tma.cuh"

namespace opm {

namespace {

constexpr int kSXL = 4;            // columns x per lane
constexpr int kSXW = 32 * kSXL;    // columns x per warp
constexpr int kSWarps = 8;         // neighbouring columns j (rows k) per CTA
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
// on), count if none.  Whole warp.
template <typename Pred>
__device__ __forceinline__ int first_index(int count, int lane, const Pred& reached) {
  int lo = 0, hi = count;  // the answer lies in [lo, hi]
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

// This lane's kSXL counts of camera row k of one frame: neighbours (VEC) or
// columns 32 apart; zeros for a missing frame.
template <bool VEC>
__device__ __forceinline__ void load_counts(const uint16_t* __restrict__ frame, size_t o, int lim, f2 (&out)[2]) {
  uint32_t w0 = 0, w1 = 0;
  if (frame) {
    const uint16_t* p = frame + o;
    if constexpr (VEC) {
      const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
      w0 = u.x, w1 = u.y;
    } else {
      if (0 < lim) w0 = __ldg(p);
      if (32 < lim) w0 |= (uint32_t)__ldg(p + 32) << 16;
      if (64 < lim) w1 = __ldg(p + 64);
      if (96 < lim) w1 |= (uint32_t)__ldg(p + 96) << 16;
    }
  }
  out[0] = u16x2_to_f2(w0);
  out[1] = u16x2_to_f2(w1);
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
__device__ __forceinline__ void fold_column(const PlanView& v, const Pair& A, const Pair& B, int j, int lane, int x0,
                                            int lim, Fold& f) {
  const Split aj = v.A[j];
  const int top = B.n != kNoPair ? B.n : A.n, bottom = A.n != kNoPair ? A.n : B.n;
  auto lower = [&](int k) {
    const Split b = v.B[k];
    return aj.i - b.i - (aj.f - b.f < 0.0f);
  };
  for (int k = first_index(v.nz, lane, [&](int i) { return lower(i) <= top; }); k < v.nz; ++k) {
    int n0;
    float w;
    plane_weight(aj, v.B[k], v.linear, n0, w);
    if (n0 < bottom) break;
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

// Row k: its columns in pair A (which come first) and pair B.
template <bool VEC>
__device__ __forceinline__ void fold_row(const PlanView& v, const Pair& A, const Pair& B, int k, int lane, int x0,
                                         int lim, Fold& f) {
  const Split b = v.B[k];
  const int top = B.n != kNoPair ? B.n : A.n, bottom = A.n != kNoPair ? A.n : B.n;
  auto lower = [&](int j) {
    const Split a = v.A[j];
    return a.i - b.i - (a.f - b.f < 0.0f);
  };
  const size_t o = (size_t)k * v.ncols + x0;
  f2 lo[2], hi[2];
  int held = kNoPair;
  for (int j = first_index(v.ny, lane, [&](int i) { return lower(i) >= bottom; }); j < v.ny; ++j) {
    int n0;
    float w;
    plane_weight(v.A[j], b, v.linear, n0, w);
    if (n0 > top) break;
    f.any = true;
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
}

template <bool VEC>
__device__ __forceinline__ void get(const float* p, int lim, float (&out)[kSXL]) {
  if constexpr (VEC) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    out[0] = q.x, out[1] = q.y, out[2] = q.z, out[3] = q.w;
  } else {
#pragma unroll
    for (int c = 0; c < kSXL; ++c) out[c] = 32 * c < lim ? p[32 * c] : 0.0f;
  }
}
template <bool VEC>
__device__ __forceinline__ void put(float* p, int lim, const float (&v)[kSXL]) {
  if constexpr (VEC) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int c = 0; c < kSXL; ++c)
      if (32 * c < lim) p[32 * c] = v[c];
  }
}
__device__ __forceinline__ void max_into(float (&a)[kSXL], const float (&b)[kSXL]) {
#pragma unroll
  for (int c = 0; c < kSXL; ++c) a[c] = fmaxf(a[c], b[c]);
}

// Which column j or row k a warp owns, and its columns x.  Blocks: x-tiles
// fastest, the columns [j0, j1) in groups of kSWarps, then the rows.
struct Place {
  bool column, live;
  int i;        // j or k
  int x0, lim;  // first column x of the lane, columns from there to the edge
};
template <bool VEC>
__device__ __forceinline__ Place place(const PlanView& v, int xtiles, int j0, int j1) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int jgroups = (j1 - j0 + kSWarps - 1) / kSWarps;
  const int g = blockIdx.x / xtiles, xb = (blockIdx.x - g * xtiles) * kSXW;
  Place p;
  p.column = g < jgroups;
  p.i = (p.column ? j0 + g * kSWarps : (g - jgroups) * kSWarps) + warp;
  p.live = p.i < (p.column ? j1 : v.nz);
  p.x0 = xb + (VEC ? lane * kSXL : lane);
  p.lim = v.nx - p.x0;
  if (VEC && p.lim <= 0) p.x0 = 0;  // reads something, writes nothing
  return p;
}

// Pair A into the outputs (any of them NULL): columns [j0, j1) hold its voxels.
template <bool VEC, bool SUM>
__global__ void __launch_bounds__(32 * kSWarps)
k_stream_pair(PlanView v, Pair A, int xtiles, int j0, int j1, float* zmip, float* zsum, float* ymip) {
  const Place p = place<VEC>(v, xtiles, j0, j1);
  if (!p.live) return;
  const int lane = threadIdx.x & 31;
  const Pair none{nullptr, nullptr, kNoPair};
  Fold f{};
  if (p.column)
    fold_column<VEC, SUM>(v, A, none, p.i, lane, p.x0, p.lim, f);
  else
    fold_row<VEC>(v, A, none, p.i, lane, p.x0, p.lim, f);
  float* out = p.column ? zmip : ymip;
  if (!f.any || p.lim <= 0) return;
  const size_t o = (size_t)p.i * v.nx + p.x0;
  float old[kSXL];
  if (out) {
    get<VEC>(out + o, p.lim, old);
    max_into(f.a, old);
    put<VEC>(out + o, p.lim, f.a);
  }
  if constexpr (SUM) {
    if (p.column) {
      get<VEC>(zsum + o, p.lim, old);
#pragma unroll
      for (int c = 0; c < kSXL; ++c) old[c] += f.s[c];
      put<VEC>(zsum + o, p.lim, old);
    }
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

template <bool VEC>
__global__ void __launch_bounds__(32 * kSWarps)
k_sliding_push(PlanView v, Pair A, Pair B, Slide s, int xtiles) {
  const Place p = place<VEC>(v, xtiles, 0, v.ny);
  if (!p.live) return;
  const int lane = threadIdx.x & 31;
  const size_t o = (p.column ? (size_t)0 : (size_t)v.ny * v.nx) + (size_t)p.i * v.nx + p.x0;
  float run[kSXL] = {}, next[kSXL] = {};
  if (p.lim > 0) {  // on their way while the run is searched
    if (!s.fresh) get<VEC>(s.run + o, p.lim, run);
    if (s.next) get<VEC>(s.next + o, p.lim, next);
  }
  Fold f{};
  if (p.column)
    fold_column<VEC, false>(v, A, B, p.i, lane, p.x0, p.lim, f);
  else
    fold_row<VEC>(v, A, B, p.i, lane, p.x0, p.lim, f);
  if (p.lim <= 0) return;
  if (s.slotA) put<VEC>(s.slotA + o, p.lim, f.a);
  if (s.slotB) put<VEC>(s.slotB + o, p.lim, f.b);
  max_into(run, f.a);
  if (s.last) max_into(run, f.b);
  if (f.any || s.fresh) put<VEC>(s.run + o, p.lim, run);
  max_into(run, next);
  max_into(run, f.b);
  put<VEC>(s.view + o, p.lim, run);
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

// Blocks for columns [j0, j1) and all rows; 0 when there are too many.
static unsigned stream_blocks(const PlanView& v, long long columns, bool rows) {
  const long long xtiles = (v.nx + kSXW - 1) / kSXW;
  const long long groups = (columns + kSWarps - 1) / kSWarps + (rows ? (v.nz + kSWarps - 1) / kSWarps : 0);
  return xtiles * groups <= 0x7fffffffLL ? (unsigned)(xtiles * groups) : 0u;
}

opm_status launch_stream_pair(const opm_plan* p, const uint16_t* lo, const uint16_t* hi, int n, float* zmip,
                              float* zsum, float* ymip, cudaStream_t s) {
  const PlanView& v = p->view;
  if (v.nz > 65535) return fail(OPM_ERR_UNSUPPORTED, "more than 65535 camera rows");
  // columns with a voxel in the pair: n0 grows with j and falls with k
  const Split b0 = p->hB.front(), b1 = p->hB.back();
  const auto lower = [](const Split& a, const Split& b) { return a.i - b.i - (a.f - b.f < 0.0f ? 1 : 0); };
  const auto first = [&](const Split& b, int least) {
    return (int)(std::partition_point(p->hA.begin(), p->hA.end(), [&](const Split& a) { return lower(a, b) < least; }) -
                 p->hA.begin());
  };
  int j0 = first(b0, n), j1 = first(b1, n + 1);
  if ((!zmip && !zsum) || j1 < j0) j1 = j0;
  const unsigned blocks = stream_blocks(v, j1 - j0, ymip != nullptr);
  if (blocks == 0) {
    if (j1 == j0 && !ymip) return OPM_OK;  // the pair has no voxel
    return fail(OPM_ERR_UNSUPPORTED, "plane-pair grid exceeds launch limits");
  }
  const bool vec = stream_vec(v, lo, hi, nullptr) && vec_out(zmip) && vec_out(zsum) && vec_out(ymip);
  const int xtiles = (v.nx + kSXW - 1) / kSXW;
  const auto kern = zsum ? (vec ? k_stream_pair<true, true> : k_stream_pair<false, true>)
                         : (vec ? k_stream_pair<true, false> : k_stream_pair<false, false>);
  kern<<<blocks, 32 * kSWarps, 0, s>>>(v, Pair{lo, hi, n}, xtiles, j0, j1, zmip, zsum, ymip);
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
  const unsigned blocks = stream_blocks(v, v.ny, true);
  if (blocks == 0) return fail(OPM_ERR_UNSUPPORTED, "sliding-view grid exceeds launch limits");
  const bool vec = stream_vec(v, A.lo, A.hi, B.hi) && per % kSXL == 0 && vec_out(run) && vec_out(slots) && vec_out(view);
  const int xtiles = (v.nx + kSXW - 1) / kSXW;
  (vec ? k_sliding_push<true> : k_sliding_push<false>)<<<blocks, 32 * kSWarps, 0, s>>>(v, A, B, sl, xtiles);
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
