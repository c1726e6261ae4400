// Full-volume deskew (Fig. 2c remap with linear interpolation between scan
// planes).  Output-write bound: every voxel is written once with streaming
// stores.  Each warp walks a run of kRunJ output columns j of one row k and
// keeps the current pair of raw planes in registers, so a raw vector is
// fetched once per plane step rather than once per voxel.  The run's planes
// and weights are worked out by the warp's lanes side by side, one column
// each, and handed round by shuffles; where the walk next steps onto the plane
// after the current pair, that plane is already on its way.
// A lane owns NH vectors of H columns x, 32 H apart, so that every load and
// store instruction of a warp covers one contiguous span.
// Bounded by DRAM: the FP32 volume of 200 x 512 x 2048 (35 deg, step 0.3, pixel
// 0.1) takes 699 us, 4.70 GB at 6.73 TB/s (718 us with the plane table read and
// each plane waited for column by column); its uint16 volume at 45 deg, 0.2,
// 0.115 325 us, 1.91 GB at 5.9 TB/s (496 us with 8-byte vectors and two trips
// per sample through the conversion unit).
#include <algorithm>

#include "opm_common.cuh"

namespace opm {

namespace {

constexpr int kThreadsX = 32;  // lanes along x
constexpr int kThreadsY = 4;   // j-runs per CTA
constexpr int kRunJ = 32;      // output columns per warp, one per lane for the plane table

// H raw elements as loaded, packed into words; VEC: one load of 8 or 16 bytes,
// else element by element.
template <typename T, int H>
struct RawVec {
  static_assert(sizeof(T) * H == 8 || sizeof(T) * H == 16, "8- or 16-byte vectors");
  uint32_t w[sizeof(T) * H / 4];
};
template <typename T>
struct RawVec<T, 1> {
  T v;
};

template <bool VEC, typename T, int H>
__device__ __forceinline__ void load_raw(const T* __restrict__ p, RawVec<T, H>& out) {
  if constexpr (H == 1) {
    out.v = __ldg(p);
  } else if constexpr (!VEC) {
#pragma unroll
    for (int i = 0; i < (int)(sizeof(out.w) / 4); ++i) {
      if constexpr (sizeof(T) == 2)
        out.w[i] = (uint32_t)__ldg(p + 2 * i) | (uint32_t)__ldg(p + 2 * i + 1) << 16;
      else
        out.w[i] = __float_as_uint(__ldg(p + i));
    }
  } else if constexpr (sizeof(T) * H == 16) {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    out.w[0] = u.x, out.w[1] = u.y, out.w[2] = u.z, out.w[3] = u.w;
  } else {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    out.w[0] = u.x, out.w[1] = u.y;
  }
}

template <typename T, int H>
__device__ __forceinline__ void zero_raw(RawVec<T, H>& out) {
  if constexpr (H == 1) {
    out.v = T(0);
  } else {
#pragma unroll
    for (int i = 0; i < (int)(sizeof(out.w) / 4); ++i) out.w[i] = 0u;
  }
}

// Raw elements as accumulator values.  uint16: 2^23 + u in the float's bit
// pattern by a byte permute, then 2^23 off again, exact and off the
// conversion unit (cvt.f32.u16 issues once in 8 cycles).
template <typename T, int H, typename Acc>
__device__ __forceinline__ void widen(const RawVec<T, H>& r, Acc (&out)[H]) {
  if constexpr (std::is_same<T, uint16_t>::value) {
#pragma unroll
    for (int i = 0; i < H; ++i) {
      uint32_t u;
      if constexpr (H == 1)
        u = 0x4B000000u | r.v;
      else
        u = __byte_perm(r.w[i / 2], 0x4B000000u, i % 2 ? 0x7632 : 0x7610);
      out[i] = __uint_as_float(u) - 8388608.0f;
    }
  } else if constexpr (H == 1) {
    out[0] = static_cast<Acc>(r.v);
  } else {
    static_assert(std::is_same<T, float>::value, "vectors of uint16 or FP32");
#pragma unroll
    for (int i = 0; i < H; ++i) out[i] = __uint_as_float(r.w[i]);
  }
}

// Two values in [0, 65535] rounded half to even, packed: adding 2^23 leaves
// the rounded integer in the low bits of the pattern.
__device__ __forceinline__ uint32_t pack_rn(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo + 8388608.0f), __float_as_uint(hi + 8388608.0f), 0x5410);
}

// Stores one vector of H output values with streaming stores.  `INSIDE`: the
// values are known to lie in [0, 65535] (interpolated uint16 counts).
template <typename Tout, int H, bool INSIDE, typename Acc>
__device__ __forceinline__ void store_vec(Tout* op, const Acc (&val)[H]) {
  if constexpr (std::is_same<Tout, uint16_t>::value && H > 1) {
    uint32_t q[H / 2];
#pragma unroll
    for (int i = 0; i < H / 2; ++i) {
      if constexpr (INSIDE)
        q[i] = pack_rn(val[2 * i], val[2 * i + 1]);
      else  // clamp; NaN maps to 0
        q[i] = pack_rn(fminf(fmaxf(val[2 * i], 0.0f), 65535.0f), fminf(fmaxf(val[2 * i + 1], 0.0f), 65535.0f));
    }
    if constexpr (H == 8)
      st_cs_v4u(op, q[0], q[1], q[2], q[3]);
    else if constexpr (H == 4)
      asm volatile("st.global.cs.v2.b32 [%0], {%1, %2};" ::"l"(op), "r"(q[0]), "r"(q[1]) : "memory");
    else
      asm volatile("st.global.cs.b32 [%0], %1;" ::"l"(op), "r"(q[0]) : "memory");
  } else if constexpr (std::is_same<Tout, uint16_t>::value) {
    const float c = INSIDE ? val[0] : fminf(fmaxf(val[0], 0.0f), 65535.0f);
    __stcs(op, (uint16_t)__float_as_uint(c + 8388608.0f));
  } else if constexpr (std::is_same<Tout, float>::value && H == 4) {
    st_cs_v4(op, val[0], val[1], val[2], val[3]);
  } else if constexpr (std::is_same<Tout, float>::value && H == 2) {
    asm volatile("st.global.cs.v2.f32 [%0], {%1, %2};" ::"l"(op), "f"(val[0]), "f"(val[1]) : "memory");
  } else {
    static_assert(H == 1, "vectors of 4 or 2 floats");
    __stcs(op, (Tout)val[0]);
  }
}

// Which planes ahead are fetched: every one (plans that never step over a plane),
// those the walk steps onto next by a mask worked out once per run, or by a look
// at the next change (the widest element-wise forms, where the mask's test turns
// the loads into predicated ones: 100 x 256 x 509 FP32 58 us against 48).
enum Ahead { kAlways, kMask, kLook };

// vol2 (uint16, may be NULL unless DUAL) receives the round-to-nearest-even
// copy of the same values in the same pass.
template <typename Tin, typename Tout, typename Acc, int H, int NH, bool DUAL, bool VEC, Ahead AHEAD>
__global__ void __launch_bounds__(kThreadsX* kThreadsY)
k_deskew(PlanView v, const Tin* __restrict__ raw, Tout* __restrict__ vol, uint16_t* __restrict__ vol2,
         int xtiles) {
  constexpr bool kInside = std::is_same<Tin, uint16_t>::value;
  const int k = blockIdx.x / xtiles;
  const int xt = blockIdx.x - k * xtiles;
  const int lane = threadIdx.x;
  int xh[NH], lim[NH];  // first column and valid columns of each vector
#pragma unroll
  for (int h = 0; h < NH; ++h) {
    xh[h] = xt * kThreadsX * H * NH + h * kThreadsX * H + lane * H;
    lim[h] = v.nx - xh[h];
  }
  const int jb = (blockIdx.y * kThreadsY + threadIdx.y) * kRunJ;
  if (jb >= v.ny) return;
  const int nj = min(kRunJ, v.ny - jb);
  const size_t plane = (size_t)v.nrows * v.ncols;
  const Tin* rowp = raw + (size_t)k * v.ncols;

  // lane l: lower plane and weight of column jb + l, and whether the walk
  // changes planes there
  int nl;
  Acc wl;
  plane_weight_t<Acc>(v.A[min(jb + lane, v.ny - 1)], v.B[k], v.linear, nl, wl);
  const int nprev = __shfl_up_sync(0xffffffffu, nl, 1);
  const unsigned change = __ballot_sync(0xffffffffu, lane == 0 || nl != nprev);
  unsigned ahead = 0;  // changes after which the walk next steps onto the plane above
  if constexpr (AHEAD == kMask) {
    const unsigned later = lane < 31 ? change >> (lane + 1) : 0u;
    const int nnext = __shfl_sync(0xffffffffu, nl, (lane + __ffs(later)) & 31);
    ahead = __ballot_sync(0xffffffffu, later && nnext == nl + 1);
  }

  auto fetch = [&](int n, RawVec<Tin, H>(&out)[NH]) {
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      if (n >= 0 && n < v.nscan && lim[h] > 0)
        load_raw<VEC, Tin, H>(rowp + (size_t)n * plane + xh[h], out[h]);
      else
        zero_raw(out[h]);
    }
  };

  Acc a[NH][H], b[NH][H], d[NH][H];
  RawVec<Tin, H> next[NH];  // plane ocur + 2, when the next change steps onto plane ocur + 1
  int ocur = -0x40000000;   // plane index held in a[] (none yet)
#pragma unroll
  for (int h = 0; h < NH; ++h)
#pragma unroll
    for (int i = 0; i < H; ++i) a[h][i] = b[h][i] = d[h][i] = Acc(0);
  size_t orow = ((size_t)k * v.ny + jb) * v.nx;

#pragma unroll 1
  for (int jj = 0; jj < nj; ++jj, orow += v.nx) {
    if ((change >> jj) & 1u) {
      const int n0 = __shfl_sync(0xffffffffu, nl, jj);
      if (n0 == ocur + 1) {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
#pragma unroll
          for (int i = 0; i < H; ++i) a[h][i] = b[h][i];
          widen<Tin, H, Acc>(next[h], b[h]);
        }
      } else {
        RawVec<Tin, H> r0[NH], r1[NH];
        fetch(n0, r0);
        fetch(n0 + 1, r1);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          widen<Tin, H, Acc>(r0[h], a[h]);
          widen<Tin, H, Acc>(r1[h], b[h]);
        }
      }
      if constexpr (AHEAD == kLook) {
        const unsigned later = jj < 31 ? change >> (jj + 1) : 0u;
        if (later && __shfl_sync(0xffffffffu, nl, jj + __ffs(later)) == n0 + 1) fetch(n0 + 2, next);
      } else {
        if (AHEAD == kAlways || ((ahead >> jj) & 1u)) fetch(n0 + 2, next);
      }
#pragma unroll
      for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int i = 0; i < H; ++i) d[h][i] = b[h][i] - a[h][i];
      ocur = n0;
    }
    const Acc w = __shfl_sync(0xffffffffu, wl, jj);
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      if (lim[h] <= 0) continue;
      Acc val[H];
#pragma unroll
      for (int i = 0; i < H; ++i) val[i] = fma(w, d[h][i], a[h][i]);
      store_vec<Tout, H, kInside>(vol + orow + xh[h], val);
      if constexpr (DUAL)
        store_vec<uint16_t, H, kInside>(vol2 + orow + xh[h], val);
    }
  }
}

// Whether every row of an array starts on a vector of H elements.
template <typename T, int H>
bool aligned(const void* q, int n) {
  return n % H == 0 && (uintptr_t)q % (sizeof(T) * H) == 0;
}

template <typename Tin, typename Tout, typename Acc, int H, int NH, bool DUAL, bool VEC>
opm_status run(const opm_plan* p, const void* raw, void* vol, void* vol2, cudaStream_t s) {
  const PlanView& v = p->view;
  const int xtiles = (v.nx + kThreadsX * H * NH - 1) / (kThreadsX * H * NH);
  const long long gx = (long long)xtiles * v.nz;
  const int gy = (v.ny + kThreadsY * kRunJ - 1) / (kThreadsY * kRunJ);
  if (gx > 0x7fffffffLL || gy > 65535)
    return fail(OPM_ERR_UNSUPPORTED, "deskew grid exceeds launch limits");
  dim3 block(kThreadsX, kThreadsY);
  dim3 grid((unsigned)gx, (unsigned)gy);
  const auto go = [&](auto ahead) {
    k_deskew<Tin, Tout, Acc, H, NH, DUAL, VEC, decltype(ahead)::value><<<grid, block, 0, s>>>(
        v, static_cast<const Tin*>(raw), static_cast<Tout*>(vol), static_cast<uint16_t*>(vol2), xtiles);
  };
  if constexpr (H == 1 && sizeof(Tin) < 8)
    go(std::integral_constant<Ahead, NH == 8 ? kLook : kMask>{});
  else if (p->unit_steps)
    go(std::integral_constant<Ahead, kAlways>{});
  else
    go(std::integral_constant<Ahead, kMask>{});
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? OPM_OK : cuda_fail(e, "launch k_deskew");
}

// Vectors of H elements when the rows of every array start on one; FP32 input
// that is only 8-byte aligned (an even width, a base off 16 bytes) in vectors of
// two; aligned outputs alone keep their vector stores and take the raw elements
// one by one.  Else one element per lane and instruction, contiguous for the
// warp, where element-wise vectors would leave strides of H between lanes.  The
// narrower forms hold 8 columns per lane where the row has them, since the walk's
// own instructions bound them.  us, 100 x 256 x w at 45 deg, step 0.2, pixel
// 0.115, element-wise half-vectors -> this: uint16 to FP32 w = 509 85 -> 38, raw
// alone off 4 bytes 39 -> 34; FP32 to FP32 w = 509 52 -> 48 (55 with 4 per lane),
// w = 506 49 -> 46; FP32 to uint16 w = 506 48 -> 42, w = 509 48 -> 49.
template <typename Tin, typename Tout, typename Acc, int H, int NH, bool DUAL = false>
opm_status run_aligned(const opm_plan* p, const void* raw, void* vol, void* vol2, cudaStream_t s) {
  const int nx = p->view.nx;
  const bool out = aligned<Tout, H>(vol, nx) && (!DUAL || aligned<uint16_t, H>(vol2, nx));
  if (out && aligned<Tin, H>(raw, nx)) return run<Tin, Tout, Acc, H, NH, DUAL, true>(p, raw, vol, vol2, s);
  if constexpr (sizeof(Tin) == 4)
    if (aligned<Tin, 2>(raw, nx) && aligned<Tout, 2>(vol, nx) && (!DUAL || aligned<uint16_t, 2>(vol2, nx)))
      return nx <= 4 * kThreadsX ? run<Tin, Tout, Acc, 2, 2, DUAL, true>(p, raw, vol, vol2, s)
                                 : run<Tin, Tout, Acc, 2, 4, DUAL, true>(p, raw, vol, vol2, s);
  if (out) return run<Tin, Tout, Acc, H, NH, DUAL, false>(p, raw, vol, vol2, s);
  if (nx <= 4 * kThreadsX) return run<Tin, Tout, Acc, 1, 4, DUAL, true>(p, raw, vol, vol2, s);
  return run<Tin, Tout, Acc, 1, 8, DUAL, true>(p, raw, vol, vol2, s);
}

// ---------------------------------------------------------------------------
// Volume and live view in one pass (uint16 input): every voxel is stored as
// k_deskew stores it, and folded into the z-MIP and y-MIP on the way.  CTA
// (32 x 8 threads): 128 columns x (4 per lane) x 32 columns j (4 per warp) x
// a chunk of kMipRows camera rows, 4 CTAs per SM.  The z-maxima of a
// thread's 4 x 4 voxels
// stay in registers across the chunk's rows and are folded into the global
// z-MIP once; the y-maxima of each row are combined across the 8 warps with
// shared-memory atomics and folded into the global y-MIP once per CTA.  All
// combines are maxima of non-negative values on their bit patterns, so the
// result does not depend on their order.
constexpr int kMipRows = 64;
constexpr int kMipWarps = 8;  // warps (runs of kMipJ columns) per CTA
constexpr int kMipJ = 4;     // columns j per thread
constexpr int kMipVec = 4;   // columns x per lane

template <bool F32, bool U16>
__global__ void __launch_bounds__(kThreadsX* kMipWarps, 4)
k_deskew_mip(PlanView v, const uint16_t* __restrict__ raw, float* __restrict__ volf, uint16_t* __restrict__ volh,
             float* __restrict__ zmip, float* __restrict__ ymip, int in_vec_ok, int out_vec_ok) {
  __shared__ float ybuf[kMipRows][kThreadsX * kMipVec];
  const int lane = threadIdx.x, w = threadIdx.y;
  const int x = blockIdx.x * kThreadsX * kMipVec + lane * kMipVec;
  const int jb = (blockIdx.y * kMipWarps + w) * kMipJ;
  const int k0 = blockIdx.z * kMipRows;
  const int k1 = min(k0 + kMipRows, v.nz);
  for (int i = threadIdx.y * kThreadsX + threadIdx.x; i < kMipRows * kThreadsX * kMipVec; i += kThreadsX * kMipWarps)
    (&ybuf[0][0])[i] = 0.0f;
  __syncthreads();
  const bool active = x < v.nx && jb < v.ny;
  const int lim = v.nx - x;  // valid columns of this lane's vector
  const bool vin = in_vec_ok && lim >= kMipVec;
  const bool vout = out_vec_ok && lim >= kMipVec;
  const size_t plane = (size_t)v.nrows * v.ncols;
  float zmax[kMipJ][kMipVec];
#pragma unroll
  for (int j = 0; j < kMipJ; ++j)
#pragma unroll
    for (int c = 0; c < kMipVec; ++c) zmax[j][c] = 0.0f;  // uint16 voxels are >= 0

#pragma unroll 1
  for (int k = k0; active && k < k1; ++k) {
    const Split b = v.B[k];
    const uint16_t* rowp = raw + (size_t)k * v.ncols + x;
    float a[kMipVec], bb[kMipVec], d[kMipVec], ym[kMipVec];
#pragma unroll
    for (int c = 0; c < kMipVec; ++c) a[c] = bb[c] = d[c] = ym[c] = 0.0f;
    int ocur = -0x40000000;
    auto fetch = [&](int n, float(&out)[kMipVec]) {
      if (n >= 0 && n < v.nscan) {
        const uint16_t* p = rowp + (size_t)n * plane;
        if (vin) {
          const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
          out[0] = (float)(u.x & 0xFFFFu);
          out[1] = (float)(u.x >> 16);
          out[2] = (float)(u.y & 0xFFFFu);
          out[3] = (float)(u.y >> 16);
        } else {
#pragma unroll
          for (int c = 0; c < kMipVec; ++c) out[c] = c < lim ? (float)__ldg(p + c) : 0.0f;
        }
      } else {
#pragma unroll
        for (int c = 0; c < kMipVec; ++c) out[c] = 0.0f;
      }
    };
#pragma unroll
    for (int jj = 0; jj < kMipJ; ++jj) {
      const int j = jb + jj;
      if (j >= v.ny) break;
      int n0;
      float wt;
      plane_weight(v.A[j], b, v.linear, n0, wt);
      if (n0 != ocur) {
        if (n0 == ocur + 1) {
#pragma unroll
          for (int c = 0; c < kMipVec; ++c) a[c] = bb[c];
        } else {
          fetch(n0, a);
        }
        fetch(n0 + 1, bb);
#pragma unroll
        for (int c = 0; c < kMipVec; ++c) d[c] = bb[c] - a[c];  // exact: integers below 2^24
        ocur = n0;
      }
      float val[kMipVec];
#pragma unroll
      for (int c = 0; c < kMipVec; ++c) {
        val[c] = fmaf(wt, d[c], a[c]);
        zmax[jj][c] = fmaxf(zmax[jj][c], val[c]);
        ym[c] = fmaxf(ym[c], val[c]);
      }
      const size_t o = ((size_t)k * v.ny + j) * v.nx + x;
      if (vout) {
        if (F32) st_cs_v4(volf + o, val[0], val[1], val[2], val[3]);
        if (U16) {
          const uint32_t lo = (uint32_t)to_u16_rn(val[0]) | ((uint32_t)to_u16_rn(val[1]) << 16);
          const uint32_t hi = (uint32_t)to_u16_rn(val[2]) | ((uint32_t)to_u16_rn(val[3]) << 16);
          asm volatile("st.global.cs.v2.b32 [%0], {%1, %2};" ::"l"(volh + o), "r"(lo), "r"(hi) : "memory");
        }
      } else {
#pragma unroll
        for (int c = 0; c < kMipVec; ++c) {
          if (c >= lim) break;
          if (F32) volf[o + c] = val[c];
          if (U16) volh[o + c] = to_u16_rn(val[c]);
        }
      }
    }
    if (ymip) {
#pragma unroll
      for (int c = 0; c < kMipVec; ++c)
        if (c < lim) atomicMax(reinterpret_cast<int*>(&ybuf[k - k0][lane * kMipVec + c]), __float_as_int(ym[c]));
    }
  }
  if (zmip && active) {
#pragma unroll
    for (int jj = 0; jj < kMipJ; ++jj) {
      const int j = jb + jj;
      if (j >= v.ny) break;
      float* zr = zmip + (size_t)j * v.nx + x;
#pragma unroll
      for (int c = 0; c < kMipVec; ++c)
        if (c < lim) atomicMax(reinterpret_cast<int*>(zr + c), __float_as_int(zmax[jj][c]));
    }
  }
  if (ymip) {
    __syncthreads();
    const int xb = blockIdx.x * kThreadsX * kMipVec;
    for (int i = threadIdx.y * kThreadsX + threadIdx.x; i < (k1 - k0) * kThreadsX * kMipVec;
         i += kThreadsX * kMipWarps) {
      const int kk = i / (kThreadsX * kMipVec), xx = i % (kThreadsX * kMipVec);
      if (xb + xx < v.nx)
        atomicMax(reinterpret_cast<int*>(ymip + (size_t)(k0 + kk) * v.nx + xb + xx), __float_as_int(ybuf[kk][xx]));
    }
  }
}

__global__ void k_zero2(float* a, long long na, float* b, long long nb) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < na || i < nb; i += stride) {
    if (a && i < na) a[i] = 0.0f;
    if (b && i < nb) b[i] = 0.0f;
  }
}

}  // namespace

opm_status launch_deskew(const opm_plan* p, const void* raw, opm_dtype in_t, void* vol,
                         opm_dtype out_t, cudaStream_t s) {
  if (in_t == OPM_U16 && out_t == OPM_F32) return run_aligned<uint16_t, float, float, 4, 2>(p, raw, vol, nullptr, s);
  if (in_t == OPM_U16 && out_t == OPM_U16) {
    // 16-byte vectors where the rows allow them
    if (aligned<uint16_t, 8>(raw, p->view.nx) && aligned<uint16_t, 8>(vol, p->view.nx))
      return run<uint16_t, uint16_t, float, 8, 1, false, true>(p, raw, vol, nullptr, s);
    return run_aligned<uint16_t, uint16_t, float, 4, 2>(p, raw, vol, nullptr, s);
  }
  if (in_t == OPM_F32 && out_t == OPM_F32) return run_aligned<float, float, float, 4, 1>(p, raw, vol, nullptr, s);
  if (in_t == OPM_F32 && out_t == OPM_U16) return run_aligned<float, uint16_t, float, 4, 1>(p, raw, vol, nullptr, s);
  if (in_t == OPM_F64 && out_t == OPM_F64) return run<double, double, double, 1, 2, false, true>(p, raw, vol, nullptr, s);
  return fail(OPM_ERR_UNSUPPORTED, "unsupported dtype pair");
}

opm_status launch_deskew_dual(const opm_plan* p, const void* raw, opm_dtype in_t, float* vol_f32, uint16_t* vol_u16,
                              cudaStream_t s) {
  if (in_t == OPM_U16) return run_aligned<uint16_t, float, float, 4, 2, true>(p, raw, vol_f32, vol_u16, s);
  if (in_t == OPM_F32) return run_aligned<float, float, float, 4, 1, true>(p, raw, vol_f32, vol_u16, s);
  return fail(OPM_ERR_UNSUPPORTED, "dual-output deskew takes uint16 or FP32 input");
}

}  // namespace opm

namespace opm {

namespace {

// The volume on the caller's stream s and the live view beside it on the
// plan's high-priority side stream, forked from and joined back into s.
// The live view's persistent kernel takes a part of its usual grid, so each SM
// also holds volume CTAs: the issue-bound projection then fills the issue
// slots the write-bound volume leaves idle.  Each kernel computes exactly what
// it computes alone.
// The two should end together: beside an FP32 volume (4 or 6 bytes a voxel) one
// projection CTA per SM, beside a uint16 volume, which is written in half the
// time, two.  us for the pair at 4 / 2 / 1 of them per SM and one after the
// other (uint16 volume + z-MIP of 1000 x 1024 x 2048, 45 deg, 0.2, 0.115):
// 3475 / 3297 / 3676 / 3746; uint16 + z + y of the 200 x 512 x 2048 live view:
// 526 / 503 / 554 / 541; FP32 + z + y of it: 824 / 792 / 785 / 843.
opm_status deskew_beside_project(const opm_plan* p, const void* raw, opm_dtype in_t, float* volf, uint16_t* volh,
                                 float* zmip, float* ymip, cudaStream_t s) {
  std::lock_guard<std::mutex> lock(p->side_mu);
  cudaError_t e = cudaEventRecord(p->fork_ev, s);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(p->side, p->fork_ev, 0);
  if (e != cudaSuccess) return cuda_fail(e, "forking the live view onto the side stream");
  opm_status st = launch_project(p, raw, in_t, zmip, nullptr, ymip, nullptr, p->side,
                                 volf ? p->lists_per_sm : p->lists_per_sm / 2);
  opm_status sv = OPM_OK;
  if (volf && volh)
    sv = launch_deskew_dual(p, raw, in_t, volf, volh, s);
  else
    sv = launch_deskew(p, raw, in_t, volf ? (void*)volf : (void*)volh, volf ? OPM_F32 : OPM_U16, s);
  // join even after a failed launch, so that s never runs ahead of the side stream
  e = cudaEventRecord(p->join_ev, p->side);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, p->join_ev, 0);
  if (st != OPM_OK) return st;
  if (sv != OPM_OK) return sv;
  return e == cudaSuccess ? OPM_OK : cuda_fail(e, "joining the side stream");
}

}  // namespace

opm_status launch_deskew_mip(const opm_plan* p, const void* raw, opm_dtype in_t, float* volf, uint16_t* volh,
                             float* zmip, float* ymip, cudaStream_t s) {
  const PlanView& v = p->view;
  if ((zmip || ymip) && p->side && !p->one_pass_fused)
    return deskew_beside_project(p, raw, in_t, volf, volh, zmip, ymip, s);
  if (in_t != OPM_U16) {
    // FP32 input: the volume, then the projections
    opm_status st = OPM_OK;
    if (volf && volh)
      st = launch_deskew_dual(p, raw, in_t, volf, volh, s);
    else
      st = launch_deskew(p, raw, in_t, volf ? (void*)volf : (void*)volh, volf ? OPM_F32 : OPM_U16, s);
    if (st != OPM_OK || (!zmip && !ymip)) return st;
    return launch_project(p, raw, in_t, zmip, nullptr, ymip, nullptr, s);
  }
  const int xtiles = (v.nx + kThreadsX * kMipVec - 1) / (kThreadsX * kMipVec);
  const int jblocks = (v.ny + kMipWarps * kMipJ - 1) / (kMipWarps * kMipJ);
  const int kchunks = (v.nz + kMipRows - 1) / kMipRows;
  if (jblocks > 65535 || kchunks > 65535) return fail(OPM_ERR_UNSUPPORTED, "deskew grid exceeds launch limits");
  if (zmip || ymip) {
    k_zero2<<<4 * 152, 256, 0, s>>>(zmip, zmip ? (long long)v.ny * v.nx : 0, ymip, ymip ? (long long)v.nz * v.nx : 0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "launch k_zero2");
  }
  const int in_vec_ok = (v.ncols % kMipVec == 0) && ((uintptr_t)raw % 8 == 0);
  const int out_vec_ok = (v.nx % kMipVec == 0) && ((uintptr_t)volf % 16 == 0) && ((uintptr_t)volh % 8 == 0);
  dim3 grid(xtiles, jblocks, kchunks), block(kThreadsX, kMipWarps);
  const uint16_t* r = static_cast<const uint16_t*>(raw);
  if (volf && volh)
    k_deskew_mip<true, true><<<grid, block, 0, s>>>(v, r, volf, volh, zmip, ymip, in_vec_ok, out_vec_ok);
  else if (volf)
    k_deskew_mip<true, false><<<grid, block, 0, s>>>(v, r, volf, volh, zmip, ymip, in_vec_ok, out_vec_ok);
  else
    k_deskew_mip<false, true><<<grid, block, 0, s>>>(v, r, volf, volh, zmip, ymip, in_vec_ok, out_vec_ok);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? OPM_OK : cuda_fail(e, "launch k_deskew_mip");
}

}  // namespace opm
