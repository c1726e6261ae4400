// Fused deskew + projection (Fig. 2d): z-MIP, z-sum, y-MIP and argmax-z of
// the deskewed volume, computed straight from the raw stack without ever
// writing the volume.
//
// Work decomposition (one CTA = 32 output columns j x 128 output columns x):
//  * Output row k of the volume reads only camera row k of the raw stack, at
//    planes n0(j,k), n0(j,k)+1 of the CTA's 32 columns: a contiguous slab of P
//    planes.  A producer warp stages that slab, {128 x, 1 row, P planes},
//    into shared memory with one TMA load per row, several rows ahead, on an
//    mbarrier ring.  Planes outside [0, nscan) arrive as TMA zero fill, which
//    is exactly the zero padding of the interpolation.
//  * Four compute warps own 8 columns j each and 4 columns x per lane.  For
//    every staged row they walk their 8 columns in order, keeping the current
//    plane pair (a, b - a) in registers: a column that moves to the next
//    plane costs one shared-memory load, so each staged raw value is
//    converted to FP32 once per warp rather than once per voxel.  Plane steps
//    come as warp-uniform bit masks from the producer.
//  * z-reductions stay in registers across rows; the y-max of each row is
//    reduced over the CTA's 32 columns in shared memory and folded into the
//    global y-MIP with one coalesced atomic max per column (max is order
//    independent, so the result is deterministic).
//  * Only rows whose band can carry non-zero weight for the tile are visited;
//    all other rows are exactly zero and enter the maxima as the value 0.
//
// Two kernels share that structure, the third does without it:
//  k_project_per   the periodic kernel (opm_periodic.cuh) for plans whose
//                  pixel/step is a compiled ratio p/q (1/3 or 1/2): the fast
//                  kernel's producer and schedule, compute warps of 32
//                  columns j x 2 columns x per lane with every plane step
//                  at a compile-time position.
//  k_project_fast  uint16 input, z-MIP and/or y-MIP, full 32-column tiles of
//                  plans whose columns never skip a plane (checked on the
//                  host with the kernel's own arithmetic).  Two rows per stage
//                  (one 3-input max per voxel pair into the z-max), packed
//                  FP32x2 FMAs, one branch per column step, and each tile's
//                  row band split into chunks (256 rows, fewer on narrow
//                  stacks) whose z-maxima combine by atomic max, which
//                  balances tiles of very different band length; a
//                  persistent grid of 4 CTAs per SM (fewer beside a
//                  volume) walks the chunks.
//  k_project_direct  every other call: z-sum, first arg-max, FP32 input, rows
//                  that are not a multiple of 16 bytes, any geometry
//                  (opm_direct.cuh, shared with the batch).  It reads global
//                  memory directly, without the ring described above.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cmath>
#include <cstring>
#include <mutex>

#include "opm_direct.cuh"
#include "opm_periodic.cuh"

namespace opm {

namespace {

struct ProjArgs {
  PlanView v;
  float* zmip;
  float* ymip;
  int P;       // staged planes per row
};

// Fast kernel, persistent: one CTA per list of the plan's balanced schedule
// (units of 256 rows of one j-tile at one x-tile).  The stage counter
// carries on across a CTA's units, so the next unit's slabs stream in while
// the current one drains.
template <bool YMIP, int S>
__global__ void __launch_bounds__(kThreads, 4)
k_project_fast(const __grid_constant__ CUtensorMap tmap, const ProjArgs args) {
  const PlanView& v = args.v;
  extern __shared__ __align__(128) unsigned char smem[];
  const FastRing<S> ring = fast_ring<S>(smem, args.P);
  fast_ring_init(ring);
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int g = 0;
  bool ok = true;
  int l = (int)blockIdx.x - (int)gridDim.x;
  int u = 0, uend = 0;
#pragma unroll 1
  while (ok) {
    if (u >= uend) {
      do {
        l += gridDim.x;
        if (l >= v.nlists) break;
        u = v.lists[l];
        uend = v.lists[l + 1];
      } while (u >= uend);
      if (u >= uend) break;
    }
    const WorkUnit un = v.units[u++];
    FastJob jb;
    jb.ks = un.ks;
    jb.ke = un.ke;
    jb.tmap = &tmap;
    jb.rows = v.frow + (size_t)un.jt * v.nz;
    jb.nlos = v.fnlo + (size_t)un.jt * v.nz;
    jb.zmip = args.zmip;
    jb.ymip = args.ymip;
    jb.nz = v.nz;
    jb.nx = v.nx;
    jb.j0 = tile_j0(un.jt, v.ny);
    jb.xbase = un.xt * kX;
    jb.P = args.P;
    if (warp == 0)
      ok = fast_produce(jb, ring, g, v.err, lane);
    else
      ok = fast_consume<YMIP>(jb, ring, g, v.err, warp - 1, lane);
  }
  if (warp == 0) fast_drain(ring, g, ok, v.err);
}

// Periodic kernel (opm_periodic.cuh): the fast kernel's schedule, tables
// and TMA ring for plans with pixel/step = Pp/Qq, with straight-line compute
// warps per phase; MINB CTAs per SM, S ring stages.
template <int Pp, int Qq, int RUN, int MINB, int S, bool YMIP, bool REP>
__global__ void __launch_bounds__(per::Cfg<RUN>::kThreads, MINB)
k_project_per(const __grid_constant__ CUtensorMap tmap, const ProjArgs args) {
  const PlanView& v = args.v;
  extern __shared__ __align__(128) unsigned char smem[];
  const PerRing ring = per_ring(smem, S, args.P);
  per_ring_init(ring, per::Cfg<RUN>::kCW);
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int g = 0;
  bool ok = true;
  int l = (int)blockIdx.x - (int)gridDim.x;
  int u = 0, uend = 0;
#pragma unroll 1
  while (ok) {
    if (u >= uend) {
      do {
        l += gridDim.x;
        if (l >= v.nlists) break;
        u = v.lists[l];
        uend = v.lists[l + 1];
      } while (u >= uend);
      if (u >= uend) break;
    }
    const WorkUnit un = v.units[u++];
    FastJob jb;
    jb.ks = un.ks;
    jb.ke = un.ke;
    jb.tmap = &tmap;
    jb.rows = v.frow + (size_t)un.jt * v.nz;
    jb.pairs = v.pairs + v.pair0[un.jt];
    jb.zmip = args.zmip;
    jb.ymip = args.ymip;
    jb.nz = v.nz;
    jb.nx = v.nx;
    jb.j0 = tile_j0(un.jt, v.ny);
    jb.xbase = un.xt * kX;
    jb.P = args.P;
    if (warp == 0)
      ok = per_produce(jb, ring, g, v.err, lane);
    else
      ok = per_consume<RUN, Pp, Qq, YMIP, REP>(jb, ring, g, v.err, warp - 1, lane);
  }
  if (warp == 0) per_drain(ring, g, ok, v.err);
}

// Direct kernel (opm_direct.cuh): one job per CTA, x-tiles fastest.
template <typename T, bool VEC, bool SUM, int ARG, bool JUMP>
__global__ void __launch_bounds__(direct::kCtaThreads, ARG == direct::kArg32 && SUM ? 1 : 2)
k_project_direct(const PlanView v, const T* __restrict__ raw, int wr, int slots, int xtiles, float* zmip, float* zsum,
                 float* ymip, int32_t* argz) {
  extern __shared__ __align__(128) unsigned char smem[];
  direct::Job jb;
  jb.raw = raw;
  jb.slots = slots;
  jb.row_pitch = v.ncols;
  jb.plane_pitch = (size_t)v.nrows * v.ncols;
  jb.A = v.A;
  jb.B = v.B;
  jb.linear = v.linear;
  jb.nscan = v.nscan;
  jb.ny = v.ny;
  jb.nz = v.nz;
  jb.nx = v.nx;
  jb.wr = wr;
  jb.jc = (int)(blockIdx.x / xtiles) * direct::cta_cols(wr);
  jb.xb = (int)(blockIdx.x % xtiles) * direct::kXW;
  jb.band = v.band[jb.jc / kTileJ];
  jb.zmip = zmip;
  jb.zsum = zsum;
  jb.ymip = ymip;
  jb.argz = argz;
  direct::tile<T, VEC, SUM, ARG, JUMP>(jb, smem);
}

// Initial values of the atomically combined outputs: the fast kernel folds
// its z-maxima into zeroed z-MIP rows; the y-MIP starts at 0 for uint16
// input (every voxel is >= 0) and at the plan's per-row value otherwise.
__global__ void k_init_outputs(PlanView v, float* zmip, float* ymip, int u16) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nzm = zmip ? (long long)v.ny * v.nx : 0;
  const long long nym = ymip ? (long long)v.nz * v.nx : 0;
  if (idx < nzm) zmip[idx] = 0.0f;
  if (idx < nym) ymip[idx] = u16 ? 0.0f : v.yinit[idx / v.nx];
}

// ------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    else
      cudaGetLastError();
  });
  return fn;
}

int max_optin_smem(int dev) {
  static int cache[64] = {0};
  if (dev < 0 || dev >= 64) return 0;
  if (!cache[dev]) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
      cudaGetLastError();
      v = 48 * 1024;
    }
    cache[dev] = v;
  }
  return cache[dev];
}

opm_status encode_raw(const PlanView& v, const void* raw, int P, CUtensorMap* map) {
  std::memset(map, 0, sizeof(*map));
  const cuuint64_t dims[3] = {(cuuint64_t)v.ncols, (cuuint64_t)v.nrows, (cuuint64_t)v.nscan};
  const cuuint64_t strides[2] = {(cuuint64_t)v.ncols * 2, (cuuint64_t)v.nrows * v.ncols * 2};
  const cuuint32_t box[3] = {(cuuint32_t)kX, 1u, (cuuint32_t)P};
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  CUresult cr = encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 3, const_cast<void*>(raw), dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (cr != CUDA_SUCCESS)
    return fail(OPM_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)cr) + ")");
  return OPM_OK;
}

template <typename K>
opm_status prepare_kernel(K kern, int dev, int* done) {
  if (dev >= 0 && dev < 64 && !done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin_smem(dev));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
    done[dev] = 1;
  }
  return OPM_OK;
}

// The periodic kernel of the plan's family.
template <int F>
opm_status launch_per_f(const opm_plan* p, const CUtensorMap& map, const ProjArgs& args, cudaStream_t s,
                        int grid_div) {
  if constexpr (F < kNumFamilies) {
    if (p->family - 1 != F) return launch_per_f<F + 1>(p, map, args, s, grid_div);
    constexpr int Pp = kFamilies[F].p, Qq = kFamilies[F].q;
    static int done[4][64] = {{0}};
    const bool ym = args.ymip != nullptr, rep = p->weights_repeat;
    constexpr int R = kPerRun, C = kPerCtasPerSm, S = kPerStages;
    const auto kern = ym ? (rep ? k_project_per<Pp, Qq, R, C, S, true, true> : k_project_per<Pp, Qq, R, C, S, true, false>)
                         : (rep ? k_project_per<Pp, Qq, R, C, S, false, true> : k_project_per<Pp, Qq, R, C, S, false, false>);
    opm_status st = prepare_kernel(kern, p->device, done[2 * ym + rep]);
    if (st != OPM_OK) return st;
    const PlanView& v = p->view;
    const int full = std::min(v.nunits, v.nlists);
    if (full == 0) return OPM_OK;
    const int grid = std::max(1, full / std::max(1, grid_div));
    kern<<<grid, per::Cfg<kPerRun>::kThreads, per::total(kPerStages, args.P), s>>>(map, args);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? OPM_OK : cuda_fail(e, "launch k_project_per");
  } else {
    return fail(OPM_ERR_INTERNAL, "plan names an unknown periodic family");
  }
}

opm_status launch_per(const opm_plan* p, const CUtensorMap& map, const ProjArgs& args, cudaStream_t s,
                      int grid_div) {
  if (!p->view.units || !p->view.lists) return fail(OPM_ERR_INTERNAL, "plan has no fast-kernel schedule");
  return launch_per_f<0>(p, map, args, s, grid_div);
}

template <int S>
opm_status launch_fast_s(const opm_plan* p, const CUtensorMap& map, const ProjArgs& args, cudaStream_t s,
                         int grid_div) {
  static_assert(fast_ring_bytes(S, 14) == (int)fast::total(S, 14), "the plan's arithmetic of the ring");
  static int done[2][64] = {{0}};
  const auto kern = args.ymip ? k_project_fast<true, S> : k_project_fast<false, S>;
  opm_status st = prepare_kernel(kern, p->device, done[args.ymip != nullptr]);
  if (st != OPM_OK) return st;
  const PlanView& v = p->view;
  const int full = std::min(v.nunits, v.nlists);
  if (full == 0) return OPM_OK;
  const int grid = std::max(1, full / std::max(1, grid_div));
  kern<<<grid, kThreads, fast::total(S, args.P), s>>>(map, args);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? OPM_OK : cuda_fail(e, "launch k_project_fast");
}

opm_status launch_fast(const opm_plan* p, const CUtensorMap& map, const ProjArgs& args, cudaStream_t s,
                       int grid_div) {
  if (p->family) return launch_per(p, map, args, s, grid_div);
  if (!p->view.units || !p->view.lists) return fail(OPM_ERR_INTERNAL, "plan has no fast-kernel schedule");
  switch (fast_stages(args.P, p->lists_per_sm / std::max(1, grid_div))) {
    case 6: return launch_fast_s<6>(p, map, args, s, grid_div);
    case 5: return launch_fast_s<5>(p, map, args, s, grid_div);
    case 4: return launch_fast_s<4>(p, map, args, s, grid_div);
    default: return launch_fast_s<3>(p, map, args, s, grid_div);
  }
}

template <typename T, bool VEC, bool SUM, int ARG>
opm_status launch_direct_as(const opm_plan* p, const void* raw, float* zmip, float* zsum, float* ymip, int32_t* argz,
                            cudaStream_t s) {
  const PlanView& v = p->view;
  const int wr = direct::row_groups(direct::grid_tiles(v.ny, v.nx)), cols = direct::cta_cols(wr);
  const long long xtiles = (v.nx + direct::kXW - 1) / direct::kXW;
  const long long nb = xtiles * ((v.ny + cols - 1) / cols);
  if (nb > 0x7fffffffLL) return fail(OPM_ERR_UNSUPPORTED, "grid too large");
  const bool jump = !p->unit_steps;
  static int done[2][64] = {{0}};
  const auto kern = jump ? k_project_direct<T, VEC, SUM, ARG, true> : k_project_direct<T, VEC, SUM, ARG, false>;
  opm_status st = prepare_kernel(kern, p->device, done[jump]);
  if (st != OPM_OK) return st;
  const int slots = direct::row_slots(jump, p->rho);
  kern<<<(unsigned)nb, direct::kCtaThreads, direct::smem_bytes<T>(slots, SUM, ARG), s>>>(
      v, static_cast<const T*>(raw), wr, slots, (int)xtiles, zmip, zsum, ymip, argz);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? OPM_OK : cuda_fail(e, "launch k_project_direct");
}

template <typename T>
opm_status launch_direct(const opm_plan* p, const void* raw, float* zmip, float* zsum, float* ymip, int32_t* argz,
                         cudaStream_t s) {
  const PlanView& v = p->view;
  const bool vec = direct::vec_rows<T>(raw, v.nx, v.ncols, (int64_t)v.nrows * v.ncols) && !p->force_generic;
  const auto go = [&](auto sm, auto ar) {
    constexpr bool SUM = decltype(sm)::value;
    constexpr int ARG = decltype(ar)::value;
    return vec ? launch_direct_as<T, true, SUM, ARG>(p, raw, zmip, zsum, ymip, argz, s)
               : launch_direct_as<T, false, SUM, ARG>(p, raw, zmip, zsum, ymip, argz, s);
  };
  const std::true_type sum;
  const std::false_type no_sum;
  const std::integral_constant<int, direct::kNoArg> no_arg;
  const std::integral_constant<int, direct::kArg32> arg32;
  const std::integral_constant<int, direct::kArg16> arg16;
  switch (direct::arg_form(argz != nullptr, zsum != nullptr, v.nz)) {
    case direct::kNoArg: return zsum ? go(sum, no_arg) : go(no_sum, no_arg);
    case direct::kArg16: return go(sum, arg16);
    default: return zsum ? go(sum, arg32) : go(no_sum, arg32);
  }
}

}  // namespace

opm_status launch_project(const opm_plan* p, const void* raw, opm_dtype in_t, float* zmip, float* zsum,
                          float* ymip, int32_t* argz, cudaStream_t s, int grid_div) {
  const PlanView& v = p->view;
  const bool u16 = in_t == OPM_U16;
  const int P = p->P;
  const int smax = max_optin_smem(p->device);
  // the TMA kernels: uint16 rows on 16 bytes, z-MIP and / or y-MIP only
  const bool fast = u16 && !zsum && !argz && p->fast_ok && v.frow && !p->force_generic && encode_fn() != nullptr &&
                    (uintptr_t)raw % 16 == 0 && (size_t)v.ncols * 2 % 16 == 0 &&
                    (int)(p->family ? per::total(kPerStages, P) : fast::total(fast_stages(P, p->lists_per_sm / std::max(1, grid_div)), P)) <= smax;

  // initial values of the atomically combined outputs
  float* zinit = fast ? zmip : nullptr;
  if (zinit || ymip) {
    const long long n = std::max(zinit ? (long long)v.ny * v.nx : 0LL, ymip ? (long long)v.nz * v.nx : 0LL);
    const long long nb = (n + 255) / 256;
    if (nb > 0x7fffffffLL) return fail(OPM_ERR_UNSUPPORTED, "grid too large");
    k_init_outputs<<<(unsigned)nb, 256, 0, s>>>(v, zinit, ymip, u16 ? 1 : 0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "launch k_init_outputs");
  }

  if (!fast)
    return u16 ? launch_direct<uint16_t>(p, raw, zmip, zsum, ymip, argz, s)
               : launch_direct<float>(p, raw, zmip, zsum, ymip, argz, s);

  ProjArgs args;
  args.v = v;
  args.zmip = zmip;
  args.ymip = ymip;
  args.P = P;
  CUtensorMap map;
  opm_status st = encode_raw(v, raw, P, &map);
  return st == OPM_OK ? launch_fast(p, map, args, s, grid_div) : st;
}

}  // namespace opm
