// Launch-shape selection and instantiation of the fused stage kernel for one
// arithmetic type.  Included once per type by mhd_stage_f64.cu / _f32.cu.
#pragma once

#include "mhd_internal.h"
#include "mhd_stage_pairs.cuh"
#include "mhd_stage_weno.cuh"

namespace mhd {

// Tiles of 3-D grids: columns of TX x TY cells marching in z (mhd_create picks the
// shape).  FP64: one CTA per SM; the SM's FP64 unit is shared by all its warps and
// one warp issues an FP64 instruction at most every 64 clocks, so the unit
// saturates only when at least four warps have FP64 work.  PLM: 32 x 8 or 16 x 16
// (211 KB of shared memory), 16 warps of 128 registers (12 of 168: 256^3 step 46.8
// instead of 44.0 ms).  WENO-Z: 32 x 8 (226 KB), 12 warps (16: 199 instead of 192 ms
// per RK3 step of 256^3), or 32 x 4 with 8 warps.  FP32 (PLM and WENO-Z): 32 x 8
// with 16 warps at 64 registers, two CTAs per SM: the kernels are bound by latency
// and issue; with 24 and 16 warps per SM the PLM kernel took 2 and 8 % longer
// (512^3).  WENO-Z launches that do not fill two CTAs per SM take one of 128
// registers (plan_stage).  2-D grids use the 32 x 8 (PLM) or 32 x 4 (WENO-Z) tile with a single
// plane; 1-D grids a 32-cell row.
template <class T, bool WENO>
constexpr int stage_warps(int ty) {
  return sizeof(T) == 8 && WENO ? (ty == 4 ? 8 : 12) : 16;
}

// Warps of a 1-D tile.  The 36 (38) cells, 34 face states and 33 faces of a 32-cell
// tile take two rounds of one warp, and a warp alone issues an FP64 instruction
// every 64 clocks whether one lane is active or all are: a second warp takes the
// second round at the same time (1024 cells, stages 1 and 2: 24 and 28 us -> 14
// and 17.5 us).  FP32 grids of more tiles than the GPU has schedulers take one
// warp: their schedulers have other tiles to issue from, and the second warp costs
// its own prologue and barriers (PLM, 20 steps: 512 tiles 0.22 ms with two warps,
// 0.25 with one; 1024 tiles 0.27, 0.26; 2048 tiles 0.43, 0.34; eight steps of
// 32768 tiles 1.45, 0.98).
constexpr int kNW1 = 2;
template <class T>
constexpr bool one_warp(const Grid& g) {
  return sizeof(T) == 4 && g.ndim == 1 && (g.n[0] + 31) / 32 > 4 * g.nsm;
}

// The dynamic shared-memory limit of a kernel is set once per device (a
// driver call per launch costs more than a small grid's kernel).  One flag
// word per kernel: the template argument is the kernel itself.
template <auto KERN>
static cudaError_t set_smem_once(size_t smem) {
  static unsigned long long done = 0;  // bit d: set on device d (d < 64)
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) done |= bit;
  return e;
}

template <class T, int TY, int NW, int STAGE, bool ZACT, bool CT = false, bool HALO = false>
static cudaError_t launch_one(const StageParams<T>& p, dim3 grid, cudaStream_t s) {
  using G = TileGeom<TY, ZACT>;
  const size_t smem = (size_t)G::WORDS * sizeof(T);
  auto kern = rk_stage_kernel<T, TY, NW, STAGE, ZACT, CT, HALO>;
  cudaError_t e = set_smem_once<rk_stage_kernel<T, TY, NW, STAGE, ZACT, CT, HALO>>(smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, NW * 32, smem, s>>>(p);
  return cudaGetLastError();
}

template <class T, bool WENO, int TX, int TY>
constexpr size_t smem_3d() {
  if constexpr (sizeof(T) == 4)
    return PairGeom<TY, WENO>::WORDS * sizeof(T);
  else if constexpr (WENO)
    return WenoGeom<TY, true>::WORDS * sizeof(T);
  else
    return TileGeom<TY, true, TX>::WORDS * sizeof(T);
}

// The 3-D stage kernels: FP64 rk_stage_kernel / rk_stage_weno_kernel, FP32
// rk_stage_pairs_kernel (mhd_stage_pairs.cuh).
template <class T, bool WENO, int STAGE, bool CT, bool HALO, int TX = 32, int TY = 8,
          int PER_SM = 2>
struct Kern3D {
  static constexpr int NW = stage_warps<T, WENO>(TY);
  static constexpr auto get() {
    if constexpr (sizeof(T) == 4)
      return rk_stage_pairs_kernel<TY, NW, STAGE, CT, HALO, WENO, PER_SM>;
    else if constexpr (WENO)
      return rk_stage_weno_kernel<T, TY, NW, STAGE, true, CT, HALO>;
    else
      return rk_stage_kernel<T, TY, NW, STAGE, true, CT, HALO, TX>;
  }
  static constexpr auto kernel = get();
  static constexpr size_t smem = smem_3d<T, WENO, TX, TY>();
  static cudaError_t prepare() { return set_smem_once<kernel>(smem); }
  static cudaError_t launch(const StageParams<T>& p, const Grid& g, int nzc, cudaStream_t s) {
    cudaError_t e = prepare();
    if (e != cudaSuccess) return e;
    const dim3 grid((g.n[0] + TX - 1) / TX, (g.n[1] + TY - 1) / TY, nzc);
    kernel<<<grid, NW * 32, smem, s>>>(p);
    return cudaGetLastError();
  }
};
template <class T, bool WENO, bool CT, bool HALO, int TX = 32, int TY = 8, int PER_SM = 2>
static cudaError_t launch_3d(int stage, const StageParams<T>& p, const Grid& g, int nzc,
                             cudaStream_t s) {
  if constexpr (sizeof(T) == 4 && WENO && PER_SM == 2) {
    if (g.per_sm == 1) return launch_3d<T, WENO, CT, HALO, TX, TY, 1>(stage, p, g, nzc, s);
  }
  if (stage == 1) return Kern3D<T, WENO, 1, CT, HALO, TX, TY, PER_SM>::launch(p, g, nzc, s);
  if (stage == 2) return Kern3D<T, WENO, 2, CT, HALO, TX, TY, PER_SM>::launch(p, g, nzc, s);
  return Kern3D<T, WENO, 3, CT, HALO, TX, TY, PER_SM>::launch(p, g, nzc, s);
}
template <class T, bool WENO, bool CT, bool HALO, int TX = 32, int TY = 8, int PER_SM = 2>
static cudaError_t prepare_3d(const Grid& g) {
  if constexpr (sizeof(T) == 4 && WENO && PER_SM == 2) {
    if (g.per_sm == 1) return prepare_3d<T, WENO, CT, HALO, TX, TY, 1>(g);
  }
  cudaError_t e = Kern3D<T, WENO, 1, CT, HALO, TX, TY, PER_SM>::prepare();
  if (e == cudaSuccess) e = Kern3D<T, WENO, 2, CT, HALO, TX, TY, PER_SM>::prepare();
  if (e == cudaSuccess) e = Kern3D<T, WENO, 3, CT, HALO, TX, TY, PER_SM>::prepare();
  return e;
}
// The FP32 kernels without halo faces address a plane with 32 bits; larger planes
// take the halo-capable ones.  (With constrained transport such a grid needs
// over 300 GB: it never reaches a launch.)
template <class T>
static bool wide_plane(const Grid& g) {
  return sizeof(T) == 4 && (long long)g.n[0] * g.n[1] * 4 >= (1ll << 32);
}

template <class T, int TY, int NW, int STAGE, bool ZACT, bool CT = false, bool HALO = false>
static cudaError_t launch_weno(const StageParams<T>& p, dim3 grid, cudaStream_t s) {
  using G = WenoGeom<TY, ZACT>;
  const size_t smem = (size_t)G::WORDS * sizeof(T);
  auto kern = rk_stage_weno_kernel<T, TY, NW, STAGE, ZACT, CT, HALO>;
  cudaError_t e = set_smem_once<rk_stage_weno_kernel<T, TY, NW, STAGE, ZACT, CT, HALO>>(smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, NW * 32, smem, s>>>(p);
  return cudaGetLastError();
}

template <class T>
void stage_shape(const Grid& g, size_t* smem, int* warps) {
  const bool weno = g.limiter == kLimWenoz;
  if (g.ndim == 3) {
    *warps = weno ? stage_warps<T, true>(g.ty) : stage_warps<T, false>(g.ty);
    *smem = weno ? (g.ty == 4 ? smem_3d<T, true, 32, 4>() : smem_3d<T, true, 32, 8>())
                 : (g.tx == 16 ? smem_3d<T, false, 16, 16>() : smem_3d<T, false, 32, 8>());
  } else if (g.ndim == 2) {
    *warps = 8;
    *smem = (weno ? WenoGeom<4, false>::WORDS : TileGeom<8, false>::WORDS) * sizeof(T);
  } else {
    *warps = one_warp<T>(g) ? 1 : kNW1;
    *smem = (weno ? WenoGeom<1, false>::WORDS : TileGeom<1, false>::WORDS) * sizeof(T);
  }
}

// Sets the shared-memory limit of every stage-kernel variant a grid launches
// (stages 1, 2, 3; constrained transport or not), so that no launch needs the
// driver call later, e.g. while a stream is being captured.
template <class T>
cudaError_t prepare_stage_kernels(const Grid& g, bool ct) {
  const bool weno = g.limiter == kLimWenoz;
  if constexpr (sizeof(T) == 8) {
    if (ct && g.ty == 4) return prepare_3d<T, true, true, false, 32, 4>(g);
  }
  if (ct) return weno ? prepare_3d<T, true, true, false>(g) : prepare_3d<T, false, true, false>(g);
  if (g.ndim == 3) {
    // FP64, and planes beyond 32-bit offsets: the halo-capable kernels (launch_stage)
    if (sizeof(T) == 8 || wide_plane<T>(g)) return prepare_stage_kernels_halo<T>(g);
    if constexpr (sizeof(T) == 4)
      return weno ? prepare_3d<T, true, false, false>(g) : prepare_3d<T, false, false, false>(g);
  }
  cudaError_t e = cudaSuccess;
  // the three stages of one variant <TY, NW> with geometry G
#define MHD_SET1(KERN, G, TY_, NW_, S_) \
  if (e == cudaSuccess) e = set_smem_once<KERN<T, TY_, NW_, S_, false, false>>((size_t)G::WORDS * sizeof(T))
#define MHD_SET3(KERN, G, TY_, NW_) \
  MHD_SET1(KERN, G, TY_, NW_, 1);   \
  MHD_SET1(KERN, G, TY_, NW_, 2);   \
  MHD_SET1(KERN, G, TY_, NW_, 3)
  using W2 = WenoGeom<4, false>;
  using W1 = WenoGeom<1, false>;
  using P2 = TileGeom<8, false>;
  using P1 = TileGeom<1, false>;
  if constexpr (sizeof(T) == 4) {
    if (weno && g.warps == 1) {
      MHD_SET3(rk_stage_weno_kernel, W1, 1, 1);
      return e;
    }
    if (g.warps == 1) {
      MHD_SET3(rk_stage_kernel, P1, 1, 1);
      return e;
    }
  }
  if (weno && g.ndim == 2) {
    MHD_SET3(rk_stage_weno_kernel, W2, 4, 8);
  } else if (weno) {
    MHD_SET3(rk_stage_weno_kernel, W1, 1, kNW1);
  } else if (g.ndim == 2) {
    MHD_SET3(rk_stage_kernel, P2, 8, 8);
  } else {
    MHD_SET3(rk_stage_kernel, P1, 1, kNW1);
  }
#undef MHD_SET3
#undef MHD_SET1
  return e;
}

// Kernel parameters shared by launch_stage and launch_stage_halo; returns
// cudaErrorInvalidValue for a bad z range.
template <class T>
static cudaError_t stage_params(StageParams<T>& p, const Grid& g, const T* win,
                                const T* un, T* uout, const StepScalars* sc,
                                unsigned long long* lam_bits, unsigned long long* floor_cnt,
                                double a_n, double a_w, int zlo, int zhi, int tz,
                                unsigned int* est_bits) {
  p.a_n = T(a_n);
  p.a_w = T(a_w);
  p.win = win;
  p.un = un;
  p.uout = uout;
  for (int d = 0; d < 3; ++d) {
    p.n[d] = g.n[d];
    p.bc_lo[d] = g.bc_lo[d];
    p.bc_hi[d] = g.bc_hi[d];
  }
  p.sy = g.n[0];
  p.sz = (long long)g.n[0] * g.n[1];
  p.sv = g.ncell;
  p.limiter = g.limiter;
  p.tz = g.ndim == 3 ? (tz > 0 ? tz : g.tz) : 1;
  p.zlo = g.ndim == 3 ? zlo : 0;
  p.zhi = g.ndim == 3 && zhi >= 0 ? zhi : g.n[2];
  if (p.zlo < 0 || p.zhi > g.n[2] || p.zlo >= p.zhi) return cudaErrorInvalidValue;
  p.ph = make_phys<T>(g);
  p.sc = sc;
  p.lam_bits = lam_bits;
  p.est_bits = est_bits;
  p.floor_cnt = floor_cnt;
  for (int d = 0; d < 3; ++d) p.bw[d] = nullptr;
  p.ctf = nullptr;
  for (int f = 0; f < 6; ++f) p.halo[f] = nullptr;
  return cudaSuccess;
}

template <class T>
cudaError_t launch_stage(const Grid& g, int stage, const T* win, const T* un, T* uout,
                         const StepScalars* sc, unsigned long long* lam_bits,
                         unsigned long long* floor_cnt, cudaStream_t stream, double a_n,
                         double a_w, const T* const* bw, T* ctf, int zlo, int zhi, int tz,
                         unsigned int* est_bits) {
  StageParams<T> p;
  cudaError_t pe = stage_params(p, g, win, un, uout, sc, lam_bits, floor_cnt, a_n, a_w, zlo,
                                zhi, tz, est_bits);
  if (pe != cudaSuccess) return pe;
  const int nzc = (p.zhi - p.zlo + p.tz - 1) / p.tz;  // z chunks of this launch
  // the FP64 last stage publishes the maximum speed estimate (speed_exact
  // finishes the maximum); it needs the estimate word
  if (sizeof(T) == 8 && stage == 2 && !ctf && !est_bits) return cudaErrorInvalidValue;
  for (int d = 0; d < 3; ++d) p.bw[d] = bw ? bw[d] : nullptr;
  p.ctf = ctf;
  if (ctf) {
    // constrained transport: 3-D grids only (checked when the context is made)
    if (g.ndim != 3 || !bw) return cudaErrorInvalidValue;
    if constexpr (sizeof(T) == 8) {
      if (g.ty == 4) return launch_3d<T, true, true, false, 32, 4>(stage, p, g, nzc, stream);
    }
    return g.limiter == kLimWenoz ? launch_3d<T, true, true, false>(stage, p, g, nzc, stream)
                                  : launch_3d<T, false, true, false>(stage, p, g, nzc, stream);
  }
  if (g.ndim == 3) {
    // FP64 GLM: always the halo-capable kernels (no halo faces here), so that a
    // grid and the blocks of its decomposition run the same code; FP32 where a
    // plane is too large for 32-bit offsets
    if (sizeof(T) == 8 || wide_plane<T>(g))
      return launch_stage_halo<T>(g, stage, win, un, uout, sc, lam_bits, floor_cnt, stream, a_n,
                                  a_w, nullptr, est_bits, zlo, zhi, tz);
    if constexpr (sizeof(T) == 4)
      return g.limiter == kLimWenoz ? launch_3d<T, true, false, false>(stage, p, g, nzc, stream)
                                    : launch_3d<T, false, false, false>(stage, p, g, nzc, stream);
  }
  if (g.limiter == kLimWenoz) {
    if (g.ndim == 2) {
      dim3 grid((g.n[0] + 31) / 32, (g.n[1] + 3) / 4, 1);
      if (stage == 1) return launch_weno<T, 4, 8, 1, false>(p, grid, stream);
      if (stage == 2) return launch_weno<T, 4, 8, 2, false>(p, grid, stream);
      return launch_weno<T, 4, 8, 3, false>(p, grid, stream);
    }
    dim3 grid((g.n[0] + 31) / 32, 1, 1);
    if constexpr (sizeof(T) == 4) {
      if (g.warps == 1) {
        if (stage == 1) return launch_weno<T, 1, 1, 1, false>(p, grid, stream);
        if (stage == 2) return launch_weno<T, 1, 1, 2, false>(p, grid, stream);
        return launch_weno<T, 1, 1, 3, false>(p, grid, stream);
      }
    }
    if (stage == 1) return launch_weno<T, 1, kNW1, 1, false>(p, grid, stream);
    if (stage == 2) return launch_weno<T, 1, kNW1, 2, false>(p, grid, stream);
    return launch_weno<T, 1, kNW1, 3, false>(p, grid, stream);
  }
  if (g.ndim == 2) {
    dim3 grid((g.n[0] + 31) / 32, (g.n[1] + 7) / 8, 1);
    if (stage == 1) return launch_one<T, 8, 8, 1, false>(p, grid, stream);
    if (stage == 2) return launch_one<T, 8, 8, 2, false>(p, grid, stream);
    return launch_one<T, 8, 8, 3, false>(p, grid, stream);
  }
  dim3 grid((g.n[0] + 31) / 32, 1, 1);
  if constexpr (sizeof(T) == 4) {
    if (g.warps == 1) {
      if (stage == 1) return launch_one<T, 1, 1, 1, false>(p, grid, stream);
      if (stage == 2) return launch_one<T, 1, 1, 2, false>(p, grid, stream);
      return launch_one<T, 1, 1, 3, false>(p, grid, stream);
    }
  }
  if (stage == 1) return launch_one<T, 1, kNW1, 1, false>(p, grid, stream);
  if (stage == 2) return launch_one<T, 1, kNW1, 2, false>(p, grid, stream);
  return launch_one<T, 1, kNW1, 3, false>(p, grid, stream);
}

// Halo faces (3-D GLM grids with kBcHalo sides): the HALO variants of the
// 3-D stage kernels, the ghost cells of those sides read from halo[f].
// Instantiated in mhd_stage_halo_f64.cu / _f32.cu only.
template <class T>
cudaError_t launch_stage_halo(const Grid& g, int stage, const T* win, const T* un, T* uout,
                              const StepScalars* sc, unsigned long long* lam_bits,
                              unsigned long long* floor_cnt, cudaStream_t stream, double a_n,
                              double a_w, const T* const* halo, unsigned int* est_bits, int zlo,
                              int zhi, int tz) {
  if (g.ndim != 3) return cudaErrorInvalidValue;
  StageParams<T> p;
  cudaError_t pe = stage_params(p, g, win, un, uout, sc, lam_bits, floor_cnt, a_n, a_w, zlo, zhi,
                                tz, est_bits);
  if (pe != cudaSuccess) return pe;
  if (sizeof(T) == 8 && stage == 2 && !est_bits) return cudaErrorInvalidValue;
  for (int f = 0; f < 6; ++f) {
    const bool lo = (f & 1) == 0;
    const int bc = lo ? g.bc_lo[f >> 1] : g.bc_hi[f >> 1];
    if (bc == kBcHalo && (!halo || !halo[f])) return cudaErrorInvalidValue;
    p.halo[f] = bc == kBcHalo ? halo[f] : nullptr;
  }
  const int nzc = (p.zhi - p.zlo + p.tz - 1) / p.tz;
  if constexpr (sizeof(T) == 8) {
    if (g.tx == 16) return launch_3d<T, false, false, true, 16, 16>(stage, p, g, nzc, stream);
    if (g.ty == 4) return launch_3d<T, true, false, true, 32, 4>(stage, p, g, nzc, stream);
  }
  return g.limiter == kLimWenoz ? launch_3d<T, true, false, true>(stage, p, g, nzc, stream)
                                : launch_3d<T, false, false, true>(stage, p, g, nzc, stream);
}

// The shared-memory limits of the HALO variants (set once, outside any capture).
template <class T>
cudaError_t prepare_stage_kernels_halo(const Grid& g) {
  if constexpr (sizeof(T) == 8) {
    if (g.tx == 16) return prepare_3d<T, false, false, true, 16, 16>(g);
    if (g.ty == 4) return prepare_3d<T, true, false, true, 32, 4>(g);
  }
  return g.limiter == kLimWenoz ? prepare_3d<T, true, false, true>(g)
                                : prepare_3d<T, false, false, true>(g);
}

}  // namespace mhd
