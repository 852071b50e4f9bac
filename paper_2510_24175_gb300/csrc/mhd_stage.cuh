// Fused Runge-Kutta stage kernel: one launch performs, for its tile of cells,
// the five per-stage steps of Section 3.2 (boundary calculation,
// cons->prim, reconstruction, Riemann solver, right-hand side) and the
// Runge-Kutta combination.  STAGE 1: out = W + dt L(W); STAGE 2 (last stage):
// out = a_n U^n + a_w (W + dt L(W)), then the GLM damping (Mignone &
// Tzeferacos 2010, Eq. 27) and the next step's max-wave-speed reduction;
// STAGE 3 (SSP-RK3 middle stage): the combination without the epilogue.
//
// Decomposition: a CTA owns a TX x TY column tile in (x, y) (32 x 8 or 16 x 16 in
// 3-D) and marches in z over p.tz planes.  Ghost zones are never stored: the boundary calculation
// is an index remap at load time (periodic: wrap; outflow: clamp to the
// nearest interior cell), so the state arrays are interior-only SoA.
//
// Per plane k, four phases separated by CTA barriers:
//   A  load + cons->prim: the tile interior of plane k+2 (into a 3-plane
//      ring) and the (x, y) halo of plane k (into halo buffers);
//   B  limited slopes, each cell and direction once: x slopes of the 34
//      cells per row, y slopes of the TY+2 rows, and -- by the thread that
//      owns the column -- the z slope of cell k+1;
//   C  face fluxes (PLM face states V -/+ sigma/2, GLM, HLLD), each face of
//      the tile once, warp-uniform direction; the column owner also computes
//      the z face k+1/2 and keeps the z data (slope, face state, flux) of its
//      column in per-owner shared slots across planes;
//   D  the column owner applies the flux divergence and the RK combination.
//
// This kernel runs FP64 grids and the 1-D and 2-D FP32 ones (3-D FP32:
// mhd_stage_pairs.cuh).  In FP64 it is bound by the SM's FP64 unit, 88 % of whose
// cycles it uses (Orszag-Tang 256^3, a step of two stages 45.0 ms); the sums,
// differences and products run as fused multiply-adds on register operands (add_f),
// and in 3-D phase D of a plane runs at the same time as A and B of the next (kRoles).
#pragma once

#include "mhd_physics.cuh"

namespace mhd {

// Per-step scalars written on the device by the step-prepare kernel.
struct StepScalars {
  double dt;         // time step of the step in progress
  double ch;         // GLM cleaning speed c_h
  double dtdx[3];    // dt / dx_d
  double damp;       // exp(-alpha c_h dt / dh_min)
  double t;          // time after this step
  double lam;        // max wave speed the step's dt was taken from
  double steps;      // number of steps since set_state
};

template <class T>
struct StageParams {
  const T* win;   // stage input W (U^n or U1)
  const T* un;    // U^n (stage 2); may alias uout
  T* uout;        // stage output
  int n[3];
  long long sy, sz, sv;  // strides of y, z, var in elements
  int bc_lo[3], bc_hi[3];
  int limiter;
  int tz;         // planes per CTA
  int zlo, zhi;   // z planes [zlo, zhi) of this launch (blockIdx.z counts tz-plane chunks)
  T a_n, a_w;     // combining stages: out = a_n U^n + a_w (W + dt L(W))
  Phys<T> ph;
  const StepScalars* sc;
  unsigned long long* lam_bits;   // stage 2: max wave speed as FP64 bits (FP32 path)
  unsigned int* est_bits;         // stage 2, FP64: max reliable FP32 speed estimate
  unsigned long long* floor_cnt;  // [3] floor activations (see count_floors)
  // constrained transport (kernels instantiated with CT = true)
  const T* bw[3];  // the stage input's face field: b_d on each cell's lower d-face
  T* ctf;          // kCtPlanes planes of ncell values (layout below)
  // halo faces (kernels instantiated with HALO = true): ghost cells beyond a
  // side whose bc is kBcHalo, per face x-, x+, y-, y+, z-, z+ (layout at
  // halo_cell below)
  const T* halo[6];
};

// HALO kernels: the address of variable 0 of cell (i, j, k) of the stage
// input and the variable stride, for indices up to GH cells outside the grid
// (GH = ghost width: 2 for PLM, 3 for WENO-Z).  A cell beyond a kBcHalo side
// comes from that face's halo buffer, which has the grid's SoA layout over
// the ghost slab: extent GH along the face normal (layer l = ghost index + GH
// on the low side, ghost index - n on the high side), the grid's extents
// along the two others.  Other out-of-range indices wrap (periodic) or clamp
// (outflow) as in remap().  The stage kernels never use a cell outside the
// grid along two axes at once, so when the chosen face's tangential indices
// are out of range the load is of an unused value and is clamped into the
// buffer; indices beyond n + GH - 1 (the unused part of a ragged tile) are
// folded first.  Every load stays in bounds.
template <int GH, class T>
__device__ __forceinline__ const T* halo_cell(const StageParams<T>& p, int i, int j, int k,
                                              long long& sv) {
  const int n0 = p.n[0], n1 = p.n[1], n2 = p.n[2];
  i = min(i, n0 + GH - 1);
  j = min(j, n1 + GH - 1);
  k = min(k, n2 + GH - 1);
  int f = -1, l = 0;
  if (k < 0 && p.bc_lo[2] == kBcHalo) {
    f = 4;
    l = k + GH;
  } else if (k >= n2 && p.bc_hi[2] == kBcHalo) {
    f = 5;
    l = k - n2;
  } else if (j < 0 && p.bc_lo[1] == kBcHalo) {
    f = 2;
    l = j + GH;
  } else if (j >= n1 && p.bc_hi[1] == kBcHalo) {
    f = 3;
    l = j - n1;
  } else if (i < 0 && p.bc_lo[0] == kBcHalo) {
    f = 0;
    l = i + GH;
  } else if (i >= n0 && p.bc_hi[0] == kBcHalo) {
    f = 1;
    l = i - n0;
  }
  if (f < 0) {
    auto wrap = [](int x, int n, int lo, int hi) {
      if (x < 0) return lo == kBcPeriodic ? x + n : 0;
      if (x >= n) return hi == kBcPeriodic ? x - n : n - 1;
      return x;
    };
    const int gx = wrap(i, n0, p.bc_lo[0], p.bc_hi[0]);
    const int gy = wrap(j, n1, p.bc_lo[1], p.bc_hi[1]);
    const int gz = wrap(k, n2, p.bc_lo[2], p.bc_hi[2]);
    sv = p.sv;
    return p.win + (long long)gz * p.sz + (long long)gy * p.sy + gx;
  }
  const int d = f >> 1;
  const int c0 = d == 0 ? l : min(max(i, 0), n0 - 1);
  const int c1 = d == 1 ? l : min(max(j, 0), n1 - 1);
  const int c2 = d == 2 ? l : min(max(k, 0), n2 - 1);
  const int e0 = d == 0 ? GH : n0, e1 = d == 1 ? GH : n1;
  const int e2 = d == 2 ? GH : n2;
  sv = (long long)e0 * e1 * e2;
  return p.halo[f] + ((long long)c2 * e1 + c1) * e0 + c0;
}

// Planes of the constrained-transport buffer written by a CT stage kernel,
// per cell: the electric field E = -v x B on the cell's lower x, y and z
// faces (the two components after the face normal in cyclic order, from the
// face flux: on a d-face E_{d+1} = F[B_{d+2}] and E_{d+2} = -F[B_{d+1}]), the
// mass flux through each of those faces (set to zero when
// |F_rho| <= delta c_h rho, delta = 1e-12 in FP64 and 1e-4 in FP32, so that
// round-off cannot pick an upwind side), and the cell-centred E.
enum : int {
  kCtXEy = 0, kCtXEz, kCtXFm, kCtYEz, kCtYEx, kCtYFm, kCtZEx, kCtZEy, kCtZFm,
  kCtEcx, kCtEcy, kCtEcz, kCtPlanes
};

template <class T>
__device__ __forceinline__ T ct_mass_flux(T f, T rho, T ch) {
  const T thr = T(sizeof(T) == 8 ? 1e-12 : 1e-4) * ch * rho;
  return tabs(f) > thr ? f : T(0);
}

// Constrained-transport data of the cell a column owner updates: the
// cell-centred E and rho (read in phase C, before the next plane's loads may
// reuse the ring slot) and the z flux through the cell's lower face.
template <class T>
struct CtCell {
  T ex, ey, ez, rho;
  T fz_bx, fz_by, fz_rho;
  __device__ __forceinline__ void from_prims(const T* v, int st) {
    const T vx = v[kVX * st], vy = v[kVY * st], vz = v[kVZ * st];
    const T bx = v[kBX * st], by = v[kBY * st], bz = v[kBZ * st];
    ex = fma_rn(vz, by, -mul_rn(vy, bz));
    ey = fma_rn(vx, bz, -mul_rn(vz, bx));
    ez = fma_rn(vy, bx, -mul_rn(vx, by));
    rho = v[kRHO * st];
  }
  // fx / fy: the x and y fluxes of the cell's lower faces (variables sx / sy
  // apart)
  __device__ __forceinline__ void write(T* ctf, long long sv, long long off, const T* fx,
                                        int sx, const T* fy, int sy, T ch) const {
    ctf[kCtXEy * sv + off] = fx[kBZ * sx];
    ctf[kCtXEz * sv + off] = -fx[kBY * sx];
    ctf[kCtXFm * sv + off] = ct_mass_flux(fx[kRHO * sx], rho, ch);
    ctf[kCtYEz * sv + off] = fy[kBX * sy];
    ctf[kCtYEx * sv + off] = -fy[kBZ * sy];
    ctf[kCtYFm * sv + off] = ct_mass_flux(fy[kRHO * sy], rho, ch);
    ctf[kCtZEx * sv + off] = fz_by;
    ctf[kCtZEy * sv + off] = -fz_bx;
    ctf[kCtZFm * sv + off] = ct_mass_flux(fz_rho, rho, ch);
    ctf[kCtEcx * sv + off] = ex;
    ctf[kCtEcy * sv + off] = ey;
    ctf[kCtEcz * sv + off] = ez;
  }
};

// Constrained transport: both sides of a d-face carry the staggered normal
// field and psi = 0 (the GLM interface step is then the identity).
template <class T>
__device__ __forceinline__ void ct_face_field(T vl[kNV], T vr[kNV], int d, T bn) {
  vl[kBX + d] = vr[kBX + d] = bn;
  vl[kPSI] = vr[kPSI] = T(0);
}

// Remaps a possibly out-of-range index (>= -2) into [0, n): periodic wraps,
// outflow clamps.  Indices beyond n+1 only occur in the unused part of a
// ragged tile and are folded to n+1 first, so every load stays in bounds.
__host__ __device__ __forceinline__ int remap(int i, int n, int lo, int hi) {
  i = min(i, n + 1);
  if (i < 0) return lo == kBcPeriodic ? i + n : 0;
  if (i >= n) return hi == kBcPeriodic ? i - n : n - 1;
  return i;
}

// Same for a three-cell-deep halo (WENO-Z; active dimensions need n >= 3).
__host__ __device__ __forceinline__ int remap3(int i, int n, int lo, int hi) {
  i = min(i, n + 2);
  if (i < 0) return lo == kBcPeriodic ? i + n : 0;
  if (i >= n) return hi == kBcPeriodic ? i - n : n - 1;
  return i;
}

template <int TY, bool ZACT, int TX_ = 32>
struct TileGeom {
  static constexpr int TX = TX_;
  static constexpr int GY = TY > 1 ? 2 : 0;
  static constexpr int NINT = TY * TX;             // interior cells per plane
  static constexpr int NXH = 4 * TY;               // x halo: columns -2, -1, 32, 33
  static constexpr int NYH = GY ? 4 * TX : 0;      // y halo: rows -2, -1, TY, TY+1
  static constexpr int NRING = ZACT ? 3 : 1;
  // shared-memory words
  // Variable stride PS of the ring slots and of the halo buffer: the x and y
  // halo cells share one buffer (x halo items first, then y halo items) with
  // the ring's stride, so every cell of the current plane is reached at a
  // compile-time stride; PS = NINT unless the halo cells are more (TY = 4)
  static constexpr int PS = NINT > NXH + NYH ? NINT : NXH + NYH;
  static constexpr int RING_W = NRING * kNV * PS;
  static constexpr int HB_W = kNV * PS;
  static constexpr int SXN = TY * (TX + 2);         // x slopes, columns -1..32
  static constexpr int SYN = GY ? (TY + 2) * TX : 0;  // y slopes, rows -1..TY
  static constexpr int FXN = TY * (TX + 1);
  static constexpr int FYN = GY ? (TY + 1) * TX : 0;
  static constexpr int Z_W = ZACT ? 3 * kNV * NINT : 0;  // z slope, z face state, z flux
  static constexpr int WORDS =
      RING_W + HB_W + kNV * SXN + kNV * SYN + kNV * FXN + kNV * FYN + Z_W;
  // phase-A items: interior, x halo, y halo
  static constexpr int NLOAD = NINT + NXH + NYH;
  // phase-C flux items [x main][y][x right edge], each segment starting on a warp:
  // a warp with both directions would run both fluxes one after the other, last
  // (16 x 16 tiles without that: 256^3 step 50.9 instead of 46.4 ms)
  static constexpr int IT_X = TY * TX;
  static constexpr int IT_Y = FYN;
  static constexpr int IT_XE0 = IT_X + (IT_Y + 31) / 32 * 32;
  static constexpr int ITEMS = IT_XE0 + TY;
};

// Half slopes of the 9 primitives of one cell from its two neighbours along a
// direction, 0 for all of them when a face density or pressure would be
// non-positive.  m, c, p: the cells (variables sm, sc, sp apart); h: variables
// sh apart.
template <class T>
__device__ __forceinline__ void cell_slopes(const T* m, int sm, const T* c, int sc, const T* p,
                                            int sp, int lim, const Phys<T>& ph, T* h, int sh) {
  T sig[kNV];
  if (lim == kLimMC) {
#pragma unroll
    for (int k = 0; k < kNV; ++k) {
      const T q = c[k * sc];
      sig[k] = half_slope_mc(sub_f(q, m[k * sm], ph), sub_f(p[k * sp], q, ph), ph);
    }
  } else if (lim == kLimMinmod) {
#pragma unroll
    for (int k = 0; k < kNV; ++k) {
      const T q = c[k * sc];
      sig[k] = half_slope_minmod(sub_f(q, m[k * sm], ph), sub_f(p[k * sp], q, ph));
    }
  } else {
#pragma unroll
    for (int k = 0; k < kNV; ++k) sig[k] = T(0);
  }
  const bool ok = gt0(sub_f(c[kRHO * sc], tabs(sig[kRHO]), ph)) &&
                  gt0(sub_f(c[kPRS * sc], tabs(sig[kPRS]), ph));
  if (!ok) {
#pragma unroll
    for (int k = 0; k < kNV; ++k) sig[k] = T(0);
  }
#pragma unroll
  for (int k = 0; k < kNV; ++k) h[k * sh] = sig[k];
}

// Named CTA barriers: n threads in all arrive or wait at barrier id.
__device__ __forceinline__ void bar_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// One tile (bx, by, bz) of one RK stage; called by every thread of a CTA of
// NW warps.  smem_raw: TileGeom::WORDS elements of T; wmax: NW doubles,
// konst (FP64): 4 doubles.
// CT (constrained transport, 3-D only): face-normal fields from p.bw, only
// rho, m and E are updated (psi is written as 0; the magnetic field is left to
// the face update), the face / cell electric fields go to p.ctf, and the last
// stage has no damping and no wave-speed reduction (done after the face update).
// HALO (3-D, not CT): ghost cells of kBcHalo sides from p.halo (halo_cell).
template <class T, int TY, int NW, int STAGE, bool ZACT, bool CT = false, bool HALO = false,
          int TX_ = 32>
__device__ __forceinline__ void stage_tile(const StageParams<T>& p, const StepScalars& sc,
                                           int bx, int by, int bz, unsigned char* smem_raw,
                                           double* wmax, double* konst = nullptr) {
  using G = TileGeom<TY, ZACT, TX_>;
  constexpr int NT = NW * 32;
  constexpr int TX = G::TX;
  constexpr int ZT0 = NT - G::NINT;  // threads ZT0.. own one tile column each
  static_assert(ZT0 >= 0, "need one thread per tile column");
  T* ring = reinterpret_cast<T*>(smem_raw);
  T* xh = ring + G::RING_W;  // x halo items (variable stride G::PS)
  T* yh = xh + G::NXH;        // y halo items (same buffer and stride)
  T* sxs = xh + G::HB_W;
  T* sys = sxs + kNV * G::SXN;
  T* Fx = sys + kNV * G::SYN;
  T* Fy = Fx + kNV * G::FXN;
  T* zS = Fy + kNV * G::FYN;  // per owner: z half slope of cell k+1
  T* zP = zS + kNV * G::NINT;  // per owner: face state V_k + sigma_k / 2
  T* zF = zP + kNV * G::NINT;  // per owner: z flux at face k-1/2

  const int tid = threadIdx.x;
  const int x0 = bx * TX;
  const int y0 = by * TY;
  const int z0 = p.zlo + bz * p.tz;
  const int z1 = min(z0 + p.tz, p.zhi);
  const int nx = p.n[0], ny = p.n[1], nz = p.n[2];
  const bool owner = tid >= ZT0;
  const int oidx = tid - ZT0;  // owned column = interior cell index r * TX + c
  const int orow = oidx / TX, ocol = oidx - (oidx / TX) * TX;

  const T ch = T(sc.ch);
  const T half_chi = T(0.5 / sc.ch);
  const T dtdx = T(sc.dtdx[0]), dtdy = T(sc.dtdx[1]), dtdz = T(sc.dtdx[2]);
  const T damp = T(sc.damp);
  // dt == 0 (a step at t_end, or one the prepare kernel turned into a no-op
  // after a non-finite wave speed): the state is copied through unchanged,
  // even where fluxes are not finite
  const bool frozen = !(sc.dt != 0.0);
  const int lim = p.limiter;
  Phys<T> ph = p.ph;
  if constexpr (TY > 1) {
    fp64_registers(ph, konst);
  } else {  // 1-D kernels wait for latency: the plain operations
    ph.one = T(1);
    ph.nzero = T(-0.0);
  }
  unsigned flags = 0;  // of the wave-speed conversions (not counted)

  auto slot = [](int zz) { return ZACT ? ((zz % 3) + 3) % 3 : 0; };
  auto ring_plane = [&](int zz) { return ring + slot(zz) * (kNV * G::PS); };

  // Floor activations are counted once per stage for each cell the tile
  // updates, from that cell's own conversion of the stage input; halo copies
  // converted by neighbouring tiles are not counted, so the counts do not
  // depend on the decomposition.  Rare: one atomic per flagged cell.
  auto count_floors = [&](unsigned fl, int zz, int r, int c) {
    if (zz < z0 || zz >= z1 || x0 + c >= nx || (G::GY && y0 + r >= ny)) return;
    if (fl & kFloorRho) atomicAdd(&p.floor_cnt[0], 1ull);
    if (fl & kFloorP) atomicAdd(&p.floor_cnt[1], 1ull);
    if (fl & kPressF64) atomicAdd(&p.floor_cnt[2], 1ull);
  };
  // offset of tile cell (r, c) of plane zz, remapped into the grid
  auto cell_off = [&](int zz, int r, int c) {
    const int gz = ZACT ? remap(zz, nz, p.bc_lo[2], p.bc_hi[2]) : 0;
    const int gx = remap(x0 + c, nx, p.bc_lo[0], p.bc_hi[0]);
    const int gy = G::GY ? remap(y0 + r, ny, p.bc_lo[1], p.bc_hi[1]) : 0;
    return (long long)gz * p.sz + (long long)gy * p.sy + gx;
  };
  // cons -> prim of cell (r, c) of plane zz into dst (variables dst_stride
  // apart); own: an interior item of the tile (counted if the tile updates it)
  auto load_cell = [&](int zz, int r, int c, T* dst, int dst_stride, bool own) {
    T u[kNV], v[kNV];
    if constexpr (HALO) {
      long long hs;
      const T* a = halo_cell<2>(p, x0 + c, y0 + r, zz, hs);
#pragma unroll
      for (int k = 0; k < kNV; ++k) u[k] = a[k * hs];
    } else {
      const long long off = cell_off(zz, r, c);
#pragma unroll
      for (int k = 0; k < kNV; ++k) u[k] = p.win[k * p.sv + off];
    }
    unsigned fl = 0;
    cons_to_prim(u, v, ph, fl);
    if (fl && own) count_floors(fl, zz, r, c);
#pragma unroll
    for (int k = 0; k < kNV; ++k) dst[k * dst_stride] = v[k];
  };
  // phase-A item: interior cell of plane zi or halo cell of plane zh
  auto load_item = [&](int it, int zi, int zh) {
    if (it < G::NINT) {
      const int r = it / TX, c = it - (it / TX) * TX;
      load_cell(zi, r, c, ring_plane(zi) + it, G::PS, true);
    } else if (it < G::NINT + G::NXH) {
      const int j = it - G::NINT;
      const int r = j >> 2, q = j & 3;
      const int c = q < 2 ? q - 2 : TX + q - 2;
      load_cell(zh, r, c, xh + j, G::PS, false);
    } else {
      const int j = it - G::NINT - G::NXH;
      const int hr = j / TX, c = j - (j / TX) * TX;
      const int r = hr < 2 ? hr - 2 : TY + hr - 2;
      load_cell(zh, r, c, yh + j, G::PS, false);
    }
  };
  // primitives of cell (r, c) of the current plane (interior in the ring slot,
  // halo in the halo buffers; variables G::PS apart)
  auto cell_ptr = [&](const T* cur, int r, int c) -> const T* {
    if (c < 0 || c >= TX) return xh + r * 4 + (c < 0 ? c + 2 : c - TX + 2);
    if (r < 0 || r >= TY) return yh + (r < 0 ? r + 2 : r - TY + 2) * TX + c;
    return cur + r * TX + c;
  };
  static_assert(sizeof(T) == 8 || !ZACT, "3-D FP32: mhd_stage_pairs.cuh");
  static_assert(!CT || ZACT, "constrained transport is 3-D only");
  static_assert(!HALO || (ZACT && !CT), "halo faces: 3-D GLM kernels only");
  // staggered normal field on the lower d-face of tile cell (r, c) of plane zz
  auto bface = [&](int d, int zz, int r, int c) -> T {
    return p.bw[d][cell_off(zz, r, c)];
  };
  CtCell<T> ctc;

  // The z march: one loop body for every plane, so that each cell's
  // conversion, slopes and z fluxes come from the same code wherever a z
  // chunk (or a block of a decomposed grid, or a launch's z range) starts --
  // a cell's result must not depend on that decomposition.  Iterations
  // k < z0 warm up: k = z0-4 and z0-3 only load planes z0-2 and z0-1 into the
  // ring, k = z0-2 sets the column owners' face state of cell z0-1, k = z0-1
  // their flux through face z0-1/2; the x, y work and the update start at
  // k = z0.  (Unrolling, and with it the peeling of warm-up iterations into
  // separate copies, is disabled.)
  constexpr int NWARM = ZACT ? 4 : 0;
  // 3-D tiles with as many other threads as owners: the owners' z slopes and
  // update (D) run at the same time as the others' loads and x, y slopes, so
  // the FP64 unit has work while loads are in flight (256^3 step 46.3 -> 44.0 ms;
  // with all slopes left to the others, whose last round is of two warps, 44.8)
  constexpr bool kRoles = ZACT && ZT0 >= G::NINT;
  SpeedMax<T> smax(ph);  // last stage: the new state's maximum wave speed
#pragma unroll 1
  for (int k = z0 - NWARM; k < z1; ++k) {
    const bool main = k >= z0;
    // ---- A: loads ---------------------------------------------------------
    // kRoles: the column owners are still in phase D of plane k-1 (it shares no
    // data with A and B) when the other warps load and go on to the slopes
    const bool roles = kRoles && main;
    const int step = roles ? ZT0 : NT;
    const int nload = main ? G::NLOAD : G::NINT;
    for (int it = roles && owner ? nload : tid; it < nload; it += step) {
      if (ZACT && it < G::NINT)
        load_item(it, k + 2, k);
      else
        load_item(it, k, k);
    }
    if (!roles) {
      __syncthreads();
    } else if (owner) {
      bar_sync(2, NT);  // the loads are done
    } else {
      bar_arrive(2, NT);
      bar_sync(1, ZT0);
    }
    if (ZACT && k < z0 - 2) continue;
    const T* cur = ring_plane(k);

    // ---- B: slopes --------------------------------------------------------
    constexpr int kSlopes = G::SXN + G::SYN;
    const int send = roles && !owner ? min(kSlopes, 2 * ZT0) : kSlopes;
    for (int it = roles && owner ? 2 * ZT0 + oidx : tid; main && it < send; it += step) {
      T* dst;
      int ds;
      const T *m, *c, *pp;
      if (it < G::SXN) {
        const int r = it / (TX + 2), cc = it - r * (TX + 2) - 1;
        m = cell_ptr(cur, r, cc - 1);
        c = cell_ptr(cur, r, cc);
        pp = cell_ptr(cur, r, cc + 1);
        dst = sxs + it;
        ds = G::SXN;
      } else {
        const int j = it - G::SXN;
        const int rr = j / TX - 1, cc = j - (j / TX) * TX;
        m = cell_ptr(cur, rr - 1, cc);
        c = cell_ptr(cur, rr, cc);
        pp = cell_ptr(cur, rr + 1, cc);
        dst = sys + j;
        ds = G::SYN;
      }
      cell_slopes(m, G::PS, c, G::PS, pp, G::PS, lim, ph, dst, ds);
    }
    if (ZACT && owner)
      cell_slopes(cur + oidx, G::PS, ring_plane(k + 1) + oidx, G::PS, ring_plane(k + 2) + oidx,
                  G::PS, lim, ph, zS + oidx, G::NINT);
    __syncthreads();

    // ---- C: fluxes --------------------------------------------------------
    for (int it = tid; main && it < G::ITEMS; it += NT) {
      T vl[kNV], vr[kNV], F[kNV];
      T* out;
      int os;
      const bool xdir = it < G::IT_X || it >= G::IT_XE0;
      if (G::IT_XE0 > G::IT_X + G::IT_Y && !xdir && it >= G::IT_X + G::IT_Y) continue;
      if (xdir) {
        int r, fi;
        if (it < G::IT_X) {
          r = it / TX;
          fi = it - r * TX;
        } else {
          r = it - G::IT_XE0;
          fi = TX;
        }
        const T* a = cell_ptr(cur, r, fi - 1);
        const T* b = cell_ptr(cur, r, fi);
        const T* ga = sxs + r * (TX + 2) + fi;      // half slope of cell fi-1
        const T* gb = ga + 1;                        // half slope of cell fi
#pragma unroll
        for (int q = 0; q < kNV; ++q) {
          vl[q] = add_f(a[q * G::PS], ga[q * G::SXN], ph);
          vr[q] = sub_f(b[q * G::PS], gb[q * G::SXN], ph);
        }
        if constexpr (CT) ct_face_field(vl, vr, 0, bface(0, k, r, fi));
        out = Fx + r * (TX + 1) + fi;
        os = G::FXN;
      } else {
        const int j = it - G::IT_X;
        const int fj = j / TX, c = j - (j / TX) * TX;
        const T* a = cell_ptr(cur, fj - 1, c);
        const T* b = cell_ptr(cur, fj, c);
        const T* ga = sys + fj * TX + c;             // half slope of row fj-1
        const T* gb = ga + TX;                       // half slope of row fj
#pragma unroll
        for (int q = 0; q < kNV; ++q) {
          vl[q] = add_f(a[q * G::PS], ga[q * G::SYN], ph);
          vr[q] = sub_f(b[q * G::PS], gb[q * G::SYN], ph);
        }
        if constexpr (CT) ct_face_field(vl, vr, 1, bface(1, k, fj, c));
        out = Fy + j;
        os = G::FYN;
      }
      // warp-uniform branch to the compile-time direction
      if (xdir)
        glm_hlld_flux<0>(vl, vr, ch, half_chi, ph, F);
      else
        glm_hlld_flux<1>(vl, vr, ch, half_chi, ph, F);
#pragma unroll
      for (int q = 0; q < kNV; ++q) out[q * os] = F[q];
    }
    T dUz[kNV];
    if constexpr (ZACT) {
      if (owner) {
        T vl[kNV], vr[kNV], F[kNV];
        const T* c = ring_plane(k + 1) + oidx;
#pragma unroll
        for (int q = 0; q < kNV; ++q) {
          vl[q] = zP[q * G::NINT + oidx];
          vr[q] = sub_f(c[q * G::PS], zS[q * G::NINT + oidx], ph);
        }
        if constexpr (CT) {
          ct_face_field(vl, vr, 2, bface(2, k + 1, orow, ocol));
          ctc.from_prims(cur + oidx, G::PS);
          ctc.fz_bx = zF[kBX * G::NINT + oidx];
          ctc.fz_by = zF[kBY * G::NINT + oidx];
          ctc.fz_rho = zF[kRHO * G::NINT + oidx];
        }
        if (k >= z0 - 1) {  // from k = z0-1 on, zP holds the face state of cell k
          glm_hlld_flux<2>(vl, vr, ch, half_chi, ph, F);
#pragma unroll
          for (int q = 0; q < kNV; ++q) {
            dUz[q] = sub_f(F[q], zF[q * G::NINT + oidx], ph);
            zF[q * G::NINT + oidx] = F[q];
          }
        }
#pragma unroll
        for (int q = 0; q < kNV; ++q)
          zP[q * G::NINT + oidx] = add_f(c[q * G::PS], zS[q * G::NINT + oidx], ph);
      }
    }
    __syncthreads();

    // ---- D: right-hand side and RK combination (column owners) -------------
    if (main && owner) {
      const int gx = x0 + ocol, gy = y0 + orow;
      const bool valid = gx < nx && gy < ny;
      T unew[kNV];
#pragma unroll
      for (int q = 0; q < kNV; ++q) unew[q] = T(0);
      if (valid) {
        const long long off = (long long)k * p.sz + (long long)gy * p.sy + gx;
        T W[kNV], un[kNV];  // (loads first: their latency is the phase's)
#pragma unroll
        for (int q = 0; q < kNV; ++q) {
          W[q] = p.win[q * p.sv + off];
          if constexpr (STAGE != 1) un[q] = p.un[q * p.sv + off];
        }
#pragma unroll
        for (int q = 0; q < kNV; ++q) {
          const T* fx = Fx + q * G::FXN + orow * (TX + 1) + ocol;
          // sums of products with their rounding fixed (mul_rn / fma_rn), so
          // every instantiation of this tile code gives the same bits
          T du = mul_f(sub_f(fx[1], fx[0], ph), dtdx, ph);
          if constexpr (G::GY > 0) {
            const T* fy = Fy + q * G::FYN + orow * TX + ocol;
            du = fma_rn(sub_f(fy[TX], fy[0], ph), dtdy, du);
          }
          if constexpr (ZACT) du = fma_rn(dUz[q], dtdz, du);
          if (frozen) du = T(0);
          unew[q] = sub_f(W[q], du, ph);
        }
        if constexpr (STAGE != 1) {
          // RK2: (U^n + s) / 2, the same value with one operation less
          if (p.a_n == T(0.5) && p.a_w == T(0.5)) {
#pragma unroll
            for (int q = 0; q < kNV; ++q)
              unew[q] = half_of(add_f(un[q], unew[q], ph));
          } else {
#pragma unroll
            for (int q = 0; q < kNV; ++q)
              unew[q] = fma_rn(p.a_n, un[q], mul_f(p.a_w, unew[q], ph));
          }
        }
        if constexpr (CT) {
#pragma unroll
          for (int q = 0; q < kNV; ++q)
            if (q != kBX && q != kBY && q != kBZ)
              p.uout[q * p.sv + off] = q == kPSI ? T(0) : unew[q];
          ctc.write(p.ctf, p.sv, off, Fx + orow * (TX + 1) + ocol, G::FXN,
                    Fy + orow * TX + ocol, G::FYN, ch);
        } else {
          if constexpr (STAGE == 2) unew[kPSI] = mul_rn(unew[kPSI], damp);
#pragma unroll
          for (int q = 0; q < kNV; ++q) p.uout[q * p.sv + off] = unew[q];
        }
      }
      if constexpr (STAGE == 2 && !CT) {  // every lane of the (whole) owner warps
        const int ndim = 1 + (G::GY > 0) + (ZACT ? 1 : 0);
        smax.update(unew, valid, ph, ndim, flags);
      }
    }
  }

  if constexpr (STAGE == 2 && !CT) {
    // block max of the wave speed -> one FP64-bit atomicMax per CTA
    double l = smax.value();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double other = __shfl_xor_sync(0xffffffffu, l, o);
      l = nan_max(l, other);
    }
    __syncthreads();
    if ((tid & 31) == 0) wmax[tid >> 5] = l;
    __syncthreads();
    if (tid == 0) {
      double m = wmax[0];
      for (int w = 1; w < NW; ++w)
        m = nan_max(m, wmax[w]);
      SpeedMax<T>::publish(m, p.lam_bits, p.est_bits);
    }
  }
  __syncthreads();  // the CTA may start another tile on the same shared memory
}

template <class T, int TY, int NW, int STAGE, bool ZACT, bool CT, bool HALO = false, int TX = 32>
__global__ void __launch_bounds__(NW * 32, 1)
    rk_stage_kernel(const StageParams<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double wmax[NW];
  __shared__ double konst[4];
  const StepScalars sc = *p.sc;
  stage_tile<T, TY, NW, STAGE, ZACT, CT, HALO, TX>(p, sc, blockIdx.x, blockIdx.y, blockIdx.z,
                                                   smem_raw, wmax, konst);
}

}  // namespace mhd
