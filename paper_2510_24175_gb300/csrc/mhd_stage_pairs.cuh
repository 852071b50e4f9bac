// Fused Runge-Kutta stage of 3-D FP32 grids: the phases of stage_tile()
// (mhd_stage.cuh) and of the WENO-Z kernel (mhd_stage_weno.cuh) on 32 x 8 column
// tiles, arranged for the FP32 kernels' bounds, latency, instruction issue and
// shared-memory wavefronts:
//   * the nine variables of a cell are kept as four pairs and one value (rho
//     vx | vy vz | Bx By | Bz p | psi), so that a cell moves in five shared-
//     memory instructions and slopes, WENO-Z values, face states and updates run
//     on packed pairs;
//   * phase B stores a cell's lower and upper face states instead of its slope,
//     and a face's flux overwrites the lower state that only that face reads (45
//     shared-memory values per face instead of 54, and no flux arrays);
//   * global addresses are a warp-uniform plane and variable base plus the
//     thread's 32-bit byte offset in the plane; the HALO form uses 64-bit ones,
//     and grids with planes of 4 GB and more take it, with or without halo faces.
// The arithmetic of a cell is that of every other instantiation, operation by
// operation (packed instructions round like scalar ones).  Turbulent box 512^3, a
// step of two stages: 25.1 ms (32.6 with scalar values, slopes in shared memory and
// 16 warps per SM; 27.7 with 32 warps); Orszag-Tang 256^3 WENO-Z with constrained
// transport, a step of three stages: 11.0 ms (13.6).
#pragma once

#include <type_traits>

#include "mhd_stage.cuh"
#include "mhd_wenoz.cuh"

namespace mhd {

template <int TY, bool WENO>
struct PairGeom {
  static constexpr int TX = 32;
  static constexpr int GH = WENO ? 3 : 2;  // ghost width
  static constexpr int NR = WENO ? 5 : 3;  // ring planes
  static constexpr int NINT = TY * TX;
  static constexpr int NXH = 2 * GH * TY;  // x halo: columns -GH..-1, 32..31+GH
  static constexpr int NYH = 2 * GH * TX;  // y halo: rows -GH..-1, TY..TY+GH-1
  static constexpr int PS = NINT > NXH + NYH ? NINT : NXH + NYH;  // cells of a set
  static constexpr int RING = NR * kNV * PS;
  static constexpr int HB = kNV * PS;
  static constexpr int XN = TY * (TX + 1);  // x faces
  static constexpr int YN = (TY + 1) * TX;  // y faces
  static constexpr int WORDS = RING + HB + 2 * kNV * (XN + YN) + 2 * kNV * NINT;
  static constexpr int NLOAD = NINT + NXH + NYH;
  static constexpr int SX = TY * (TX + 2);  // x face-state items, columns -1..32
  static constexpr int SY0 = (SX + 31) / 32 * 32;  // y items start on a warp
  static constexpr int SY = (TY + 2) * TX;  // y face-state items, rows -1..TY
  static constexpr int ITEMS = XN + YN;     // flux items: [x main][y][x right edge]
};

// The nine values of cell i of a set of S cells at b.
template <int S>
__device__ __forceinline__ void ld9(const float* b, int i, float v[kNV]) {
  const float2* q = reinterpret_cast<const float2*>(b) + i;
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    const float2 t = q[n * S];
    v[2 * n] = t.x;
    v[2 * n + 1] = t.y;
  }
  v[8] = b[8 * S + i];
}
template <int S>
__device__ __forceinline__ void st9(float* b, int i, const float v[kNV]) {
  float2* q = reinterpret_cast<float2*>(b) + i;
#pragma unroll
  for (int n = 0; n < 4; ++n) q[n * S] = make_float2(v[2 * n], v[2 * n + 1]);
  b[8 * S + i] = v[8];
}

// Pairwise 9-vector operations (the last element alone).
__device__ __forceinline__ void add9(const float a[kNV], const float b[kNV], float c[kNV]) {
#pragma unroll
  for (int n = 0; n < 8; n += 2) {
    const f2 t = f2(a[n], a[n + 1]) + f2(b[n], b[n + 1]);
    c[n] = t.v.x;
    c[n + 1] = t.v.y;
  }
  c[8] = a[8] + b[8];
}
__device__ __forceinline__ void sub9(const float a[kNV], const float b[kNV], float c[kNV]) {
#pragma unroll
  for (int n = 0; n < 8; n += 2) {
    const f2 t = f2(a[n], a[n + 1]) - f2(b[n], b[n + 1]);
    c[n] = t.v.x;
    c[n + 1] = t.v.y;
  }
  c[8] = a[8] - b[8];
}
// c = a * s + c
__device__ __forceinline__ void fma9(const float a[kNV], float s, float c[kNV]) {
#pragma unroll
  for (int n = 0; n < 8; n += 2) {
    const f2 t = fma_rn(f2(a[n], a[n + 1]), f2(s), f2(c[n], c[n + 1]));
    c[n] = t.v.x;
    c[n + 1] = t.v.y;
  }
  c[8] = fma_rn(a[8], s, c[8]);
}
__device__ __forceinline__ void mul9(const float a[kNV], float s, float c[kNV]) {
#pragma unroll
  for (int n = 0; n < 8; n += 2) {
    const f2 t = mul_rn(f2(a[n], a[n + 1]), f2(s));
    c[n] = t.v.x;
    c[n + 1] = t.v.y;
  }
  c[8] = mul_rn(a[8], s);
}

// Face values of the cell q with neighbours m, p along a direction: lo at its
// lower, hi at its upper face (half slopes as cell_slopes() takes them).
__device__ __forceinline__ void face_pair(const float m[kNV], const float q[kNV],
                                          const float p[kNV], int lim, float lo[kNV],
                                          float hi[kNV]) {
  float dm[kNV], dp[kNV], h[kNV];
  sub9(q, m, dm);
  sub9(p, q, dp);
  if (lim == kLimMC) {
    float c[kNV], up[kNV], dn[kNV];
    add9(dm, dp, c);
    mul9(c, 0.25f, c);
#pragma unroll
    for (int k = 0; k < kNV; ++k) {  // half_slope_mc
      up[k] = fmaxf(min3(dm[k], dp[k], c[k]), 0.0f);
      dn[k] = fminf(max3(dm[k], dp[k], c[k]), 0.0f);
    }
    add9(up, dn, h);
  } else if (lim == kLimMinmod) {
#pragma unroll
    for (int k = 0; k < kNV; ++k) h[k] = half_slope_minmod(dm[k], dp[k]);
  } else {
#pragma unroll
    for (int k = 0; k < kNV; ++k) h[k] = 0.0f;
  }
  if (!(q[kRHO] - fabsf(h[kRHO]) > 0.0f && q[kPRS] - fabsf(h[kPRS]) > 0.0f)) {
#pragma unroll
    for (int k = 0; k < kNV; ++k) h[k] = 0.0f;
  }
  sub9(q, h, lo);
  add9(q, h, hi);
}

// Face values of a cell from the cells at(j) (base, index) along a direction, j =
// 0 the cell itself: PLM (WENO = false) or WENO-Z, with the flat fallback on
// a non-positive face density or pressure.
template <bool WENO, int PS, class At>
__device__ __forceinline__ void face_states(At at, int lim, float lo[kNV], float hi[kNV]) {
  if constexpr (!WENO) {
    float m[kNV], q[kNV], n[kNV];
    const auto cm = at(-1), cq = at(0), cn = at(1);
    ld9<PS>(cm.b, cm.i, m);
    ld9<PS>(cq.b, cq.i, q);
    ld9<PS>(cn.b, cn.i, n);
    face_pair(m, q, n, lim, lo, hi);
  } else {
    decltype(at(0)) c[5] = {at(-2), at(-1), at(0), at(1), at(2)};
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      f2 f[5], a, b;
#pragma unroll
      for (int j = 0; j < 5; ++j) f[j] = f2(reinterpret_cast<const float2*>(c[j].b)[n * PS + c[j].i]);
      wenoz_pair(f, a, b);
      lo[2 * n] = a.v.x;
      lo[2 * n + 1] = a.v.y;
      hi[2 * n] = b.v.x;
      hi[2 * n + 1] = b.v.y;
    }
    f2 f[5], a, b;
#pragma unroll
    for (int j = 0; j < 5; ++j) f[j] = f2(c[j].b[8 * PS + c[j].i]);
    wenoz_pair(f, a, b);
    lo[8] = a.v.x;
    hi[8] = b.v.x;
    if (!(lo[kRHO] > 0.0f && hi[kRHO] > 0.0f && lo[kPRS] > 0.0f && hi[kPRS] > 0.0f)) {
      ld9<PS>(c[2].b, c[2].i, lo);
#pragma unroll
      for (int k = 0; k < kNV; ++k) hi[k] = lo[k];
    }
  }
}
struct CellRef {  // cell i of the set at b
  const float* b;
  int i;
};

// One tile (bx, by, bz) of one RK stage (see stage_tile()); smem: PairGeom words.
template <int TY, int NW, int STAGE, bool CT, bool HALO, bool WENO>
__device__ __forceinline__ void stage_tile_pairs(const StageParams<float>& p,
                                                 const StepScalars& sc, int bx, int by, int bz,
                                                 float* smem, double* wmax) {
  using G = PairGeom<TY, WENO>;
  constexpr int NT = NW * 32, TX = G::TX, PS = G::PS, NI = G::NINT, GH = G::GH;
  constexpr int ZT0 = NT - NI;  // threads ZT0.. own one tile column each
  constexpr int NA = (G::NLOAD + NT - 1) / NT;
  static_assert(ZT0 >= 0, "need one thread per tile column");
  static_assert(!HALO || !CT, "halo faces: GLM kernels only");
  float* ring = smem;
  float* hb = ring + G::RING;          // x halo cells, then y halo cells
  float* xU = hb + G::HB;              // upper x states of columns -1..31, at the face
  float* xL = xU + kNV * G::XN;        // lower x states of columns 0..32, then fluxes
  float* yU = xL + kNV * G::XN;        // the same for y, rows -1..TY
  float* yL = yU + kNV * G::YN;
  float* zP = yL + kNV * G::YN;        // per owner: upper z state of cell k
  float* zF = zP + kNV * NI;           // per owner: z flux at face k-1/2

  const int tid = threadIdx.x;
  const int x0 = bx * TX, y0 = by * TY;
  const int z0 = p.zlo + bz * p.tz;
  const int z1 = min(z0 + p.tz, p.zhi);
  const int nx = p.n[0], ny = p.n[1];
  const bool owner = tid >= ZT0;
  const int oidx = tid - ZT0;
  const int orow = oidx / TX, ocol = oidx - (oidx / TX) * TX;
  const float ch = float(sc.ch);
  const float half_chi = float(0.5 / sc.ch);
  const bool frozen = !(sc.dt != 0.0);  // see stage_tile()
  const Phys<float> ph = p.ph;
  unsigned flags = 0;  // of the wave-speed conversions (not counted)
  SpeedMax<float> smax(ph);

  auto ring_plane = [&](int zz) { return ring + ((zz + 2 * G::NR) % G::NR) * (kNV * PS); };
  auto wrap = [](int i, int n, int lo, int hi) {
    return GH == 2 ? remap(i, n, lo, hi) : remap3(i, n, lo, hi);
  };
  // in-plane offset of tile cell (r, c), remapped into the grid, in bytes
  auto plane_off = [&](int r, int c) {
    const int gx = wrap(x0 + c, nx, p.bc_lo[0], p.bc_hi[0]);
    const int gy = wrap(y0 + r, ny, p.bc_lo[1], p.bc_hi[1]);
    return (unsigned)(gy * (unsigned)nx + gx) * 4u;
  };
  auto plane_z = [&](int zz) {
    return (long long)wrap(zz, p.n[2], p.bc_lo[2], p.bc_hi[2]) * p.sz;
  };
  using Off = std::conditional_t<HALO, unsigned long long, unsigned>;
  auto ldg = [](const float* base, Off off) {
    return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + off);
  };
  auto stg = [](float* base, Off off, float v) {
    *reinterpret_cast<float*>(reinterpret_cast<char*>(base) + off) = v;
  };
  // Load items: the tile's interior, its x halo, its y halo.  Item it: tile cell
  // (r, c); the thread's items are the same in every plane.
  auto load_rc = [&](int it, int& r, int& c) {
    if (it < NI) {
      r = it / TX;
      c = it - r * TX;
    } else if (it < NI + G::NXH) {
      const int j = it - NI;
      r = j / (2 * GH);
      const int q = j - r * (2 * GH);
      c = q < GH ? q - GH : TX + q - GH;
    } else {
      const int j = it - NI - G::NXH, hr = j / TX;
      c = j - hr * TX;
      r = hr < GH ? hr - GH : TY + hr - GH;
    }
  };
  unsigned aoff[NA];
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    int r = 0, c = 0;
    load_rc(min(tid + a * NT, G::NLOAD - 1), r, c);
    aoff[a] = HALO ? 0u : plane_off(r, c);
  }
  // cons -> prim of load item it (interior: of plane zi; halo: of plane zh);
  // floor activations of the cells the tile updates are counted (rare)
  auto load_item = [&](int it, unsigned off, int zi, int zh) {
    const bool own = it < NI;
    const int zz = own ? zi : zh;
    float u[kNV], v[kNV];
    if constexpr (HALO) {
      int r, c;
      load_rc(it, r, c);
      long long hs;
      const float* a = halo_cell<GH>(p, x0 + c, y0 + r, zz, hs);
#pragma unroll
      for (int k = 0; k < kNV; ++k) u[k] = a[k * hs];
    } else {
      // (the two planes' bases are warp-uniform, the item's choice is not)
      const float* bi = p.win + plane_z(zi);
      const float* bh = p.win + plane_z(zh);
      if (own) {
#pragma unroll
        for (int k = 0; k < kNV; ++k) u[k] = ldg(bi + k * p.sv, off);
      } else {
#pragma unroll
        for (int k = 0; k < kNV; ++k) u[k] = ldg(bh + k * p.sv, off);
      }
    }
    unsigned fl = 0;
    cons_to_prim(u, v, ph, fl);
    if (own)
      st9<PS>(ring_plane(zi), it, v);
    else
      st9<PS>(hb, it - NI, v);
    if (fl && own) {
      int r, c;
      load_rc(it, r, c);
      if (zz >= z0 && zz < z1 && x0 + c < nx && y0 + r < ny) {
        if (fl & kFloorRho) atomicAdd(&p.floor_cnt[0], 1ull);
        if (fl & kFloorP) atomicAdd(&p.floor_cnt[1], 1ull);
        if (fl & kPressF64) atomicAdd(&p.floor_cnt[2], 1ull);
      }
    }
  };
  // staggered normal field on the lower d-face of tile cell (r, c) of plane zz
  auto bface = [&](int d, int zz, int r, int c) {
    return ldg(p.bw[d] + plane_z(zz), plane_off(r, c));
  };
  CtCell<float> ctc;
  const bool valid = owner && x0 + ocol < nx && y0 + orow < ny;
  const Off doff = (Off(y0 + orow) * Off(nx) + Off(x0 + ocol)) * 4u;

  // The z march; warm-up iterations as in stage_tile().
#pragma unroll 1
  for (int k = z0 - 2 * GH; k < z1; ++k) {
    const bool main = k >= z0;
    // ---- A: loads: interior of plane k+GH, halo of plane k -----------------
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      const int it = tid + a * NT;
      if (it < (main ? G::NLOAD : NI)) load_item(it, aoff[a], k + GH, k);
    }
    __syncthreads();
    if (k < z0 - 2) continue;
    const float* cur = ring_plane(k);

    // ---- B: face states of x and y -----------------------------------------
    for (int it = tid; main && it < G::SY0 + G::SY; it += NT) {
      float lo[kNV], hi[kNV];
      if (it < G::SX) {
        const int r = it / (TX + 2), c = it - r * (TX + 2) - 1;
        face_states<WENO, PS>(
            [&](int j) {
              const int cc = c + j;
              const bool h = cc < 0 || cc >= TX;
              return CellRef{h ? hb : cur, h ? r * (2 * GH) + (cc < 0 ? cc + GH : cc - TX + GH)
                                             : r * TX + cc};
            },
            p.limiter, lo, hi);
        const int f = r * (TX + 1) + c;  // lower face of the cell
        if (c >= 0) st9<G::XN>(xL, f, lo);
        if (c < TX) st9<G::XN>(xU, f + 1, hi);
      } else if (it >= G::SY0) {
        const int j0 = it - G::SY0;
        const int r = j0 / TX - 1, c = j0 - (j0 / TX) * TX;
        face_states<WENO, PS>(
            [&](int j) {
              const int rr = r + j;
              const bool h = rr < 0 || rr >= TY;
              return CellRef{h ? hb : cur,
                             h ? G::NXH + (rr < 0 ? rr + GH : rr - TY + GH) * TX + c : rr * TX + c};
            },
            p.limiter, lo, hi);
        const int f = r * TX + c;
        if (r >= 0) st9<G::YN>(yL, f, lo);
        if (r < TY) st9<G::YN>(yU, f + TX, hi);
      }
    }
    __syncthreads();

    // ---- C: fluxes ----------------------------------------------------------
    for (int it = tid; main && it < G::ITEMS; it += NT) {
      float vl[kNV], vr[kNV], F[kNV];
      const bool xdir = it < NI || it >= NI + G::YN;
      if (xdir) {
        const int r = it < NI ? it / TX : it - (NI + G::YN);
        const int fi = it < NI ? it - r * TX : TX;
        const int f = r * (TX + 1) + fi;
        ld9<G::XN>(xU, f, vl);
        ld9<G::XN>(xL, f, vr);
        if constexpr (CT) ct_face_field(vl, vr, 0, bface(0, k, r, fi));
        glm_hlld_flux<0>(vl, vr, ch, half_chi, ph, F);
        st9<G::XN>(xL, f, F);
      } else {
        const int f = it - NI;
        ld9<G::YN>(yU, f, vl);
        ld9<G::YN>(yL, f, vr);
        if constexpr (CT) ct_face_field(vl, vr, 1, bface(1, k, f / TX, f - (f / TX) * TX));
        glm_hlld_flux<1>(vl, vr, ch, half_chi, ph, F);
        st9<G::YN>(yL, f, F);
      }
    }
    float dUz[kNV];
    if (owner) {
      float vl[kNV], vr[kNV], hi[kNV];
      if constexpr (CT) {
        float q[kNV];
        ld9<PS>(cur, oidx, q);
        ctc.from_prims(q, 1);
      }
      face_states<WENO, PS>([&](int j) { return CellRef{ring_plane(k + 1 + j), oidx}; }, p.limiter,
                            vr, hi);
      ld9<NI>(zP, oidx, vl);
      st9<NI>(zP, oidx, hi);
      if (k >= z0 - 1) {  // from k = z0-1 on, zP holds the upper state of cell k
        float F[kNV], F0[kNV];
        if constexpr (CT) ct_face_field(vl, vr, 2, bface(2, k + 1, orow, ocol));
        glm_hlld_flux<2>(vl, vr, ch, half_chi, ph, F);
        ld9<NI>(zF, oidx, F0);
        if constexpr (CT) {
          ctc.fz_bx = F0[kBX];
          ctc.fz_by = F0[kBY];
          ctc.fz_rho = F0[kRHO];
        }
        sub9(F, F0, dUz);
        st9<NI>(zF, oidx, F);
      }
    }
    __syncthreads();

    // ---- D: right-hand side and RK combination (column owners) --------------
    if (main && valid) {
      float f0[kNV], f1[kNV], du[kNV], u[kNV];
      const float* wb = p.win + (long long)k * p.sz;
      float* ob = p.uout + (long long)k * p.sz;
#pragma unroll
      for (int q = 0; q < kNV; ++q) u[q] = ldg(wb + q * p.sv, doff);
      float un[kNV];
      if constexpr (STAGE != 1) {
        const float* nb = p.un + (long long)k * p.sz;
#pragma unroll
        for (int q = 0; q < kNV; ++q) un[q] = ldg(nb + q * p.sv, doff);
      }
      const int fx = orow * (TX + 1) + ocol, fy = orow * TX + ocol;
      ld9<G::XN>(xL, fx, f0);
      ld9<G::XN>(xL, fx + 1, f1);
      sub9(f1, f0, du);
      mul9(du, float(sc.dtdx[0]), du);
      if constexpr (CT) {
        float g0[kNV];
        ld9<G::YN>(yL, fy, g0);
        ctc.write(p.ctf + (long long)k * p.sz, p.sv, doff / 4u, f0, 1, g0, 1, ch);
      }
      ld9<G::YN>(yL, fy, f0);
      ld9<G::YN>(yL, fy + TX, f1);
      sub9(f1, f0, f1);
      fma9(f1, float(sc.dtdx[1]), du);
      fma9(dUz, float(sc.dtdx[2]), du);
      if (frozen) {
#pragma unroll
        for (int q = 0; q < kNV; ++q) du[q] = 0.0f;
      }
      sub9(u, du, u);
      if constexpr (STAGE != 1) {
        mul9(u, p.a_w, u);
        fma9(un, p.a_n, u);
      }
      if constexpr (CT) {
#pragma unroll
        for (int q = 0; q < kNV; ++q)
          if (q < kBX || q > kBZ) stg(ob + q * p.sv, doff, q == kPSI ? 0.0f : u[q]);
      } else {
        if constexpr (STAGE == 2) u[kPSI] = mul_rn(u[kPSI], float(sc.damp));
#pragma unroll
        for (int q = 0; q < kNV; ++q) stg(ob + q * p.sv, doff, u[q]);
        if constexpr (STAGE == 2) smax.update(u, true, ph, 3, flags);
      }
    }
  }

  if constexpr (STAGE == 2 && !CT) {
    // block max of the wave speed -> one atomicMax per CTA
    double l = smax.value();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l = nan_max(l, __shfl_xor_sync(0xffffffffu, l, o));
    __syncthreads();
    if ((tid & 31) == 0) wmax[tid >> 5] = l;
    __syncthreads();
    if (tid == 0) {
      double m = wmax[0];
      for (int w = 1; w < NW; ++w) m = nan_max(m, wmax[w]);
      SpeedMax<float>::publish(m, p.lam_bits, p.est_bits);
    }
  }
  __syncthreads();  // the CTA may start another tile on the same shared memory
}

// PER_SM: CTAs per SM (2: 64 registers a thread, 1: 128).
template <int TY, int NW, int STAGE, bool CT, bool HALO, bool WENO, int PER_SM>
__global__ void __launch_bounds__(NW * 32, PER_SM)
    rk_stage_pairs_kernel(const StageParams<float> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double wmax[NW];
  const StepScalars sc = *p.sc;
  stage_tile_pairs<TY, NW, STAGE, CT, HALO, WENO>(p, sc, blockIdx.x, blockIdx.y, blockIdx.z,
                                                  reinterpret_cast<float*>(smem_raw), wmax);
}

}  // namespace mhd
