// Fused Runge-Kutta stage kernel with WENO-Z reconstruction (the
// reconstruction of the paper's own runs, Section 4.2): WENO-Z weights of
// Borges, Carmona, Costa & Don (2008) with exponent 1 and the candidate
// stencils and smoothness indicators of Jiang & Shu (1996), applied to the
// primitive variables.  Same phases as the PLM kernel (mhd_stage.cuh):
//   A  load + cons->prim: interior of plane k+3 (5-plane ring) and the
//      (x, y) halo of plane k (three cells deep);
//   B  the two face values of each cell and direction, once: x for the 34
//      cells of each row, y for the TY+2 rows, z (column owners) for cell k+1;
//      a cell whose face density or pressure would be <= 0 keeps its flat
//      value;
//   C  face fluxes (GLM + HLLD), each face of the tile once; column owners also
//      the z face k+1/2;
//   D  flux divergence + Runge-Kutta combination (+ damping and the wave-speed
//      reduction in the last stage).
// A face's flux overwrites the minus value that only this face reads, and the
// owners keep their z values in registers from B to C, so a 32 x 8 FP64 tile fits
// in shared memory (226 KB).  Bound by the FP64 unit: Orszag-Tang 256^3, a step of
// three stages 189 ms (335 with 32 x 4 tiles, scaled second differences, CUDA's
// divisions and roots and the longer HLLD).  FP64 grids and the 1-D and 2-D FP32
// ones (3-D FP32: mhd_stage_pairs.cuh).
#pragma once

#include "mhd_stage.cuh"
#include "mhd_wenoz.cuh"

namespace mhd {

// Face values of all 9 primitives of one cell from five cells c[0..4]
// (variables stride[j] apart); flat fallback on non-positive face density
// or pressure.  FP32 reconstructs the variables in pairs (0, 1) ... (6, 7).
template <class T>
__device__ __forceinline__ void cell_weno(const T* const c[5], const int st[5],
                                          const Phys<T>& ph, const WenoConst<T>& w,
                                          T M[kNV], T P[kNV]) {
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int k = 0; k + 1 < kNV; k += 2) {
      f2 f[5], m, p;
#pragma unroll
      for (int j = 0; j < 5; ++j) f[j] = f2(c[j][k * st[j]], c[j][(k + 1) * st[j]]);
      wenoz_pair(f, m, p);
      M[k] = m.v.x;
      M[k + 1] = m.v.y;
      P[k] = p.v.x;
      P[k + 1] = p.v.y;
    }
    f2 f[5], m, p;
#pragma unroll
    for (int j = 0; j < 5; ++j) f[j] = f2(c[j][(kNV - 1) * st[j]]);
    wenoz_pair(f, m, p);
    M[kNV - 1] = m.v.x;
    P[kNV - 1] = p.v.x;
  } else {
#pragma unroll
    for (int k = 0; k < kNV; ++k) {
      T f[5];
#pragma unroll
      for (int j = 0; j < 5; ++j) f[j] = c[j][k * st[j]];
      wenoz_pair(f, ph, w, M[k], P[k]);
    }
  }
  const bool ok = gt0(M[kRHO]) && gt0(P[kRHO]) && gt0(M[kPRS]) && gt0(P[kPRS]);
  if (!ok) {
#pragma unroll
    for (int k = 0; k < kNV; ++k) M[k] = P[k] = c[2][k * st[2]];
  }
}

template <int TY, bool ZACT>
struct WenoGeom {
  static constexpr int TX = 32;
  static constexpr int GY = TY > 1 ? 3 : 0;
  static constexpr int NINT = TY * TX;
  static constexpr int NXH = 6 * TY;               // x halo: columns -3..-1, 32..34
  static constexpr int NYH = GY ? 6 * TX : 0;      // y halo: rows -3..-1, TY..TY+2
  static constexpr int NRING = ZACT ? 5 : 1;
  static constexpr int RING_W = NRING * kNV * NINT;
  static constexpr int XH_W = kNV * NXH;
  static constexpr int YH_W = kNV * NYH;
  static constexpr int SXN = TY * (TX + 2);           // x face-value items, columns -1..32
  static constexpr int SYN = GY ? (TY + 2) * TX : 0;  // y face-value items, rows -1..TY
  static constexpr int FXN = TY * (TX + 1);           // x faces
  static constexpr int FYN = GY ? (TY + 1) * TX : 0;  // y faces
  static constexpr int Z_W = ZACT ? 2 * kNV * NINT : 0;  // zP, zF per owner
  static constexpr int WORDS = RING_W + XH_W + YH_W + 2 * kNV * FXN + 2 * kNV * FYN + Z_W;
  static constexpr int NLOAD = NINT + NXH + NYH;
  static constexpr int IT_X = TY * TX;
  static constexpr int IT_Y = FYN;
  static constexpr int IT_XE = TY;
  static constexpr int ITEMS = IT_X + IT_Y + IT_XE;
};

// CT: constrained transport, HALO: halo faces, as in stage_tile() (mhd_stage.cuh).
template <class T, int TY, int NW, int STAGE, bool ZACT, bool CT, bool HALO = false>
__global__ void __launch_bounds__(NW * 32, 1)
    rk_stage_weno_kernel(const StageParams<T> p) {
  using G = WenoGeom<TY, ZACT>;
  constexpr int NT = NW * 32;
  constexpr int TX = G::TX;
  constexpr int ZT0 = NT - G::NINT;
  static_assert(ZT0 >= 0, "need one thread per tile column");
  static_assert(sizeof(T) == 8 || !ZACT, "3-D FP32: mhd_stage_pairs.cuh");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double wmax[NW];
  T* ring = reinterpret_cast<T*>(smem_raw);
  T* xh = ring + G::RING_W;
  T* yh = xh + G::XH_W;
  T* xU = yh + G::YH_W;        // per x face: plus value of the cell below it
  T* Fx = xU + kNV * G::FXN;   // per x face: minus value of the cell above it, then its flux
  T* yU = Fx + kNV * G::FXN;   // the same for y
  T* Fy = yU + kNV * G::FYN;
  T* zP = Fy + kNV * G::FYN;   // per owner: plus-face value of cell k
  T* zF = zP + kNV * G::NINT;  // per owner: z flux at face k-1/2

  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * TX;
  const int y0 = blockIdx.y * TY;
  const int z0 = p.zlo + blockIdx.z * p.tz;
  const int z1 = min(z0 + p.tz, p.zhi);
  const int nx = p.n[0], ny = p.n[1], nz = p.n[2];
  const bool owner = tid >= ZT0;
  const int oidx = tid - ZT0;
  const int orow = oidx / TX, ocol = oidx - (oidx / TX) * TX;

  const StepScalars sc = *p.sc;
  const T ch = T(sc.ch);
  const T half_chi = T(0.5 / sc.ch);
  const T dtdx = T(sc.dtdx[0]), dtdy = T(sc.dtdx[1]), dtdz = T(sc.dtdx[2]);
  const T damp = T(sc.damp);
  const bool frozen = !(sc.dt != 0.0);
  __shared__ double konst[8];
  Phys<T> ph = p.ph;
  if constexpr (sizeof(T) == 8) {
    if (threadIdx.x == 0) WenoConst<T>::fill(konst + 4);
  }
  fp64_registers(ph, konst);  // (synchronises)
  if constexpr (TY == 1) {  // 1-D kernels wait for latency: the plain operations
    ph.one = T(1);
    ph.nzero = T(-0.0);
  }
  const WenoConst<T> wk(konst + 4);
  unsigned flags = 0;  // of the wave-speed conversions (not counted)

  auto slot = [](int zz) { return ZACT ? ((zz % 5) + 5) % 5 : 0; };
  auto ring_plane = [&](int zz) { return ring + slot(zz) * (kNV * G::NINT); };

  // floor activations: once per stage for each cell the tile updates, from
  // its own conversion (as in the PLM stage kernel)
  auto count_floors = [&](unsigned fl, int zz, int r, int c) {
    if (zz < z0 || zz >= z1 || x0 + c >= nx || (G::GY && y0 + r >= ny)) return;
    if (fl & kFloorRho) atomicAdd(&p.floor_cnt[0], 1ull);
    if (fl & kFloorP) atomicAdd(&p.floor_cnt[1], 1ull);
    if (fl & kPressF64) atomicAdd(&p.floor_cnt[2], 1ull);
  };
  // offset of tile cell (r, c) of plane zz, remapped into the grid
  auto cell_off = [&](int zz, int r, int c) {
    const int gz = ZACT ? remap3(zz, nz, p.bc_lo[2], p.bc_hi[2]) : 0;
    const int gx = remap3(x0 + c, nx, p.bc_lo[0], p.bc_hi[0]);
    const int gy = G::GY ? remap3(y0 + r, ny, p.bc_lo[1], p.bc_hi[1]) : 0;
    return (long long)gz * p.sz + (long long)gy * p.sy + gx;
  };
  auto load_cell = [&](int zz, int r, int c, T* dst, int dst_stride, bool own) {
    T u[kNV], v[kNV];
    if constexpr (HALO) {
      long long hs;
      const T* a = halo_cell<3>(p, x0 + c, y0 + r, zz, hs);
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
  auto load_item = [&](int it, int zi, int zh) {
    if (it < G::NINT) {
      const int r = it / TX, c = it - (it / TX) * TX;
      load_cell(zi, r, c, ring_plane(zi) + it, G::NINT, true);
    } else if (it < G::NINT + G::NXH) {
      const int j = it - G::NINT;
      const int r = j / 6, q = j - (j / 6) * 6;
      const int c = q < 3 ? q - 3 : TX + q - 3;
      load_cell(zh, r, c, xh + j, G::NXH, false);
    } else {
      const int j = it - G::NINT - G::NXH;
      const int hr = j / TX, c = j - (j / TX) * TX;
      const int r = hr < 3 ? hr - 3 : TY + hr - 3;
      load_cell(zh, r, c, yh + j, G::NYH, false);
    }
  };
  auto cell_ptr = [&](const T* cur, int r, int c, int* st) -> const T* {
    if (c < 0 || c >= TX) {
      *st = G::NXH;
      return xh + r * 6 + (c < 0 ? c + 3 : c - TX + 3);
    }
    if (r < 0 || r >= TY) {
      *st = G::NYH;
      return yh + (r < 0 ? r + 3 : r - TY + 3) * TX + c;
    }
    *st = G::NINT;
    return cur + r * TX + c;
  };
  static_assert(!CT || ZACT, "constrained transport is 3-D only");
  static_assert(!HALO || (ZACT && !CT), "halo faces: 3-D GLM kernels only");
  // staggered normal field on the lower d-face of tile cell (r, c) of plane zz
  auto bface = [&](int d, int zz, int r, int c) -> T {
    return p.bw[d][cell_off(zz, r, c)];
  };
  CtCell<T> ctc;
  // face values of the owned column's cell in plane zc (planes zc-2..zc+2)
  auto z_cell = [&](int zc, T M[kNV], T P[kNV]) {
    const T* c[5];
    int st[5];
    for (int j = 0; j < 5; ++j) {
      c[j] = ring_plane(zc - 2 + j) + oidx;
      st[j] = G::NINT;
    }
    cell_weno(c, st, ph, wk, M, P);
  };

  // The z march: one loop body for every plane (see stage_tile in
  // mhd_stage.cuh), so a cell's result does not depend on where a z chunk,
  // block or launch range starts.  Warm-up: k = z0-6 .. z0-3 only load
  // planes z0-3 .. z0 into the ring, k = z0-2 computes the column owners'
  // face values of cell z0-1, k = z0-1 their flux through face z0-1/2; the
  // x, y work and the update start at k = z0.
  constexpr int NWARM = ZACT ? 6 : 0;
  // 3-D tiles: the warps without columns take the first kB rounds of the x, y
  // values and the first kC of the fluxes, the owners the rest besides their z
  // work, so that no phase ends in a round of a few warps (dealt out evenly with
  // z on top: 256^3 RK3 step 192 instead of 189 ms)
  constexpr bool kDeal = ZACT && ZT0 > 0;
  constexpr int kB = (G::SXN + G::SYN + G::NINT + NT - 1) / NT;
  constexpr int kC = (G::ITEMS + G::NINT + NT - 1) / NT;
  const int first = kDeal && owner ? oidx : tid, step = !kDeal ? NT : owner ? G::NINT : ZT0;
  SpeedMax<T> smax(ph);  // last stage: the new state's maximum wave speed
#pragma unroll 1
  for (int k = z0 - NWARM; k < z1; ++k) {
    const bool main = k >= z0;
    // ---- A: loads ---------------------------------------------------------
    const int nload = main ? G::NLOAD : G::NINT;
    for (int it = tid; it < nload; it += NT) {
      if (ZACT && it < G::NINT)
        load_item(it, k + 3, k);
      else
        load_item(it, k, k);
    }
    __syncthreads();
    if (ZACT && k < z0 - 2) continue;
    const T* cur = ring_plane(k);

    // ---- B: face values ---------------------------------------------------
    constexpr int kValues = G::SXN + G::SYN;
    const int vend = kDeal && !owner ? min(kValues, kB * ZT0) : kValues;
    for (int it = (kDeal && owner ? kB * ZT0 : 0) + first; main && it < vend; it += step) {
      const T* c[5];
      int st[5];
      T M[kNV], P[kNV];
      T *dM, *dP;  // the cell's lower and upper face
      int ds;
      bool lower, upper;
      if (it < G::SXN) {
        const int r = it / (TX + 2), cc = it - r * (TX + 2) - 1;
        for (int j = 0; j < 5; ++j) c[j] = cell_ptr(cur, r, cc - 2 + j, &st[j]);
        const int f = r * (TX + 1) + cc;
        dM = Fx + f;
        dP = xU + f + 1;
        ds = G::FXN;
        lower = cc >= 0;
        upper = cc < TX;
      } else {
        const int j0 = it - G::SXN;
        const int rr = j0 / TX - 1, cc = j0 - (j0 / TX) * TX;
        for (int j = 0; j < 5; ++j) c[j] = cell_ptr(cur, rr - 2 + j, cc, &st[j]);
        const int f = rr * TX + cc;
        dM = Fy + f;
        dP = yU + f + TX;
        ds = G::FYN;
        lower = rr >= 0;
        upper = rr < TY;
      }
      cell_weno(c, st, ph, wk, M, P);
      if (lower) {
#pragma unroll
        for (int q = 0; q < kNV; ++q) dM[q * ds] = M[q];
      }
      if (upper) {
#pragma unroll
        for (int q = 0; q < kNV; ++q) dP[q * ds] = P[q];
      }
    }
    T zm[kNV], zp[kNV];  // the owned column's face values of cell k+1
    if (ZACT && owner) z_cell(k + 1, zm, zp);
    __syncthreads();

    // ---- C: fluxes: the owners' z face, then x and y ------------------------
    T dUz[kNV];
    if constexpr (ZACT) {
      if (owner) {
        if (k >= z0 - 1) {  // from k = z0-1 on, zP holds the plus value of cell k
          T vl[kNV], F[kNV];
#pragma unroll
          for (int q = 0; q < kNV; ++q) vl[q] = zP[q * G::NINT + oidx];
          if constexpr (CT) {
            ct_face_field(vl, zm, 2, bface(2, k + 1, orow, ocol));
            ctc.from_prims(cur + oidx, G::NINT);
            ctc.fz_bx = zF[kBX * G::NINT + oidx];
            ctc.fz_by = zF[kBY * G::NINT + oidx];
            ctc.fz_rho = zF[kRHO * G::NINT + oidx];
          }
          glm_hlld_flux<2>(vl, zm, ch, half_chi, ph, F);
#pragma unroll
          for (int q = 0; q < kNV; ++q) {
            dUz[q] = sub_f(F[q], zF[q * G::NINT + oidx], ph);
            zF[q * G::NINT + oidx] = F[q];
          }
        }
#pragma unroll
        for (int q = 0; q < kNV; ++q) zP[q * G::NINT + oidx] = zp[q];
      }
    }
    const int fend = kDeal && !owner ? min(G::ITEMS, kC * ZT0) : G::ITEMS;
    for (int it = (kDeal && owner ? kC * ZT0 : 0) + first; main && it < fend; it += step) {
      T vl[kNV], vr[kNV], F[kNV];
      const T* up;
      T* out;
      int os;
      const bool xdir = it < G::IT_X || it >= G::IT_X + G::IT_Y;
      if (xdir) {
        int r, fi;
        if (it < G::IT_X) {
          r = it / TX;
          fi = it - r * TX;
        } else {
          r = it - (G::IT_X + G::IT_Y);
          fi = TX;
        }
        const int f = r * (TX + 1) + fi;
        up = xU + f;
        out = Fx + f;
        os = G::FXN;
#pragma unroll
        for (int q = 0; q < kNV; ++q) {
          vl[q] = up[q * G::FXN];
          vr[q] = out[q * G::FXN];
        }
        if constexpr (CT) ct_face_field(vl, vr, 0, bface(0, k, r, fi));
      } else {
        const int f = it - G::IT_X;
        up = yU + f;
        out = Fy + f;
        os = G::FYN;
#pragma unroll
        for (int q = 0; q < kNV; ++q) {
          vl[q] = up[q * G::FYN];
          vr[q] = out[q * G::FYN];
        }
        if constexpr (CT) ct_face_field(vl, vr, 1, bface(1, k, f / TX, f - (f / TX) * TX));
      }
      if (xdir)
        glm_hlld_flux<0>(vl, vr, ch, half_chi, ph, F);
      else
        glm_hlld_flux<1>(vl, vr, ch, half_chi, ph, F);
#pragma unroll
      for (int q = 0; q < kNV; ++q) out[q * os] = F[q];
    }
    __syncthreads();

    // ---- D: right-hand side and Runge-Kutta combination --------------------
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
    double l = smax.value();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l = nan_max(l, __shfl_xor_sync(0xffffffffu, l, o));
    __syncthreads();
    if ((tid & 31) == 0) wmax[tid >> 5] = l;
    __syncthreads();
    if (tid == 0) {
      double m = wmax[0];
      for (int w = 1; w < NW; ++w) m = nan_max(m, wmax[w]);
      SpeedMax<T>::publish(m, p.lam_bits, p.est_bits);
    }
  }
}

}  // namespace mhd
