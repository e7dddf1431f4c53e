// pf.cuh -- the primitive, predictor and Riemann-solver passes of the patch
// advance (A of the paper's Sec. 2.2 life cycle) fused into one kernel, with
// the predicted face states kept on chip; the staged k_update then finishes
// the step from the fluxes this kernel stores.  Included by advance.cuh
// inside its per-build namespace.
//
// A work item is an x-y tile of tx x ty cells (at most TX x TY, the host
// splits each patch's UB+1 region into tiles of near-equal extents) and a
// chunk [z0, z1) of its planes.  A block has one thread per tile cell, one
// per cell of the tile's lower x column and lower y row (the left neighbours
// whose upper face states the tile's lowest faces need) and up to a warp or
// two more; the shared-memory arrays are laid out for the largest tile.
// Marching along z, for each plane zc:
//   1. every thread runs the predictor of its cell on plane zc (limited
//      slopes, Hancock increment, six predicted face states) from the rings of
//      primitives W.  A tile cell keeps its own lower states and its upper z state
//      in registers; the upper x and y states, which neighbours read, go to
//      shared memory;
//   2. the block loads plane zc + 2 into the rings (primitives and cell EMFs E^n
//      over the tile grown by two cells below and one above), a cell to each
//      tile thread and the rest to the other threads, and each tile thread takes
//      its cell's three lower faces: the CT half-step normal field from E^n, the
//      HLLD flux, stored in the staged layout (vector groups) for k_update and
//      the captures.
// A barrier after each.  W has three planes (plane zc - 1 is done with once the
// predictor has run), E^n four (the faces read zc - 1 to zc + 1).
//
// Bound by instruction issue (59% of the slots at 17 warps per SM): 240 MB per
// 128^3 launch in FP32, 13% of the copy rate.  Both types keep the staged
// kernels' expressions, order and bits: which kernels advance a call depends on its
// captures, update boxes and size, and neighbouring patches in different
// calls have to agree on their shared faces.  2,627 warp instructions per 32
// cells and 266 us at 128^3 in FP32, where k_prim, k_pred and k_flux take 276
// us and move 1.28 GB.  FP32 expressions of its own (conserved face states
// shared between a face's flux and its predicted state, the star state's physical flux,
// four of E^n a face) took 2,480 and 207 us, but a state that differs by rounding.
// Tried and slower, in that form: 256 threads with tiles of 15 x 15
// (the loads lack threads: 368 against 345 us a step), the next plane's reads held
// in registers across the x face (398 us), one item chain per resident block
// with equal shares (359 us; neighbouring tiles then run at different planes).
// Tiles overlap only in the predictor of their lower column and row.
#pragma once

template <int TX, int TY> struct PfLayout {
  static constexpr int NC = TX * TY;             // tile cells
  // threads: the tile's, its lower row's and left column's, in whole warps, and
  // for the largest tile a warp that only loads
  static constexpr int NT = (NC + TX + TY + 31) / 32 * 32 + (NC == 256 ? 32 : 0);
  static constexpr int PX = TX + 3, PY = TY + 3; // W / E^n region: x0-2 .. x0+TX
  static constexpr int G = PX * PY;
  static constexpr int NXU = (TX + 1) * TY;      // upper x states: cells x0-1 .. x0+TX-1
  static constexpr int NYU = TX * (TY + 1);      // upper y states: rows y0-1 .. y0+TY-1
  // offsets in elements
  static constexpr int W = 0;                    // [3][8][G]
  static constexpr int EN = W + 3 * 8 * G;       // [4][3][G]
  static constexpr int XU = EN + 4 * 3 * G;      // [7][NXU]
  static constexpr int YU = XU + 7 * NXU;        // [7][NYU]
  static constexpr int TOTAL = YU + 7 * NYU;
};

// The value of x, which the compiler does not see through.  The staged kernels
// pass slopes and face states through memory; here they stay in registers, where
// FP32 multiply-adds would be contracted across them and the bits would differ.
__device__ __forceinline__ float opaque(float x) {
  asm("" : "+f"(x));
  return x;
}
__device__ __forceinline__ double opaque(double x) { return x; }  // (the contracted FP64 build may)

// Limited slope of component q along axis d of the cell at ring position s of
// plane W0 (Wm, Wp: the planes below and above).
template <typename R, int TX, int TY>
__device__ __forceinline__ R pf_slope(const R* W0, const R* Wm, const R* Wp, int s, int d, int q, R w, int lim) {
  using L = PfLayout<TX, TY>;
  const int so = d == 0 ? 1 : L::PX;
  const R wm = d == 2 ? Wm[q * L::G + s] : W0[q * L::G + s - so];
  const R wp = d == 2 ? Wp[q * L::G + s] : W0[q * L::G + s + so];
  return limiter(lim, w - wm, wp - w);
}

// The predictor of one cell from the W ring: put(f, pw) takes the six
// predicted face states (f = 2 axis + side, primitives in xyz order), again
// with the cell's own w after the second positivity rule; duk is the Hancock
// increment (zero after that fallback) for the reference EMF.
template <typename R, int TX, int TY, typename Put>
__device__ __forceinline__ void pf_predict(const R* __restrict__ sm, int s, int zc, const SolverConsts<R>& sc,
                                           const StepDt<R>& st, R (&duk)[8], R (&w)[8], const Put& put) {
  using L = PfLayout<TX, TY>;
  const R* W0 = sm + L::W + (zc % 3) * 8 * L::G;
  const R* Wm = sm + L::W + ((zc + 2) % 3) * 8 * L::G;
  const R* Wp = sm + L::W + ((zc + 1) % 3) * 8 * L::G;
#pragma unroll
  for (int q = 0; q < 8; ++q) w[q] = W0[q * L::G + s];
  bool bad = false, bad2 = false;
  R du[8], dw[3][8];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int q = 0; q < 8; ++q) dw[d][q] = opaque(pf_slope<R, TX, TY>(W0, Wm, Wp, s, d, q, w[q], sc.limiter));
    if (face_rule1(w, dw[d])) bad = true;
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) du[q] = R(0);
  if (bad) {
    // first positivity rule: zero slopes (24 selects, where selecting w for each
    // face state takes 96; the increment is then +0 and the states are U(w))
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int q = 0; q < 8; ++q) dw[d][q] = R(0);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    R fwm[8], fwp[8], fm[8], fp[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      fwm[q] = w[q] - R(0.5) * dw[d][q];
      fwp[q] = w[q] + R(0.5) * dw[d][q];
    }
    flux_xyz(d, fwp, sc.igm1, fp);
    flux_xyz(d, fwm, sc.igm1, fm);
#pragma unroll
    for (int q = 0; q < 8; ++q) du[q] = du[q] - st.hdtdx[d] * (fp[q] - fm[q]);
  }
  // the face states anew, as the staged predictor takes them (not merged with
  // the flux's, which would change what is contracted)
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int q = 0; q < 8; ++q) dw[d][q] = opaque(dw[d][q]);
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    const int d = f / 2;
    R fw[8], u[8], pw[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) fw[q] = f % 2 ? w[q] + R(0.5) * dw[d][q] : w[q] - R(0.5) * dw[d][q];
    prim2cons(fw, sc.igm1, u);
#pragma unroll
    for (int q = 0; q < 8; ++q) u[q] = u[q] + du[q];
    cons2prim(u, sc.gm1, pw);
    if (!(pw[0] > R(0)) || !(pw[4] > R(0))) bad2 = true;
    put(f, pw);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) duk[q] = du[q];
  if (bad2) {  // second positivity rule: first order
#pragma unroll
    for (int f = 0; f < 6; ++f) put(f, w);
#pragma unroll
    for (int q = 0; q < 8; ++q) duk[q] = R(0);
  }
}

// The cell EMF E^n_a at ring position s of plane z.
template <typename R, int TX, int TY> __device__ __forceinline__ R pf_en(const R* __restrict__ sm, int a, int s, int z) {
  using L = PfLayout<TX, TY>;
  return sm[L::EN + ((z & 3) * 3 + a) * L::G + s];
}

// E^n average at the axis-a edge stored at ring position s of plane z (the
// four cells around it, the staged expression and order).
template <typename R, int TX, int TY, int a>
__device__ __forceinline__ R pf_edge(const R* __restrict__ sm, int s, int z) {
  using L = PfLayout<TX, TY>;
  constexpr int b = (a + 1) % 3, cc = (a + 2) % 3;
  constexpr int so[3] = {1, L::PX, 0}, zo[3] = {0, 0, 1};
  const R e00 = pf_en<R, TX, TY>(sm, a, s - so[b] - so[cc], z - zo[b] - zo[cc]);
  const R e10 = pf_en<R, TX, TY>(sm, a, s - so[cc], z - zo[cc]);
  const R e01 = pf_en<R, TX, TY>(sm, a, s - so[b], z - zo[b]);
  const R e11 = pf_en<R, TX, TY>(sm, a, s, z);
  return Tr<R>::quarter(e00 + e10 + e01 + e11);
}

// The flux of the axis-d lower face of a tile cell (element x, ring position
// s of plane zc) between the face states lf and rf (7 values in the face's
// rotated frame): the CT half-step normal field from edge averages of E^n,
// then HLLD.
template <typename R, int TX, int TY, int d>
__device__ __forceinline__ void pf_face(const R* __restrict__ sm, const DPatch& p, const StepDt<R>& st,
                                        const SolverConsts<R>& sc, R* scr, int64_t x, int s, int zc, const R (&lf)[7],
                                        const R (&rf)[7]) {
  using L = PfLayout<TX, TY>;
  constexpr int b = (d + 1) % 3, cc = (d + 2) % 3;
  constexpr int so[3] = {1, L::PX, 0}, zo[3] = {0, 0, 1};
  const R dEc = pf_edge<R, TX, TY, cc>(sm, s + so[b], zc + zo[b]) - pf_edge<R, TX, TY, cc>(sm, s, zc);
  const R dEb = pf_edge<R, TX, TY, b>(sm, s + so[cc], zc + zo[cc]) - pf_edge<R, TX, TY, b>(sm, s, zc);
  const R bh = ((const R*)p.B[d])[x] - (st.hdtdx[b] * dEc - st.hdtdx[cc] * dEb);
  const R Lf[8] = {lf[0], lf[1], lf[2], lf[3], lf[4], R(0), lf[5], lf[6]};
  const R Rf[8] = {rf[0], rf[1], rf[2], rf[3], rf[4], R(0), rf[5], rf[6]};
  R fr[8], f[8], upw;
  hlld<R, kFastRecip>(d, Lf, Rf, bh, sc.gamma, sc.igm1, sc.eps_up, sc.emf != 1, fr, &upw);
  rot_out(d, fr, f);
  f[5 + d] = upw;
  VecIO<R>::store8(arr(scr, p, SC_F + d * 8), p.snelem, x, f);
}

template <typename R, int TX, int TY, int MINB>
__global__ void __launch_bounds__(PfLayout<TX, TY>::NT, MINB)
    k_pf(const DPatch* __restrict__ P, const FusedItem* __restrict__ items, R* scr, const R* __restrict__ K,
         SolverConsts<R> sc, int* status) {
  using L = PfLayout<TX, TY>;
  extern __shared__ __align__(16) unsigned char pf_smem[];
  R* sm = reinterpret_cast<R*>(pf_smem);
  const FusedItem it = items[blockIdx.x];
  const DPatch& p = P[it.patch];
  const StepDt<R> st(K, it.patch);
  const int x0 = it.x0, y0 = it.y0, z0 = it.z0, z1 = it.z1, tx = it.tx, ty = it.ty;
  const int nc = tx * ty;                   // tile cells
  const int lo = p.g - p.k;                 // update box
  const int hix = p.g + p.n[0] - 1 + p.k, hiy = p.g + p.n[1] - 1 + p.k, hiz = p.g + p.n[2] - 1 + p.k;
  // this thread's predictor cell: tile, lower row (y0 - 1), left column
  // (x0 - 1) or none
  const int t = threadIdx.x;
  int cx = x0 - 2, cy = y0 - 2;
  const bool tile = t < nc;
  if (tile) {
    cx = x0 + t % tx;
    cy = y0 + t / tx;
  } else if (t < nc + tx) {
    cx = x0 + (t - nc);
    cy = y0 - 1;
  } else if (t < nc + tx + ty) {
    cx = x0 - 1;
    cy = y0 + (t - nc - tx);
  }
  // inside UB+1: the predictor is defined there
  const bool act = t < nc + tx + ty && cx >= lo - 1 && cx <= hix + 1 && cy >= lo - 1 && cy <= hiy + 1;
  // this thread's lower faces, on planes where the axis allows
  const bool facet = tile && cx <= hix + 1 && cy <= hiy + 1;
  const int s = (cy - (y0 - 2)) * L::PX + (cx - (x0 - 2));
  const int zstart = z0 - 1 >= lo - 1 ? z0 - 1 : z0;
  const int64_t s1 = p.s1, s2 = p.s2;
  const int rx = tx + 3, nr = rx * (ty + 3);
  // primitives and E^n of the ring cells rr, rr + step, ... of plane zl
  auto load_cells = [&](int zl, int rr, int step) {
    if (zl < lo - 2 || zl > hiz + 2) return;
    R* W = sm + L::W + (zl % 3) * 8 * L::G;
    R* En = sm + L::EN + (zl & 3) * 3 * L::G;
    for (; rr < nr; rr += step) {
      int lx;
      const int ly = divmod24(rr, rx, lx);
      const int r = ly * L::PX + lx;
      const int gx = x0 - 2 + lx, gy = y0 - 2 + ly;
      if (gx < lo - 2 || gx > hix + 2 || gy < lo - 2 || gy > hiy + 2) continue;
      R w[8];
      load_prim(p, (int64_t)gx + (int64_t)gy * s1 + (int64_t)zl * s2, sc, w);
      if (sc.rho_floor > R(0) && !(w[0] >= sc.rho_floor)) w[0] = sc.rho_floor;
      if (sc.p_floor > R(0) && !(w[4] >= sc.p_floor)) w[4] = sc.p_floor;
#pragma unroll
      for (int q = 0; q < 8; ++q) W[q * L::G + r] = w[q];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int b = (a + 1) % 3, cc = (a + 2) % 3;
        En[a * L::G + r] = w[1 + cc] * w[5 + b] - w[1 + b] * w[5 + cc];
      }
      if (!(w[0] > R(0)) || !(w[4] > R(0))) raise_status(status, -4);
    }
  };
  for (int zl = zstart - 1; zl <= zstart + 1; ++zl) load_cells(zl, t, L::NT);
  __syncthreads();
  R zlow[7];  // this tile cell's upper z state on plane zc - 1
#pragma unroll
  for (int q = 0; q < 7; ++q) zlow[q] = R(0);
  for (int zc = zstart; zc < z1; ++zc) {
    // predictor of this thread's cell on plane zc; a tile cell keeps its
    // lower states and its upper z state
    R own[3][7], zup[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) zup[q] = own[0][q] = own[1][q] = own[2][q] = R(0);
    if (act) {
      R duk[8], w[8];
      R* const xu = sm + L::XU + (cy - y0) * (TX + 1) + (cx - (x0 - 1));
      R* const yu = sm + L::YU + (cy - (y0 - 1)) * TX + (cx - x0);
      const bool px = cy >= y0, py = cx >= x0;  // not the lower row, not the left column
      pf_predict<R, TX, TY>(sm, s, zc, sc, st, duk, w, [&](int f, const R (&pw)[8]) {
        const int d = f >> 1, t1 = (d + 1) % 3, t2 = (d + 2) % 3;
        const R v[7] = {opaque(pw[0]), opaque(pw[1 + d]), opaque(pw[1 + t1]), opaque(pw[1 + t2]),
                        opaque(pw[4]), opaque(pw[5 + t1]), opaque(pw[5 + t2])};
        if (f == 1) {
          if (px) {
#pragma unroll
            for (int q = 0; q < 7; ++q) xu[q * L::NXU] = v[q];
          }
        } else if (f == 3) {
          if (py) {
#pragma unroll
            for (int q = 0; q < 7; ++q) yu[q * L::NYU] = v[q];
          }
        } else {
#pragma unroll
          for (int q = 0; q < 7; ++q) (f == 5 ? zup : own[d])[q] = v[q];
        }
      });
      if (tile && sc.emf != 1 && zc >= z0) {
        // reference cell EMF from U^{n+1/2}, read by the upwinded EMF average
        const int64_t x = (int64_t)cx + (int64_t)cy * s1 + (int64_t)zc * s2;
        reference_emf(p, x, scr, sc, w, duk);
      }
    }
    __syncthreads();
    // the faces of plane zc, and the ring's next plane
    const bool next = zc + 1 < z1;
    const bool faces = facet && zc >= z0;
    const int64_t x = (int64_t)cx + (int64_t)cy * s1 + (int64_t)zc * s2;
    if (next) load_cells(zc + 2, t, tile ? nr : L::NT - nc);
    if (faces && zc >= lo && zc > zstart) pf_face<R, TX, TY, 2>(sm, p, st, sc, scr, x, s, zc, zlow, own[2]);
    R left[7];
    if (faces && cx >= lo) {
      const R* xu = sm + L::XU + (cy - y0) * (TX + 1) + (cx - x0);  // cell cx - 1
#pragma unroll
      for (int q = 0; q < 7; ++q) left[q] = xu[q * L::NXU];
      pf_face<R, TX, TY, 0>(sm, p, st, sc, scr, x, s, zc, left, own[0]);
    }
    if (faces && cy >= lo) {
      const R* yu = sm + L::YU + (cy - y0) * TX + (cx - x0);        // row cy - 1
#pragma unroll
      for (int q = 0; q < 7; ++q) left[q] = yu[q * L::NYU];
      pf_face<R, TX, TY, 1>(sm, p, st, sc, scr, x, s, zc, left, own[1]);
    }
#pragma unroll
    for (int q = 0; q < 7; ++q) zlow[q] = zup[q];
    // the next plane's predictor reads the ring and replaces the upper states
    __syncthreads();
  }
}
