// Fused persistent FP32 stage kernels for 16^3 and 16^2 blocks with a limiter of
// two ghost cells.
//
// What bounds them is instruction issue (the state moves at a fifth of the HBM
// rate, 62% of the issue slots are used), so the layout is chosen for
// instructions per cell at 16 warps an SM:
//   - a cell's limited slopes are evaluated once and give both of its face
//     states; the state that the next cell's face needs goes through the
//     face-flux array (x, y) or stays in a register (z, along the march);
//   - planes keep two variables next to each other, so that the slopes of two
//     variables are one packed evaluation on 8-byte shared-memory reads;
//   - 3D: the x and the y face of a cell are solved together, one per lane of the
//     packed instructions (HLLD: 196 instructions a face, against 233 with the two
//     sides of one face in the lanes); the z face with its two sides in the lanes;
//   - a face flux is evaluated once per block, by the thread of the cell above
//     the face; the 32 faces on the +x/+y boundary by one of warps 4 .. 7 with the
//     same code (warps 0 .. 3 convert the halo), the slopes of the cells around the
//     block by all warps.  A ninth warp for them would take the registers from 128
//     to 96 a thread;
//   - planes are copied one iteration ahead of their conversion.
// Against one slope a face and 272 threads with one barrier a plane: 58 -> 49
// warp instructions a cell and stage without the waits, a stage of 256^3 cells
// 1.48 -> 1.22 ms, a step of the 3D AMR blast (75 M cells) 21.4 -> 18.0 ms, of 256
// 2D instances (15.4 M cells) 3.67 -> 3.26 ms.  Two cells a thread (x, x + 1 in the
// lanes, 168 registers, 10 warps an SM) needed 44 instructions but issued in 35%
// of the slots: 26.5 ms.
//
// 3D: one CTA of 256 threads (a column each) per block, two CTAs an SM, marching
// over z with a ring of four primitive planes with their two-cell x/y halo.
// Iteration z, with planes z and z+1 converted and the copies of plane z+2 issued:
//   x and y slopes of plane z, states handed over;
//   arrive 1; convert plane z+2 (own cell; threads 0 .. 127 one halo cell) in
//   place; issue the copies of U0 of plane z and of plane z+3; wait 1;
//   x and y fluxes of plane z into the flux arrays;
//   arrive 2; z slopes of cell z+1, flux of face z+1/2 (own column); wait 2;
//   update of plane z.
// The two barriers are split (mbarriers, one arrival per warp), so that a warp
// works on its own column while the others catch up: the warps of the block
// boundary have up to 250 instructions more in a plane.  The flux arrays are
// double-buffered by plane parity: the states of plane z+1 are handed over after
// both waits of plane z, i.e. once every warp has updated plane z-1.  After wait 2
// every warp is done with the neighbours in plane z, whose ring slot is refilled
// in the next iteration.
#pragma once

#include "physics_f2.cuh"

namespace amrvac {

constexpr int F2_T = FB * FB;
constexpr int F2_PW = FB + 2 * NG;
constexpr int F2_NH = 4 * NG * FB;  // halo cells of a plane

// one plane of cells: the variables (rho, p), (vx, vy), (vz, Bz), (Bx, By) in
// pairs, psi by itself
struct F2Plane {
  float2 pr[4][F2_PW][F2_PW];
  float psi[F2_PW][F2_PW];
};
__host__ __device__ constexpr int f2_first(int k) { return k == 0 ? 0 : k == 1 ? 1 : k == 2 ? 3 : 5; }
__host__ __device__ constexpr int f2_second(int k) { return k == 0 ? 4 : k == 1 ? 2 : k == 2 ? 7 : 6; }
__device__ __forceinline__ float* f2_at(F2Plane& p, int v, int j, int i) {
  if (v == 8) return &p.psi[j][i];
  const int k = v == 0 || v == 4 ? 0 : v == 1 || v == 2 ? 1 : v == 3 || v == 7 ? 2 : 3;
  return reinterpret_cast<float*>(&p.pr[k][j][i]) + (v == f2_first(k) ? 0 : 1);
}

using F2Fx = float[NV][FB][FXW];
using F2Fy = float[NV][FB + 1][FXW];

struct FusedF2Smem {
  F2Plane plane[4];
  F2Fx fx[2];
  F2Fy fy[2];
  float u0[NV][FB * FB];
  float red[F2_T / 32][2];
  unsigned long long bar[2];
  int next;
};

struct Fused2dF2Smem {
  F2Plane tile[2];  // by block parity: conserved, converted in place
  float u0[2][NV][FB * FB];
  F2Fx fx[2];
  F2Fy fy[2];
  unsigned long long bar[3];
  int first[2];
  int next[2];
};

// A split barrier of the CTA's warps: every warp arrives once a phase, waits
// come later.  The wait is bounded (a lost arrival would latch
// AMRVAC_E_TIMEOUT, not hang).
__device__ __forceinline__ void f2_bar_init(unsigned long long* bar) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(a), "r"(F2_T / 32) : "memory");
}
__device__ __forceinline__ void f2_arrive(unsigned long long* bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
    asm volatile("{\n.reg .b64 t;\nmbarrier.arrive.shared.b64 t, [%0];\n}" ::"r"(a) : "memory");
  }
}
__device__ __forceinline__ void f2_wait(unsigned long long* bar, int parity, int* err, int b) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  for (int n = 0; n < (1 << 20); n++) {
    int done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared.b64 p, [%1], %2;\n"
        "selp.b32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return;
  }
  latch_error(err, AMRVAC_E_TIMEOUT, b, threadIdx.x, 0);
}

// Halo cell h (0 .. 127) of a plane: x halo, then y halo
__device__ __forceinline__ void f2_halo_xy(int h, int& hx, int& hy) {
  if (h < F2_NH / 2) {
    const int side = h / (NG * FB), r = h % (NG * FB);
    hy = r / NG;
    hx = side ? FB + r % NG : -NG + r % NG;
  } else {
    const int u = h - F2_NH / 2, side = u / (NG * FB), r = u % (NG * FB);
    hx = r % FB;
    hy = side ? FB + r / FB : -NG + r / FB;
  }
}

struct F2Prim {
  const StageParams* sp;
  double gammad;
  float gm1f;
  bool ff;
};

// conserved -> primitive of cell (j, i) of a plane, in place; true when it is
// small (Sect. 7.4)
__device__ __forceinline__ bool f2_convert(F2Plane& P, int j, int i, int flip, const F2Prim& c) {
  float u[NV], w[NV];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const float2 t = P.pr[k][j][i];
    u[f2_first(k)] = t.x;
    u[f2_second(k)] = t.y;
  }
  const float ir = 1.f / u[0];
  w[0] = u[0];
#pragma unroll
  for (int v = 1; v < 4; v++) w[v] = u[v] * ir;
  if (c.ff)
    w[4] = pressure_ff(c.gm1f, u, w[1], w[2], w[3]);
  else
    w[4] = pressure_of(c.gammad, u, w[1], w[2], w[3]);
#pragma unroll
  for (int v = 5; v < 8; v++) w[v] = u[v];
  if (flip) wall_flip(flip, w);
  *f2_at(P, 4, j, i) = w[4];
  P.pr[1][j][i] = make_float2(w[1], w[2]);
  if (flip) {
    P.pr[2][j][i] = make_float2(w[3], w[7]);
    P.pr[3][j][i] = make_float2(w[5], w[6]);
  } else {
    *f2_at(P, 3, j, i) = w[3];
  }
  return c.sp->check_small &&
         is_small_prim(w[0], w[4], c.sp->small_density_f, c.sp->small_pressure_f);
}

// the variable pairs of a plane
#define F2_PAIRS(k, va, vb) constexpr int va##_[4] = {0, 1, 3, 5}, vb##_[4] = {4, 2, 7, 6}; \
  const int va = va##_[k], vb = vb##_[k]

// x and y slopes of one plane of primitives, by all threads: the states at the
// low faces of cell (x, y) stay in lox and loy, those at its high faces go to
// the neighbour through fx and fy.  The cells around the block are shared by the
// warps: their states at faces 0 go to fx and fy too, those at faces 16 to the
// column F2_HLO of the flux arrays that no face uses.
constexpr int F2_HLO = FB + 1;

template <int LIM>
__device__ __forceinline__ void f2_xy_slopes(const F2Plane& P, F2Fx& fx, F2Fy& fy, int x, int y,
                                             int lim, SymLim sl, float* lox, float* loy) {
  const int X = x + NG, Y = y + NG;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    F2_PAIRS(k, va, vb);
    const float2 c = P.pr[k][Y][X];
    float2 s, t;  // increments to the low and the high face
    cell_increments2<LIM>(P.pr[k][Y][X - 1], c, P.pr[k][Y][X + 1], lim, sl, s, t);
    lox[va] = c.x - s.x;
    lox[vb] = c.y - s.y;
    fx[va][y][x + 1] = c.x + t.x;
    fx[vb][y][x + 1] = c.y + t.y;
    cell_increments2<LIM>(P.pr[k][Y - 1][X], c, P.pr[k][Y + 1][X], lim, sl, s, t);
    loy[va] = c.x - s.x;
    loy[vb] = c.y - s.y;
    fy[va][y + 1][x] = c.x + t.x;
    fy[vb][y + 1][x] = c.y + t.y;
  }
  {
    // psi: its x and y slopes in the two lanes
    const float c = P.psi[Y][X];
    float2 s, t;
    cell_increments2<LIM>(make_float2(P.psi[Y][X - 1], P.psi[Y - 1][X]), sp2(c),
                          make_float2(P.psi[Y][X + 1], P.psi[Y + 1][X]), lim, sl, s, t);
    lox[8] = c - s.x;
    loy[8] = c - s.y;
    fx[8][y][x + 1] = c + t.x;
    fy[8][y + 1][x] = c + t.y;
  }
  {
    // the cells around the block: warp w the pair w & 3 of the cells -1 (w < 4) or
    // 16, lane r < 16 in row r along x, lane 16 + r in column r along y; no branch,
    // so that these slopes overlap with the others
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = lane & 15, k = warp & 3;
    const bool ydir = lane >= 16, far = warp >= 4;
    const int st = ydir ? F2_PW : 1, base = ydir ? r + NG : (r + NG) * F2_PW;
    const int os = ydir ? (FB + 1) * FXW : FB * FXW;
    float* near = ydir ? &fy[0][0][r] : &fx[0][r][0];
    float* hlo = ydir ? &fy[0][r][F2_HLO] : &fx[0][r][F2_HLO];
    const float2* p = &P.pr[0][0][0] + k * F2_PW * F2_PW + base + (far ? FB + NG - 1 : NG - 2) * st;
    const float2 c = p[st];
    float2 s, t;
    cell_increments2<LIM>(p[0], c, p[2 * st], lim, sl, s, t);
    float* out = far ? hlo : near;
    out[f2_first(k) * os] = far ? c.x - s.x : c.x + t.x;
    out[f2_second(k) * os] = far ? c.y - s.y : c.y + t.y;
    if (warp == 7) {  // psi of cells -1 and 16 in the two lanes
      const float* q = &P.psi[0][0] + base;
      const float2 d = make_float2(q[(NG - 1) * st], q[(FB + NG) * st]);
      cell_increments2<LIM>(make_float2(q[(NG - 2) * st], q[(FB + NG - 1) * st]), d,
                            make_float2(q[NG * st], q[(FB + NG + 1) * st]), lim, sl, s, t);
      near[8 * os] = d.x + t.x;
      hlo[8 * os] = d.y - s.y;
    }
  }
}

// the x and y fluxes, thread (x, y) the faces on the low side of its cell, both at
// once; the warp of `boundary` then, lane r < 16, the +x boundary face of row r
// and the +y boundary face of column r with the same code (a plane's code has to
// stay in the instruction cache).  keep(face, cell, f) sees every flux on the
// block boundary.
template <int FLUX, class Keep>
__device__ __forceinline__ void f2_xy_solve(F2Plane& P, F2Fx& fx, F2Fy& fy, int x, int y,
                                            bool boundary, const float* lox, const float* loy,
                                            const FaceConst2& fc, Keep keep) {
  constexpr int SX = FB * FXW, SY = (FB + 1) * FXW;
  float2 wr[NV];
#pragma unroll
  for (int c = 0; c < NV; c++) wr[c] = make_float2(lox[c], loy[yface_var(c)]);
  float *ax = &fx[0][y][x], *ay = &fy[0][y][x];
  const int lane = threadIdx.x & 31;
  // cells above the x face and above the y face
  int jx = y + NG, ix = x + NG, jy = y + NG, iy = x + NG;
  const int last = boundary && lane < 16;
#pragma unroll 1
  for (int pass = 0; pass <= last; pass++) {
    float2 wl[NV], f[NV];
    if (pass) {
      ax = &fx[0][lane][FB];
      ay = &fy[0][FB][lane];
      const float *hx = &fx[0][lane][F2_HLO], *hy = &fy[0][lane][F2_HLO];
#pragma unroll
      for (int c = 0; c < NV; c++) wr[c] = make_float2(hx[c * SX], hy[yface_var(c) * SY]);
      jx = iy = lane + NG;
      ix = jy = FB + NG;
    }
#pragma unroll
    for (int c = 0; c < NV; c++) wl[c] = make_float2(ax[c * SX], ay[yface_var(c) * SY]);
    // first order where a state is not positive (or NaN)
    const bool bx = !(wl[0].x > 0.f) || !(wl[4].x > 0.f) || !(wr[0].x > 0.f) || !(wr[4].x > 0.f);
    const bool by = !(wl[0].y > 0.f) || !(wl[4].y > 0.f) || !(wr[0].y > 0.f) || !(wr[4].y > 0.f);
    if (bx || by) {
#pragma unroll
      for (int c = 0; c < NV; c++) {
        const int d = yface_var(c);
        if (bx) {
          wl[c].x = *f2_at(P, c, jx, ix - 1);
          wr[c].x = *f2_at(P, c, jx, ix);
        }
        if (by) {
          wl[c].y = *f2_at(P, d, jy - 1, iy);
          wr[c].y = *f2_at(P, d, jy, iy);
        }
      }
    }
    face_flux_xy<FLUX>(wl, wr, fc, f);
#pragma unroll
    for (int c = 0; c < NV; c++) {
      ax[c * SX] = f[c].x;
      ay[yface_var(c) * SY] = f[c].y;
    }
    if (pass || x == 0) {
      float g[NV];
#pragma unroll
      for (int c = 0; c < NV; c++) g[c] = f[c].x;
      keep(pass, pass ? lane : y, g);
    }
    if (pass || y == 0) {
      float g[NV];
#pragma unroll
      for (int c = 0; c < NV; c++) g[yface_var(c)] = f[c].y;
      keep(2 + pass, pass ? lane : x, g);
    }
  }
}

// The same fluxes with one face at a time, its two sides in the lanes: more
// instructions (233 a face against 196 with HLLD) in shorter chains, the better one
// where a block is a single plane (see k_fused2d_f2).
template <int FLUX, class Keep>
__device__ __forceinline__ void f2_xy_solve_sides(F2Plane& P, F2Fx& fx, F2Fy& fy, int x, int y,
                                                  bool boundary, const float* lox,
                                                  const float* loy, const FaceConst2& fc,
                                                  Keep keep) {
  const int X = x + NG, Y = y + NG;
  float2 w[NV];
  float f[NV];
  auto cells = [&](int j, int i, int dj, int di) {  // first order: the cells on both sides
#pragma unroll
    for (int v = 0; v < NV; v++) w[v] = make_float2(*f2_at(P, v, j - dj, i - di), *f2_at(P, v, j, i));
  };
#pragma unroll
  for (int v = 0; v < NV; v++) w[v] = make_float2(fx[v][y][x], lox[v]);
  if (not_positive2(w)) cells(Y, X, 0, 1);
  face_flux2<0, FLUX>(w, fc, f);
#pragma unroll
  for (int v = 0; v < NV; v++) fx[v][y][x] = f[v];
  if (x == 0) keep(0, y, f);
#pragma unroll
  for (int v = 0; v < NV; v++) w[v] = make_float2(fy[v][y][x], loy[v]);
  if (not_positive2(w)) cells(Y, X, 1, 0);
  face_flux2<1, FLUX>(w, fc, f);
#pragma unroll
  for (int v = 0; v < NV; v++) fy[v][y][x] = f[v];
  if (y == 0) keep(2, x, f);
  if (boundary) {
    // the faces 16, one a lane (x faces, then y faces), in the face's local frame
    // (component c is variable var(c))
    const int lane = threadIdx.x & 31, r = lane & 15;
    const bool ydir = lane >= 16;
    auto var = [&](int c) { return ydir ? yface_var(c) : c; };
    float* out = ydir ? &fy[0][FB][r] : &fx[0][r][FB];
    const float* hlo = ydir ? &fy[0][r][F2_HLO] : &fx[0][r][F2_HLO];
    const int os = ydir ? (FB + 1) * FXW : FB * FXW;
#pragma unroll
    for (int c = 0; c < NV; c++) w[c] = make_float2(out[var(c) * os], hlo[var(c) * os]);
    if (not_positive2(w)) {
      if (ydir) {
        float2 g[NV];
        cells(FB + NG, r + NG, 1, 0);
#pragma unroll
        for (int c = 0; c < NV; c++) g[c] = w[yface_var(c)];
#pragma unroll
        for (int c = 0; c < NV; c++) w[c] = g[c];
      } else {
        cells(r + NG, FB + NG, 0, 1);
      }
    }
    face_flux2<0, FLUX>(w, fc, f);
#pragma unroll
    for (int c = 0; c < NV; c++) out[var(c) * os] = f[c];
    float g[NV];  // in variable order
#pragma unroll
    for (int c = 0; c < NV; c++) g[yface_var(c)] = f[c];
#pragma unroll
    for (int c = 0; c < NV; c++) g[c] = ydir ? g[c] : f[c];
    keep(ydir ? 3 : 1, r, g);
  }
}

template <int LIM, int FLUX, bool FULL>
__global__ void __launch_bounds__(F2_T, 2)
    k_fused_f2(DevMesh M, const float* U0, const float* __restrict__ Uk, const float* U2,
               float* out, float* out2, const int* __restrict__ work, int nwork,
               const float* __restrict__ gslab, int* __restrict__ counter, StageParams sp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  FusedF2Smem& S = *reinterpret_cast<FusedF2Smem*>(smraw);
  constexpr int PL = FB * FB;
  constexpr int SLAB_FACE = NV * NG * PL;  // one face: [v][layer][t2][t1]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int x = lane & 15, y = fused_row(warp, lane);
  const size_t vs = (size_t)M.nblocks * M.ncell;
  const bool ff = sp.pressure_ff != 0;
  const SymLim sl = sym_lim(sp.limiter);
  const bool halo = tid < F2_NH;
  int hx = 0, hy = 0;
  if (halo) f2_halo_xy(tid, hx, hy);
  if (tid == 0) {
    f2_bar_init(&S.bar[0]);
    f2_bar_init(&S.bar[1]);
  }
  __syncthreads();

  // work distribution: static (CTA i takes items i, i + grid, ...) or dynamic
  // (each CTA draws its next item from a counter the host zeroes per launch)
  auto next_work = [&](int wi) -> int {
    if (!counter) return wi + gridDim.x;
    __syncthreads();
    if (tid == 0) S.next = atomicAdd(counter, 1);
    __syncthreads();
    return S.next;
  };
  for (int wi = counter ? next_work(0) : blockIdx.x; wi < nwork; wi = next_work(wi)) {
    const int b = work[wi];
    const int q = M.blk[b * 5], L = M.blk[b * 5 + 1];
    const double gammad = ff ? 0.0 : M.gamma[q];
    const float* lc = M.lcf + (q * MAXLEV + L) * LC_N;
    const float g = lc[LC_G], gm1f = lc[LC_GM1];
    const float idd[3] = {lc[LC_IDX], lc[LC_IDX + 1], lc[LC_IDX + 2]};
    const size_t own = (size_t)b * M.ncell + y * FB + x;  // own cell of plane 0
    float smx = 0.f, cmx = 0.f;  // CFL terms of the new state (last stage)

    if (lc[LC_SKIP] != 0.f) {
      // finished instance: copied through unchanged
      for (int z = 0; z < FB; z++) {
        float u[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) {
          const size_t at = (size_t)v * vs + own + z * PL;
          u[v] = Uk[at];
          out[at] = u[v];
          if (FULL && sp.has2) out2[at] = u[v];
        }
        if (sp.epilogue) cfl_terms<float, 3>(u, gammad, g, ff, gm1f, idd, smx, cmx);
      }
    } else {
      const float dt = lc[LC_DT], damp = lc[LC_DAMP];
      const FaceConst2 fc = face_const2(g, lc[LC_CH], sp.glm);
      // neighbour codes: a level-change face reads its ghost slab (code -3 -
      // slab); (FULL) a symmetric wall reads the block's own mirrored cells: bit
      // f of wmask marks face f, whose code becomes the outflow one
      int wmask = 0;
      auto nbr = [&](int f) {
        int code = M.nbr[b * 6 + f];
        if (FULL && code == NBR_WALL) {
          code = NBR_OUTFLOW;
          wmask |= 1 << f;
        }
        return code == NBR_GENERAL ? -3 - M.gface[b * 6 + f] : code;
      };
      int nb[6];
#pragma unroll
      for (int f = 0; f < 6; f++) nb[f] = nbr(f);
      // this thread's halo cell (x or y ghost layers): its values in plane 0, and
      // the strides to the next variable and the next plane
      const float* hp = Uk;
      size_t hvs = vs;
      int hzs = PL, hflip = 0;
      if (halo) {
        const bool xf = tid < F2_NH / 2;
        const int n = xf ? hx : hy, t1 = xf ? hy : hx;
        const int f = (xf ? 0 : 2) + (n < 0 ? 0 : 1);
        const int code = xf ? (n < 0 ? nb[0] : nb[1]) : (n < 0 ? nb[2] : nb[3]);
        if (code <= -3) {
          hp = gslab + (size_t)(-3 - code) * SLAB_FACE + (n < 0 ? n + NG : n - FB) * PL + t1;
          hvs = NG * PL;
          hzs = FB;
        } else {
          int nn = code >= 0 ? (n < 0 ? n + FB : n - FB) : (n < 0 ? 0 : FB - 1);
          if (FULL && ((wmask >> f) & 1)) {
            nn = n < 0 ? -1 - n : 2 * FB - 1 - n;
            hflip = 1 << (f >> 1);
          }
          hp = Uk + (size_t)(code >= 0 ? code : b) * M.ncell + (xf ? t1 * FB + nn : nn * FB + t1);
        }
      }
      // copies of plane pz (-2 .. 17) into its ring slot
      auto issue_plane = [&](int pz) {
        F2Plane& P = S.plane[pz & 3];
        const float* src = Uk + own;
        size_t st = vs;
        if (pz >= 0 && pz < FB) {
          src += pz * PL;
        } else {
          const int code = pz < 0 ? nb[4] : nb[5];
          if (code <= -3) {
            src = gslab + (size_t)(-3 - code) * SLAB_FACE + (pz < 0 ? pz + NG : pz - FB) * PL +
                  y * FB + x;
            st = NG * PL;
          } else {
            int nn = code >= 0 ? (pz & (FB - 1)) : (pz < 0 ? 0 : FB - 1);
            if (FULL && (wmask & (pz < 0 ? 16 : 32))) nn = pz < 0 ? -1 - pz : 2 * FB - 1 - pz;
            src = Uk + (size_t)(code >= 0 ? code : b) * M.ncell + nn * PL + y * FB + x;
          }
        }
#pragma unroll
        for (int v = 0; v < NV; v++)
          cp_async_elem_after_reads(f2_at(P, v, y + NG, x + NG), src + v * st);
        if (halo && pz >= 0 && pz < FB) {
          const float* hs = hp + pz * hzs;
#pragma unroll
          for (int v = 0; v < NV; v++)
            cp_async_elem_after_reads(f2_at(P, v, hy + NG, hx + NG), hs + v * hvs);
        }
      };
      const F2Prim pc = {&sp, gammad, gm1f, ff};
      auto convert = [&](int pz) {
        F2Plane& P = S.plane[pz & 3];
        const int flip = FULL && ((pz < 0 && (wmask & 16)) || (pz >= FB && (wmask & 32))) ? 4 : 0;
        bool bad = f2_convert(P, y + NG, x + NG, flip, pc);
        if (halo && pz >= 0 && pz < FB) bad |= f2_convert(P, hy + NG, hx + NG, hflip, pc);
        if (bad) latch_error(M.err, AMRVAC_E_SMALL_VALUES, b, tid, 0);
      };
      // z faces of the own column: wz[v] = (state of cell zc-1, of cell zc) at the
      // face below plane zc; zslopes leaves the state of cell zc at its upper face
      // in hi
      float2 wz[NV];
      auto zslopes = [&](int zc, float* hi) {
        const F2Plane &A = S.plane[(zc - 1) & 3], &B = S.plane[zc & 3], &C = S.plane[(zc + 1) & 3];
        float2 s, t;
#pragma unroll
        for (int k = 0; k < 4; k++) {
          F2_PAIRS(k, va, vb);
          const float2 c = B.pr[k][y + NG][x + NG];
          cell_increments2<LIM>(A.pr[k][y + NG][x + NG], c, C.pr[k][y + NG][x + NG], sp.limiter,
                                sl, s, t);
          wz[va].y = c.x - s.x;
          wz[vb].y = c.y - s.y;
          hi[va] = c.x + t.x;
          hi[vb] = c.y + t.y;
        }
        const float c = B.psi[y + NG][x + NG];
        cell_increments2<LIM>(sp2(A.psi[y + NG][x + NG]), sp2(c), sp2(C.psi[y + NG][x + NG]),
                              sp.limiter, sl, s, t);
        wz[8].y = c - s.x;
        hi[8] = c + t.x;
      };
      auto zflux = [&](int zc, float* f) {
        float hi[NV];
        zslopes(zc, hi);
        if (not_positive2(wz)) {
          const F2Plane &A = S.plane[(zc - 1) & 3], &B = S.plane[zc & 3];
#pragma unroll
          for (int k = 0; k < 4; k++) {
            F2_PAIRS(k, va, vb);
            const float2 a = A.pr[k][y + NG][x + NG], c = B.pr[k][y + NG][x + NG];
            wz[va] = make_float2(a.x, c.x);
            wz[vb] = make_float2(a.y, c.y);
          }
          wz[8] = make_float2(A.psi[y + NG][x + NG], B.psi[y + NG][x + NG]);
        }
        face_flux2<2, FLUX>(wz, fc, f);
#pragma unroll
        for (int v = 0; v < NV; v++) wz[v].x = hi[v];
      };
      auto keep = [&](int face, int idx, const float* f) {
        if (!FULL || !sp.reflux) return;
        const int code = face == 0   ? nb[0]
                         : face == 1 ? nb[1]
                         : face == 2 ? nb[2]
                         : face == 3 ? nb[3]
                         : face == 4 ? nb[4]
                                     : nb[5];
        if (code <= -3) keep_face_flux(M, code, idx, f);
      };

      float fzp[NV];
#pragma unroll 1
      for (int pz = -NG; pz < NG; pz++) issue_plane(pz);
      cp_async_commit();
      cp_async_wait_all();
#pragma unroll 1
      for (int pz = -NG; pz < NG; pz++) convert(pz);
      {
        float hi[NV];
        zslopes(-1, hi);
#pragma unroll
        for (int v = 0; v < NV; v++) wz[v].x = hi[v];
      }
      zflux(0, fzp);
      keep(4, y * FB + x, fzp);
      issue_plane(2);  // into the slot of plane -2, read by this thread only
      cp_async_commit();
      __syncthreads();  // planes 0 and 1 with their halos

      float lox[NV], loy[NV];
      auto slopes = [&](int z) {
        f2_xy_slopes<LIM>(S.plane[z & 3], S.fx[z & 1], S.fy[z & 1], x, y, sp.limiter, sl, lox,
                          loy);
      };
#pragma unroll 1
      for (int z = 0; z < FB; z++) {
        const int fb = z & 1;
        const size_t at0 = own + z * PL;
        slopes(z);
        f2_arrive(&S.bar[0]);
        cp_async_wait_all();  // plane z + 2, issued one iteration ago
        convert(z + 2);
        if (!sp.plain) {
#pragma unroll
          for (int v = 0; v < NV; v++)
            cp_async_elem_after_reads(&S.u0[v][tid], U0 + at0 + v * vs);
        }
        cp_async_commit();
        if (z + 3 < FB + NG) issue_plane(z + 3);
        cp_async_commit();
        f2_wait(&S.bar[0], fb, M.err, b);
        f2_xy_solve<FLUX>(S.plane[z & 3], S.fx[fb], S.fy[fb], x, y, warp == 4 + ((z + 2) & 3), lox,
                          loy, fc,
                          [&](int face, int t, const float* f) { keep(face, z * FB + t, f); });
        f2_arrive(&S.bar[1]);
        float uk[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) uk[v] = Uk[at0 + v * vs];
        float acc[NV];
        {
          float fz[NV];
          zflux(z + 1, fz);
          if (z == FB - 1) keep(5, y * FB + x, fz);
#pragma unroll
          for (int v = 0; v < NV; v++) {
            acc[v] = (fz[v] - fzp[v]) * idd[2];
            fzp[v] = fz[v];
          }
        }
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");  // U0 of plane z
        f2_wait(&S.bar[1], fb, M.err, b);

        float un[NV];
#pragma unroll
        for (int v = 0; v < NV; v++) {
          float a = fmaf(S.fx[fb][v][y][x + 1] - S.fx[fb][v][y][x], idd[0], acc[v]);
          a = fmaf(S.fy[fb][v][y + 1][x] - S.fy[fb][v][y][x], idd[1], a);
          const size_t at = at0 + v * vs;
          float ut = fmaf(-dt, a, uk[v]);
          if (v == 8) ut = ut * damp;
          un[v] = sp.plain ? ut : fmaf(sp.af, S.u0[v][tid], sp.bf * ut);
          if (FULL && sp.has2) {
            // SSPRK(5,4) stage 3: w = a2 U2 + b2 (Uk + c2 dt L); U2 is out's
            // register and out2 is U0's, both read above before their writes
            float ut2 = fmaf(-lc[LC_DT2], a, uk[v]);
            if (v == 8) ut2 = ut2 * lc[LC_DAMP2];
            out2[at] = sp.a2f * U2[at] + sp.b2f * ut2;
          }
          out[at] = un[v];
        }
        if (sp.epilogue) cfl_terms<float, 3>(un, gammad, g, ff, gm1f, idd, smx, cmx);
      }
    }
    if (sp.epilogue) {
      // maximum of the two CFL terms
      __syncthreads();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        smx = fmaxf(smx, __shfl_xor_sync(0xffffffffu, smx, o));
        cmx = fmaxf(cmx, __shfl_xor_sync(0xffffffffu, cmx, o));
      }
      if (lane == 0) {
        S.red[warp][0] = smx;
        S.red[warp][1] = cmx;
      }
      __syncthreads();
      if (tid < 2) {
        float a = S.red[0][tid];
        for (int w = 1; w < F2_T / 32; w++) a = fmaxf(a, S.red[w][tid]);
        M.part[(size_t)b * NPART + tid] = a;
      }
    }
  }
}

// 2D: a 16^2 block is one plane, so the CTA pipelines over its work list: the
// next block (with halo, and U0 for stages k > 0) is copied into the other of
// two slots and converted while the current one is computed.  Block n, converted:
//   wait 0; x and y slopes, states handed over                     arrive 1
//   issue the copies of block n+1;
//   wait 1; x and y fluxes                                         arrive 2
//   convert block n+1 in place (own cell, keeping its conserved values; threads
//   0 .. 127 one halo cell)                                        arrive 0
//   wait 2; update of block n.
// Slot n+1 was last read by the fluxes of block n-1, which every thread finished
// before wait 2 of that block; the flux arrays are double-buffered (see above).
template <int LIM, int FLUX, bool FULL>
__global__ void __launch_bounds__(F2_T, 2)
    k_fused2d_f2(DevMesh M, const float* U0, const float* __restrict__ Uk, const float* U2,
                 float* out, float* out2, const int* __restrict__ work, int nwork,
                 const float* __restrict__ gslab, int* __restrict__ counter, StageParams sp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  Fused2dF2Smem& S = *reinterpret_cast<Fused2dF2Smem*>(smraw);
  constexpr int SLAB_FACE = NV * NG * FB;  // one face: [v][layer][t1]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int x = lane & 15, y = fused_row(warp, lane);
  const size_t vs = (size_t)M.nblocks * M.ncell;
  const bool ff = sp.pressure_ff != 0;
  const SymLim sl = sym_lim(sp.limiter);
  const bool halo = tid < F2_NH;
  int hx = 0, hy = 0;
  if (halo) f2_halo_xy(tid, hx, hy);
  const bool xf = tid < F2_NH / 2;
  const int hn = xf ? hx : hy, ht = xf ? hy : hx;
  const int hface = (xf ? 0 : 2) + (hn < 0 ? 0 : 1);

  // copies of block bb into slot s
  auto issue = [&](int bb, int s) {
    const size_t own = (size_t)bb * M.ncell + y * FB + x;
    F2Plane& P = S.tile[s];
#pragma unroll
    for (int v = 0; v < NV; v++)
      cp_async_elem_after_reads(f2_at(P, v, y + NG, x + NG), Uk + own + v * vs);
    if (!sp.plain) {
#pragma unroll
      for (int v = 0; v < NV; v++) cp_async_elem_after_reads(&S.u0[s][v][tid], U0 + own + v * vs);
    }
    if (halo) {
      const float* src;
      size_t st = vs;
      const int code = M.nbr[bb * 6 + hface];
      if (code == NBR_GENERAL) {
        src = gslab + (size_t)M.gface[bb * 6 + hface] * SLAB_FACE +
              (hn < 0 ? hn + NG : hn - FB) * FB + ht;
        st = NG * FB;
      } else {
        int nn = code >= 0 ? (hn & (FB - 1)) : (hn < 0 ? 0 : FB - 1);
        if (FULL && code == NBR_WALL) nn = hn < 0 ? -1 - hn : 2 * FB - 1 - hn;
        src = Uk + (size_t)(code >= 0 ? code : bb) * M.ncell + (xf ? ht * FB + nn : nn * FB + ht);
      }
#pragma unroll
      for (int v = 0; v < NV; v++)
        cp_async_elem_after_reads(f2_at(P, v, hy + NG, hx + NG), src + v * st);
    }
    cp_async_commit();
  };

  // work items: static (i, i + grid, ...) or drawn from the counter; the item
  // after next is fetched by thread 0 between two barriers of a block
  int wi, wn;
  if (tid == 0) {
    for (int k = 0; k < 3; k++) f2_bar_init(&S.bar[k]);
    if (counter) {
      S.first[0] = atomicAdd(counter, 1);
      S.first[1] = atomicAdd(counter, 1);
    }
  }
  __syncthreads();
  if (counter) {
    wi = S.first[0];
    wn = S.first[1];
  } else {
    wi = blockIdx.x;
    wn = wi + gridDim.x;
  }
  // once its copies have landed: the conserved values of the own cell of block bb
  // (slot s) into u, and the conversion of the own and the halo cell
  auto convert = [&](int bb, int s, float* u) {
    F2Plane& P = S.tile[s];
    const int q = M.blk[bb * 5], L = M.blk[bb * 5 + 1];
    const float* lc = M.lcf + (q * MAXLEV + L) * LC_N;
    const double gammad = ff ? 0.0 : M.gamma[q];
#pragma unroll
    for (int v = 0; v < NV; v++) u[v] = f2_at(P, v, y + NG, x + NG)[0];
    if (lc[LC_SKIP] != 0.f) return;
    const F2Prim pc = {&sp, gammad, lc[LC_GM1], ff};
    bool bad = f2_convert(P, y + NG, x + NG, 0, pc);
    if (halo) {
      const int flip = FULL && M.nbr[bb * 6 + hface] == NBR_WALL ? 1 << (hface >> 1) : 0;
      bad |= f2_convert(P, hy + NG, hx + NG, flip, pc);
    }
    if (bad) latch_error(M.err, AMRVAC_E_SMALL_VALUES, bb, tid, 0);
  };
  float uk[NV];
  if (wi < nwork) {
    issue(work[wi], 0);
    cp_async_wait_all();
    convert(work[wi], 0, uk);
    f2_arrive(&S.bar[0]);
  }

  for (int it = 0; wi < nwork; it++) {
    const int s = it & 1;
    const int b = work[wi];
    const int q = M.blk[b * 5], L = M.blk[b * 5 + 1];
    const double gammad = ff ? 0.0 : M.gamma[q];
    const float* lc = M.lcf + (q * MAXLEV + L) * LC_N;
    const float g = lc[LC_G], gm1f = lc[LC_GM1];
    const float idd[3] = {lc[LC_IDX], lc[LC_IDX + 1], 0.f};
    const bool skip = lc[LC_SKIP] != 0.f;
    float smx = 0.f, cmx = 0.f;
    double* part_b = M.part + (size_t)b * NPART;
    f2_wait(&S.bar[0], s, M.err, b);
    if (tid == 0) {
      if (sp.epilogue) part_b[0] = part_b[1] = 0.0;
      if (counter) S.next[s] = atomicAdd(counter, 1);
    }
    float lox[NV], loy[NV];
    if (!skip)
      f2_xy_slopes<LIM>(S.tile[s], S.fx[s], S.fy[s], x, y, sp.limiter, sl, lox, loy);
    f2_arrive(&S.bar[1]);
    if (wn < nwork) issue(work[wn], s ^ 1);
    f2_wait(&S.bar[1], s, M.err, b);
    if (!skip)
      f2_xy_solve_sides<FLUX>(S.tile[s], S.fx[s], S.fy[s], x, y, warp == 4 + (it & 3), lox, loy,
                        face_const2(g, lc[LC_CH], sp.glm),
                        [&](int face, int t, const float* f) {
                          if (FULL && sp.reflux && M.nbr[b * 6 + face] == NBR_GENERAL)
                            keep_face_flux(M, -3 - M.gface[b * 6 + face], t, f);
                        });
    f2_arrive(&S.bar[2]);
    const int wnn = counter ? S.next[s] : wn + gridDim.x;
    float un_k[NV];  // conserved values of the next block's own cell
    if (wn < nwork) {
      cp_async_wait_all();
      convert(work[wn], s ^ 1, un_k);
      f2_arrive(&S.bar[0]);
    }
    f2_wait(&S.bar[2], s, M.err, b);
    const float dt = lc[LC_DT], damp = lc[LC_DAMP];
    float un[NV];
#pragma unroll
    for (int v = 0; v < NV; v++) {
      const size_t at = (size_t)v * vs + (size_t)b * M.ncell + y * FB + x;
      if (skip) {  // finished instance: copied through unchanged
        un[v] = uk[v];
        if (FULL && sp.has2) out2[at] = uk[v];
      } else {
        float a = (S.fx[s][v][y][x + 1] - S.fx[s][v][y][x]) * idd[0];
        a = fmaf(S.fy[s][v][y + 1][x] - S.fy[s][v][y][x], idd[1], a);
        float ut = fmaf(-dt, a, uk[v]);
        if (v == 8) ut = ut * damp;
        un[v] = sp.plain ? ut : fmaf(sp.af, S.u0[s][v][tid], sp.bf * ut);
        if (FULL && sp.has2) {
          // SSPRK(5,4) stage 3: w = a2 U2 + b2 (Uk + c2 dt L); U2 is out's
          // register (read here before its write), out2 is U0's (in smem)
          float ut2 = fmaf(-lc[LC_DT2], a, uk[v]);
          if (v == 8) ut2 = ut2 * lc[LC_DAMP2];
          out2[at] = sp.a2f * U2[at] + sp.b2f * ut2;
        }
      }
      out[at] = un[v];
    }
    if (sp.epilogue) {
      cfl_terms<float, 2>(un, gammad, g, ff, gm1f, idd, smx, cmx);
      warp_max2_atomic(smx, cmx, part_b);
    }
#pragma unroll
    for (int v = 0; v < NV; v++) uk[v] = un_k[v];
    wi = wn;
    wn = wnn;
  }
}

}  // namespace amrvac
