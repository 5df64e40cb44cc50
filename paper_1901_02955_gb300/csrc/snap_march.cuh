// snap_march.cuh -- the 3-D stage as a march along z (inviscid layouts). Included by the 3-D
// translation units kern_*3d.cu.
//
// A CTA owns TX x TY columns (one thread each, a warp per x row) of a chunk of levels and walks
// up the chunk one level at a time. Shared memory keeps the primitives of the last five levels of
// the owned columns (the z window of every thread's own column, and the level being finished,
// which the x and y windows read together with that level's x and y halo). Per level k: the
// level k + 3 and the halo of level k are converted; each thread reconstructs its cell of level
// k + 1 along z and solves the face k + 1/2 (no exchange: the left state stays with the thread
// from the level before), then reconstructs its cell of level k along x and y; neighbours hand
// over left states and face fluxes through shared memory; the cell is finished and stored.
//
// Why: the tile kernel (8 x 8 x 4 cells) converts 4 cells and reconstructs 4 windows per owned
// cell where the method needs 1 and 3; the march converts about 2.1 and reconstructs 3.4. The
// stage is bound by instruction issue, so the work saved is time saved.
#pragma once
#include "snap_stage.cuh"

namespace snap {

template <class R, class L, class T>
struct MarchSmem {
  static constexpr int NC = T::TX * T::TY;
  // primitives: five levels of x rows with room for both x halos (an x window then has unit
  // stride), after them the current level's y halo
  static constexpr int BX = T::TX + 6, NL = BX * T::TY, HY = 5 * NL, NP = HY + 6 * T::TX;
  // left states, then fluxes, of the current level's x faces and y faces
  static constexpr int FY = (T::TX + 1) * T::TY, NE = FY + T::TX * (T::TY + 1);
  // right states of the faces at the tile's far x and y sides
  static constexpr int NX = T::TY + T::TX;
  static constexpr size_t bytes(int n) { return (sizeof(R) * L::NV * n + 15) / 16 * 16; }
  static constexpr size_t e_off = bytes(NP), x_off = e_off + bytes(NE), q_off = x_off + bytes(NX);
  static constexpr size_t red_off = q_off + bytes(NC);
  static constexpr size_t dom_off = red_off + 32 * sizeof(double);
  using Dom = DomLocal<R, T::TZ + 7>;  // levels z0 - 3 .. z0 + TZ + 3
  static constexpr size_t total = dom_off + (sizeof(Dom) + 15) / 16 * 16;
  // location of (x, y) of the level whose rows start at cur: its row (a ragged tile's far y halo
  // lies in the rows it does not own), else the y halo
  static __host__ __device__ __forceinline__ int at(int cur, int x, int y) {
    if ((unsigned)y >= (unsigned)T::TY) return HY + (y < 0 ? y + 3 : y - T::TY + 3) * T::TX + x;
    return cur + y * BX + x + 3;
  }
};

// One stage over the CTA's tiles. RES as for stage_tiles (cells written during the launch are
// read past L1, the CFL maximum goes to rate_next).
template <class R, class L, class T, bool MICRO, bool RES = false>
__device__ __forceinline__ void march_tiles(const StageArgs &a, const int stage,
                                            unsigned char *smem) {
  using M = MarchSmem<R, L, T>;
  using P = Prof<R>;
  constexpr int NV = L::NV, TX = T::TX, TY = T::TY, NT = T::NT, NC = M::NC;
  constexpr int NW = NT / 32;
  static_assert(TX == 32 && NT == NC && NT >= 6 * TX + 6 * TY, "a warp per x row; a thread per halo cell");
  using V = SV<R, NV>;
  R *s_p = reinterpret_cast<R *>(smem);
  R *s_e = reinterpret_cast<R *>(smem + M::e_off);
  R *s_x = reinterpret_cast<R *>(smem + M::x_off);
  R *s_q = reinterpret_cast<R *>(smem + M::q_off);  // left z state of the face above, per column
  double *s_red = reinterpret_cast<double *>(smem + M::red_off);
  R *s_dt = reinterpret_cast<R *>(s_red + 31);  // the time step in the kernel's type
  typename M::Dom &S = *reinterpret_cast<typename M::Dom *>(smem + M::dom_off);
  // the stage's input, Y^n and output at the tile's first column and level 0
  void **s_buf = reinterpret_cast<void **>(s_red + 28);
  const Phys &ph = a.ph;
  const CstT<R> &C = cst<R>(a);
  const R weps = C.weno_eps;
  const int tid = threadIdx.x, lx = tid % TX, ly = tid / TX;
  const int col = ly * M::BX + lx + 3;  // the thread's column within a level

  for (int tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    const int dm = find_domain(a.tile_domain, a.ndom, tile);
    const DomDev &D = a.doms[dm];
    const int nx = D.nx, ny = D.ny, nz = D.nz;
    const int lt = tile - D.tile_begin;
    const int cz = D.cz;  // levels per tile, at most T::TZ
    int ix, iy, iz;
    tile_coords(D, lt, ix, iy, iz);
    const int x0 = ix * TX, y0 = iy * TY, z0 = iz * cz;
    const int ex = min(TX, nx - x0), ey = min(TY, ny - y0), ez = min(cz, nz - z0);
    const R *Ys = reinterpret_cast<const R *>(a.buf_s ? a.buf_s : D.buf[stage]);
    double dt0 = 0.0;  // waited for after the columns' first levels
    if (tid == 0) dt0 = stage_dt<RES>(a, D, stage, lt, s_red[0]);
    S.fill(D, z0 - 3, tid);
    if (tid >= 8 && tid < 11) {
      const int i = tid - 8;  // input, Y^n, output
      const void *o = i == 0 ? a.buf_s : (i == 1 ? a.buf_n : a.buf_o);
      const int def = i == 0 ? stage : (i == 1 ? 0 : (stage + 1) % 3);
      s_buf[i] = (R *)(o ? o : D.buf[def]) + ((long long)y0 * nx + x0);
    }
    __syncthreads();
    const bool own = lx < ex && ly < ey;
    R rate_max = R(0);
    R Fz[NV];  // flux through the lower face of the level to be finished next

    // the thread's column one level on, and its cell of a level's x and y halo (thread h of the
    // first 6 TX + 6 TY): where they come from, and the conserved values as loaded
    HaloCell<R> hh = {};
    R yc[NV], yh[NV];
    int hx = 0, hy = 0;
    bool has_h = false;
    if (tid < 6 * TX) {
      const int r = tid / TX;
      hx = tid % TX;
      hy = r < 3 ? r - 3 : ey + r - 3;
      has_h = hx < ex;
    } else if (tid < 6 * TX + 6 * TY) {
      const int r = (tid - 6 * TX) % 6;
      hy = (tid - 6 * TX) / 6;
      hx = r < 3 ? r - 3 : ex + r - 3;
      has_h = hy < ey;
    }
    const int hdir = tid < 6 * TX ? 1 : 0;
    if (has_h) hh = halo_cell<R>(a, D, stage, Ys, x0 + hx, y0 + hy, z0, hdir);
    const int hstep = has_h ? int(hh.stride / nz) : 0, plane = nx * ny;  // one level
    const int at_col = ly * nx + lx;  // the thread's column from s_buf
    auto load_column = [&](int k) {  // the z sides are walls: beyond them the mirrored level
      const int gz = k < 0 ? -1 - k : (k >= nz ? 2 * nz - 1 - k : k);
      load_fields<R, NV, RES>((const R *)s_buf[0] + ((long long)gz * plane + at_col),
                              (long long)plane * nz, yc);
    };
    auto store_column = [&](int k, int slot) {
      R x[NV], pt;
      HaloCell<R> hc;
      hc.gz = k < 0 ? -1 - k : (k >= nz ? 2 * nz - 1 - k : k);
      hc.flip = hc.gz != k;
      hc.side = k < 0 ? 4 : 5;
      halo_prim<R, L>(S, ph, C, hc, 2, yc, x, pt);
      V::store(s_p, slot * M::NL + col, M::NP, x);
    };
    if (own) {
#pragma unroll 1
      for (int j = -3; j < 1; ++j) {
        load_column(z0 + j);
        store_column(z0 + j, j + 3);
      }
      load_column(z0 + 1);
    }
    if (tid == 0) {
      s_red[0] = dt0;
      *s_dt = R(dt0);
    }
    // level z0 + j is in slot (j + 3) mod 5. Two rounds ahead of the first level only build its
    // lower z face.
    int b = 0;  // slot of level k - 1
#pragma unroll 1
    for (int kk = -2; kk < ez; ++kk) {
      const int k = z0 + kk;
      const bool body = kk >= 0;
      int slot[5];  // levels k - 1 .. k + 3
#pragma unroll
      for (int i = 0; i < 5; ++i) slot[i] = b + i < 5 ? b + i : b + i - 5;
      b = slot[1];
      const int cur = slot[1] * M::NL;
      // ---- A. convert what was loaded a level ago: the next level of the columns and the halo
      // of this level
      if (own) store_column(k + 3, slot[4]);
      if (body) {
        if (has_h) {
          R q[NV], pt;
          hh.gz = k;
          halo_prim<R, L>(S, ph, C, hh, hdir, yh, q, pt);
          V::store(s_p, M::at(cur, hx, hy), M::NP, q);
          hh.src += hstep;
        }
        __syncthreads();
      }
      // ---- B. reconstruction: z of level k + 1 with the face below it, x and y of level k
      if (body) {
        // the cells next to the tile: rows y = -1 and y = ey (warps 0 and 1), columns x = -1 and
        // x = ex (warp 2), of which the tile's outer faces need one state each
        const int w = tid / 32, lane = tid % 32;
        if (w < 3) {
          const bool row = w < 2, far = row ? w == 1 : lane >= TY;
          const int x = row ? lane : (far ? ex : -1);
          const int y = row ? (far ? ey : -1) : lane % TY;
          if (row ? x < ex : (lane < 2 * TY && y < ey)) {
            R QM[NV], QP[NV];
            int o[5];
#pragma unroll
            for (int i = 0; i < 5; ++i)
              o[i] = M::at(cur, row ? x : x + i - 2, row ? y + i - 2 : y);
            recon_window<R, NV>(s_p, o, M::NP, weps, QM, QP);
            if (far)
              V::store(s_x, row ? TY + x : y, M::NX, QP);
            else
              V::store(s_e, row ? M::FY + x : y * (TX + 1), M::NE, QM);
          }
        }
      }
      R Fn[NV], QY[NV];
      if (own) {
        R QM[NV], QP[NV];
        int o[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) o[i] = slot[i] * M::NL + col;
        recon_window<R, NV>(s_p, o, M::NP, weps, QM, QP);
        if (kk > -2) {
          R QL[NV];
          V::load(s_q, tid, NC, QL);
          const R pref = P::pf(S, k + 1);
          lmars<R, L>(C, QL, QP, 2, pref, Fn);
          if constexpr (L::MOIST && MICRO) {
            // no condensate passes a wall (both z sides are)
            if (ph.sediment && k + 1 != 0 && k + 1 != nz) sediment_flux<R, L>(C, QL, QP, pref, Fn);
          }
        }
        V::store(s_q, tid, NC, QM);
        if (body) {
#pragma unroll
          for (int i = 0; i < 5; ++i) o[i] = cur + col + i - 2;
          recon_window<R, NV>(s_p, o, M::NP, weps, QM, QP);
          V::store(s_e, ly * (TX + 1) + lx + 1, M::NE, QM);
          // the right state of the cell's lower x face waits in the column's own place of level
          // k - 1, which nothing reads any more
          V::store(s_p, slot[0] * M::NL + col, M::NP, QP);
#pragma unroll
          for (int i = 0; i < 5; ++i) o[i] = M::at(cur, lx, ly + i - 2);
          recon_window<R, NV>(s_p, o, M::NP, weps, QM, QY);
          V::store(s_e, M::FY + (ly + 1) * TX + lx, M::NE, QM);
        }
      }
      if (!body) {
#pragma unroll
        for (int v = 0; v < NV; ++v) Fz[v] = Fn[v];
        if (own) load_column(k + 4);
        if (kk == -1 && has_h) load_fields<R, NV, RES>(hh.src, (long long)hstep * nz, yh);
        continue;
      }
      __syncthreads();
      // ---- C. x and y fluxes, each written over its left state
      const R pref = P::pc(S, k);
      if (own) {
        R QL[NV], QR[NV], F[NV];
        int f = M::FY + ly * TX + lx;
        V::load(s_e, f, M::NE, QL);
        lmars<R, L>(C, QL, QY, 1, pref, F);
        V::store(s_e, f, M::NE, F);
        f = ly * (TX + 1) + lx;
        V::load(s_e, f, M::NE, QL);
        V::load(s_p, slot[0] * M::NL + col, M::NP, QR);
        lmars<R, L>(C, QL, QR, 0, pref, F);
        V::store(s_e, f, M::NE, F);
      }
      {
        const int w = tid / 32, lane = tid % 32;
        if (w >= NW - 2) {  // the far y side (last warp) and the far x side (the one before)
          const bool row = w == NW - 1;
          if (lane < (row ? ex : ey)) {
            R QL[NV], QR[NV], F[NV];
            const int f = row ? M::FY + ey * TX + lane : lane * (TX + 1) + ex;
            V::load(s_e, f, M::NE, QL);
            V::load(s_x, row ? TY + lane : lane, M::NX, QR);
            if (row)
              lmars<R, L>(C, QL, QR, 1, pref, F);
            else
              lmars<R, L>(C, QL, QR, 0, pref, F);
            V::store(s_e, f, M::NE, F);
          }
        }
      }
      // the cell's stage input and Y^n: on their way while the CTA meets
      const long long g = (long long)k * plane + at_col, ncell = (long long)plane * nz;
      R ys[NV], yn[NV];
      if (own) {
        load_fields<R, NV, RES>((const R *)s_buf[0] + g, ncell, ys);
        if (stage != 0) load_fields<R, NV, RES>((const R *)s_buf[1] + g, ncell, yn);
      }
      __syncthreads();
      // ---- D. divergence, sources, stage combine, store; the loads of the next round go first
      if (kk + 1 < ez) {
        if (own) load_column(k + 4);
        if (has_h) load_fields<R, NV, RES>(hh.src, (long long)hstep * nz, yh);
      }
      if (own) {
        const R dt = *s_dt;
        R acc[NV], F0[NV], F1[NV], yo[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = R(0);
        V::load(s_e, ly * (TX + 1) + lx, M::NE, F0);
        V::load(s_e, ly * (TX + 1) + lx + 1, M::NE, F1);
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] -= (F1[v] - F0[v]) * P::ih(S, 0);
        V::load(s_e, M::FY + ly * TX + lx, M::NE, F0);
        V::load(s_e, M::FY + (ly + 1) * TX + lx, M::NE, F1);
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] -= (F1[v] - F0[v]) * P::ih(S, 1);
        R mb = R(0), mt = R(0);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          acc[v] -= (Fn[v] - Fz[v]) * P::ih(S, 2);
          if (v < L::IM0) mb += Fz[v], mt += Fn[v];
          Fz[v] = Fn[v];
        }
        finish_cell<R, L, MICRO>(a, S, ph, C, stage, dt, k, ys, acc, mb, mt,
                                 [&](int v) { return yn[v]; }, yo);
        R *out = (R *)s_buf[2] + g;
#pragma unroll
        for (int v = 0; v < NV; ++v, out += ncell) *out = yo[v];
        if (stage == 2)
          rate_max = fmax(rate_max, cell_rate_r<R, L>(C, yo, P::er(S, k), P::ih(S, 0),
                                                      P::ih(S, 1), P::ih(S, 2)));
      }
    }
    if (stage == 2) {
      double bm;
      if constexpr (sizeof(R) == 4)
        bm = double(block_max_f(rate_max, reinterpret_cast<float *>(s_red + 1)));
      else
        bm = block_max(rate_max, s_red + 1);
      if (tid == 0)
        atomicMax(RES ? D.rate_next : D.rate, (unsigned long long)__double_as_longlong(bm));
    }
    __syncthreads();
  }
}

}  // namespace snap
