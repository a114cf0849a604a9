// dmr_multi.cuh -- several EM steps in one launch (K coarse steps of an FP32 run).
//
// A launch per EM step costs a fixed 3 us or so (launch, one chain of loads,
// stores, the grid's completion) whatever its bytes, and streams the whole
// state once.  Here a launch advances K coarse steps:
//
//  * Tiles (k_multi).  The coarse mesh away from the fine rectangle is cut into
//    tiles; a block holds its tile and K more cells on every side in registers,
//    steps it K times and stores the tile (the halo's values are computed
//    redundantly; each step spoils one more cell of it).  Reads level n,
//    writes level n + K into the other buffer parity, as the one-step launches
//    do.  Two node columns per lane (float2 loads), x neighbours by shuffle,
//    the rows next to another warp's through shared memory, one block barrier
//    per step.  Issue slots are 58 % used (2 blocks of 15 warps per SM), the FP64
//    pipe 35 % (the E^2 sums: 16 cycles per warp and SM for a fused multiply-add,
//    19 for an add, 16 for a conversion, hence to_f64); the rest waits for a tile's
//    loads, shuffles and the step's barrier.  1024^2 with its period end: 11.4 us
//    per step with one launch each, 6.6 us with K = 4 (with one block of 32 warps
//    per SM 8.5 us, with the conversion instruction 8.2 us); 512^2: 1.7 us of tiles
//    per step at K = 8.
//
//  * Fine tiles (k_fine).  The r sub-steps of a larger fine mesh in one launch of
//    such tiles after the coarse step's launch; the coarse-fine sides blend the
//    coarse lines of both levels, the last sub-step writes the fine->coarse
//    means.  2048 x 1024, a quarter of it refined: 392 us per coarse step at
//    r = 4 with one launch per sub-step, 211 us here; r = 2: 78 to 62 us.  Issue
//    slots 67 % used on 1200^2 fine cells (blocks of 10 warps), 46 % on 800^2 (one
//    block of 26 warps per SM, 1.9 waves).
//
//  * The near region (k_near).  The fine rectangle with its r sub-steps per
//    coarse step and the coarse nodes up to 2K + 1 around it live in one
//    16-block cluster, E in shared memory and the rest in registers, each
//    block with a slab of rows; border rows, the coarse-fine lines and the
//    fine->coarse means go to the other blocks by distributed shared memory,
//    with one cluster barrier (0.3 us) per sub-step.  It stores the coarse
//    nodes up to K around the rectangle (what the tiles, which know nothing of
//    the fine mesh, get wrong) and the fine mesh, and runs beside the tiles on a
//    stream of its own.  Bound by latency (a warp is at barriers 44 % of its
//    time, waiting for instructions 12 %; a fourth of the issue slots used): 3.7 us per coarse step at r = 2 with a 64^2 patch, where the
//    one-step launches take 4.5 + 2.9 us.
//
// 512^2 with a 64^2 patch: 8.2 us per coarse step with one launch per step and
// sub-step, 4.4 us here (K = 8); 96^2 whole in the cluster: 6.0 to 3.4 us.
//
// Every element goes through the helpers of dmr_kernels.cuh in the order of
// the one-step launches, so both give the same bits.
#pragma once
#include "dmr_kernels.cuh"

namespace dmr {

enum { BC_FROZEN = 3 };   // side of a near-region window that is not a side of the mesh

// |E^n|^2 at node (i, j) from the edges around it (incident added to Ey),
// one-sided at the mesh's sides, as em_strips takes it
template <class T>
__device__ __forceinline__ T node_sample(int i, int j, int nx, int ny, T exl, T exc, T eyp, T eyc, T inc) {
  T sx, sy;
  if (i > 0 && i < nx) sx = sq_mean(exl, exc);
  else if (i > 0) sx = exl * exl;
  else sx = exc * exc;
  const T e = eyp + inc, f = eyc + inc;
  if (j > 0 && j < ny) sy = sq_mean(e, f);
  else if (j > 0) sy = e * e;
  else sy = f * f;
  return sx + sy;
}

// What the steps of one mesh share: the fields it starts from, where the new
// level goes, the coefficients and the phase of the incident wave.
template <class T>
struct MultiMesh {
  Mesh<T> m;
  T* d[5];             // Ex, Ey, Hz, vx, vy of the new level
  Step<T> c;           // coefficients (its level-dependent fields unused)
  const T *ps, *pc;    // sin / cos of w t per step of a period
  int q0, N;           // step of the period at the start, steps per period
};

template <class T>
struct MultiArgs {
  MultiMesh<T> C;
  int K;               // coarse steps
  // tiles
  int hx;              // halo columns (K rounded up to the columns per lane)
  int tw, th, gx, gy;  // nodes a tile owns, tiles across and up
  int z0, z1, z2, z3;  // nodes (i0, j0, i1, j1) the near region stores; z0 > z2: none
};

// The fine mesh's r sub-steps of one coarse step in tiles (k_fine): its sides,
// the coarse lines around it (levels n and n + 1) and the fine->coarse means.
template <class T>
struct FineArgs {
  int mode[4];                 // BC_MUR or BC_CFB
  const T *old_line[4], *new_line[4];
  int stride[4], len[4], start[4];
  int r;
  T frac[17];                  // k / r
  RestrW<T> W;
};

// The near region (see above).  Its coarse window is a mesh of its own: nodes
// [wi, wi + wnx] x [wj, wj + wny], sides Mur where they are the domain's,
// frozen elsewhere.
template <class T>
struct NearArgs {
  MultiMesh<T> F;
  int r, restr;                // refinement; E means go back to the coarse mesh
  int I0, J0, I1, J1;
  int wi, wj, wnx, wny;
  int cmode[4], fmode[4];
  int crow, frow;              // cell rows per block (coarse window, fine rectangle)
  int jlo, jhi, ilo, ihi;      // restricted coarse Ex rows, Ey columns
  T rinv;
  T frac[17];                  // k / r: FP64 divisions are slow software sequences here
};

// ---------------------------------------------------------------------------
// Tiles
// ---------------------------------------------------------------------------
template <class T, int C> struct TileVec;
template <> struct TileVec<float, 2> {
  static __device__ __forceinline__ void ld(const float* q, float* v) {
    const float2 t = *reinterpret_cast<const float2*>(q);
    v[0] = t.x; v[1] = t.y;
  }
  static __device__ __forceinline__ void st(float* q, const float* v) {
    *reinterpret_cast<float2*>(q) = make_float2(v[0], v[1]);
  }
};

// shared memory of a tile block: two sets of three rows per warp (the top
// row's Ex and Ey, the bottom row's Ex), then the incident field per step
// and column
template <class T, int C>
__host__ __device__ constexpr size_t tile_smem(int warps, int K) {
  return ((size_t)2 * 3 * warps + K) * 32 * C * sizeof(T);
}

template <class T, int C>
__host__ __device__ constexpr size_t fine_smem(int warps, int R, int K) {
  const size_t step = tile_smem<T, C>(warps, K) + (size_t)4 * (32 * C + R * warps) * sizeof(T);
  const size_t means = (size_t)2 * 32 * C * R * warps * sizeof(T);
  return step > means ? step : means;
}

// One tile: lane l holds columns ox + C l .., warp w rows oy + R w ... .
// EDGE: the tile touches a side of the mesh; its origin is then moved inside
// so that the mesh's first / last row is the tile's first / last row (rows 0,
// 1 and ny - 1, ny in one thread each, for the Mur sides).  FINE: the fine
// mesh over one coarse step; its coarse-fine sides take Eq. 5b from the lines
// of levels n and n + 1 (interpolated in space once, blended in time per
// sub-step), and the last sub-step's E goes to the coarse mesh (a8).
template <class T, int C, int R, bool EDGE, bool FINE>
__device__ __forceinline__ void multi_tile(const MultiArgs<T>& A, const FineArgs<T>* Fp, int bx, int by, int ox, int oy,
                                           T* sm) {
  const MultiMesh<T>& M = A.C;
  const Mesh<T>& m = M.m;
  const Step<T>& c = M.c;
  static_assert(C == 2, "float2 and double2 accesses");
  constexpr int W = 32 * C;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int nx = m.nx, ny = m.ny, p = m.p, K = A.K;
  const int i0 = ox + C * lane, j0 = oy + R * w;
  const int ax = bx * A.tw, ay = by * A.th;
  const int ae = min(ax + A.tw, nx + 1), be = min(ay + A.th, ny + 1);   // owned [ax, ae) x [ay, be)
  T* rows = sm;                                    // [parity][warp][3][W]
  T* incs = sm + (size_t)2 * 3 * nw * W;           // [step][W]
  const int Ht = R * nw;
  T* lines = incs + (size_t)K * W;                 // FINE: bottom, top [W][2], left, right [Ht][2]
  // what no EM launch writes may be read before the previous launch is done:
  // the incident field's tables and the density
  for (int q = threadIdx.x; q < K * W; q += blockDim.x) {
    const int s = q / W, x = min(ox + (q - s * W), nx);
    int lev = M.q0 + s;
    while (lev >= M.N) lev -= M.N;
    incs[q] = c.E0 * (M.ps[lev] * c.ckx[x] - M.pc[lev] * c.skx[x]);
  }
  auto ld = [&](const T* a, int j, T* v) {
    if constexpr (EDGE) {
#pragma unroll
      for (int k = 0; k < C; ++k) v[k] = (i0 + k <= nx && j <= ny) ? a[j * p + i0 + k] : T(0);
    } else {
      TileVec<T, C>::ld(a + j * p + i0, v);
    }
  };
  T cnx[R][C], cny[R][C];
  {
    T n[R + 1][C];
#pragma unroll
    for (int q = 0; q <= R; ++q) ld(m.n, min(j0 + q, ny), n[q]);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const T nr = __shfl_down_sync(0xffffffffu, n[q][0], 1);
#pragma unroll
      for (int k = 0; k < C; ++k) {
        cnx[q][k] = c.cj * (n[q][k] + (k + 1 < C ? n[q][k + 1 < C ? k + 1 : k] : nr));
        cny[q][k] = c.cj * (n[q][k] + n[q + 1][k]);
      }
    }
  }
  pdl_enter();
  if constexpr (FINE && EDGE) {
    const FineArgs<T>& F = *Fp;
    for (int q = threadIdx.x; q < 2 * W + 2 * Ht; q += blockDim.x) {
      const int sd = q < W ? SIDE_BOTTOM : q < 2 * W ? SIDE_TOP : q < 2 * W + Ht ? SIDE_LEFT : SIDE_RIGHT;
      const bool hor = q < 2 * W;
      const int e = q < W ? q : q < 2 * W ? q - W : q < 2 * W + Ht ? q - 2 * W : q - 2 * W - Ht;
      const int smp = (hor ? ox : oy) + e;
      const bool here = sd == SIDE_BOTTOM ? oy == 0 : sd == SIDE_TOP ? oy + Ht > ny : sd == SIDE_LEFT ? ox == 0 : ox + W > nx;
      if (F.mode[sd] != BC_CFB || !here || smp >= (hor ? nx : ny)) continue;
      // fine sample at coarse position start + (2 smp + 1 - r)/(2r), clamped (cfb_pos)
      const int num = 2 * smp + 1 - F.r, den = 2 * F.r;
      const int fl = num >= 0 ? num / den : -((-num + den - 1) / den);
      int i = F.start[sd] + fl;
      T xp = (T)(num - fl * den) / (T)den;
      if (i < 0) { i = 0; xp = T(0); }
      if (i > F.len[sd] - 2) { i = F.len[sd] - 2; xp = T(1); }
      const T *o = F.old_line[sd], *l = F.new_line[sd];
      const int st = F.stride[sd];
      lines[2 * q] = o[i * st] * (T(1) - xp) + o[(i + 1) * st] * xp;
      lines[2 * q + 1] = l[i * st] * (T(1) - xp) + l[(i + 1) * st] * xp;
    }
  }
  T ex[R][C], ey[R][C], hz[R][C], vx[R][C], vy[R][C], hzb[C];
  double s2[R][C];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int j = j0 + q;
    ld(m.Ex, j, ex[q]);
    ld(m.Ey, j, ey[q]);
    ld(m.Hz, j, hz[q]);
    ld(m.vx, j, vx[q]);
    ld(m.vy, j, vy[q]);
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const int i = i0 + k;
      s2[q][k] = (i >= ax && i < ae && j >= ay && j < be) ? m.S2[j * p + i] : 0.0;
    }
  }
  if (j0 > 0) {
    ld(m.Hz, j0 - 1, hzb);
  } else {
#pragma unroll
    for (int k = 0; k < C; ++k) hzb[k] = T(0);
  }
  const bool sampled = j0 < be && j0 + R > ay;     // the warp has owned rows
  // rows next to the neighbouring warps: parity 0
  auto put = [&](int par) {
    T* r = rows + ((size_t)par * nw + w) * 3 * W + C * lane;
    TileVec<T, C>::st(r, ex[R - 1]);
    TileVec<T, C>::st(r + W, ey[R - 1]);
    TileVec<T, C>::st(r + 2 * W, ex[0]);
  };
  put(0);
  __syncthreads();
  int lev = M.q0;
  for (int s = 0; s < K; ++s) {
    T exb[C], eyb[C], exa[C], inc[C];
    {
      const T* r = rows + (size_t)(s & 1) * nw * 3 * W + C * lane;
      const int wb = max(w - 1, 0), wa = min(w + 1, nw - 1);
      TileVec<T, C>::ld(r + (size_t)wb * 3 * W, exb);
      TileVec<T, C>::ld(r + (size_t)wb * 3 * W + W, eyb);
      TileVec<T, C>::ld(r + (size_t)wa * 3 * W + 2 * W, exa);
      TileVec<T, C>::ld(incs + s * W + C * lane, inc);
    }
    // ---- H (Eq. 2): the row below the warp's, then the warp's
    {
      const T r0 = __shfl_down_sync(0xffffffffu, eyb[0], 1);
#pragma unroll
      for (int k = 0; k < C; ++k)
        hzb[k] = upd_h(c, hzb[k], ((k + 1 < C ? eyb[k + 1 < C ? k + 1 : k] : r0) - eyb[k]) - (ex[0][k] - exb[k]));
    }
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const T r0 = __shfl_down_sync(0xffffffffu, ey[q][0], 1);
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const T exn = q + 1 < R ? ex[q + 1 < R ? q + 1 : q][k] : exa[k];
        hz[q][k] = upd_h(c, hz[q][k], ((k + 1 < C ? ey[q][k + 1 < C ? k + 1 : k] : r0) - ey[q][k]) - (exn - ex[q][k]));
      }
    }
    const bool accum = lev != 0 && sampled;
    T b0[C], b1[C], t0[C], t1[C];                  // old Ex of the first and last two rows (Mur)
    if constexpr (EDGE) {
#pragma unroll
      for (int k = 0; k < C; ++k) {
        b0[k] = ex[0][k]; b1[k] = ex[1][k];
        t0[k] = ex[R - 1][k]; t1[k] = ex[R - 2][k];
      }
    }
    // ---- E^2 sample of level n, then v (Eq. 3) and E (Eq. 1), from the top row down
#pragma unroll
    for (int q = R - 1; q >= 0; --q) {
      const T exl0 = __shfl_up_sync(0xffffffffu, ex[q][C - 1], 1);
      const T hzl0 = __shfl_up_sync(0xffffffffu, hz[q][C - 1], 1);
      T oy_[C];                                     // old Ey of the row
#pragma unroll
      for (int k = 0; k < C; ++k) oy_[k] = ey[q][k];
      if (accum) {
#pragma unroll
        for (int k = 0; k < C; ++k) {
          const T exl = k > 0 ? ex[q][k > 0 ? k - 1 : 0] : exl0;
          const T eyp = q > 0 ? ey[q > 0 ? q - 1 : 0][k] : eyb[k];
          if constexpr (EDGE) {
            s2[q][k] += to_f64(node_sample(i0 + k, j0 + q, nx, ny, exl, ex[q][k], eyp, ey[q][k], inc[k]));
          } else {
            s2[q][k] = add_sample(s2[q][k], exl, ex[q][k], eyp + inc[k], ey[q][k] + inc[k]);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const T hzp = q > 0 ? hz[q > 0 ? q - 1 : 0][k] : hzb[k];
        const T hzl = k > 0 ? hz[q][k > 0 ? k - 1 : 0] : hzl0;
        vx[q][k] = upd_v(c, vx[q][k], ex[q][k]);
        ex[q][k] = mad_(cnx[q][k], vx[q][k], mad_(c.ce, hz[q][k] - hzp, ex[q][k]));
        vy[q][k] = upd_v(c, vy[q][k], ey[q][k] + inc[k]);
        ey[q][k] = mad_(cny[q][k], vy[q][k], mad_(-c.ce, hz[q][k] - hzl, ey[q][k]));
      }
      if constexpr (EDGE) {
        // sides left / right: Eq. 5b, or Mur from the neighbouring column's old and new Ey
        const bool cl = FINE && Fp->mode[SIDE_LEFT] == BC_CFB, cr = FINE && Fp->mode[SIDE_RIGHT] == BC_CFB;
        const T oll = __shfl_up_sync(0xffffffffu, oy_[C - 1], 1), nll = __shfl_up_sync(0xffffffffu, ey[q][C - 1], 1);
        if (i0 == 0 && !cl) ey[q][0] = oy_[1] + c.mur * (ey[q][1] - oy_[0]);
#pragma unroll
        for (int k = 0; k < C; ++k)
          if (i0 + k == nx && !cr)
            ey[q][k] = k > 0 ? oy_[0] + c.mur * (ey[q][0] - oy_[k]) : oll + c.mur * (nll - oy_[k]);
        if constexpr (FINE) {
          const T f = Fp->frac[s + 1];
          const T* l = lines + 4 * W + 2 * (R * w + q);
          if (i0 == 0 && cl) ey[q][0] = (T(1) - f) * l[0] + f * l[1];
#pragma unroll
          for (int k = 0; k < C; ++k)
            if (i0 + k == nx && cr) ey[q][k] = (T(1) - f) * l[2 * Ht] + f * l[2 * Ht + 1];
        }
      }
    }
    if constexpr (EDGE) {
      if (j0 == 0) {
        const bool cb = FINE && Fp->mode[SIDE_BOTTOM] == BC_CFB;
        const T f = FINE ? Fp->frac[s + 1] : T(0);
        const T* l = lines + 2 * C * lane;
#pragma unroll
        for (int k = 0; k < C; ++k)
          ex[0][k] = cb ? (T(1) - f) * l[2 * k] + f * l[2 * k + 1] : b1[k] + c.mur * (ex[1][k] - b0[k]);
      }
      if (j0 + R - 1 == ny) {
        const bool ct = FINE && Fp->mode[SIDE_TOP] == BC_CFB;
        const T f = FINE ? Fp->frac[s + 1] : T(0);
        const T* l = lines + 2 * W + 2 * C * lane;
#pragma unroll
        for (int k = 0; k < C; ++k)
          ex[R - 1][k] = ct ? (T(1) - f) * l[2 * k] + f * l[2 * k + 1] : t1[k] + c.mur * (ex[R - 2][k] - t0[k]);
      }
    }
    if (++lev == M.N) lev = 0;
    if (s + 1 < K) {
      put((s + 1) & 1);
      __syncthreads();
    }
  }
  // ---- the owned nodes, except those the near region stores
  const bool plain = !EDGE && (ae <= A.z0 || ax > A.z2 || be <= A.z1 || ay > A.z3);
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int j = j0 + q, id = j * p + i0;
    if (j < ay || j >= be) continue;
    if (plain) {
      // the owned columns start and end at multiples of C
      if (i0 >= ax && i0 < ae) {
        TileVec<T, C>::st(M.d[0] + id, ex[q]);
        TileVec<T, C>::st(M.d[1] + id, ey[q]);
        TileVec<T, C>::st(M.d[2] + id, hz[q]);
        TileVec<T, C>::st(M.d[3] + id, vx[q]);
        TileVec<T, C>::st(M.d[4] + id, vy[q]);
        *reinterpret_cast<double2*>(m.S2 + id) = make_double2(s2[q][0], s2[q][1]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const int i = i0 + k;
        if (i < ax || i >= ae || (i >= A.z0 && i <= A.z2 && j >= A.z1 && j <= A.z3)) continue;
        if (i < nx) { M.d[0][id + k] = ex[q][k]; M.d[3][id + k] = vx[q][k]; }
        if (j < ny) { M.d[1][id + k] = ey[q][k]; M.d[4][id + k] = vy[q][k]; }
        if (i < nx && j < ny) M.d[2][id + k] = hz[q][k];
        m.S2[id + k] = s2[q][k];
      }
    }
  }
  if constexpr (FINE) {
    // a8: the means of r collinear fine edges, in the order of em_strips; the
    // owned columns and rows start at multiples of r
    const RestrW<T>& Wr = Fp->W;
    if (!Wr.on) return;
    __syncthreads();                               // the rows of the last sub-step have been read
    T *sx = sm, *sy = sm + (size_t)W * Ht;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      TileVec<T, C>::st(sx + (R * w + q) * W + C * lane, ex[q]);
      TileVec<T, C>::st(sy + (R * w + q) * W + C * lane, ey[q]);
    }
    __syncthreads();
    const int r = Fp->r, hx = (ae - ax + r - 1) / r, hy = (be - ay + r - 1) / r;   // group heads
    const unsigned mul = 0xffffffffu / (unsigned)hx + 1u;
    for (int e = threadIdx.x; e < hx * hy; e += blockDim.x) {
      const int gy = hx > 1 ? (int)__umulhi((unsigned)e, mul) : e, gx = e - gy * hx;
      const int i = ax + r * gx, j = ay + r * gy, I = Wr.I0 + i / r, J = Wr.J0 + j / r;
      const int at = (j - oy) * W + i - ox;
      if (i < nx && J >= Wr.jlo && J <= Wr.jhi) {
        T acc = sx[at];
        for (int u = 1; u < r; ++u) acc = acc + sx[at + u];
        Wr.cEx[J * Wr.cp + I] = acc * Wr.rinv;
      }
      if (j < ny && I >= Wr.ilo && I <= Wr.ihi) {
        T acc = sy[at];
        for (int u = 1; u < r; ++u) acc = acc + sy[at + u * W];
        Wr.cEy[J * Wr.cp + I] = acc * Wr.rinv;
      }
    }
  }
}

// block `t` of the tiles
template <class T, int C, int R, bool FINE = false>
__device__ __forceinline__ void multi_tiles(const MultiArgs<T>& A, int t, T* sm, const FineArgs<T>* Fp = nullptr) {
  const int by = t / A.gx, bx = t - by * A.gx;
  if (by >= A.gy) return;
  constexpr int W = 32 * C;
  const int nx = A.C.m.nx, ny = A.C.m.ny, H = R * (int)(blockDim.x >> 5);
  const int xmax = (nx + 1 - W + C - 1) / C * C;     // origin of the last column of tiles
  const int ox = max(min(bx * A.tw - A.hx, xmax), 0);
  const int oy = max(min(by * A.th - A.K, ny + 1 - H), 0);
  if (bx * A.tw >= A.z0 && min(bx * A.tw + A.tw, nx + 1) - 1 <= A.z2 && by * A.th >= A.z1 &&
      min(by * A.th + A.th, ny + 1) - 1 <= A.z3)
    return;                                          // all of it belongs to the near region
  if (ox == 0 || ox + W > nx || oy == 0 || oy + H > ny) multi_tile<T, C, R, true, FINE>(A, Fp, bx, by, ox, oy, sm);
  else multi_tile<T, C, R, false, FINE>(A, Fp, bx, by, ox, oy, sm);
}

// ---------------------------------------------------------------------------
// The near region
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ int cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Shared memory of a block of the cluster, in elements of T from its start.
// Per mesh: Ex and Ey of the block's node rows, twice (a sub-step reads one
// copy and writes the other), with the row below (row -1) and rows above;
// everything else of a node is in the registers of the warp that owns it.
struct Slab {
  int ex, ey;                            // row -1 of copy 0; copy 1 is `plane` further
  int cols, plane;
  int nx, ny, j0, nr, per, last;         // own node rows [j0, j0 + nr); per: cell rows per block; last: the last block with rows
  int x0, y0;                            // the mesh's origin in the arrays
  int si0, sj0, si1, sj1;                // nodes the near region stores
};

constexpr int kNearPad = 8;              // rows past the own ones that a unit may read

// A border value of a block after a sub-step: what it is (IT_MUR: the Mur
// edge y from the edge x next to it; IT_PUSH: the old and the new value of
// coarse edge x to place y of blocks z; IT_LINE: the coarse-fine edge y, sample
// x), Ey or Ex, and whether the block above keeps a copy (of column IT_COL).
enum { IT_MUR = 0, IT_PUSH = 1, IT_LINE = 2, IT_OP = 3, IT_Y = 4, IT_UP = 8, IT_DEF = 16, IT_FINE = 32, IT_COL = 8 };
// places for items: the coarse-fine edges (at most two rows and two columns of
// a block's fine nodes), then the other items of both meshes: as many fine ones
// (Mur sides), the coarse window's sides, the lines
__host__ __device__ constexpr int near_edges_max(int nfx, int frow) { return 2 * (nfx + 1) + 2 * (frow + 2); }
__host__ __device__ constexpr int near_items_max(int wnx, int crow, int nfx, int frow, int ni, int nj) {
  return 2 * near_edges_max(nfx, frow) + 2 * (wnx + 1) + 2 * (crow + 2) + 2 * (ni + 2) + 2 * (nj + 2);
}

// shared memory of a slab in elements
__host__ __device__ constexpr int slab_rows(int per) { return per + 2 + kNearPad; }
template <class T>
__host__ __device__ constexpr size_t near_smem(int wnx, int crow, int nfx, int frow, int r, int ni, int nj, int K) {
  const size_t e = (size_t)4 * slab_rows(crow) * (wnx + 1) + (size_t)4 * slab_rows(frow) * (nfx + 1) +
                   4 * (ni + 2) + 4 * (nj + 2) + nfx + frow + 3 + (size_t)2 * K * (r + 1);
  return e * sizeof(T) + (nfx + frow + 3) * sizeof(int) + (size_t)near_items_max(wnx, crow, nfx, frow, ni, nj) * sizeof(int4) + 64;
}

// warps that a slab with up to `rows` rows takes: 30 node columns each (lane 0
// and lane 31 hold the halo columns, as in em_strips) times R rows
__host__ __device__ constexpr int near_units(int cols, int rows, int R) {
  return ((cols + STRIP_W - 1) / STRIP_W) * ((rows + R - 1) / R);
}

template <class T, int R>
struct Unit {
  int at;                     // the lane's column in the first row, from a copy's start
  int below;                  // to Ey of the row below (the row itself at the mesh's first row)
  int top;                    // row of the unit that is the mesh's last node row (or none)
  unsigned st;                // rows whose x edge (bit q) / y edge (bit 16 + q) takes Eq. 1 here
  int qup, qdn;               // row that the block above / below keeps a copy of (or none)
  bool on_l, on_r;            // first / last node column of the mesh
  T hz[R], vx[R], vy[R], cx[R], cy[R], hzb;   // cx, cy = cj (n_a + n_b); hzb: Hz of the row below
  T ck, sk;                   // cos(k x), sin(k x)
  double s2[R];
};

// stores to the shared memory of block `rank` of the cluster; at: byte
// address of the same place in this block's
__device__ __forceinline__ unsigned cluster_at(unsigned at, int rank) {
  unsigned o;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(at), "r"(rank));
  return o;
}
__device__ __forceinline__ void cluster_st(unsigned at, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(at), "f"(v) : "memory");
}

// What a block needs besides its slabs: the coarse-fine lines, (old, new)
// coarse tangential E per side from one sample before the rectangle to one
// after; per fine sample (of the columns, then of the block's rows from the
// one below on) its position and weight (Eq. 5b).
struct NearPlace {
  int b, t, l, r;       // lines: bottom, top, left, right
  int wx;               // weights
  int ph;               // phases
  int nfx;
  const int* pos;
};

template <class T>
__device__ __forceinline__ T line_value(const T* sm, const NearPlace& L, int line, int e, T frac) {
  const T* v = sm + line + 2 * L.pos[e];
  const T xp = sm[L.wx + e], one = T(1);
  const T lo = v[0] * (one - xp) + v[2] * xp;
  const T ln = v[1] * (one - xp) + v[3] * xp;
  return (one - frac) * lo + frac * ln;
}

// One EM step of a unit: Eqs. 1-3 and the E^2 sample from one copy of E
// (at ox, oy) into the other (at wx, wy), and the border rows to the blocks
// that keep a copy (up, dn: byte addresses of their copies' border rows).  No
// branches: the sides and the coarse-fine lines are the items' business.
template <class T, int R>
__device__ __forceinline__ void near_step(T* sm, int ox, int oy, int wx, int wy, int cols, Unit<T, R>& n, const Step<T>& c,
                                          bool accum, T sp, T cp, unsigned upx, unsigned upy, unsigned dnx) {
  const T* Ex = sm + ox + n.at;
  const T* Ey = sm + oy + n.at;
  T* Wx = sm + wx + n.at;
  T* Wy = sm + wy + n.at;
  const T exb = Ex[-cols];
  const T eyb = Ey[n.below];
  T ex[R + 1], ey[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    ex[q] = Ex[q * cols];
    ey[q] = Ey[q * cols];
  }
  ex[R] = Ex[R * cols];
  const T inc = c.E0 * (sp * n.ck - cp * n.sk);
  n.hzb = upd_h(c, n.hzb, (__shfl_down_sync(0xffffffffu, eyb, 1) - eyb) - (ex[0] - exb));
#pragma unroll
  for (int q = 0; q < R; ++q)
    n.hz[q] = upd_h(c, n.hz[q], (__shfl_down_sync(0xffffffffu, ey[q], 1) - ey[q]) - (ex[q + 1] - ex[q]));
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const T hzl = __shfl_up_sync(0xffffffffu, n.hz[q], 1);
    const T exl = __shfl_up_sync(0xffffffffu, ex[q], 1);
    const T eym = q > 0 ? ey[q > 0 ? q - 1 : 0] : eyb;
    const T hzp = q > 0 ? n.hz[q > 0 ? q - 1 : 0] : n.hzb;
    if (accum) {
      // at a side both edges of a pair are the one that is there
      // ((a^2 + a^2) / 2 = a^2 exactly)
      n.s2[q] = add_sample(n.s2[q], n.on_l ? ex[q] : exl, n.on_r ? exl : ex[q], eym + inc,
                           (q == n.top ? eym : ey[q]) + inc);
    }
    n.vx[q] = upd_v(c, n.vx[q], ex[q]);
    n.vy[q] = upd_v(c, n.vy[q], ey[q] + inc);
    const T enx = mad_(n.cx[q], n.vx[q], mad_(c.ce, n.hz[q] - hzp, ex[q]));
    const T eny = mad_(n.cy[q], n.vy[q], mad_(-c.ce, n.hz[q] - hzl, ey[q]));
    const bool sx_ = n.st & (1u << q), sy_ = n.st & (0x10000u << q);
    if (sx_) Wx[q * cols] = enx;
    if (sy_) Wy[q * cols] = eny;
    if (q == n.qup) {
      if (sx_) cluster_st(upx, enx);
      if (sy_) cluster_st(upy, eny);
    }
    if (q == n.qdn && sx_) cluster_st(dnx, enx);
  }
}

// The border items it[0 .. n) of both meshes after a sub-step; fo, co: the copy
// of each mesh's E that the sub-step read (it wrote the other one).
template <class T>
__device__ __forceinline__ void near_items(const Slab& Fs, const Slab& Cs, T* sm, unsigned sa, const int4* it, int n, int fo,
                                           int co, T fmur, T cmur, int above) {
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int4 q = it[e];
    const int m = q.w;
    const bool f = m & IT_FINE, y = m & IT_Y;
    const int plane = f ? Fs.plane : Cs.plane, o = f ? fo : co;
    const int arr = f ? (y ? Fs.ey : Fs.ex) : (y ? Cs.ey : Cs.ex);
    const T* O = sm + arr + o * plane;
    const int wo = arr + (o ^ 1) * plane;
    T* W = sm + wo;
    const T old = O[q.x], nw = W[q.x];
    if ((m & IT_OP) == IT_PUSH) {
      for (int b = q.z >> 8; b <= (q.z & 255); ++b) {
        const unsigned d = cluster_at(sa + (unsigned)(q.y * sizeof(T)), b);
        cluster_st(d, old);
        cluster_st(d + (unsigned)sizeof(T), nw);
      }
    } else {
      const T v = old + (f ? fmur : cmur) * (nw - O[q.y]);
      W[q.y] = v;
      if (m & IT_UP) cluster_st(cluster_at(sa + (unsigned)((wo + (m >> IT_COL)) * sizeof(T)), above), v);
    }
  }
}

// The coarse-fine sides of the fine mesh (Eq. 5b) in copy w.  def: the first
// sub-step's, evaluated at the start of the second one (its coarse E^{n+1}
// came from other blocks during the first), with the row below.
template <class T>
__device__ __forceinline__ void near_sides(const Slab& S, T* sm, unsigned sa, const int4* it, int n, int w, T frac, bool def,
                                           int above, const NearPlace& L) {
  const int pw = w * S.plane;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int4 q = it[e];
    const int m = q.w, arr = ((m & IT_Y) ? S.ey : S.ex) + pw;
    if (!def && (m & IT_DEF)) continue;
    const T v = line_value(sm, L, q.z, q.x, frac);
    sm[arr + q.y] = v;
    if (!def && (m & IT_UP)) cluster_st(cluster_at(sa + (unsigned)((arr + (m >> IT_COL)) * sizeof(T)), above), v);
  }
}

// The items of a mesh into it[], its coarse-fine edges into il[]; n, nl: counts
template <class T, bool COARSE>
__device__ __forceinline__ void slab_items(const Slab& S, const Slab& Fs, const NearArgs<T>& N, const int* mode, int rank,
                                           const NearPlace& L, int4* it, int* n, int4* il, int* nl) {
  const int cols = S.cols, nx = S.nx, ny = S.ny, t = threadIdx.x, nt = blockDim.x, f = COARSE ? 0 : IT_FINE;
  const int lr = S.nr - 1;
  if (S.nr == 0) return;
  auto at = [&](int row, int i) { return (row + 1) * cols + i; };
  auto add = [&](int a, int b, int c, int m) { it[atomicAdd(n, 1)] = make_int4(a, b, c, m | f); };
  auto line = [&](int a, int b, int c, int m) { il[atomicAdd(nl, 1)] = make_int4(a, b, c, m | IT_LINE); };
  for (int i = t; i < nx; i += nt) {
    if (S.j0 == 0) {
      if (mode[SIDE_BOTTOM] == BC_MUR) add(at(1, i), at(0, i), 0, IT_MUR);
      if (mode[SIDE_BOTTOM] == BC_CFB) line(i, at(0, i), L.b, 0);
    }
    if (rank == S.last) {
      if (mode[SIDE_TOP] == BC_MUR) add(at(lr - 1, i), at(lr, i), 0, IT_MUR);
      if (mode[SIDE_TOP] == BC_CFB) line(i, at(lr, i), L.t, 0);
    }
  }
  for (int e = t; e < 2 * (S.nr + 1); e += nt) {
    const int row = (e >> 1) - 1, j = S.j0 + row;
    if (j < 0 || j >= ny) continue;
    const int sd = (e & 1) ? SIDE_RIGHT : SIDE_LEFT, i = (e & 1) ? nx : 0, i1 = (e & 1) ? nx - 1 : 1;
    const int m = IT_Y | (i << IT_COL) | (row == lr && rank < S.last ? IT_UP : 0);
    if (mode[sd] == BC_MUR && row >= 0) add(at(row, i1), at(row, i), 0, IT_MUR | m);
    if (mode[sd] == BC_CFB) line(L.nfx + row + 1, at(row, i), (e & 1) ? L.r : L.l, m | (row < 0 ? IT_DEF : 0));
  }
  if (COARSE) {
    const int ni = N.I1 - N.I0, nj = N.J1 - N.J0;
    for (int e = t; e < 2 * (ni + 2); e += nt) {
      const int I = e >> 1, sd = (e & 1) ? SIDE_TOP : SIDE_BOTTOM;
      const int i = N.I0 - 1 + I - N.wi, row = ((e & 1) ? N.J1 : N.J0) - N.wj - S.j0;
      if (N.fmode[sd] != BC_CFB || i < 0 || i >= nx || row < 0 || row >= S.nr) continue;
      const int b = (e & 1) ? Fs.last : 0;
      add(at(row, i), ((e & 1) ? L.t : L.b) + 2 * I, (b << 8) | b, IT_PUSH);
    }
    for (int e = t; e < 2 * (nj + 2); e += nt) {
      const int J = e >> 1, sd = (e & 1) ? SIDE_RIGHT : SIDE_LEFT;
      const int i = ((e & 1) ? N.I1 : N.I0) - N.wi, row = N.J0 - 1 + J - N.wj - S.j0;
      if (N.fmode[sd] != BC_CFB || row < 0 || row >= S.nr || S.j0 + row >= ny) continue;
      // the blocks with a fine row (or the row below theirs) in the coarse
      // cells from one below the sample to two above it
      const int cpb = N.frow / N.r;
      add(at(row, i), ((e & 1) ? L.r : L.l) + 2 * J, ((max(J - 2, 0) / cpb) << 8) | (min(J + 1, nj - 1) / cpb),
          IT_PUSH | IT_Y);
    }
  }
}

__device__ __forceinline__ void slab_place(Slab& S, int nx, int ny, int per, int rank, int* at) {
  S.nx = nx; S.ny = ny; S.per = per;
  S.cols = nx + 1;
  S.last = (ny - 1) / per;
  S.j0 = min(rank * per, ny);
  S.nr = rank > S.last ? 0 : min(S.j0 + per, ny) - S.j0 + (rank == S.last ? 1 : 0);
  S.plane = slab_rows(per) * S.cols;
  S.ex = *at;
  S.ey = *at + 2 * S.plane;
  *at += 4 * S.plane;
}

// unit u of a slab: its place, and what no EM launch writes (the density and
// the incident tables)
template <class T, int R>
__device__ __forceinline__ void unit_const(const Slab& S, Unit<T, R>& n, const MultiMesh<T>& M, int u, int rank, int* ri,
                                           int* rrow) {
  const int sx = (S.cols + STRIP_W - 1) / STRIP_W, g = u / sx, lane = threadIdx.x & 31;
  const int i = (u - g * sx) * STRIP_W - 1 + lane, row0 = g * R;
  const bool own = lane >= 1 && lane <= STRIP_W && i <= S.nx;
  const int ic = min(max(i, 0), S.nx), p = M.m.p;
  *ri = own ? i : -1 - ic;
  *rrow = row0;
  n.at = (row0 + 1) * S.cols + ic;
  n.below = S.j0 + row0 > 0 ? -S.cols : 0;
  n.top = S.ny - S.j0 - row0;
  n.on_l = i == 0;
  n.on_r = i == S.nx;
  n.qup = rank < S.last ? S.nr - 1 - row0 : -1;
  n.qdn = rank > 0 ? -row0 : -1;
  n.st = 0u;
  n.ck = M.c.ckx[S.x0 + ic];
  n.sk = M.c.skx[S.x0 + ic];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    n.cx[q] = n.cy[q] = T(0);
    const int row = row0 + q, j = S.j0 + row;
    if (row >= S.nr) continue;
    if (own && i < S.nx && j > 0 && j < S.ny) n.st |= 1u << q;
    if (own && i > 0 && i < S.nx && j < S.ny) n.st |= 0x10000u << q;
    const int at = (S.y0 + j) * p + S.x0 + ic;
    const T v = M.m.n[at];
    if (ic < S.nx) n.cx[q] = M.c.cj * (v + M.m.n[at + 1]);
    if (j < S.ny) n.cy[q] = M.c.cj * (v + M.m.n[at + p]);
  }
}

template <class T, int R>
__device__ __forceinline__ void unit_load(const Slab& S, Unit<T, R>& n, const MultiMesh<T>& M, int ri, int row0) {
  const int p = M.m.p, i = ri >= 0 ? ri : -1 - ri;
  const bool x = i < S.nx;
  n.hzb = T(0);
  if (x && S.j0 + row0 > 0 && row0 < S.nr) n.hzb = M.m.Hz[(S.y0 + S.j0 + row0 - 1) * p + S.x0 + i];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    n.hz[q] = n.vx[q] = n.vy[q] = T(0);
    n.s2[q] = 0.0;
    const int row = row0 + q, j = S.j0 + row;
    if (row >= S.nr) continue;
    const int at = (S.y0 + j) * p + S.x0 + i;
    if (x && j < S.ny) n.hz[q] = M.m.Hz[at];
    if (x) n.vx[q] = M.m.vx[at];
    if (j < S.ny) n.vy[q] = M.m.vy[at];
    if (ri >= S.si0 && ri <= S.si1 && j >= S.sj0 && j <= S.sj1) n.s2[q] = M.m.S2[at];
  }
}

// E of a slab's rows and the rows just outside, into both copies
template <class T>
__device__ __forceinline__ void slab_load(const Slab& S, const MultiMesh<T>& M, T* sm, int rank) {
  if (S.nr == 0) return;
  const int cols = S.cols, p = M.m.p, w = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31;
  const int r0 = S.j0 > 0 ? -1 : 0, r1 = rank < S.last ? S.nr : S.nr - 1;
  for (int row = r0 + w; row <= r1; row += nw) {
    const int j = S.j0 + row;
    for (int i = lane; i < cols; i += 32) {
      const int at = (S.y0 + j) * p + S.x0 + i, o = (row + 1) * cols + i;
      const T x = i < S.nx ? M.m.Ex[at] : T(0), y = j < S.ny ? M.m.Ey[at] : T(0);
      sm[S.ex + o] = x; sm[S.ex + S.plane + o] = x;
      sm[S.ey + o] = y; sm[S.ey + S.plane + o] = y;
    }
  }
}

template <class T, int R>
__device__ __forceinline__ void unit_store(const Slab& S, const Unit<T, R>& n, const MultiMesh<T>& M, const T* sm, int par,
                                           int i, int row0) {
  const int p = M.m.p;
  if (i < S.si0 || i > S.si1) return;
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int row = row0 + q, j = S.j0 + row;
    if (row >= S.nr || j < S.sj0 || j > S.sj1) continue;
    const int at = (S.y0 + j) * p + S.x0 + i, o = par * S.plane + n.at + q * S.cols;
    if (i < S.nx) { M.d[0][at] = sm[S.ex + o]; M.d[3][at] = n.vx[q]; }
    if (j < S.ny) { M.d[1][at] = sm[S.ey + o]; M.d[4][at] = n.vy[q]; }
    if (i < S.nx && j < S.ny) M.d[2][at] = n.hz[q];
    M.m.S2[at] = n.s2[q];
  }
}

__device__ __forceinline__ unsigned div_mul(unsigned d) { return 0xffffffffu / d + 1u; }

// a restricted coarse edge's new value to the block that owns its row, and
// to the neighbours that keep a copy of the row (copy par)
template <class T>
__device__ __forceinline__ void near_put_coarse(const Slab& S, unsigned sa, unsigned mul, int par, bool x, int i, int j,
                                                T v) {
  const int q = (int)__umulhi((unsigned)min(j, S.ny - 1), mul), row = j - q * S.per;
  const unsigned a = sa + (unsigned)(((x ? S.ex : S.ey) + par * S.plane + i) * sizeof(T));
  cluster_st(cluster_at(a + (unsigned)((row + 1) * S.cols * sizeof(T)), q), v);
  if (x && row == 0 && q > 0) cluster_st(cluster_at(a + (unsigned)((S.per + 1) * S.cols * sizeof(T)), q - 1), v);
  if (row == S.per - 1 && q < S.last) cluster_st(cluster_at(a, q + 1), v);
}

// R: rows per warp.  The first warps of a block step its share of the fine
// mesh, the next ones its share of the coarse window.
template <class T, int R>
__device__ __forceinline__ void multi_near(const MultiArgs<T>& A, const NearArgs<T>& N, char* smem) {
  __shared__ int cnt[4];      // fine items, coarse-fine edges, items of both meshes
  static_assert(R <= kNearPad, "rows past the own ones");
  const int rank = (int)cluster_rank(), nt = blockDim.x, t = threadIdx.x, r = N.r, K = A.K, w = t >> 5;
  const int ni = N.I1 - N.I0, nj = N.J1 - N.J0, nfx = r * ni, nfy = r * nj;
  T* sm = reinterpret_cast<T*>(smem);
  const unsigned sa = (unsigned)__cvta_generic_to_shared(sm);
  Slab Cs, Fs;
  int at = 0;
  slab_place(Cs, N.wnx, N.wny, N.crow, rank, &at);
  slab_place(Fs, nfx, nfy, N.frow, rank, &at);
  Cs.x0 = N.wi; Cs.y0 = N.wj; Fs.x0 = Fs.y0 = 0;
  Cs.si0 = A.z0 - N.wi; Cs.sj0 = A.z1 - N.wj; Cs.si1 = A.z2 - N.wi; Cs.sj1 = A.z3 - N.wj;
  Fs.si0 = Fs.sj0 = 0; Fs.si1 = nfx; Fs.sj1 = nfy;
  NearPlace L;
  L.b = at; L.t = L.b + 2 * (ni + 2); L.l = L.t + 2 * (ni + 2); L.r = L.l + 2 * (nj + 2);
  L.wx = L.r + 2 * (nj + 2);
  L.ph = L.wx + nfx + N.frow + 3;   // sin, cos per coarse step, then per fine sub-step
  L.nfx = nfx;
  int* pos = reinterpret_cast<int*>(sm + L.ph + 2 * K * (r + 1));
  L.pos = pos;
  int4* itl = reinterpret_cast<int4*>(((uintptr_t)(pos + nfx + N.frow + 3) + 15) & ~(uintptr_t)15);
  int4* itf = itl + near_edges_max(nfx, N.frow);
  if (t < 4) cnt[t] = 0;
  // ---- tables
  for (int s = t; s < K * (r + 1); s += nt) {
    const bool co = s < K;
    const MultiMesh<T>& M = co ? A.C : N.F;
    const int lev = (M.q0 + (co ? s : s - K)) % M.N;
    sm[L.ph + 2 * s] = M.ps[lev];
    sm[L.ph + 2 * s + 1] = M.pc[lev];
  }
  // Eq. 5b positions: fine sample q at coarse position start + (2q + 1 - r)/(2r),
  // clamped to the coarse line (cfb_pos)
  for (int e = t; e < nfx + Fs.nr + 1; e += nt) {
    const bool x = e < nfx;
    const int s = x ? e : Fs.j0 + e - nfx - 1, start = x ? N.I0 : N.J0, len = x ? A.C.m.nx : A.C.m.ny;
    const int num = 2 * s + 1 - r, den = 2 * r;
    const int fl = num >= 0 ? num / den : -((-num + den - 1) / den);
    int i = start + fl;
    T v = (T)(num - fl * den) / (T)den;
    if (i < 0) { i = 0; v = T(0); }
    if (i > len - 2) { i = len - 2; v = T(1); }
    pos[e] = s < 0 ? 0 : i - (start - 1);
    sm[L.wx + e] = v;
  }
  const int uf = near_units(Fs.cols, Fs.nr, R), uc = near_units(Cs.cols, Cs.nr, R);
  const bool fine = w < uf, coarse = !fine && w < uf + uc;
  Unit<T, R> n{};
  int ui = 0, urow = 0;
  if (fine) unit_const(Fs, n, N.F, w, rank, &ui, &urow);
  else if (coarse) unit_const(Cs, n, A.C, w - uf, rank, &ui, &urow);
  __syncthreads();            // cnt
  slab_items<T, false>(Fs, Fs, N, N.fmode, rank, L, itf, cnt, itl, cnt + 1);
  __syncthreads();            // the fine items first: the sub-steps after the first have no others
  if (t == 0) cnt[2] = cnt[0];
  __syncthreads();
  slab_items<T, true>(Cs, Fs, N, N.cmode, rank, L, itf, cnt + 2, itl, cnt + 3);
  pdl_enter();
  if (fine) unit_load(Fs, n, N.F, ui, urow);
  else if (coarse) unit_load(Cs, n, A.C, ui, urow);
  slab_load(Cs, A.C, sm, rank);
  slab_load(Fs, N.F, sm, rank);
  cluster_sync();     // every block's shared memory is ready (and its loads done)
  const unsigned cmul = div_mul((unsigned)N.crow), nmul = div_mul((unsigned)(ni + 1));
  const int fr = Fs.nr / r, top = Fs.nr > 0 && rank == Fs.last;   // coarse rows with fine rows here
  // the lane's column in the copy 0 border rows of the blocks above and below
  const int col = fine ? n.at - (urow + 1) * Fs.cols : n.at - (urow + 1) * Cs.cols;
  const int bx = fine ? Fs.ex : Cs.ex, by = fine ? Fs.ey : Cs.ey;
  const unsigned ax = sa + (unsigned)((bx + col) * sizeof(T)), ay = sa + (unsigned)((by + col) * sizeof(T));
  const int above = min(rank + 1, cluster_size() - 1);
  const unsigned upx = cluster_at(ax, above), upy = cluster_at(ay, above);
  const unsigned dnx = cluster_at(ax + (unsigned)((fine ? (Fs.per + 1) * Fs.cols : (Cs.per + 1) * Cs.cols) * sizeof(T)),
                                  max(rank - 1, 0));
  bool nmur = false;   // restricted edges among the items
  for (int q = 0; q < 4; ++q) nmur = nmur || N.fmode[q] == BC_MUR;
  const int nitf = cnt[0], nitl = cnt[1], nit = cnt[2];
  int pc = 0, pf = 0, qc = A.C.q0 % A.C.N, qf = N.F.q0 % N.F.N;
  for (int s = 0; s < K; ++s) {
    for (int k = 1; k <= r; ++k) {
      if (k == 2 && nitl) {
        near_sides(Fs, sm, sa, itl, nitl, pf, N.frac[1], true, above, L);
        __syncthreads();
      }
      if (fine || (coarse && k == 1)) {
        const int o = fine ? pf * Fs.plane : pc * Cs.plane, v = fine ? (pf ^ 1) * Fs.plane : (pc ^ 1) * Cs.plane;
        const T* pq = sm + L.ph + (fine ? 2 * (K + s * r + k - 1) : 2 * s);
        const unsigned vb = (unsigned)(v * sizeof(T));
        near_step<T, R>(sm, bx + o, by + o, bx + v, by + v, fine ? Fs.cols : Cs.cols, n, fine ? N.F.c : A.C.c,
                        (fine ? qf : qc) != 0, pq[0], pq[1], upx + vb, upy + vb, dnx + vb);
      }
      const int ni_ = k == 1 ? nit : nitf;
      if (ni_ || (k > 1 && nitl)) {
        __syncthreads();
        near_items(Fs, Cs, sm, sa, itf, ni_, pf, pc, N.F.c.mur, A.C.c.mur, above);
        if (k > 1) near_sides(Fs, sm, sa, itl, nitl, pf ^ 1, N.frac[k], false, above, L);
      }
      if (k == 1) pc ^= 1;
      pf ^= 1;
      if (k == r && N.restr && Fs.nr) {
        // a8: the means of r collinear fine edges, in the order of em_strips
        if (nmur || !(ni_ || nitl)) __syncthreads();
        for (int e = t; e < (fr + top) * (ni + 1); e += nt) {
          const int a = (int)__umulhi((unsigned)e, nmul), I = e - a * (ni + 1);
          const int gi = N.I0 + I, gj = N.J0 + Fs.j0 / r + a;
          const T* f = sm + Fs.ex + pf * Fs.plane + (1 + a * r) * Fs.cols + r * I;
          if (I < ni && gj >= N.jlo && gj <= N.jhi) {
            T acc = f[0];
            for (int u = 1; u < r; ++u) acc = acc + f[u];
            near_put_coarse(Cs, sa, cmul, pc, true, gi - N.wi, gj - N.wj, acc * N.rinv);
          }
          if (a < fr && gi >= N.ilo && gi <= N.ihi) {
            const T* g = f + (Fs.ey - Fs.ex);
            T acc = g[0];
            for (int u = 1; u < r; ++u) acc = acc + g[u * Fs.cols];
            near_put_coarse(Cs, sa, cmul, pc, false, gi - N.wi, gj - N.wj, acc * N.rinv);
          }
        }
      }
      cluster_sync();
      if (++qf == N.F.N) qf = 0;
    }
    if (++qc == A.C.N) qc = 0;
  }
  if (fine) unit_store(Fs, n, N.F, sm, pf, ui, urow);
  else if (coarse) unit_store(Cs, n, A.C, sm, pc, ui, urow);
}

// ---------------------------------------------------------------------------
// Launches
// ---------------------------------------------------------------------------
extern __shared__ __align__(16) char multi_smem[];

// the tiles of the coarse mesh (all of it without a fine rectangle)
template <class T, int C, int R, int TH>
__global__ void __launch_bounds__(TH) k_multi(MultiArgs<T> A) {
  multi_tiles<T, C, R>(A, (int)blockIdx.x, reinterpret_cast<T*>(multi_smem));
}

// the r sub-steps of a fine mesh in one coarse step
template <class T, int C, int R, int TH>
__global__ void __launch_bounds__(TH) k_fine(MultiArgs<T> A, const __grid_constant__ FineArgs<T> F) {
  multi_tiles<T, C, R, true>(A, (int)blockIdx.x, reinterpret_cast<T*>(multi_smem), &F);
}

// the near region: one cluster
template <class T, int R, int TH>
__global__ void __launch_bounds__(TH) k_near(MultiArgs<T> A, NearArgs<T> N) {
  multi_near<T, R>(A, N, multi_smem);
}

// The same for the runs of a batch: their arguments in the launch's parameters
// (a block copies its run's into shared memory), tiles of run q from block
// off[q] on, one cluster per run.
constexpr int kMultiRuns = 40;
template <class T>
struct MultiBatch {
  int nruns, off[kMultiRuns + 1];
  MultiArgs<T> a[kMultiRuns];
  NearArgs<T> n[kMultiRuns];
};
static_assert(sizeof(MultiBatch<float>) <= 32764, "kernel parameters");

template <class A>
__device__ __forceinline__ void multi_stage(A* dst, const A& src) {
  static_assert(sizeof(A) % 4 == 0, "words");
  const int* s = reinterpret_cast<const int*>(&src);
  for (int q = threadIdx.x; q < (int)(sizeof(A) / 4); q += blockDim.x) reinterpret_cast<int*>(dst)[q] = s[q];
}

template <class T, int C, int R, int TH>
__global__ void __launch_bounds__(TH) k_multi_batch(const __grid_constant__ MultiBatch<T> B) {
  __shared__ MultiArgs<T> A;
  int q = 0;
  while (q + 1 < B.nruns && (int)blockIdx.x >= B.off[q + 1]) ++q;
  multi_stage(&A, B.a[q]);
  __syncthreads();
  multi_tiles<T, C, R>(A, (int)blockIdx.x - B.off[q], reinterpret_cast<T*>(multi_smem));
}

template <class T, int R, int TH>
__global__ void __launch_bounds__(TH) k_near_batch(const __grid_constant__ MultiBatch<T> B) {
  __shared__ MultiArgs<T> A;
  __shared__ NearArgs<T> N;
  const int q = (int)blockIdx.x / cluster_size();
  multi_stage(&A, B.a[q]);
  multi_stage(&N, B.n[q]);
  __syncthreads();
  multi_near<T, R>(A, N, multi_smem);
}

}  // namespace dmr
