// dmr_adjoint.cuh -- hand-written reverse-mode (adjoint) kernels of the DMR
// time step with the refinement schedule held fixed.
//
// Each forward operation of dmr_kernels.cuh is transposed in gather form
// where every output has one writer (no atomics), and scatter form with
// atomics where several fine samples map to one coarse sample (Eq. 5a/5b
// transposes).  Notation: a* is the adjoint (dL/d*) of a forward variable.
//
// Forward EM step at level l (see k_em), per mesh:
//   S2 += e2(E^l)                       (if the level is an E^2 sample)
//   H'  = H - ch curlE(E^l)
//   v'  = va v - vb (E^l + inc)
//   E'  = E^l + ce curlH(H') + cj (n_a + n_b) v'          interior edges
//   E'_b = E^l_1 + mur (E'_1 - E^l_b)                      Mur sides
//   E'_b = Eq. 5b(coarse E^n, coarse E^{n+1})              coarse-fine sides
// Reverse: Mur^T, Eq. 5b^T (scatter to coarse), E^T, v^T, H^T, S2^T.
#pragma once
#include "dmr_kernels.cuh"

namespace dmr {

// Tape copies of a recorded step in one launch: job q copies n16[q] 16-byte
// words from src[q] to dst[q] (blockIdx.y = job, grid-stride along x).
constexpr int kTapeJobs = 16;
struct TapeJobs {
  const int4* src[kTapeJobs];
  int4* dst[kTapeJobs];
  long long n16[kTapeJobs];
  int n;
};

__global__ void ka_tape_gather(TapeJobs J) {
  const int q = blockIdx.y;
  if (q >= J.n) return;
  const int4* __restrict__ s = J.src[q];
  int4* __restrict__ d = J.dst[q];
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < J.n16[q]; k += stride) d[k] = s[k];
}

template <class T>
struct AdjM {
  const T *aEx_in, *aEy_in;   // adjoint of E^{l+1}
  T *aEx_out, *aEy_out;       // adjoint of E^l (accumulated with +=)
  const T* aHz;               // adjoint of H^{l+1/2} (ka_eh: before the step's own curl share)
  T* aHz_out;                 // ka_eh: adjoint of H^{l-1/2} (the other buffer of the pair)
  T *avx, *avy;               // adjoint of v^{l+1/2} in, of v^{l-1/2} out (in place)
  T* an;                      // adjoint of n (accumulated)
  const T* aS2;               // adjoint of the period's S2 sum (nodes)
  int nx, ny, p;
};

template <class T>
struct FwdM {                 // recorded forward values of the step
  const T *Ex, *Ey;           // E^l as the step used it
  const T *vx, *vy;           // v^{l+1/2}
  const T* n;
};

struct Modes { int m[4]; };

__device__ __forceinline__ double block_sum_d(double v) { return block_sum(v); }

// Coarse side of a reversed coarse step (nullptrs / off on a fine mesh or
// without a rectangle):
//  * the Eq. 5b^T shares of the coarse tangential E^n along the rectangle's
//    coarse-fine sides, gathered by ka_cfb into line buffers (indexed along
//    the line) instead of the edge adjoints: the coarse ka_e adds them to
//    the edges it writes and clears them;
//  * a8^T: the adjoint of a restricted coarse E^n edge goes to its r fine
//    edges (1/r each; the fine E^n adjoint) and the coarse edge keeps 0.
template <class T>
struct CoarseT {
  int side_on[4], side_at[4];   // lines of the coarse-fine sides (row bottom/top, column left/right)
  T* side[4];
  int restr;                     // a8 is transposed at this step
  int I0, J0, I1, J1, r, jlo, jhi, ilo, ihi;
  T *fEx, *fEy;                  // the fine E^n adjoint
  int fp;
};

// Node (i, j) of a reversed EM step: the adjoint of H^{l-1/2} at cell (i, j)
// (from the other H buffer, re-evaluated at the two neighbouring cells the
// edges of the node need), then the gather of aE^l (edges (i, j)), av, an;
// returns the node's E0 share.  The edge adjoints of E^l are stored (the
// output buffer is not cleared before); with a CoarseT the side shares are
// added and a8 transposed.
// Bound by latency: a reversed coarse step is a chain of r + 1 launches of few
// blocks each.  So all loads come first and none is behind a branch that
// differs within a block: absent edges count 0, the Mur rows' shares are
// selects, and 64 registers hold what is in flight.  (With the loads where the
// formulas need them, behind the edge tests, the compiler kept 32 registers and
// a thread made one trip to L2 after the other: 13.9 us per launch cold, of 12
// blocks as of 580.)  near_mur (the block holds nodes whose edges reach a Mur
// row's share) is the same for the whole block.  512^2, r = 2, 512 steps recorded
// and reversed, FP32: 27.8 to 23.1 ms, 21.3 ms with the Mur sides' loads and the
// fine edges' read-modify-writes out of the other blocks' chains; 40 x 32 in
// FP64, 128 steps: 10.7 to 9.4 ms.
template <class T>
__device__ __forceinline__ T ka_e_node(const AdjM<T>& a, const FwdM<T>& f, const Step<T>& c, const Modes& md,
                                       const CoarseT<T>& ct, bool near_mur, int i, int j) {
  const int nx = a.nx, ny = a.ny, p = a.p;
  if (i > nx || j > ny) return T(0);
  const int id = j * p + i;
  const bool xe = i < nx, ye = j < ny;
  auto ld = [](const T* q, bool v) { return v ? *q : T(0); };
  // edges whose E' the interior formula gives: 0 < j < ny (x), 0 < i < nx (y)
  const bool jin = j > 0 && j < ny, iin = i > 0 && i < nx;
  const bool jdn = j > 1, jup = j + 1 < ny, ilf = i > 1, irt = i + 1 < nx;   // the same one row / column on
  T x00 = ld(a.aEx_in + id, xe && jin);
  T x0p = ld(a.aEx_in + id + p, xe && jup);
  T x0m = ld(a.aEx_in + id - p, xe && jdn);
  T xm0 = ld(a.aEx_in + id - 1, i > 0 && jin);
  T xmp = ld(a.aEx_in + id + p - 1, i > 0 && jup);
  T y00 = ld(a.aEy_in + id, ye && iin);
  T yp0 = ld(a.aEy_in + id + 1, ye && irt);
  T ym0 = ld(a.aEy_in + id - 1, ye && ilf);
  T y0m = ld(a.aEy_in + id - p, j > 0 && iin);
  T ypm = ld(a.aEy_in + id - p + 1, j > 0 && irt);
  const T hz00 = ld(a.aHz + id, xe && ye);
  const T hz0m = ld(a.aHz + id - p, xe && j > 0);
  const T hzm0 = ld(a.aHz + id - 1, ye && i > 0);
  const T avx0 = ld(a.avx + id, xe), avy0 = ld(a.avy + id, ye), an0 = a.an[id];
  const T n00 = f.n[id], np0 = ld(f.n + id + 1, xe), n0p = ld(f.n + id + p, ye);
  const T vx0 = ld(f.vx + id, xe && jin), vxm = ld(f.vx + id - 1, i > 0 && jin);
  const T vy0 = ld(f.vy + id, ye && iin), vym = ld(f.vy + id - p, j > 0 && iin);
  const T ckx = c.ckx[i], skx = c.skx[i];
  const T ex = ld(f.Ex + id, c.accum && xe), ey0 = ld(f.Ey + id, c.accum && ye);
  const T s00 = ld(a.aS2 + id, c.accum), sp0 = ld(a.aS2 + id + 1, c.accum && xe), s0p = ld(a.aS2 + id + p, c.accum && ye);
  const bool s_b = xe && ct.side_on[SIDE_BOTTOM] && j == ct.side_at[SIDE_BOTTOM];
  const bool s_t = xe && ct.side_on[SIDE_TOP] && j == ct.side_at[SIDE_TOP];
  const bool s_l = ye && ct.side_on[SIDE_LEFT] && i == ct.side_at[SIDE_LEFT];
  const bool s_r = ye && ct.side_on[SIDE_RIGHT] && i == ct.side_at[SIDE_RIGHT];
  const T v_b = ld(ct.side[SIDE_BOTTOM] + i, s_b), v_t = ld(ct.side[SIDE_TOP] + i, s_t);
  const T v_l = ld(ct.side[SIDE_LEFT] + j, s_l), v_r = ld(ct.side[SIDE_RIGHT] + j, s_r);
  // ---- Mur sides: row 1 of Ex gave mur E' to row 0 (and so on), so its adjoint
  // takes mur times row 0's; bx0, bxm: row 0 or ny of columns i, i - 1, by0, bym:
  // column 0 or nx of rows j, j - 1
  const bool mb = md.m[SIDE_BOTTOM] == BC_MUR && j <= 2, mt = md.m[SIDE_TOP] == BC_MUR && j >= ny - 2;
  const bool ml = md.m[SIDE_LEFT] == BC_MUR && i <= 2, mr = md.m[SIDE_RIGHT] == BC_MUR && i >= nx - 2;
  T b0 = T(0), t0 = T(0), l0 = T(0), r0 = T(0);
  if (near_mur) {   // the same for the whole block
    b0 = ld(a.aEx_in + i, mb && xe);
    const T bm = ld(a.aEx_in + i - 1, mb && i > 0);
    t0 = ld(a.aEx_in + ny * p + i, mt && xe);
    const T tm = ld(a.aEx_in + ny * p + i - 1, mt && i > 0);
    l0 = ld(a.aEy_in + j * p, ml && ye);
    const T lm = ld(a.aEy_in + (j - 1) * p, ml && j > 0);
    r0 = ld(a.aEy_in + j * p + nx, mr && ye);
    const T rm = ld(a.aEy_in + (j - 1) * p + nx, mr && j > 0);
    auto mur = [&](T v, bool on, T w) { return on ? v + c.mur * w : v; };
    x00 = mur(mur(x00, mb && j == 1, b0), mt && j == ny - 1, t0);
    x0p = mur(mur(x0p, mb && j == 0, b0), mt && j == ny - 2, t0);
    x0m = mur(mur(x0m, mb && j == 2, b0), mt && j == ny, t0);
    xm0 = mur(mur(xm0, mb && j == 1, bm), mt && j == ny - 1, tm);
    xmp = mur(mur(xmp, mb && j == 0, bm), mt && j == ny - 2, tm);
    y00 = mur(mur(y00, ml && i == 1, l0), mr && i == nx - 1, r0);
    yp0 = mur(mur(yp0, ml && i == 0, l0), mr && i == nx - 2, r0);
    ym0 = mur(mur(ym0, ml && i == 2, l0), mr && i == nx, r0);
    y0m = mur(mur(y0m, ml && i == 1, lm), mr && i == nx - 1, rm);
    ypm = mur(mur(ypm, ml && i == 0, lm), mr && i == nx - 2, rm);
  }
  // ---- adjoint of H^{l-1/2} at the cells (i, j), (i, j - 1), (i - 1, j): that
  // of H^{l+1/2} plus ce curlH^T(aE') over the interior edges
  const T h00 = (xe && ye) ? hz00 + c.ce * (x00 - x0p - y00 + yp0) : T(0);
  const T h0m = (xe && j > 0) ? hz0m + c.ce * (x0m - x00 - y0m + ypm) : T(0);
  const T hm0 = (ye && i > 0) ? hzm0 + c.ce * (xm0 - xmp - ym0 + y00) : T(0);
  T e0 = T(0), an_acc = vx0 * x00;
  an_acc = an_acc + vxm * xm0;
  // ---- x edge (i, j)
  T outx, avx1;
  {
    const T avt = avx0 + c.cj * (n00 + np0) * x00;
    T out = x00;
    if (j == 1 && mb) out = out + b0;
    if (j == ny - 1 && mt) out = out + t0;
    if (j == 0 && mb) out = -c.mur * b0;
    if (j == ny && mt) out = -c.mur * t0;
    out = out - c.vb * avt;
    out = out - c.ch * (h00 - h0m);
    if (c.accum) {
      const T wl = (i > 0) ? T(0.5) : T(1);                 // node i: this is its right edge
      const T wr = (i + 1 < nx) ? T(0.5) : T(1);            // node i+1: its left edge
      out = out + T(2) * ex * (s00 * wl + sp0 * wr);
    }
    avx1 = c.va * avt;
    if (s_b) out = v_b + out;
    if (s_t) out = v_t + out;
    outx = out;
  }
  // ---- y edge (i, j)
  an_acc = an_acc + vy0 * y00;
  an_acc = an_acc + vym * y0m;
  T outy, avy1;
  {
    const T phi = c.sphi * ckx - c.cphi * skx;
    const T avt = avy0 + c.cj * (n00 + n0p) * y00;
    T out = y00;
    if (i == 1 && ml) out = out + l0;
    if (i == nx - 1 && mr) out = out + r0;
    if (i == 0 && ml) out = -c.mur * l0;
    if (i == nx && mr) out = -c.mur * r0;
    out = out - c.vb * avt;
    if (ye) e0 -= c.vb * avt * phi;
    out = out - c.ch * (hm0 - h00);
    if (c.accum && ye) {
      const T ey = ey0 + c.E0 * phi;
      const T wb = (j > 0) ? T(0.5) : T(1);
      const T wt = (j + 1 < ny) ? T(0.5) : T(1);
      const T g = T(2) * ey * (s00 * wb + s0p * wt);
      out = out + g;
      e0 += g * phi;
    }
    avy1 = c.va * avt;
    if (s_l) out = v_l + out;
    if (s_r) out = v_r + out;
    outy = out;
  }
  // ---- a8 transposed: the adjoint of a restricted coarse edge goes to its r
  // fine edges; the first two of each are loaded before anything is stored
  const bool gx = ct.restr && xe && i >= ct.I0 && i < ct.I1 && j >= ct.jlo && j <= ct.jhi;
  const bool gy = ct.restr && ye && j >= ct.J0 && j < ct.J1 && i >= ct.ilo && i <= ct.ihi;
  T* const dx = ct.fEx + ((ptrdiff_t)(ct.r * (j - ct.J0)) * ct.fp + ct.r * (i - ct.I0));
  T* const dy = ct.fEy + ((ptrdiff_t)(ct.r * (j - ct.J0)) * ct.fp + ct.r * (i - ct.I0));
  const T dx0 = ld(dx, gx), dx1 = ld(dx + 1, gx), dy0 = ld(dy, gy), dy1 = ld(dy + ct.fp, gy);
  // ---- stores
  if (xe && ye) a.aHz_out[id] = h00;
  a.an[id] = an0 + c.cj * an_acc;
  if (xe) {
    a.avx[id] = avx1;
    if (s_b) ct.side[SIDE_BOTTOM][i] = T(0);
    if (s_t) ct.side[SIDE_TOP][i] = T(0);
    if (gx) {
      const T t = outx / (T)ct.r;
      dx[0] = dx0 + t;
      dx[1] = dx1 + t;
      for (int q = 2; q < ct.r; ++q) dx[q] += t;
      outx = T(0);
    }
    a.aEx_out[id] = outx;
  }
  if (ye) {
    a.avy[id] = avy1;
    if (s_l) ct.side[SIDE_LEFT][j] = T(0);
    if (s_r) ct.side[SIDE_RIGHT][j] = T(0);
    if (gy) {
      const T t = outy / (T)ct.r;
      dy[0] = dy0 + t;
      dy[ct.fp] = dy1 + t;
      for (int q = 2; q < ct.r; ++q) dy[(size_t)q * ct.fp] += t;
      outy = T(0);
    }
    a.aEy_out[id] = outy;
  }
  return e0;
}

// Eq. 5b^T: the adjoint of each coarse-fine boundary edge of the fine mesh goes
// to the coarse tangential E before (old) and after (new) the coarse step.
template <class T>
struct CfbT {
  int mode[4], start[4], len[4], at[4];
  int r;
  T frac;
  T *new_x, *new_y;                   // coarse adjoint arrays of E^{n+1}
  T* old_line[4];                     // E^n shares, per side along its line (CoarseT::side)
  int cp;                             // coarse pitch
};

// Eq. 5b^T of sample q of side SD, if q lies on it; else q is reduced by the
// side's length and false returned.
template <int SD, class T>
__device__ __forceinline__ bool ka_cfb_side(const AdjM<T>& a, const CfbT<T>& b, int& q) {
  if (b.mode[SD] != BC_CFB) return false;
  constexpr bool xs = SD == SIDE_BOTTOM || SD == SIDE_TOP;
  const int nfx = a.nx, nfy = a.ny, p = a.p;
  const int len = xs ? nfx : nfy;
  if (q >= len) { q -= len; return false; }
  T t;
  if (SD == SIDE_BOTTOM) t = a.aEx_in[q];
  else if (SD == SIDE_TOP) t = a.aEx_in[nfy * p + q];
  else if (SD == SIDE_LEFT) t = a.aEy_in[q * p];
  else t = a.aEy_in[q * p + nfx];
  const int num = 2 * q + 1 - b.r, den = 2 * b.r;
  const int fl = (num >= 0) ? num / den : -((-num + den - 1) / den);
  int i0 = b.start[SD] + fl;
  T xp = (T)(num - fl * den) / (T)den;
  if (i0 < 0) { i0 = 0; xp = T(0); }
  if (i0 > b.len[SD] - 2) { i0 = b.len[SD] - 2; xp = T(1); }
  const T one = T(1);
  const T wo0 = (one - b.frac) * (one - xp), wo1 = (one - b.frac) * xp;
  const T wn0 = b.frac * (one - xp), wn1 = b.frac * xp;
  size_t s0, s1;
  T* n;
  if (xs) {
    s0 = (size_t)b.at[SD] * b.cp + i0; s1 = s0 + 1; n = b.new_x;
  } else {
    s0 = (size_t)i0 * b.cp + b.at[SD]; s1 = s0 + b.cp; n = b.new_y;
  }
  atomicAdd(b.old_line[SD] + i0, wo0 * t);
  atomicAdd(b.old_line[SD] + i0 + 1, wo1 * t);
  atomicAdd(n + s0, wn0 * t);
  atomicAdd(n + s1, wn1 * t);
  return true;
}

// Eq. 5b^T of side sample q (the sides in the order bottom, top, left, right)
template <class T>
__device__ __forceinline__ void ka_cfb_sample(const AdjM<T>& a, const CfbT<T>& b, int q) {
  if (ka_cfb_side<SIDE_BOTTOM>(a, b, q)) return;
  if (ka_cfb_side<SIDE_TOP>(a, b, q)) return;
  if (ka_cfb_side<SIDE_LEFT>(a, b, q)) return;
  ka_cfb_side<SIDE_RIGHT>(a, b, q);
}

// A rectangle of node blocks of one mesh in a reversed EM step: blocks
// (bx0 + k % nbx, by0 + k / nbx), each TX x TY nodes, except those inside the
// skip box [sx0, sx1] x [sy0, sy1] (sx0 > sx1: none skipped).
template <class T>
struct NodePart {
  AdjM<T> a;
  FwdM<T> f;
  Step<T> c;
  Modes md;
  CoarseT<T> ct;
  int bx0, by0, nbx, nby;
  int sx0, sx1, sy0, sy1;
};

// Node block k of a part: ka_e_node over its nodes, E0 share summed in FP64.
template <class T>
__device__ __forceinline__ void ka_part_block(const NodePart<T>& P, int k, double* e0acc) {
  const int by = P.by0 + k / P.nbx, bx = P.bx0 + k % P.nbx;
  if (bx >= P.sx0 && bx <= P.sx1 && by >= P.sy0 && by <= P.sy1) return;   // whole block
  const bool near_mur = (P.md.m[SIDE_LEFT] == BC_MUR && bx * TX <= 2) ||
                        (P.md.m[SIDE_RIGHT] == BC_MUR && bx * TX + TX - 1 >= P.a.nx - 2) ||
                        (P.md.m[SIDE_BOTTOM] == BC_MUR && by * TY <= 2) ||
                        (P.md.m[SIDE_TOP] == BC_MUR && by * TY + TY - 1 >= P.a.ny - 2);
  const T e0 = ka_e_node(P.a, P.f, P.c, P.md, P.ct, near_mur, bx * TX + (int)threadIdx.x,
                         by * TY + (int)threadIdx.y);
  const double s = block_sum_d((double)e0);
  if (threadIdx.x == 0 && threadIdx.y == 0 && s != 0.0) atomicAdd(e0acc, s);
}

// One launch of a reversed EM step: the node blocks of part P0 (nb0 blocks),
// then the Eq. 5b^T side samples of P0's fine mesh (ncfb blocks of TX * TY
// samples; they read aE' and add to coarse adjoints only), then the node
// blocks of part P1 (nb1 blocks): coarse nodes away from the rectangle run
// beside the fine sub-steps of the same coarse step, which neither read nor
// write them.
template <class T>
__global__ void __launch_bounds__(TX * TY, sizeof(T) == 4 ? 4 : 2) ka_eh(NodePart<T> P0, NodePart<T> P1, CfbT<T> cb, int nb0, int ncfb,
                                                 double* e0acc) {
  const int blk = (int)blockIdx.x;
  if (blk < nb0) {
    ka_part_block(P0, blk, e0acc);
  } else if (blk < nb0 + ncfb) {
    ka_cfb_sample(P0.a, cb, (blk - nb0) * TX * TY + (int)(threadIdx.y * TX + threadIdx.x));
  } else {
    ka_part_block(P1, blk - nb0 - ncfb, e0acc);
  }
}

// a8^T for E: the adjoint of a restricted coarse edge goes to its r fine edges
// (1/r each) and is cleared on the coarse mesh.
template <class T>
__global__ void ka_restrict(T* cEx, T* cEy, int cp, T* fEx, T* fEy, int fp, int I0, int J0, int I1,
                            int J1, int r, int jlo, int jhi, int ilo, int ihi) {
  const int i = I0 + blockIdx.x * blockDim.x + threadIdx.x;
  const int j = J0 + blockIdx.y * blockDim.y + threadIdx.y;
  if (i > I1 || j > J1) return;
  const int fa = r * (i - I0), fb = r * (j - J0);
  if (i < I1 && j >= jlo && j <= jhi) {
    const T t = cEx[j * cp + i] / (T)r;
    T* d = fEx + (size_t)fb * fp + fa;
    for (int q = 0; q < r; ++q) d[q] += t;
    cEx[j * cp + i] = T(0);
  }
  if (j < J1 && i >= ilo && i <= ihi) {
    const T t = cEy[j * cp + i] / (T)r;
    T* d = fEy + (size_t)fb * fp + fa;
    for (int q = 0; q < r; ++q) d[(size_t)q * fp] += t;
    cEy[j * cp + i] = T(0);
  }
}

// S2^T for one sample level: aE += 2 E_total aS2 (node weights), E0 share.
template <class T>
__global__ void ka_s2(T* aEx, T* aEy, const T* Ex, const T* Ey, const T* aS2, Step<T> c, int nx,
                      int ny, int p, double* e0acc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  double e0 = 0.0;
  if (i <= nx && j <= ny) {
    const int id = j * p + i;
    if (i < nx) {
      const T wl = (i > 0) ? T(0.5) : T(1);
      const T wr = (i + 1 < nx) ? T(0.5) : T(1);
      aEx[id] += T(2) * Ex[id] * (aS2[id] * wl + aS2[id + 1] * wr);
    }
    if (j < ny) {
      const T phi = c.sphi * c.ckx[i] - c.cphi * c.skx[i];
      const T ey = Ey[id] + c.E0 * phi;
      const T wb = (j > 0) ? T(0.5) : T(1);
      const T wt = (j + 1 < ny) ? T(0.5) : T(1);
      const T g = T(2) * ey * (aS2[id] * wb + aS2[id + p] * wt);
      aEy[id] += g;
      e0 += (double)g * (double)phi;
    }
  }
  const double s = block_sum_d(e0);
  if (threadIdx.x == 0 && threadIdx.y == 0 && s != 0.0) atomicAdd(e0acc, s);
}

// ---------------------------------------------------------------------------
// Continuity step (Eq. 4) reverse
// ---------------------------------------------------------------------------
// Per node: nu_net, D_eff and the derivatives the reverse sweep needs,
// evaluated exactly as k_rates does for the values.
template <class T>
__global__ void ka_rates_d(const T* n, const double* S2f, Dens d, double A1, int nx, int ny, int p, T* D,
                           T* nu, T* dDdn, T* dDdnu, T* dnudS2, T* nu_s) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i > nx || j > ny) return;
  const int id = j * p + i;
  const double s2 = S2f[id];
  const double e2 = eeff2_of(s2, d);
  const double eeff = sqrt(e2);
  const T x = ehp_of<T>(e2, d);
  T nui = T(0), dn = T(0), per_s = T(0);
  if (d.model == 1) {
    // Townsend form: nu = A p exp(-Bp/E) mu_e E, d nu/d S2 = nu (1 + Bp/E) / (2 S2)
    const T ee = sqrt((T)e2);
    if (ee > T(0)) {
      const T ex = exp(-(T)d.tBp / ee);
      nui = (T)d.A * ex * (T)d.mu_e * ee;
      per_s = (T)A1 * ex * (T)d.mu_e * ee;
      dn = (T)((double)nui * (1.0 + d.tBp / (double)ee) / (2.0 * s2));
    }
  } else if (x > T(0)) {
    const T ex = exp(T(-73.0) * pow(x, T(-0.44)));
    nui = (T)d.A * ex;
    per_s = (T)A1 * ex;
    // d nu / d S2 = nu 73 0.44 x^-1.44 (dx/dS2), dx/dS2 = 1 / (2 hp eeff N g)
    dn = (T)((double)nui * 73.0 * 0.44 * pow((double)x, -1.44) / (2.0 * d.hp * eeff * d.N * d.g));
  }
  const T nv = n[id];
  const T wp2 = nv * (T)d.wp2c;
  const T num = nui * (T)d.nu_m * (T)d.De + wp2 * (T)d.Da;
  const T den = nui * (T)d.nu_m + wp2;
  T Dv, gn = T(0), gnu = T(0);
  if (den == T(0)) {
    Dv = (T)d.De;
  } else {
    Dv = num / den;
    gn = (T)d.wp2c * ((T)d.Da - Dv) / den;
    gnu = (T)d.nu_m * ((T)d.De - Dv) / den;
  }
  D[id] = Dv;
  nu[id] = nui - (T)d.nu_a;
  dDdn[id] = gn;
  dDdnu[id] = gnu;
  dnudS2[id] = dn;
  nu_s[id] = per_s;
}

// Gather of a_n (old density), a_S2f and the s_nu share from a_n' (new
// density).  `dir` nodes of the fine mesh were set from the coarse mesh and do
// not depend on the fine density (their a_n' has been moved already).
template <class T>
__global__ void ka_density(const T* n, const T* D, const T* nu, const T* dDdn, const T* dDdnu,
                           const T* dnudS2, const T* nu_s, const T* an_new, T* an_old, T* aS2,
                           Dens d, Dir<T> dir, int nx, int ny, int p, double* snu_acc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  double sacc = 0.0;
  if (i <= nx && j <= ny) {
    const int id = j * p + i;
    auto isdir = [&](int a, int b) {
      return (dir.on[SIDE_BOTTOM] && b == 0) || (dir.on[SIDE_TOP] && b == ny) ||
             (dir.on[SIDE_LEFT] && a == 0) || (dir.on[SIDE_RIGHT] && a == nx);
    };
    const T T_ = (T)d.T, dx2 = (T)d.dx2, r = (T)d.r_ei;
    const T nk = n[id], Dk = D[id];
    T a_n = T(0), a_nu = T(0);
    const int nb_i[4] = {i + 1, i - 1, i, i};
    const int nb_j[4] = {j, j, j + 1, j - 1};
    const bool self_live = !isdir(i, j);
    const T ak = self_live ? an_new[id] : T(0);
    // own update
    if (self_live) {
      T dself = T(0), dnu = T(0);
      for (int f = 0; f < 4; ++f) {
        const int a = nb_i[f], b = nb_j[f];
        if (a < 0 || a > nx || b < 0 || b > ny) continue;
        const int fid = b * p + a;
        dself = dself + (T(0.5) * dDdn[id] * (n[fid] - nk) - T(0.5) * (Dk + D[fid]));
        dnu = dnu + T(0.5) * dDdnu[id] * (n[fid] - nk);
      }
      a_n = a_n + ak * (T(1) + T_ * (dself / dx2 + nu[id] - T(2) * r * nk));
      a_nu = a_nu + ak * T_ * (dnu / dx2 + nk);
    }
    // neighbours' updates that read this node
    for (int f = 0; f < 4; ++f) {
      const int a = nb_i[f], b = nb_j[f];
      if (a < 0 || a > nx || b < 0 || b > ny) continue;
      if (isdir(a, b)) continue;
      const int fid = b * p + a;
      const T af = an_new[fid];
      a_n = a_n + af * T_ * (T(0.5) * (D[fid] + Dk) + T(0.5) * dDdn[id] * (nk - n[fid])) / dx2;
      a_nu = a_nu + af * T_ * T(0.5) * dDdnu[id] * (nk - n[fid]) / dx2;
    }
    an_old[id] = a_n;
    aS2[id] = a_nu * dnudS2[id];
    sacc = (double)a_nu * (double)nu_s[id];
  }
  const double s = block_sum_d(sacc);
  if (threadIdx.x == 0 && threadIdx.y == 0 && s != 0.0) atomicAdd(snu_acc, s);
}

// a10^T: fine Dirichlet nodes took the new coarse density along the side
// (same side priority as k_density); their adjoint moves to the coarse mesh.
// Here dir.line[] point into the coarse adjoint array.
template <class T>
__global__ void ka_dir(T* an_f, int nfx, int nfy, int fp, Dir<T> dir) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i > nfx || j > nfy) return;
  int sd = -1, q = 0;
  if (dir.on[SIDE_BOTTOM] && j == 0) { sd = SIDE_BOTTOM; q = i; }
  else if (dir.on[SIDE_TOP] && j == nfy) { sd = SIDE_TOP; q = i; }
  else if (dir.on[SIDE_LEFT] && i == 0) { sd = SIDE_LEFT; q = j; }
  else if (dir.on[SIDE_RIGHT] && i == nfx) { sd = SIDE_RIGHT; q = j; }
  if (sd < 0) return;
  const int id = j * fp + i;
  const T t = an_f[id];
  an_f[id] = T(0);
  double pos = (double)dir.start[sd] + (double)q / (double)dir.r;
  int i0 = (int)floor(pos);
  double w = pos - (double)i0;
  if (i0 < 0) { i0 = 0; w = 0.0; }
  if (i0 > dir.len[sd] - 2) { i0 = dir.len[sd] - 2; w = 1.0; }
  const T xp = (T)w;
  const int s = dir.stride[sd];
  T* l = const_cast<T*>(dir.line[sd]);
  atomicAdd(l + (size_t)i0 * s, t * (T(1) - xp));
  atomicAdd(l + (size_t)(i0 + 1) * s, t * xp);
}

// injection^T (commit^T): coarse nodes of the closed rectangle took the fine
// value; their adjoint goes to the coinciding fine node.
template <class T>
__global__ void ka_inject(T* an_c, int cp, T* an_f, int fp, int I0, int J0, int I1, int J1, int r) {
  const int i = I0 + blockIdx.x * blockDim.x + threadIdx.x;
  const int j = J0 + blockIdx.y * blockDim.y + threadIdx.y;
  if (i > I1 || j > J1) return;
  const int cid = j * cp + i;
  an_f[(size_t)(r * (j - J0)) * fp + r * (i - I0)] += an_c[cid];
  an_c[cid] = T(0);
}

// a12^T: growth copied the old fine data and filled the rest bilinearly from
// the coarse mesh.  Adjoint: copy back to the old layout, scatter the rest.
template <class T>
struct ExpT {
  const T *nEx, *nEy, *nHz, *nvx, *nvy, *nn;   // adjoints in the new layout
  T *oEx, *oEy, *oHz, *ovx, *ovy, *on;         // adjoints in the old layout (written)
  T *cEx, *cEy, *cHz, *cvx, *cvy, *cn;         // coarse adjoints (atomic +=)
  int nnx, nny, np, onx, ony, op, cnx, cny, cp;
  int I0, J0, oI0, oJ0, r;
};

template <class T>
__device__ __forceinline__ void bilin_t(T* F, int p, int Lx, int Ly, double u, double v, T t) {
  int i0 = (int)floor(u);
  double fu = u - (double)i0;
  if (i0 < 0) { i0 = 0; fu = 0.0; }
  if (i0 > Lx - 2) { i0 = Lx - 2; fu = 1.0; }
  int j0 = (int)floor(v);
  double fv = v - (double)j0;
  if (j0 < 0) { j0 = 0; fv = 0.0; }
  if (j0 > Ly - 2) { j0 = Ly - 2; fv = 1.0; }
  T* r0 = F + (size_t)j0 * p;
  T* r1 = r0 + p;
  atomicAdd(r0 + i0, t * (T)((1.0 - fu) * (1.0 - fv)));
  atomicAdd(r0 + i0 + 1, t * (T)(fu * (1.0 - fv)));
  atomicAdd(r1 + i0, t * (T)((1.0 - fu) * fv));
  atomicAdd(r1 + i0 + 1, t * (T)(fu * fv));
}

template <class T>
__global__ void ka_expand(ExpT<T> e) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = blockIdx.y * blockDim.y + threadIdx.y;
  if (a > e.nnx || b > e.nny) return;
  const int sa = a - e.r * (e.oI0 - e.I0), sb = b - e.r * (e.oJ0 - e.J0);
  const int id = b * e.np + a;
  const double rr = (double)e.r;
  const double xn = (double)e.I0 + (double)a / rr, yn = (double)e.J0 + (double)b / rr;
  const double xh = ((double)e.I0 + ((double)a + 0.5) / rr) - 0.5;
  const double yh = ((double)e.J0 + ((double)b + 0.5) / rr) - 0.5;
  const bool in_x = sa >= 0 && sa < e.onx, in_xn = sa >= 0 && sa <= e.onx;
  const bool in_y = sb >= 0 && sb < e.ony, in_yn = sb >= 0 && sb <= e.ony;
  const int oid = sb * e.op + sa;
  if (a < e.nnx) {
    if (in_x && in_yn) { e.oEx[oid] = e.nEx[id]; e.ovx[oid] = e.nvx[id]; }
    else {
      bilin_t(e.cEx, e.cp, e.cnx, e.cny + 1, xh, yn, e.nEx[id]);
      bilin_t(e.cvx, e.cp, e.cnx, e.cny + 1, xh, yn, e.nvx[id]);
    }
  }
  if (b < e.nny) {
    if (in_xn && in_y) { e.oEy[oid] = e.nEy[id]; e.ovy[oid] = e.nvy[id]; }
    else {
      bilin_t(e.cEy, e.cp, e.cnx + 1, e.cny, xn, yh, e.nEy[id]);
      bilin_t(e.cvy, e.cp, e.cnx + 1, e.cny, xn, yh, e.nvy[id]);
    }
  }
  if (a < e.nnx && b < e.nny) {
    if (in_x && in_y) e.oHz[oid] = e.nHz[id];
    else bilin_t(e.cHz, e.cp, e.cnx, e.cny, xh, yh, e.nHz[id]);
  }
  if (in_xn && in_yn) e.on[oid] = e.nn[id];
  else bilin_t(e.cn, e.cp, e.cnx + 1, e.cny + 1, xn, yn, e.nn[id]);
}

}  // namespace dmr
