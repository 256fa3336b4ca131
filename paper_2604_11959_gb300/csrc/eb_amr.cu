// eb_amr.cu -- two-level static refinement (Sec. 4.3): the coarse level of a
// refinement ratio of 2 in every direction, built from the fine level by
// merging its cells, and the restriction of a fine state to the coarse level.
//
// A coarse CV of any grid is a block of 2 x 2 x 2 cells of the fine c grid:
// cells 2I, 2I + 1 along x for the c grid and 2I - 1, 2I for the u grid (the
// right half of coarse cell I - 1 and the left half of cell I), likewise
// along y for v and along z for w; fine cells below the bottom or above the
// top of the domain hold no fluid and take no part in the class.  Merging:
//   volume fraction   the mean of the 8 fine ones, the centroid their
//                     volume-weighted mean position;
//   face fraction     the mean of the 4 fine faces on the coarse low face,
//                     the centroid their area-weighted mean position;
//   EB area           the sum of the fine ones (a quarter of it in units of
//                     the coarse dx dy), the centroid their area-weighted mean;
//   EB normal         the direction of the area-weighted sum of the fine EB
//                     normals: the boundary of the fluid in the CV is closed,
//                     so that sum is sum_d (open area of the high d-face - open
//                     area of the low d-face) e_d;
//   class             covered or regular when all its fine cells inside the
//                     domain are, else cut.
// Positions are offsets from the CV (or face) centre in grid units of its
// level: a fine cell's centre lies at -1/2 or +1/2 fine units from the coarse
// CV centre along each axis, and a fine unit is half a coarse one.
#include "eb_handle.cuh"

#include <algorithm>

using namespace ebh;

namespace {

// the fine c-grid cell (i, j, k): class (-1 outside the domain in z) and, with
// V, its moments in the record layout of the geometry kernels (alpha, cent[3],
// beta[3], fcent[6], nrm[3], aeb, ebc[3])
struct FineC {
  Dims D;
  GridDev G;
};

template <bool V>
__device__ inline int fine_cell(const FineC &F, int i, int j, int k, double v[20]) {
  if (V)
    for (int q = 0; q < 20; ++q) v[q] = 0.0;
  if (k < 0 || k >= F.D.nz) return -1;
  const int col = wrapi(i, F.D.nx) + F.D.nx * wrapi(j, F.D.ny);
  const int kc = F.G.kcov[col], kx = F.G.kxt[col];
  if (k < kc) return EBK_COVERED;
  if (k >= kx) {
    if (V) v[0] = v[4] = v[5] = v[6] = 1.0;
    return EBK_REGULAR;
  }
  const long long r = F.G.roff[col] + (k - kc), n = F.G.nrec;
  if (V) {
    v[0] = F.G.alpha[r];
    for (int d = 0; d < 3; ++d) {
      v[1 + d] = F.G.cent[d * n + r];
      v[4 + d] = F.G.beta[d * n + r];
      v[13 + d] = F.G.nrm[d * n + r];
      v[17 + d] = F.G.ebc[d * n + r];
    }
    for (int q = 0; q < 6; ++q) v[7 + q] = F.G.fcent[q * n + r];
    v[16] = F.G.aeb[r];
  }
  return F.G.flag[r];
}

// open fraction of the low d-face of fine cell (i, j, k); the lid above the
// top is open, the floor below the bottom closed
__device__ inline double fine_low_face(const FineC &F, int i, int j, int k, int d) {
  if (k >= F.D.nz) return d == 2 ? 1.0 : 0.0;
  double v[20];
  if (fine_cell<true>(F, i, j, k, v) < 0) return 0.0;
  return v[4 + d];
}

// first fine cell of the block of coarse CV (I, J, K) of grid g
__device__ inline void block_origin(int g, int I, int J, int K, int f0[3]) {
  f0[0] = 2 * I - (g == 1);
  f0[1] = 2 * J - (g == 2);
  f0[2] = 2 * K - (g == 3);
}

__device__ inline int coarse_class(const FineC &F, int g, int I, int J, int K) {
  int f0[3];
  block_origin(g, I, J, K, f0);
  int nin = 0, ncov = 0, nreg = 0;
  double v[20];
  for (int c = 0; c < 2; ++c)
    for (int b = 0; b < 2; ++b)
      for (int a = 0; a < 2; ++a) {
        const int cls = fine_cell<false>(F, f0[0] + a, f0[1] + b, f0[2] + c, v);
        if (cls < 0) continue;
        ++nin;
        ncov += cls == EBK_COVERED;
        nreg += cls == EBK_REGULAR;
      }
  return ncov == nin ? EBK_COVERED : (nreg == nin ? EBK_REGULAR : EBK_CUT);
}

__global__ void k_coarse_bounds(FineC F, Dims Dc, int g, int *kcov, int *kreg) {
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= Dc.nx * Dc.ny) return;
  const int I = col % Dc.nx, J = col / Dc.nx;
  const int nzg = nzg_of(Dc, g);
  int kc = 0;
  while (kc < nzg && coarse_class(F, g, I, J, kc) == EBK_COVERED) ++kc;
  int kr = nzg;
  while (kr > kc && coarse_class(F, g, I, J, kr - 1) == EBK_REGULAR) --kr;
  kcov[col] = kc;
  kreg[col] = kr;
}

// the merged moments of coarse CV (I, J, K) of grid g, record layout
__device__ inline void merge_cv(const FineC &F, const Dims &Dc, int g, int I, int J, int K, double out[20]) {
  int f0[3];
  block_origin(g, I, J, K, f0);
  double vol = 0, m[3] = {0, 0, 0}, eba = 0, eb[3] = {0, 0, 0};
  double fa[3] = {0, 0, 0}, f1[3] = {0, 0, 0}, f2[3] = {0, 0, 0}, fh[3] = {0, 0, 0};
  double v[20];
  for (int c = 0; c < 2; ++c)
    for (int b = 0; b < 2; ++b)
      for (int a = 0; a < 2; ++a) {
        if (fine_cell<true>(F, f0[0] + a, f0[1] + b, f0[2] + c, v) < 0) continue;
        const int q[3] = {a, b, c};
        const double o[3] = {a - 0.5, b - 0.5, c - 0.5};
        vol += v[0];
        eba += v[16];
        for (int d = 0; d < 3; ++d) {
          m[d] += v[0] * (o[d] + v[1 + d]);
          eb[d] += v[16] * (o[d] + v[17 + d]);
        }
        for (int d = 0; d < 3; ++d) {
          if (q[d] != 0) continue;   // the fine cells on the coarse low d-face
          const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
          const double be = v[4 + d];
          fa[d] += be;
          f1[d] += be * (o[t1] + v[7 + 2 * d]);
          f2[d] += be * (o[t2] + v[8 + 2 * d]);
        }
      }
  // open areas of the coarse high faces: the low faces of the fine cells two
  // beyond the block's first along d
  for (int d = 0; d < 3; ++d)
    for (int u = 0; u < 2; ++u)
      for (int w = 0; w < 2; ++w) {
        int p[3] = {f0[0], f0[1], f0[2]};
        const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
        p[d] += 2;
        p[t1] += u;
        p[t2] += w;
        fh[d] += fine_low_face(F, p[0], p[1], p[2], d);
      }
  const double Af[3] = {F.D.dy * F.D.dz, F.D.dx * F.D.dz, F.D.dx * F.D.dy};
  out[0] = vol / 8.0;
  double nv[3], nn = 0.0;
  for (int d = 0; d < 3; ++d) {
    out[1 + d] = vol > 0 ? 0.5 * m[d] / vol : 0.0;
    out[4 + d] = fa[d] / 4.0;
    out[7 + 2 * d] = fa[d] > 0 ? 0.5 * f1[d] / fa[d] : 0.0;
    out[8 + 2 * d] = fa[d] > 0 ? 0.5 * f2[d] / fa[d] : 0.0;
    out[17 + d] = eba > 0 ? 0.5 * eb[d] / eba : 0.0;
    nv[d] = (fh[d] - fa[d]) * Af[d];
    nn += nv[d] * nv[d];
  }
  nn = sqrt(nn);
  for (int d = 0; d < 3; ++d) out[13 + d] = (eba > 0 && nn > 0) ? nv[d] / nn : 0.0;
  out[16] = eba / 4.0;
}

__global__ void k_coarse_geometry(FineC F, Dims Dc, int g, GridDev G) {
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= Dc.nx * Dc.ny) return;
  const int I = col % Dc.nx, J = col / Dc.nx;
  const long long n = G.nrec;
  for (int k = G.kcov[col]; k < G.kxt[col]; ++k) {
    const long long r = G.roff[col] + (k - G.kcov[col]);
    double v[20];
    merge_cv(F, Dc, g, I, J, k, v);
    G.flag[r] = (uint8_t)coarse_class(F, g, I, J, k);
    G.alpha[r] = v[0];
    for (int d = 0; d < 3; ++d) {
      G.cent[d * n + r] = v[1 + d];
      G.beta[d * n + r] = v[4 + d];
      G.nrm[d * n + r] = v[13 + d];
      G.ebc[d * n + r] = v[17 + d];
    }
    for (int q = 0; q < 6; ++q) G.fcent[q * n + r] = v[7 + q];
    G.aeb[r] = v[16];
    G.alpha_f[r] = (float)v[0];
    for (int d = 0; d < 3; ++d) G.beta_f[d * n + r] = (float)v[4 + d];
    for (int q = 0; q < 6; ++q) G.fcent_f[q * n + r] = (float)v[7 + q];
  }
}

__global__ void k_subsample_heights(const double *hf, Dims Df, double *hc, Dims Dc) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long n = (long long)(Dc.nx + 1) * (Dc.ny + 1);
  if (t >= n) return;
  const int I = (int)(t % (Dc.nx + 1)), J = (int)(t / (Dc.nx + 1));
  hc[t] = hf[(long long)(2 * J) * (Df.nx + 1) + 2 * I];
}

// Restriction: coarse value = (sum of w times fine value) / (sum of w), with
// w the fine volume fractions (c grid) or the fine low-face fractions of the
// 4 fine faces on the coarse face (face grids), in double; the states hold
// perturbations about per-level profiles of their own level (pf fine, pc
// coarse; zeros where none), so the profiles' weighted mean minus the coarse
// profile is added.  The fine handle may be an x-window of the fine level:
// its local column q is global fine column fx0 + q (mod nxg); coarse columns
// I0 .. I0 + ncols - 1 (mod the coarse nx) are restricted.  CVs without fine
// fluid or open area keep their value.
template <typename T>
struct RestrictArgs {
  FineC F;
  Dims Dc;
  const T *uf[5];
  T *uc[5];
  const double *pf[5], *pc[5];   // per-level profiles (nullptr: none)
  int fx0, nxg, I0, ncols;
};

// s + e = a + b exactly (float; Knuth's branch-free two-sum)
__device__ inline void two_sum(float a, float b, float &s, float &e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// A constant of a level: in double and, for the float path, as the nearest
// float and the rest.
struct LevelConst {
  double d;
  float hi, lo;
};
template <typename T>
__device__ inline void level_const(double d, LevelConst &c) {
  c.d = d;
  if constexpr (sizeof(T) == sizeof(float)) {
    c.hi = (float)d;
    c.lo = (float)(d - (double)c.hi);
  }
}

// the mean of N values (a power of two) plus a level constant, in double
template <int N, typename T>
__device__ inline double mean_double(const T (&v)[N], const LevelConst &c) {
  double s = (double)v[0];
#pragma unroll
  for (int q = 1; q < N; ++q) s += (double)v[q];
  return s * (1.0 / N) + c.d;
}
// The same rounded to the state's type.  FP64 instructions would bound both
// kernels on the float path, so there N times the value is first formed as t +
// rest, every addition's rounding error kept (the errors' own roundings, and
// what two floats leave of the constant, are added up as a bound); where both
// ends of rest +- bound round to the same float, that is the rounded value (the
// rounding test of Ziv, ACM Trans. Math. Softw. 17, 1991; plain means, whose
// bound is mostly zero, may then end on ties).  Otherwise, and where anything is
// infinite, NaN or overflows (every such comparison is false) or the scaled
// value could be subnormal, sure becomes false, and the caller forms its
// values by mean_double: all of a thread's after one test, so that their loads
// stay together.
// the sum of N floats as s + rest, up to bound; pairs first: a short chain
struct PairSum {
  float s, rest, bound;
};
template <int N>
__device__ inline PairSum pair_sum(const float *v) {
  if constexpr (N == 1) {
    return PairSum{v[0], 0.f, 0.f};
  } else {
    const PairSum a = pair_sum<N / 2>(v), b = pair_sum<N / 2>(v + N / 2);
    PairSum o{0.f, 0.f, 0.f};
    if constexpr (N == 2) {
      two_sum(a.s, b.s, o.s, o.rest);
    } else {
      float e, f, r1, r2;
      two_sum(a.s, b.s, o.s, e);
      two_sum(a.rest, b.rest, f, r1);
      two_sum(f, e, o.rest, r2);
      o.bound = __fadd_ru(__fadd_ru(a.bound, b.bound), __fadd_ru(fabsf(r1), fabsf(r2)));
    }
    return o;
  }
}
template <bool CONST, int N>
__device__ inline double mean_plus(const double (&v)[N], const LevelConst &c, bool &) {
  return mean_double(v, c);
}
template <bool CONST, int N>   // CONST false: c is zero
__device__ inline float mean_plus(const float (&v)[N], const LevelConst &c, bool &sure) {
  if (!CONST && N == 1) return v[0];
  const PairSum p = pair_sum<N>(v);
  float t = p.s, rest = p.rest, bound = p.bound;
  if constexpr (CONST) {   // (products with N are exact)
    float e, r;
    two_sum(t, N * c.hi, t, e);
    if constexpr (N > 1) {
      two_sum(rest, e, rest, r);
      bound = __fadd_ru(bound, fabsf(r));
    } else {
      rest = e;
    }
    two_sum(rest, N * c.lo, rest, r);
    bound = __fadd_ru(bound, fabsf(r));
    bound = __fmaf_ru(fabsf(N * c.hi), 0x1p-47f, bound);
  }
  const float a = __fadd_rn(t, __fsub_rd(rest, bound)), b = __fadd_rn(t, __fadd_ru(rest, bound));
  sure = sure && a == b && (fabsf(a) >= 0x1p-100f || a == 0.f);
  return a * (1.f / N);
}

// The coarse CVs at (I, J, K) of all five fields where fine cells are cut or
// covered: the eight fine cells' fractions are looked up once (one chain of
// column, offset and record loads), then weight every field in double.
template <typename T>
__device__ inline void restrict_cut(const RestrictArgs<T> &R, const int cols[4], long long b0, int K, long long tc) {
  const FineC &F = R.F;
  const Dims &Df = F.D;
  const int *kv = F.G.kcov;
  if (min(min(kv[cols[0]], kv[cols[1]]), min(kv[cols[2]], kv[cols[3]])) > 2 * K + 1) return;   // all covered
  double w[4][8];   // volume fraction, low x, y, z face fractions of fine cell a + 2 b + 4 c
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int col = cols[q], kc = F.G.kcov[col], kx = F.G.kxt[col];
    const long long ro = F.G.roff[col];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int k = 2 * K + c, e = q + 4 * c;
      const bool rec = k >= kc && k < kx;
      const long long r = ro + (k - kc);
#pragma unroll
      for (int m = 0; m < 4; ++m)
        w[m][e] = rec ? (m ? F.G.beta[(m - 1) * F.G.nrec + r] : F.G.alpha[r]) : (k < kc ? 0.0 : 1.0);
    }
  }
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    const int m = f <= 1 ? 0 : f - 1;
    double ws = 0.0, s = 0.0, sp = 0.0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (m && ((e >> (m - 1)) & 1)) continue;   // a face field: the four cells on the coarse low face
      const double we = w[m][e];
      ws += we;
      s += we * (double)R.uf[f][b0 + cols[e & 3] + (e >> 2) * Df.nxy];
      if (R.pf[f]) sp += we * R.pf[f][2 * K + (e >> 2)];
    }
    if (ws > 0.0) {
      double val = s / ws;
      if (R.pf[f]) val += sp / ws;
      if (R.pc[f]) val -= R.pc[f][K];
      R.uc[f][tc] = (T)val;
    }
  }
}

// All five fields of one coarse level per blockIdx.y (the lid face above the
// top level keeps its value).  Where the four fine columns are regular, every
// value is a plain mean of 8 (4) fine ones plus a constant of the level, formed
// almost without FP64 on the float path.  Latency and the FP64 sums over the cut
// cells bound it: 64 x 256 x 128 fine cells onto 32 x 128 x 64 take 36 us, their
// 47 MB would take 7 (130 us for one launch per field with double sums over
// looked-up fractions).
template <typename T>
__global__ void __launch_bounds__(256) k_restrict(const __grid_constant__ RestrictArgs<T> R) {
  const Dims &Dc = R.Dc, &Df = R.F.D;
  __shared__ LevelConst lc[4];   // per field: mean fine profile minus the coarse one
  const LevelConst none{0.0, 0.f, 0.f};
  const unsigned n = (unsigned)R.ncols * (unsigned)Dc.ny;
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = (int)(t / (unsigned)R.ncols), It = (int)(t - (unsigned)J * (unsigned)R.ncols);
  const int I = wrapi(R.I0 + It, Dc.nx);
  for (int K = blockIdx.y; K < Dc.nz; K += gridDim.y) {
    __syncthreads();
    if (threadIdx.x < 4) {
      const int f = threadIdx.x;
      double d = 0.0;
      if (R.pf[f]) d += 0.5 * (R.pf[f][2 * K] + R.pf[f][2 * K + 1]);
      if (R.pc[f]) d -= R.pc[f][K];
      level_const<T>(d, lc[f]);
    }
    __syncthreads();
    if (t >= n) continue;
    const long long tc = I + (long long)Dc.nx * J + Dc.nxy * K;
    const int x0 = wrapi(2 * I - R.fx0, R.nxg), x1 = wrapi(2 * I + 1 - R.fx0, R.nxg);
    const int c00 = x0 + Df.nx * (2 * J), c10 = x1 + Df.nx * (2 * J), c01 = c00 + Df.nx, c11 = c10 + Df.nx;
    const int *kx = R.F.G.kxt;
    if (max(max(kx[c00], kx[c10]), max(kx[c01], kx[c11])) > 2 * K) {
      const int cols[4] = {c00, c10, c01, c11};
      restrict_cut(R, cols, Df.nxy * (2LL * K), K, tc);
      continue;
    }
    const long long b0 = Df.nxy * (2LL * K), b1 = b0 + Df.nxy;
    const T *r = R.uf[0], *h = R.uf[1], *u = R.uf[2], *v = R.uf[3], *w = R.uf[4];
    const T vr[8] = {r[b0 + c00], r[b0 + c10], r[b0 + c01], r[b0 + c11],
                     r[b1 + c00], r[b1 + c10], r[b1 + c01], r[b1 + c11]};
    const T vh[8] = {h[b0 + c00], h[b0 + c10], h[b0 + c01], h[b0 + c11],
                     h[b1 + c00], h[b1 + c10], h[b1 + c01], h[b1 + c11]};
    const T vu[4] = {u[b0 + c00], u[b0 + c01], u[b1 + c00], u[b1 + c01]};
    const T vv[4] = {v[b0 + c00], v[b0 + c10], v[b1 + c00], v[b1 + c10]};
    const T vw[4] = {w[b0 + c00], w[b0 + c10], w[b0 + c01], w[b0 + c11]};
    bool sure = true;
    T o[5] = {mean_plus<true>(vr, lc[0], sure), mean_plus<true>(vh, lc[1], sure), mean_plus<true>(vu, lc[2], sure),
              mean_plus<true>(vv, lc[3], sure), mean_plus<false>(vw, none, sure)};
    if (!sure) {
      o[0] = (T)mean_double(vr, lc[0]);
      o[1] = (T)mean_double(vh, lc[1]);
      o[2] = (T)mean_double(vu, lc[2]);
      o[3] = (T)mean_double(vv, lc[3]);
      o[4] = (T)mean_double(vw, none);
    }
#pragma unroll
    for (int f = 0; f < 5; ++f) R.uc[f][tc] = o[f];
  }
}

// Prolongation onto the fine handle's columns outside [lo, hi) (local
// indices): every fine CV takes the value of the coarse CV it lies in; a fine
// face of a face grid on a coarse face takes that face's value, one halfway
// between two coarse faces (odd fine index along the face's axis) their mean;
// full values (state plus profile) are interpolated, with one rounding of the
// double value.
template <typename T>
struct ProlongArgs {
  Dims Df, Dc;
  const T *uc[5];
  T *uf[5];
  const double *pf[5], *pc[5];
  int fx0, nxg, lo, hi;
};

// One fine level per blockIdx.y, all five fields of the columns outside [lo,
// hi) (the level above the top holds rho*w only).  A value costs one addition
// of the level's profile difference (as on the restriction's float path, almost
// without FP64).  24 of 88 columns x 256 x 128: 17 us, latency (127 us for one
// launch per field over all columns); a whole level of 256 x 256 x 128: 101 us for
// 189 MB, instructions.
template <typename T>
__global__ void __launch_bounds__(256) k_prolong(const __grid_constant__ ProlongArgs<T> P) {
  const Dims &Df = P.Df, &Dc = P.Dc;
  __shared__ LevelConst lc[4];   // per field: coarse profile minus the fine one
  const LevelConst none{0.0, 0.f, 0.f};
  const unsigned cols = (unsigned)(Df.nx - (P.hi - P.lo));
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = (int)(t / cols);
  int i = (int)(t - (unsigned)j * cols);
  if (i >= P.lo) i += P.hi - P.lo;   // the owned columns are left out
  const int gi = wrapi(P.fx0 + i, P.nxg);
  const int I = gi / 2, J = j / 2;
  for (int k = blockIdx.y; k <= Df.nz; k += gridDim.y) {
    const int K = k / 2;
    __syncthreads();
    if (threadIdx.x < 4 && k < Df.nz) {
      const int f = threadIdx.x;
      double d = 0.0;
      if (P.pc[f]) d += P.pc[f][K];
      if (P.pf[f]) d -= P.pf[f][k];
      level_const<T>(d, lc[f]);
    }
    __syncthreads();
    if (t >= cols * (unsigned)Df.ny) continue;
    const long long c = I + (long long)Dc.nx * J + Dc.nxy * K;
    const long long q = i + (long long)Df.nx * j + Df.nxy * k;
    // one coarse value, or the two coarse faces around an odd fine face (else twice the same)
    const bool cell = k < Df.nz, oddu = gi & 1, oddv = j & 1, oddw = k & 1;
    T vr[1] = {T(0)}, vh[1] = {T(0)}, vu[2] = {T(0), T(0)}, vv[2] = {T(0), T(0)}, vw[2];
    if (cell) {
      vr[0] = P.uc[0][c];
      vh[0] = P.uc[1][c];
      vu[0] = vu[1] = P.uc[2][c];
      vv[0] = vv[1] = P.uc[3][c];
      if (oddu) vu[1] = P.uc[2][c - I + wrapi(I + 1, Dc.nx)];
      if (oddv) vv[1] = P.uc[3][c + (long long)Dc.nx * (wrapi(J + 1, Dc.ny) - J)];
    }
    vw[0] = vw[1] = P.uc[4][c];
    if (oddw) vw[1] = P.uc[4][c + Dc.nxy];
    T o[5];
    bool sure = sizeof(T) == sizeof(float);
    if (sure) {
      o[0] = mean_plus<true>(vr, lc[0], sure);
      o[1] = mean_plus<true>(vh, lc[1], sure);
      o[2] = mean_plus<true>(vu, lc[2], sure);
      o[3] = mean_plus<true>(vv, lc[3], sure);
      o[4] = mean_plus<false>(vw, none, sure);
    }
    if (!sure) {
      auto one = [](const T (&v)[2], bool odd, const LevelConst &k) -> T {   // (twice a large value may overflow)
        return (T)(odd ? mean_double(v, k) : (double)v[0] + k.d);
      };
      o[0] = (T)mean_double(vr, lc[0]);
      o[1] = (T)mean_double(vh, lc[1]);
      o[2] = one(vu, oddu, lc[2]);
      o[3] = one(vv, oddv, lc[3]);
      o[4] = one(vw, oddw, none);
    }
    if (k < Df.nz) {
#pragma unroll
      for (int f = 0; f < 4; ++f) P.uf[f][q] = o[f];
    }
    P.uf[4][q] = o[4];
  }
}

}  // namespace

void launch_coarse_bounds(const Dims &Df, const GridDev &Gf, const Dims &Dc, int g, int *kcov, int *kreg,
                          cudaStream_t s) {
  FineC F{Df, Gf};
  k_coarse_bounds<<<(unsigned)((Dc.nxy + 127) / 128), 128, 0, s>>>(F, Dc, g, kcov, kreg);
}

void launch_coarse_geometry(const Dims &Df, const GridDev &Gf, const Dims &Dc, int g, const GridDev &Gc,
                            cudaStream_t s) {
  FineC F{Df, Gf};
  k_coarse_geometry<<<(unsigned)((Dc.nxy + 63) / 64), 64, 0, s>>>(F, Dc, g, Gc);
}

void launch_subsample_heights(const double *hf, const Dims &Df, double *hc, const Dims &Dc, cudaStream_t s) {
  const long long n = (long long)(Dc.nx + 1) * (Dc.ny + 1);
  k_subsample_heights<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(hf, Df, hc, Dc);
}

template <typename T>
static void restrict_t(eb_geom fine, eb_geom coarse, const eb_state *Uf, eb_state *Uc, int fx0, int lo, int hi,
                       cudaStream_t s) {
  RestrictArgs<T> R;
  R.F = FineC{fine->D, fine->G[0]};
  R.Dc = coarse->D;
  R.nxg = 2 * coarse->D.nx;
  R.fx0 = wrapi(fx0, R.nxg);
  R.I0 = wrapi(R.fx0 + lo, R.nxg) / 2;
  R.ncols = (hi - lo) / 2;
  void **uf = state_ptrs(Uf), **uc = state_ptrs(Uc);
  for (int f = 0; f < 5; ++f) {
    R.uf[f] = (const T *)uf[f];
    R.uc[f] = (T *)uc[f];
    R.pf[f] = f <= 3 ? fine->ref_d[f] : nullptr;
    R.pc[f] = f <= 3 ? coarse->ref_d[f] : nullptr;
  }
  const long long n = (long long)R.ncols * coarse->D.ny;
  const unsigned gy = (unsigned)std::min(coarse->D.nz, 65535);
  if (n > 0) k_restrict<T><<<dim3((unsigned)((n + 255) / 256), gy, 1), 256, 0, s>>>(R);
}

template <typename T>
static void prolong_t(eb_geom coarse, const eb_state *Uc, eb_geom fine, eb_state *Uf, int fx0, int lo, int hi,
                      cudaStream_t s) {
  ProlongArgs<T> P;
  P.Df = fine->D;
  P.Dc = coarse->D;
  P.nxg = 2 * coarse->D.nx;
  P.fx0 = wrapi(fx0, P.nxg);
  P.lo = lo;
  P.hi = hi;
  void **uf = state_ptrs(Uf), **uc = state_ptrs(Uc);
  for (int f = 0; f < 5; ++f) {
    P.uc[f] = (const T *)uc[f];
    P.uf[f] = (T *)uf[f];
    P.pf[f] = f <= 3 ? fine->ref_d[f] : nullptr;
    P.pc[f] = f <= 3 ? coarse->ref_d[f] : nullptr;
  }
  const long long n = (long long)(fine->D.nx - (hi - lo)) * fine->D.ny;
  const unsigned gy = (unsigned)std::min(fine->D.nz + 1, 65535);
  if (n > 0) k_prolong<T><<<dim3((unsigned)((n + 255) / 256), gy, 1), 256, 0, s>>>(P);
}

// the fine handle is the coarse level's fine level over fine columns fx0 ..
// fx0 + nx - 1 (mod 2 nx_c), full y and z
static eb_status check_levels(eb_geom fine, eb_geom coarse, const eb_state *Uf, const eb_state *Uc, int lo, int hi) {
  if (!fine || !coarse) return fail(EB_ERR_INVALID_ARG, "NULL handle");
  if (fine->D.ny != 2 * coarse->D.ny || fine->D.nz != 2 * coarse->D.nz || fine->D.nx > 2 * coarse->D.nx)
    return fail(EB_ERR_INVALID_ARG, "the fine handle must be an x-window of the coarse handle's fine level");
  if (fabs(2.0 * fine->D.dx - coarse->D.dx) > 1e-12 * coarse->D.dx ||
      fabs(2.0 * fine->D.dy - coarse->D.dy) > 1e-12 * coarse->D.dy ||
      fabs(2.0 * fine->D.dz - coarse->D.dz) > 1e-12 * coarse->D.dz)
    return fail(EB_ERR_INVALID_ARG, "the fine cells must be half the coarse ones");
  if (fine->prec != coarse->prec) return fail(EB_ERR_INVALID_ARG, "the handles differ in precision");
  if (lo < 0 || hi > fine->D.nx || lo > hi) return fail(EB_ERR_INVALID_ARG, "column range outside the fine handle");
  const size_t es = fine->prec == EB_F64 ? 8 : 4;
  if (!state_ok(Uf, es) || !state_ok(Uc, es)) return fail(EB_ERR_INVALID_ARG, "state pointer NULL or misaligned");
  return EB_OK;
}

eb_status eb_restrict(eb_geom fine, eb_geom coarse, const eb_state *Uf, eb_state *Uc, int fine_x0, int lo, int hi,
                      void *stream) {
  eb_status st = check_levels(fine, coarse, Uf, Uc, lo, hi);
  if (st != EB_OK) return st;
  if ((lo % 2) || (hi % 2) || ((fine_x0 % 2 + 2) % 2))
    return fail(EB_ERR_INVALID_ARG, "restriction columns must start on even fine columns");
  cudaStream_t s = as_stream(stream);
  if (fine->prec == EB_F64) restrict_t<double>(fine, coarse, Uf, Uc, fine_x0, lo, hi, s);
  else restrict_t<float>(fine, coarse, Uf, Uc, fine_x0, lo, hi, s);
  CUDA_TRY(cudaGetLastError(), "restriction");
  return EB_OK;
}

eb_status eb_prolong(eb_geom coarse, const eb_state *Uc, eb_geom fine, eb_state *Uf, int fine_x0, int lo, int hi,
                     void *stream) {
  eb_status st = check_levels(fine, coarse, Uf, Uc, lo, hi);
  if (st != EB_OK) return st;
  cudaStream_t s = as_stream(stream);
  if (fine->prec == EB_F64) prolong_t<double>(coarse, Uc, fine, Uf, fine_x0, lo, hi, s);
  else prolong_t<float>(coarse, Uc, fine, Uf, fine_x0, lo, hi, s);
  CUDA_TRY(cudaGetLastError(), "prolongation");
  return EB_OK;
}
