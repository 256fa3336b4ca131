// eb_project.cu -- the anelastic projection (Sec. 2.2, Algorithm 2 step 5)
// and the anelastic step.
//
// The constraint div(rho0 u) = 0 is imposed on the face momenta with the
// cut-cell divergence of the flux update,
//   D(m)_c = sum_d (beta_d,hi m_d,hi - beta_d,lo m_d,lo) / delta_d,
// beta the open fractions of the c-cell's faces (walls closed).  With the
// face gradient G(phi) = (phi_R - phi_L) / delta_d, the correction
// m <- m* - dt G(phi) removes the divergence when L phi = D(G(phi)) = D(m*)/dt.
// L is the beta-weighted 7-point operator: symmetric, negative semi-definite,
// null space the constants (the fluid above a height-function terrain is
// connected), so the mean of the right-hand side (rounding only) is removed
// and -L phi = -rhs is solved by Jacobi-preconditioned conjugate gradients
// in FP64 to a relative residual.
//
// Every kernel runs on a fixed grid of nb blocks with grid-stride loops and
// writes one partial sum per block; a consumer block adds the nb partials in
// a fixed order, so the solve is deterministic.  Convergence is detected on
// the device (the kernels of later iterations return at once) and read by
// the host every 32 iterations (every 4 with the multigrid preconditioner).
#include "eb_handle.cuh"

#include <math.h>

#include <algorithm>

using namespace ebh;

namespace {

constexpr int PB = 256;   // threads per block of every projection kernel

enum { S_SUM = 0, S_BB = 1, S_PQ = 2, S_RR = 3, S_RZ0 = 4, S_RZ1 = 5, S_CNT = 6, S_TMP = 7 };

__device__ inline double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the block (PB threads in any shape); one thread writes it to part[blockIdx.x].
__device__ inline void block_partial(double v, double *part) {
  __shared__ double s[PB / 32];
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  v = warp_sum(v);
  if ((tid & 31) == 0) s[tid >> 5] = v;
  __syncthreads();
  if (tid < 32) {
    double a = tid < PB / 32 ? s[tid] : 0.0;
    a = warp_sum(a);
    if (tid == 0) part[blockIdx.x] = a;
  }
}

// Total of nb partial sums, the same bits in every block.
__device__ inline double total(const double *part, int nb) {
  __shared__ double t;
  __syncthreads();
  if (threadIdx.x < 32) {
    double a = 0.0;
    for (int q = threadIdx.x; q < nb; q += 32) a += part[q];
    a = warp_sum(a);
    if (threadIdx.x == 0) t = a;
  }
  __syncthreads();
  return t;
}

struct Nbr {
  long long xm, xp, ym, yp;
  int k;
};

__device__ inline Nbr neighbours(const Dims &D, long long c) {
  int i, j, k;
  split_index(D, (unsigned)c, i, j, k);
  Nbr n;
  n.xm = i == 0 ? c + D.nx - 1 : c - 1;
  n.xp = i == D.nx - 1 ? c - (D.nx - 1) : c + 1;
  n.ym = j == 0 ? c + (long long)D.nx * (D.ny - 1) : c - D.nx;
  n.yp = j == D.ny - 1 ? c - (long long)D.nx * (D.ny - 1) : c + D.nx;
  n.k = k;
  return n;
}

struct Op {
  Dims D;
  const double *bx, *by, *bz, *d, *id;
  const double *ax, *ay, *az;   // open fractions times 1 / delta^2 (set-up)
  double ix2, iy2, iz2;   // 1 / delta^2
  // (-L p)_c for an active cell: one product and six fused multiply-adds
  // (FP64 arithmetic, not HBM, bounds this on the GPU)
  __device__ inline double apply(const double *p, long long c, const Nbr &n) const {
    const double azl = az[c];
    const double azh = n.k + 1 < D.nz ? az[c + D.nxy] : 0.0;
    double v = d[c] * p[c];
    v = fma(-ax[c], p[n.xm], v);
    v = fma(-ax[n.xp], p[n.xp], v);
    v = fma(-ay[c], p[n.ym], v);
    v = fma(-ay[n.yp], p[n.yp], v);
    if (azl > 0.0) v = fma(-azl, p[c - D.nxy], v);
    if (azh > 0.0) v = fma(-azh, p[c + D.nxy], v);
    return v;
  }
};

__global__ void k_recip(long long N, const double *d, double *id) {
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB)
    id[c] = d[c] > 0.0 ? 1.0 / d[c] : 0.0;
}

__global__ void k_scale(long long N, const double *b, double s, double *a) {
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) a[c] = b[c] * s;
}

__global__ void k_wall(Dims D, double *bz) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c < D.nxy) bz[c] = 0.0;   // z = 0 carries no flux
}

__global__ void k_diag(Op O, double *d, double *part) {
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  double cnt = 0.0;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    const Nbr n = neighbours(D, c);
    const double bzh = n.k + 1 < D.nz ? O.bz[c + D.nxy] : 0.0;
    const double v = (O.bx[c] + O.bx[n.xp]) * O.ix2 + (O.by[c] + O.by[n.yp]) * O.iy2 + (O.bz[c] + bzh) * O.iz2;
    d[c] = v;
    cnt += v > 0.0 ? 1.0 : 0.0;
  }
  block_partial(cnt, part);
}

// rhs = D(m) / dt on the active cells
template <typename T>
__global__ void k_rhs(Op O, const T *mu, const T *mv, const T *mw, double idt, double *rhs, double *part) {
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  double sum = 0.0;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    double v = 0.0;
    if (O.d[c] > 0.0) {
      const Nbr n = neighbours(D, c);
      const double bzh = n.k + 1 < D.nz ? O.bz[c + D.nxy] : 0.0;
      const double dx = O.bx[n.xp] * (double)mu[n.xp] - O.bx[c] * (double)mu[c];
      const double dy = O.by[n.yp] * (double)mv[n.yp] - O.by[c] * (double)mv[c];
      const double dz = bzh * (double)mw[c + D.nxy] - O.bz[c] * (double)mw[c];
      v = (dx * D.idx + dy * D.idy + dz * D.idz) * idt;
    }
    rhs[c] = v;
    sum += v;
  }
  block_partial(sum, part);
}

// remove the mean of the right-hand side over the active cells
__global__ void k_center(Op O, double *rhs, const double *psum, const double *pcnt, int nb, double *pbb) {
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  const double mean = total(psum, nb) / fmax(1.0, total(pcnt, nb));
  double bb = 0.0;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    if (O.d[c] > 0.0) {
      const double v = rhs[c] - mean;
      rhs[c] = v;
      bb += v * v;
    }
  }
  block_partial(bb, pbb);
}

// r = -rhs - A x, z = r / d, p = z
__global__ void k_init(Op O, const double *x, const double *rhs, double *r, float *rf, double *z, double *p,
                       double *prz, double *prr) {
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  double rz = 0.0, rr = 0.0;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    double rv = 0.0, zv = 0.0;
    if (O.d[c] > 0.0) {
      rv = -rhs[c] - O.apply(x, c, neighbours(D, c));
      zv = rv * O.id[c];
    }
    r[c] = rv;
    if (rf) rf[c] = (float)rv;   // the V-cycle's right-hand side
    z[c] = zv;
    p[c] = zv;
    rz += rv * zv;
    rr += rv * rv;
  }
  block_partial(rz, prz);
  __syncthreads();
  block_partial(rr, prr);
}

// q = A p
__global__ void k_apply(Op O, const double *p, double *q, double *ppq, const int *conv) {
  if (*conv) return;
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  double pq = 0.0;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    double v = 0.0;
    if (O.d[c] > 0.0) v = O.apply(p, c, neighbours(D, c));
    q[c] = v;
    pq += p[c] * v;
  }
  block_partial(pq, ppq);
}

// alpha = rz / pq; x += alpha p; r -= alpha q; z = r / d (Jacobi; the
// multigrid preconditioner forms z and r.z afterwards)
template <bool JAC>
__global__ void k_update(Op O, double *x, const double *p, const double *q, double *r, float *rf, double *z,
                         const double *ppq, const double *prz, int nrz, double *prz_next, double *prr, int nb,
                         const int *conv) {
  if (*conv) return;
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  const double alpha = total(prz, nrz) / total(ppq, nb);
  double rz = 0.0, rr = 0.0;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    if (O.d[c] > 0.0) {
      x[c] += alpha * p[c];
      const double rv = r[c] - alpha * q[c];
      r[c] = rv;
      if (!JAC) rf[c] = (float)rv;
      if (JAC) {
        const double zv = rv * O.id[c];
        z[c] = zv;
        rz += rv * zv;
      }
      rr += rv * rv;
    }
  }
  if (JAC) {
    block_partial(rz, prz_next);
    __syncthreads();
  }
  block_partial(rr, prr);
}

// convergence test; else p = z + (rz_next / rz) p
__global__ void k_direction(Op O, double *p, const double *z, const double *prz, const double *prz_next,
                            int nrz, const double *prr, int nb, double thr2, int it, int *conv) {
  if (*conv) return;
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  const double rr = total(prr, nb);
  if (rr <= thr2) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *conv = it + 1;
    return;
  }
  const double beta = total(prz_next, nrz) / total(prz, nrz);
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB)
    p[c] = z[c] + beta * p[c];
}

// m -= dt G(x) on the open faces
template <typename T>
__global__ void k_correct(Op O, const double *x, double dt, T *mu, T *mv, T *mw) {
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    const Nbr n = neighbours(D, c);
    if (O.bx[c] > 0.0) mu[c] = (T)((double)mu[c] - dt * (x[c] - x[n.xm]) * D.idx);
    if (O.by[c] > 0.0) mv[c] = (T)((double)mv[c] - dt * (x[c] - x[n.ym]) * D.idy);
    if (n.k >= 1 && O.bz[c] > 0.0) mw[c] = (T)((double)mw[c] - dt * (x[c] - x[c - D.nxy]) * D.idz);
  }
}

// ---------------------------------------------------------------------------
// Multigrid preconditioner (EB_PRECOND_MG): z = V(r), one V-cycle in FP32
// (FP64 arithmetic is scarce on this GPU; the outer conjugate gradients stay
// in FP64).  Damped Jacobi with the same weight and the same number of
// sweeps before and after the coarse correction (three on the finest grid,
// where they cut 18 iterations to 16 at rtol 1e-10 on the 192x192x96 random
// terrain for a shorter solve; two on the coarser grids), restriction = 1/8
// of the transpose of the injection
// prolongation, and a fixed number of Jacobi sweeps from zero on the
// coarsest grid: up to float rounding V is a fixed symmetric positive
// semi-definite operator, as conjugate gradients need.
// ---------------------------------------------------------------------------
// Jacobi weight: the rows of the operator have off-diagonal magnitudes
// summing to the diagonal, so the eigenvalues of D^-1 A lie in [0, 2] and any
// weight below 1 keeps the smoother convergent and the V-cycle definite; 0.9
// took the 192x192x96 random terrain's projection from 16 iterations (0.8) to
// 13 at rtol 1e-10, 0.95 back up to 17.
constexpr float MG_OMEGA = 0.9f;
// Jacobi sweeps from zero on the coarsest grid (even: the result ends in x).
// Any count gives a positive operator (the weight keeps 1 - w*lambda in
// (-1, 1]); on the 192x192x96 random terrain 8 to 64 sweeps all needed 13
// outer iterations, and fewer sweeps cost less (16: 7.6 ms, 64: 8.0 ms).
constexpr int MG_COARSE_SWEEPS = 16;

// The operator of one level.  From kreg[column] up, every face of the cells
// within two columns is fully open (the terrain lies below), so there, away
// from the floor and the lid, the kernels read no coefficient at all.
struct Op32 {
  Dims D;
  const float *bx, *by, *bz;   // low-face open fractions
  const float *wi;             // MG_OMEGA / diagonal (0 off the active cells)
  const int *kreg;
  float ix2, iy2, iz2;
  // off-diagonal sum and diagonal of cell c (grid-stride form; coarsest grids and set-up)
  __device__ inline void parts(const float *x, long long c, float &S, float &d) const {
    const Nbr n = neighbours(D, c);
    const float axl = bx[c] * ix2, axh = bx[n.xp] * ix2, ayl = by[c] * iy2, ayh = by[n.yp] * iy2;
    const float azl = bz[c] * iz2, azh = n.k + 1 < D.nz ? bz[c + D.nxy] * iz2 : 0.f;
    d = axl + axh + ayl + ayh + azl + azh;
    S = axl * x[n.xm] + axh * x[n.xp] + ayl * x[n.ym] + ayh * x[n.yp];
    if (azl > 0.f) S += azl * x[c - D.nxy];
    if (azh > 0.f) S += azh * x[c + D.nxy];
  }
  __device__ inline float diag(long long c) const {
    const Nbr n = neighbours(D, c);
    const float azh = n.k + 1 < D.nz ? bz[c + D.nxy] * iz2 : 0.f;
    return (bx[c] + bx[n.xp]) * ix2 + (by[c] + by[n.yp]) * iy2 + bz[c] * iz2 + azh;
  }
};

__global__ void k_mg_winv(Op32 L, float *wi) {
  const long long N = L.D.nxy * L.D.nz;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    const float d = L.diag(c);
    wi[c] = d > 0.f ? MG_OMEGA / d : 0.f;
  }
}

// top[col]: the level from which every low face of the column's cells is
// fully open (the floor's z face apart)
template <typename F>
__global__ void k_open_top(Dims D, const F *bx, const F *by, const F *bz, int *top) {
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= D.nxy) return;
  int k = D.nz;
  while (k > 0) {
    const long long c = col + D.nxy * (long long)(k - 1);
    if (bx[c] != F(1) || by[c] != F(1) || (k > 1 && bz[c] != F(1))) break;
    --k;
  }
  top[col] = k;
}
__global__ void k_open_box(Dims D, const int *top, int *kreg) {
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= D.nxy) return;
  const int i = col % D.nx, j = col / D.nx;
  int k = 0;
  for (int dj = -2; dj <= 2; ++dj)
    for (int di = -2; di <= 2; ++di) k = max(k, top[wrapmod(i + di, D.nx) + D.nx * wrapmod(j + dj, D.ny)]);
  kreg[col] = k;
}

// level 0: float copies of the open fractions
__global__ void k_mg_copy(long long N, const double *bx, const double *by, const double *bz, float *fx, float *fy,
                          float *fz) {
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    fx[c] = (float)bx[c];
    fy[c] = (float)by[c];
    fz[c] = (float)bz[c];
  }
}

// coarse open fractions: the mean over the four fine faces a coarse face covers
__global__ void k_mg_coarsen(Op32 F, Dims C, float *bx, float *by, float *bz) {
  const long long N = C.nxy * C.nz;
  const long long sy = F.D.nx, sz = F.D.nxy;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    int I, J, K;
    split_index(C, (unsigned)c, I, J, K);
    const long long f = 2LL * I + sy * 2LL * J + sz * 2LL * K;
    bx[c] = 0.25f * (F.bx[f] + F.bx[f + sy] + F.bx[f + sz] + F.bx[f + sy + sz]);
    by[c] = 0.25f * (F.by[f] + F.by[f + 1] + F.by[f + sz] + F.by[f + 1 + sz]);
    bz[c] = 0.25f * (F.bz[f] + F.bz[f + 1] + F.bz[f + sy] + F.bz[f + 1 + sy]);
  }
}

// V adjacent values of a row
template <int V>
struct Vec {
  float v[V];
};
template <int V>
__device__ inline Vec<V> ldv(const float *p) {
  Vec<V> o;
  if constexpr (V == 4) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    o.v[0] = t.x, o.v[1] = t.y, o.v[2] = t.z, o.v[3] = t.w;
  } else if constexpr (V == 2) {
    const float2 t = *reinterpret_cast<const float2 *>(p);
    o.v[0] = t.x, o.v[1] = t.y;
  } else {
    o.v[0] = p[0];
  }
  return o;
}
template <int V>
__device__ inline void stv(float *p, const Vec<V> &a) {
  if constexpr (V == 4) *reinterpret_cast<float4 *>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
  else if constexpr (V == 2) *reinterpret_cast<float2 *>(p) = make_float2(a.v[0], a.v[1]);
  else p[0] = a.v[0];
}

// Work split of the marching kernels: a thread owns V adjacent columns of one
// row and walks a slab of levels; a block is MBX x MBY threads.
constexpr int MBX = 16, MBY = 16;
static_assert(MBX * MBY == PB, "block sums take PB threads");
struct Slabs {
  int nbx, nby, nz;   // blocks along x and y, slabs
  int blocks() const { return nbx * nby * nz; }
};
// enough slabs for about 1536 threads per SM, down to one level each on the
// small grids, where latency is all that counts
inline Slabs slabs_of(const Dims &D, int V, int sms) {
  Slabs S;
  S.nbx = (D.nx / V + MBX - 1) / MBX;
  S.nby = (D.ny + MBY - 1) / MBY;
  const int plane = S.nbx * S.nby;
  S.nz = std::max(1, std::min(D.nz, (6 * sms + plane - 1) / plane));
  return S;
}
// a thread's columns: offsets within a plane of its own row, the rows beside
// it and the cells left and right of its V
struct Cols {
  int i, j, c, ym, yp, xl, xr, k0, k1;
  bool in;
};
template <int V>
__device__ inline Cols cols_of(const Dims &D, const Slabs &S) {
  Cols q;
  const int sl = blockIdx.x / (S.nbx * S.nby), b = blockIdx.x - sl * S.nbx * S.nby;
  const int by = b / S.nbx, bx = b - by * S.nbx;
  q.i = V * (bx * MBX + (int)threadIdx.x);
  q.j = by * MBY + (int)threadIdx.y;
  q.in = q.i < D.nx && q.j < D.ny;
  if (!q.in) q.i = q.j = 0;
  const int row = D.nx * q.j;
  q.c = q.i + row;
  q.ym = q.i + (q.j == 0 ? D.nx * (D.ny - 1) : row - D.nx);
  q.yp = q.i + (q.j == D.ny - 1 ? 0 : row + D.nx);
  q.xl = row + (q.i == 0 ? D.nx - 1 : q.i - 1);
  q.xr = row + (q.i + V == D.nx ? 0 : q.i + V);
  q.k0 = (int)((long long)D.nz * sl / S.nz);
  q.k1 = (int)((long long)D.nz * (sl + 1) / S.nz);
  return q;
}

// One damped Jacobi sweep, xout = (1 - w) x + w (b + S(x)) / d, of
//   FIRST    x = w b / d, the sweep from zero (so two sweeps in one pass),
//   PLAIN    x = xin,
//   PROLONG  x = xin + the parent's coarse correction (injection; inactive
//            cells are never read with a nonzero coefficient).
// FINAL: the finest level's last sweep, which writes the FP64 z and the block
// partials of r.z.
// L2 bandwidth bounds it (16 bytes per cell; the level's arrays stay in the
// 129 MB L2): V = 4 columns per thread with 16-byte accesses, the z
// neighbours carried in registers, no coefficients above the terrain.
// 192x192x96: 11 us (PLAIN), 18 (FIRST, two sweeps), 16 (PROLONG); one cell
// per thread with index splits and six coefficient loads took 29 per sweep
// and 12 for the prolongation.
enum { FIRST = 0, PLAIN = 1, PROLONG = 2 };
template <int V, int MODE, bool FINAL>
__global__ void __launch_bounds__(MBX * MBY) k_mg_sweep(const __grid_constant__ Op32 L,
                                                        const __grid_constant__ Slabs SL,
                                                        const float *__restrict__ xin, const float *__restrict__ xc,
                                                        const __grid_constant__ Dims C, float *__restrict__ xout,
                                                        double *__restrict__ zout, const double *__restrict__ r,
                                                        const float *__restrict__ b, double *prz, const int *conv) {
  if (*conv) return;
  const Dims &D = L.D;
  const Cols q = cols_of<V>(D, SL);
  const float wreg = MG_OMEGA / (2.f * (L.ix2 + L.iy2 + L.iz2));
  int kr = 0;
#pragma unroll
  for (int e = 0; e < V; ++e) kr = max(kr, L.kreg[q.c + e]);
  // plane offset of the parent of plane offset o in row j (PROLONG)
  auto parent = [&](int i, int j) { return (i >> 1) + C.nx * (j >> 1); };
  const int pc = parent(q.i, q.j), pym = parent(q.i, q.j == 0 ? D.ny - 1 : q.j - 1),
            pyp = parent(q.i, q.j == D.ny - 1 ? 0 : q.j + 1), pxl = parent(q.i == 0 ? D.nx - 1 : q.i - 1, q.j),
            pxr = parent(q.i + V == D.nx ? 0 : q.i + V, q.j);
  // x of V cells at plane offset o (parents from po) / of one cell
  auto vec = [&](int k, int o, int po, bool reg) -> Vec<V> {
    const long long t = D.nxy * (long long)k + o;
    Vec<V> a;
    if constexpr (MODE == FIRST) {
      a = ldv<V>(b + t);
      if (reg) {
#pragma unroll
        for (int e = 0; e < V; ++e) a.v[e] *= wreg;
      } else {
        const Vec<V> w = ldv<V>(L.wi + t);
#pragma unroll
        for (int e = 0; e < V; ++e) a.v[e] *= w.v[e];
      }
    } else {
      a = ldv<V>(xin + t);
      if constexpr (MODE == PROLONG) {
        const float *p = xc + C.nxy * (long long)(k >> 1) + po;
#pragma unroll
        for (int e = 0; e < V; ++e) a.v[e] += p[e >> 1];
      }
    }
    return a;
  };
  auto one = [&](int k, int o, int po, bool reg) -> float {
    const long long t = D.nxy * (long long)k + o;
    if constexpr (MODE == FIRST) return b[t] * (reg ? wreg : L.wi[t]);
    else if constexpr (MODE == PROLONG) return xin[t] + xc[C.nxy * (long long)(k >> 1) + po];
    else return xin[t];
  };
  double rz = 0.0;
  if (q.in) {
    Vec<V> xm, x0, xp;
#pragma unroll
    for (int e = 0; e < V; ++e) xm.v[e] = xp.v[e] = 0.f;
    if (q.k0 > 0) xm = vec(q.k0 - 1, q.c, pc, false);
    x0 = vec(q.k0, q.c, pc, false);
#pragma unroll 2
    for (int k = q.k0; k < q.k1; ++k) {   // two levels' loads in flight
      const bool reg = k > kr && k < D.nz - 2;   // open faces in this cell and in its neighbours
      const long long t = D.nxy * (long long)k;
      if (k + 1 < D.nz) xp = vec(k + 1, q.c, pc, reg);
      const Vec<V> ym = vec(k, q.ym, pym, reg), yp = vec(k, q.yp, pyp, reg);
      const float xl = one(k, q.xl, pxl, reg), xr = one(k, q.xr, pxr, reg);
      const Vec<V> bv = ldv<V>(b + t + q.c);
      Vec<V> o;
      if (reg) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const float S = L.ix2 * ((e ? x0.v[e ? e - 1 : 0] : xl) + (e + 1 < V ? x0.v[e + 1 < V ? e + 1 : 0] : xr)) +
                          L.iy2 * (ym.v[e] + yp.v[e]) + L.iz2 * (xm.v[e] + xp.v[e]);
          o.v[e] = (1.f - MG_OMEGA) * x0.v[e] + wreg * (bv.v[e] + S);
        }
      } else {
        const Vec<V> bx = ldv<V>(L.bx + t + q.c), yl = ldv<V>(L.by + t + q.c), yh = ldv<V>(L.by + t + q.yp),
                     zl = ldv<V>(L.bz + t + q.c), wi = ldv<V>(L.wi + t + q.c);
        Vec<V> zh;
#pragma unroll
        for (int e = 0; e < V; ++e) zh.v[e] = 0.f;
        if (k + 1 < D.nz) zh = ldv<V>(L.bz + t + D.nxy + q.c);
        const float bxr = L.bx[t + q.xr];
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const float S = L.ix2 * (bx.v[e] * (e ? x0.v[e ? e - 1 : 0] : xl) +
                                   (e + 1 < V ? bx.v[e + 1 < V ? e + 1 : 0] * x0.v[e + 1 < V ? e + 1 : 0] : bxr * xr)) +
                          L.iy2 * (yl.v[e] * ym.v[e] + yh.v[e] * yp.v[e]) +
                          L.iz2 * (zl.v[e] * xm.v[e] + zh.v[e] * xp.v[e]);
          o.v[e] = wi.v[e] > 0.f ? (1.f - MG_OMEGA) * x0.v[e] + wi.v[e] * (bv.v[e] + S) : 0.f;
        }
      }
      if constexpr (FINAL) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const double z = (double)o.v[e];
          zout[t + q.c + e] = z;
          rz += r[t + q.c + e] * z;
        }
      } else {
        stv<V>(xout + t + q.c, o);
      }
      xm = x0;
      x0 = xp;
    }
  }
  if constexpr (FINAL) block_partial(rz, prz);
}

// Coarse right-hand side: the mean of the eight children's residuals b - A x.
// A thread forms V / 2 coarse cells per coarse level from V columns x 2 rows.
// 192x192x96: 11 us (one coarse cell per thread: 25).
template <int V>
__global__ void __launch_bounds__(MBX * MBY) k_mg_restrict(const __grid_constant__ Op32 F, const float *x,
                                                           const float *b, const __grid_constant__ Dims C,
                                                           float *bc, int kper, const int *conv) {
  if (*conv) return;
  const Dims &D = F.D;
  const int g = D.nx / V;   // groups of V columns per row
  const long long t = blockIdx.x * (long long)(MBX * MBY) + threadIdx.y * MBX + threadIdx.x;
  const long long plane = (long long)g * C.ny;
  const int sl = (int)(t / plane), u = (int)(t - sl * plane);
  const int J = u / g, i = V * (u - J * g);
  const float dreg = 2.f * (F.ix2 + F.iy2 + F.iz2);
  const int K0 = sl * kper, K1 = min(C.nz, K0 + kper);
  if (K0 >= C.nz) return;
  int kr = 0;
#pragma unroll
  for (int e = 0; e < V; ++e) kr = max(kr, max(F.kreg[i + e + D.nx * (2 * J)], F.kreg[i + e + D.nx * (2 * J + 1)]));
  for (int K = K0; K < K1; ++K) {
    float sum[V / 2];
#pragma unroll
    for (int e = 0; e < V / 2; ++e) sum[e] = 0.f;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int k = 2 * K + (h >> 1), j = 2 * J + (h & 1);
      const int row = D.nx * j, o = i + row;
      const int om = i + (j == 0 ? D.nx * (D.ny - 1) : row - D.nx), op = i + (j == D.ny - 1 ? 0 : row + D.nx);
      const int ol = row + (i == 0 ? D.nx - 1 : i - 1), orr = row + (i + V == D.nx ? 0 : i + V);
      const long long pl = D.nxy * (long long)k;
      const Vec<V> x0 = ldv<V>(x + pl + o), ym = ldv<V>(x + pl + om), yp = ldv<V>(x + pl + op), bv = ldv<V>(b + pl + o);
      Vec<V> xm, xp;
#pragma unroll
      for (int e = 0; e < V; ++e) xm.v[e] = xp.v[e] = 0.f;
      if (k > 0) xm = ldv<V>(x + pl - D.nxy + o);
      if (k + 1 < D.nz) xp = ldv<V>(x + pl + D.nxy + o);
      const float xl = x[pl + ol], xr = x[pl + orr];
      if (k >= kr && k > 0 && k < D.nz - 1) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const float S = F.ix2 * ((e ? x0.v[e ? e - 1 : 0] : xl) + (e + 1 < V ? x0.v[e + 1 < V ? e + 1 : 0] : xr)) +
                          F.iy2 * (ym.v[e] + yp.v[e]) + F.iz2 * (xm.v[e] + xp.v[e]);
          sum[e / 2] += bv.v[e] - dreg * x0.v[e] + S;
        }
      } else {
        const Vec<V> bx = ldv<V>(F.bx + pl + o), yl = ldv<V>(F.by + pl + o), yh = ldv<V>(F.by + pl + op),
                     zl = ldv<V>(F.bz + pl + o);
        Vec<V> zh;
#pragma unroll
        for (int e = 0; e < V; ++e) zh.v[e] = 0.f;
        if (k + 1 < D.nz) zh = ldv<V>(F.bz + pl + D.nxy + o);
        const float bxr = F.bx[pl + orr];
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const float axl = F.ix2 * bx.v[e], axh = F.ix2 * (e + 1 < V ? bx.v[e + 1 < V ? e + 1 : 0] : bxr);
          const float ayl = F.iy2 * yl.v[e], ayh = F.iy2 * yh.v[e], azl = F.iz2 * zl.v[e], azh = F.iz2 * zh.v[e];
          const float d = axl + axh + ayl + ayh + azl + azh;
          const float S = axl * (e ? x0.v[e ? e - 1 : 0] : xl) + axh * (e + 1 < V ? x0.v[e + 1 < V ? e + 1 : 0] : xr) +
                          ayl * ym.v[e] + ayh * yp.v[e] + azl * xm.v[e] + azh * xp.v[e];
          if (d > 0.f) sum[e / 2] += bv.v[e] - d * x0.v[e] + S;
        }
      }
    }
    float *dst = bc + C.nxy * (long long)K + (long long)C.nx * J + (i >> 1);
#pragma unroll
    for (int e = 0; e < V / 2; ++e) dst[e] = 0.125f * sum[e];
  }
}

// The lower part of the V-cycle (every level from lt down, each at most
// MG_LOWER_CELLS cells) in one block, which holds the levels' fractions,
// diagonals, right-hand sides and corrections in shared memory: the same
// sweeps, restrictions, coarsest sweeps and prolongations as the multi-block
// kernels, separated by block barriers instead of launches.  A serial chain
// of about 30 block-wide passes bounds it, so a pass costs little: a thread
// walks up whole columns with the z neighbours in registers and its row
// offsets formed once.  Shared memory: seven floats per cell, at most
// MG_LOWER_CELLS (1 + 1/8 + ...) cells.  Only a coarsest grid that cannot be
// coarsened to MG_LOWER_CELLS runs from global memory (SMEM false).
// 24x24x12 and below: 34 us (48 from global memory, a cell per thread).
constexpr long long MG_LOWER_CELLS = 7000;
constexpr int MG_LOWER_SMEM = (int)(MG_LOWER_CELLS * 8 / 7 + 8) * 28;
struct MgLower {
  Op32 L[kMgMaxLevels];
  float *x[kMgMaxLevels], *t[kMgMaxLevels], *b[kMgMaxLevels];
  int lt, top;
};

// One level as the block sees it.  On the SMEM path the pointers are built
// from the shared array itself, so that every access compiles to a
// shared-memory one.
struct LowerLevel {
  int nx, ny, nz, n;
  FastDiv fnx, fnxy;
  float ix2, iy2, iz2;
  float *bx, *by, *bz, *wi, *x, *t, *b;
};
template <bool SMEM>
__device__ __forceinline__ LowerLevel lower_level(const MgLower &M, int l, float *smem) {
  LowerLevel V;
  const Op32 &L = M.L[l];
  V.nx = L.D.nx, V.ny = L.D.ny, V.nz = L.D.nz, V.n = (int)(L.D.nxy * L.D.nz);
  V.fnx = L.D.fnx, V.fnxy = L.D.fnxy;
  V.ix2 = L.ix2, V.iy2 = L.iy2, V.iz2 = L.iz2;
  if constexpr (SMEM) {
    int o = 0;
    for (int q = M.lt; q < l; ++q) o += 7 * (int)(M.L[q].D.nxy * M.L[q].D.nz);
    float *q = smem + o;
    V.bx = q, V.by = q + V.n, V.bz = q + 2 * V.n, V.wi = q + 3 * V.n;
    V.x = q + 4 * V.n, V.t = q + 5 * V.n, V.b = q + 6 * V.n;
  } else {
    V.bx = const_cast<float *>(L.bx), V.by = const_cast<float *>(L.by), V.bz = const_cast<float *>(L.bz);
    V.wi = const_cast<float *>(L.wi);
    V.x = M.x[l], V.t = M.t[l], V.b = M.b[l];
  }
  return V;
}

// out = one sweep of xin, or (RES) the residual b - A xin.  A thread takes a
// column, or a run of levels of it where the block has threads for more.
template <bool RES>
__device__ __forceinline__ void lower_pass(const LowerLevel &L, const float *__restrict__ xin,
                                           float *__restrict__ out) {
  const int nx = L.nx, ny = L.ny, nz = L.nz, nxy = nx * ny;
  const float *__restrict__ bx = L.bx, *__restrict__ by = L.by, *__restrict__ bz = L.bz, *__restrict__ wi = L.wi,
                            *__restrict__ b = L.b;
  const int per = nxy >= (int)blockDim.x ? nz : max(1, (nz * nxy + (int)blockDim.x - 1) / (int)blockDim.x);
  for (int u = threadIdx.x; u < nxy * ((nz + per - 1) / per); u += blockDim.x) {
    const int seg = (int)L.fnxy.div((unsigned)u), col = u - seg * nxy, k0 = seg * per, k1 = min(nz, k0 + per);
    const int j = (int)L.fnx.div((unsigned)col), i = col - j * nx;
    const int xl = i == 0 ? nx - 1 : -1, xr = i == nx - 1 ? 1 - nx : 1;
    const int ym = j == 0 ? nx * (ny - 1) : -nx, yp = j == ny - 1 ? -nx * (ny - 1) : nx;
    int c = col + nxy * k0;
    float xm = k0 > 0 ? xin[c - nxy] : 0.f, x0 = xin[c], zl = bz[c];
#pragma unroll 3
    for (int k = k0; k < k1; ++k, c += nxy) {
      const bool up = k + 1 < nz;
      const float zh = up ? bz[c + nxy] : 0.f, xp = up ? xin[c + nxy] : 0.f;
      const float bxl = bx[c], bxr = bx[c + xr], byl = by[c], byr = by[c + yp], w = wi[c];
      const float S = L.ix2 * (bxl * xin[c + xl] + bxr * xin[c + xr]) + L.iy2 * (byl * xin[c + ym] + byr * xin[c + yp]) +
                      L.iz2 * (zl * xm + zh * xp);
      float v;
      if (RES) v = b[c] - (L.ix2 * (bxl + bxr) + L.iy2 * (byl + byr) + L.iz2 * (zl + zh)) * x0 + S;
      else v = (1.f - MG_OMEGA) * x0 + w * (b[c] + S);
      out[c] = w > 0.f ? v : 0.f;
      xm = x0;
      x0 = xp;
      zl = zh;
    }
  }
  __syncthreads();
}
// the sweep from zero
__device__ __forceinline__ void lower_first(const LowerLevel &L, float *__restrict__ out) {
  const float *__restrict__ wi = L.wi, *__restrict__ b = L.b;
#pragma unroll 4
  for (int c = threadIdx.x; c < L.n; c += blockDim.x) out[c] = wi[c] * b[c];
  __syncthreads();
}

template <bool SMEM>
__global__ void __launch_bounds__(1024) k_mg_lower(const __grid_constant__ MgLower M, const int *conv) {
  if (*conv) return;
  extern __shared__ float lower_smem[];
  const int lt = M.lt, top = M.top;
  if constexpr (SMEM) {
    for (int l = lt; l <= top; ++l) {
      const LowerLevel V = lower_level<true>(M, l, lower_smem);
      const float *__restrict__ gx = M.L[l].bx, *__restrict__ gy = M.L[l].by, *__restrict__ gz = M.L[l].bz,
                                *__restrict__ gw = M.L[l].wi, *__restrict__ gb = M.b[l];
#pragma unroll 4
      for (int c = threadIdx.x; c < V.n; c += blockDim.x) {
        const float a0 = gx[c], a1 = gy[c], a2 = gz[c], a3 = gw[c], a4 = l == lt ? gb[c] : 0.f;
        V.bx[c] = a0, V.by[c] = a1, V.bz[c] = a2, V.wi[c] = a3, V.b[c] = a4;
      }
    }
    __syncthreads();
  }
  for (int l = lt; l < top; ++l) {
    const LowerLevel V = lower_level<SMEM>(M, l, lower_smem), W = lower_level<SMEM>(M, l + 1, lower_smem);
    lower_first(V, V.t);
    lower_pass<false>(V, V.t, V.x);
    lower_pass<true>(V, V.x, V.t);
    const int sy = V.nx, sz = V.nx * V.ny;
    for (int c = threadIdx.x; c < W.n; c += blockDim.x) {   // the children's mean, as k_mg_restrict
      const int K = (int)W.fnxy.div((unsigned)c), col = c - K * W.nx * W.ny;
      const int J = (int)W.fnx.div((unsigned)col), I = col - J * W.nx;
      const float *f = V.t + 2 * I + sy * 2 * J + sz * 2 * K;
      W.b[c] = 0.125f * (((f[0] + f[1]) + (f[sy] + f[sy + 1])) +
                         ((f[sz] + f[sz + 1]) + (f[sz + sy] + f[sz + sy + 1])));
    }
    __syncthreads();
  }
  {
    const LowerLevel V = lower_level<SMEM>(M, top, lower_smem);
    lower_first(V, V.t);
    for (int sw = 1; sw < MG_COARSE_SWEEPS; ++sw)   // coarsest sweeps; the result ends in x
      lower_pass<false>(V, (sw & 1) ? V.t : V.x, (sw & 1) ? V.x : V.t);
  }
  for (int l = top - 1; l >= lt; --l) {
    const LowerLevel V = lower_level<SMEM>(M, l, lower_smem), W = lower_level<SMEM>(M, l + 1, lower_smem);
    for (int c = threadIdx.x; c < V.n; c += blockDim.x) {   // the parent's correction, as PROLONG
      const int k = (int)V.fnxy.div((unsigned)c), col = c - k * V.nx * V.ny;
      const int j = (int)V.fnx.div((unsigned)col), i = col - j * V.nx;
      V.x[c] += W.x[(i >> 1) + W.nx * ((j >> 1) + W.ny * (k >> 1))];
    }
    __syncthreads();
    lower_pass<false>(V, V.x, V.t);
    lower_pass<false>(V, V.t, V.x);
  }
  if constexpr (SMEM) {
    const LowerLevel V = lower_level<true>(M, lt, lower_smem);
    for (int c = threadIdx.x; c < V.n; c += blockDim.x) M.x[lt][c] = V.x[c];
  }
}

Op32 level_op(const MgLevel &L) {
  Op32 O;
  O.D = L.D;
  O.bx = L.bx;
  O.by = L.by;
  O.bz = L.bz;
  O.wi = L.wi;
  O.kreg = L.kreg;
  O.ix2 = L.ix2;
  O.iy2 = L.iy2;
  O.iz2 = L.iz2;
  return O;
}

// sizes of the levels (level 0 = the cell grid); false if multigrid does not apply
bool mg_plan(const Dims &D, int dims[kMgMaxLevels][3], int &nlev) {
  int nx = D.nx, ny = D.ny, nz = D.nz;
  nlev = 0;
  dims[nlev][0] = nx, dims[nlev][1] = ny, dims[nlev][2] = nz, ++nlev;
  while (nlev < kMgMaxLevels && (long long)nx * ny * nz > 512 && nx % 2 == 0 && ny % 2 == 0 && nz % 2 == 0 &&
         nx >= 4 && ny >= 4 && nz >= 4) {
    nx /= 2, ny /= 2, nz /= 2;
    dims[nlev][0] = nx, dims[nlev][1] = ny, dims[nlev][2] = nz, ++nlev;
  }
  return nlev >= 2 && (long long)nx * ny * nz <= 32768;
}

Op make_op(eb_geom g) {
  Op O;
  O.D = g->D;
  O.bx = g->pw.bx;
  O.by = g->pw.by;
  O.bz = g->pw.bz;
  O.d = g->pw.d;
  O.id = g->pw.id;
  O.ax = g->pw.ax;
  O.ay = g->pw.ay;
  O.az = g->pw.az;
  O.ix2 = g->D.idx * g->D.idx;
  O.iy2 = g->D.idy * g->D.idy;
  O.iz2 = g->D.idz * g->D.idz;
  return O;
}

// work space and the fixed part of the operator, on the first call
eb_status setup(eb_geom g, cudaStream_t s) {
  ProjWork &w = g->pw;
  if (w.ready) return EB_OK;
  const Dims &D = g->D;
  const long long N = D.nxy * D.nz;
  int dev = 0, sms = 0;
  CUDA_TRY(cudaGetDevice(&dev), "device");
  CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "device");
  w.nb = (int)std::max(1LL, std::min<long long>(4LL * std::max(sms, 1), (N + PB - 1) / PB));
  for (double **a : {&w.bx, &w.by, &w.bz, &w.ax, &w.ay, &w.az, &w.d, &w.id, &w.rhs, &w.r, &w.z, &w.p, &w.q, &w.x})
    CUDA_TRY(g->alloc(a, N), "alloc projection work space");
  CUDA_TRY(g->alloc(&w.part, 8LL * w.nb), "alloc projection work space");
  CUDA_TRY(g->alloc(&w.conv, 1), "alloc projection work space");
  CUDA_TRY(cudaMallocHost(&w.host, sizeof(double) * (size_t)w.nb), "alloc pinned scratch");
  launch_export_geometry(g->h, D, 0, g->G[0], EB_X_BETA_X, w.bx, s);
  launch_export_geometry(g->h, D, 0, g->G[0], EB_X_BETA_Y, w.by, s);
  launch_export_geometry(g->h, D, 0, g->G[0], EB_X_BETA_Z, w.bz, s);
  k_wall<<<(unsigned)((D.nxy + 255) / 256), 256, 0, s>>>(D, w.bz);
  k_scale<<<w.nb, PB, 0, s>>>(N, w.bx, D.idx * D.idx, w.ax);
  k_scale<<<w.nb, PB, 0, s>>>(N, w.by, D.idy * D.idy, w.ay);
  k_scale<<<w.nb, PB, 0, s>>>(N, w.bz, D.idz * D.idz, w.az);
  k_diag<<<w.nb, PB, 0, s>>>(make_op(g), w.d, w.part + S_CNT * w.nb);
  k_recip<<<w.nb, PB, 0, s>>>(N, w.d, w.id);
  CUDA_TRY(cudaMemcpyAsync(w.host, w.part + S_CNT * w.nb, sizeof(double) * w.nb, cudaMemcpyDeviceToHost, s),
           "count active cells");
  CUDA_TRY(cudaStreamSynchronize(s), "count active cells");
  double cnt = 0.0;
  for (int q = 0; q < w.nb; ++q) cnt += w.host[q];
  w.nact = (long long)cnt;
  w.ready = true;
  return EB_OK;
}

int final_blocks(eb_geom g);

// the multigrid hierarchy, on the first projection that uses it
eb_status mg_setup(eb_geom g, cudaStream_t s) {
  ProjWork &w = g->pw;
  if (w.nlev) return EB_OK;
  int dims[kMgMaxLevels][3], nlev = 0;
  if (!mg_plan(g->D, dims, nlev)) return fail(EB_ERR_INVALID_ARG, "grid cannot be coarsened for multigrid");
  const Op O0 = make_op(g);
  MgLevel &L0 = w.lev[0];
  L0.D = g->D;
  L0.ix2 = (float)O0.ix2, L0.iy2 = (float)O0.iy2, L0.iz2 = (float)O0.iz2;
  L0.nb = w.nb;
  const long long N0 = g->D.nxy * g->D.nz;
  for (float **a : {&L0.bx, &L0.by, &L0.bz, &L0.x, &L0.t, &L0.b, &L0.wi})
    CUDA_TRY(g->alloc(a, N0), "alloc multigrid level");
  k_mg_copy<<<L0.nb, PB, 0, s>>>(N0, w.bx, w.by, w.bz, L0.bx, L0.by, L0.bz);
  // MG_OMEGA / diagonal and the open levels of a level whose fractions are set
  auto finish = [&](MgLevel &L) -> cudaError_t {
    cudaError_t e = g->alloc(&L.kreg, L.D.nxy);
    int *top = nullptr;
    if (e == cudaSuccess) e = cudaMalloc(&top, sizeof(int) * (size_t)L.D.nxy);
    if (e != cudaSuccess) return e;
    const unsigned nb = (unsigned)((L.D.nxy + 127) / 128);
    k_mg_winv<<<L.nb, PB, 0, s>>>(level_op(L), L.wi);
    k_open_top<float><<<nb, 128, 0, s>>>(L.D, L.bx, L.by, L.bz, top);
    k_open_box<<<nb, 128, 0, s>>>(L.D, top, L.kreg);
    e = cudaStreamSynchronize(s);
    cudaFree(top);
    return e;
  };
  CUDA_TRY(finish(L0), "multigrid set-up");
  for (int l = 1; l < nlev; ++l) {
    MgLevel &L = w.lev[l];
    const MgLevel &F = w.lev[l - 1];
    Dims &C = L.D;
    C = F.D;
    C.nx = dims[l][0], C.ny = dims[l][1], C.nz = dims[l][2];
    C.nxy = (long long)C.nx * C.ny;
    C.dx = 2 * F.D.dx, C.dy = 2 * F.D.dy, C.dz = 2 * F.D.dz;
    C.idx = 0.5 * F.D.idx, C.idy = 0.5 * F.D.idy, C.idz = 0.5 * F.D.idz;
    C.fnx.init((unsigned)C.nx);
    C.fny.init((unsigned)C.ny);
    C.fnxy.init((unsigned)C.nxy);
    L.ix2 = 0.25f * F.ix2, L.iy2 = 0.25f * F.iy2, L.iz2 = 0.25f * F.iz2;
    const long long N = C.nxy * C.nz;
    L.nb = (int)std::max(1LL, std::min<long long>(w.nb, (N + PB - 1) / PB));
    for (float **a : {&L.bx, &L.by, &L.bz, &L.x, &L.t, &L.b, &L.wi})
      CUDA_TRY(g->alloc(a, N), "alloc multigrid level");
    k_mg_coarsen<<<L.nb, PB, 0, s>>>(level_op(F), C, L.bx, L.by, L.bz);
    CUDA_TRY(finish(L), "multigrid set-up");
  }
  w.nrz = final_blocks(g);
  CUDA_TRY(g->alloc(&w.part_rz, 2LL * w.nrz), "alloc projection work space");
  CUDA_TRY(cudaGetLastError(), "multigrid set-up");
  w.nlev = nlev;
  return EB_OK;
}

// columns per thread of a level's marching kernels
inline int level_v(const MgLevel &L) {
  if (L.D.nxy * L.D.nz < 4LL * MBX * MBY * ebk_sm_count()) return 1;   // too few threads otherwise
  return L.D.nx % 4 == 0 ? 4 : L.D.nx % 2 == 0 ? 2 : 1;
}

template <int MODE, bool FINAL>
void sweep(const MgLevel &L, const float *xin, const MgLevel *coarse, float *xout, double *zout, const double *r,
           double *prz, const int *conv, cudaStream_t s) {
  const int V = level_v(L);
  const Slabs S = slabs_of(L.D, V, ebk_sm_count());
  const Op32 O = level_op(L);
  const Dims C = coarse ? coarse->D : L.D;
  const float *xc = coarse ? coarse->x : nullptr;
  const dim3 blk(MBX, MBY, 1);
  if (V == 4) k_mg_sweep<4, MODE, FINAL><<<S.blocks(), blk, 0, s>>>(O, S, xin, xc, C, xout, zout, r, L.b, prz, conv);
  else if (V == 2) k_mg_sweep<2, MODE, FINAL><<<S.blocks(), blk, 0, s>>>(O, S, xin, xc, C, xout, zout, r, L.b, prz, conv);
  else k_mg_sweep<1, MODE, FINAL><<<S.blocks(), blk, 0, s>>>(O, S, xin, xc, C, xout, zout, r, L.b, prz, conv);
}

// from a level with an even number of columns (it is coarsened)
void restrict_residual(const MgLevel &F, const float *x, const MgLevel &C, const int *conv, cudaStream_t s) {
  const int V = F.D.nx % 4 == 0 ? 4 : 2;
  const long long plane = (long long)(F.D.nx / V) * C.D.ny;
  // two coarse levels per thread where that leaves about a wave of threads
  const int kper = plane * C.D.nz >= 2LL * 2048 * ebk_sm_count() ? 2 : 1;
  const long long n = plane * ((C.D.nz + kper - 1) / kper);
  const unsigned nb = (unsigned)((n + MBX * MBY - 1) / (MBX * MBY));
  if (V == 4) k_mg_restrict<4><<<nb, dim3(MBX, MBY, 1), 0, s>>>(level_op(F), x, F.b, C.D, C.b, kper, conv);
  else k_mg_restrict<2><<<nb, dim3(MBX, MBY, 1), 0, s>>>(level_op(F), x, F.b, C.D, C.b, kper, conv);
}

// blocks of the sweep that forms r.z (its partial sums)
int final_blocks(eb_geom g) {
  const MgLevel &L = g->pw.lev[0];
  return slabs_of(L.D, level_v(L), ebk_sm_count()).blocks();
}

// z = V(r) (r in FP64 and, as the finest level's right-hand side, in float)
// and the partial sums of r.z into prz
void vcycle(eb_geom g, const double *r, double *z, double *prz, cudaStream_t s) {
  ProjWork &w = g->pw;
  const MgLevel *L = w.lev;
  const int top = w.nlev - 1;
  // levels lt .. top (at most MG_LOWER_CELLS cells each) run in one block; level 0 never does
  int lt = top;
  while (lt > 1 && L[lt - 1].D.nxy * L[lt - 1].D.nz <= MG_LOWER_CELLS) --lt;
  // sweeps before and after the coarse correction: three on the finest level, two below
  sweep<FIRST, false>(L[0], nullptr, nullptr, L[0].t, nullptr, nullptr, nullptr, w.conv, s);
  sweep<PLAIN, false>(L[0], L[0].t, nullptr, L[0].x, nullptr, nullptr, nullptr, w.conv, s);
  restrict_residual(L[0], L[0].x, L[1], w.conv, s);
  for (int l = 1; l < lt; ++l) {
    sweep<FIRST, false>(L[l], nullptr, nullptr, L[l].x, nullptr, nullptr, nullptr, w.conv, s);
    restrict_residual(L[l], L[l].x, L[l + 1], w.conv, s);
  }
  {
    MgLower M;
    for (int l = lt; l <= top; ++l) {
      M.L[l] = level_op(L[l]);
      M.x[l] = L[l].x;
      M.t[l] = L[l].t;
      M.b[l] = L[l].b;
    }
    M.lt = lt;
    M.top = top;
    static unsigned long long attr = 0;
    ebk_smem_limit(k_mg_lower<true>, MG_LOWER_SMEM, attr);
    if (L[lt].D.nxy * L[lt].D.nz <= MG_LOWER_CELLS) k_mg_lower<true><<<1, 1024, MG_LOWER_SMEM, s>>>(M, w.conv);
    else k_mg_lower<false><<<1, 1024, 0, s>>>(M, w.conv);
  }
  for (int l = lt - 1; l >= 1; --l) {
    sweep<PROLONG, false>(L[l], L[l].x, &L[l + 1], L[l].t, nullptr, nullptr, nullptr, w.conv, s);
    sweep<PLAIN, false>(L[l], L[l].t, nullptr, L[l].x, nullptr, nullptr, nullptr, w.conv, s);
  }
  sweep<PROLONG, false>(L[0], L[0].x, &L[1], L[0].t, nullptr, nullptr, nullptr, w.conv, s);
  sweep<PLAIN, false>(L[0], L[0].t, nullptr, L[0].x, nullptr, nullptr, nullptr, w.conv, s);
  sweep<PLAIN, true>(L[0], L[0].x, nullptr, nullptr, z, r, prz, w.conv, s);
}

double host_total(eb_geom g, int slot, cudaStream_t s, cudaError_t &e) {
  ProjWork &w = g->pw;
  e = cudaMemcpyAsync(w.host, w.part + slot * w.nb, sizeof(double) * w.nb, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  double t = 0.0;
  for (int q = 0; q < w.nb; ++q) t += w.host[q];
  return t;
}

template <typename T>
void launch_rhs(eb_geom g, void *const mom[3], double dt, cudaStream_t s) {
  ProjWork &w = g->pw;
  k_rhs<T><<<w.nb, PB, 0, s>>>(make_op(g), (const T *)mom[0], (const T *)mom[1], (const T *)mom[2], 1.0 / dt, w.rhs,
                               w.part + S_SUM * w.nb);
}

template <typename T>
void launch_correct(eb_geom g, void *const mom[3], double dt, cudaStream_t s) {
  ProjWork &w = g->pw;
  k_correct<T><<<w.nb, PB, 0, s>>>(make_op(g), w.x, dt, (T *)mom[0], (T *)mom[1], (T *)mom[2]);
}

}  // namespace

eb_status eb_project_rhs(eb_geom g, void *const mom[3], double dt, double *rms, cudaStream_t s) {
  if (g->has_wind_ref)
    return fail(EB_ERR_STATE, "the projection needs full momenta: this handle has a background momentum profile");
  if (g->src_flags)
    return fail(EB_ERR_STATE, "the anelastic calls take no compressible sources: this handle has them switched on");
  eb_status st = setup(g, s);
  if (st != EB_OK) return st;
  ProjWork &w = g->pw;
  if (g->prec == EB_F64) launch_rhs<double>(g, mom, dt, s);
  else launch_rhs<float>(g, mom, dt, s);
  k_center<<<w.nb, PB, 0, s>>>(make_op(g), w.rhs, w.part + S_SUM * w.nb, w.part + S_CNT * w.nb, w.nb,
                               w.part + S_BB * w.nb);
  cudaError_t e = cudaSuccess;
  const double bb = host_total(g, S_BB, s, e);
  CUDA_TRY(e, "right-hand side");
  if (rms) *rms = w.nact > 0 ? sqrt(bb / (double)w.nact) : 0.0;
  return EB_OK;
}

eb_status eb_project_impl(eb_geom g, void *const mom[3], double dt, double rtol, int maxit, const double *phi0,
                          double *phi_out, int *iters, double *relres, cudaStream_t s, bool correct) {
  if (g->has_wind_ref)
    return fail(EB_ERR_STATE, "the projection needs full momenta: this handle has a background momentum profile");
  if (g->src_flags)
    return fail(EB_ERR_STATE, "the anelastic calls take no compressible sources: this handle has them switched on");
  eb_status st = setup(g, s);
  if (st != EB_OK) return st;
  ProjWork &w = g->pw;
  const Dims &D = g->D;
  const long long N = D.nxy * D.nz;
  const Op O = make_op(g);
  if (g->prec == EB_F64) launch_rhs<double>(g, mom, dt, s);
  else launch_rhs<float>(g, mom, dt, s);
  k_center<<<w.nb, PB, 0, s>>>(O, w.rhs, w.part + S_SUM * w.nb, w.part + S_CNT * w.nb, w.nb, w.part + S_BB * w.nb);
  if (phi0) CUDA_TRY(cudaMemcpyAsync(w.x, phi0, sizeof(double) * N, cudaMemcpyDeviceToDevice, s), "initial guess");
  else CUDA_TRY(cudaMemsetAsync(w.x, 0, sizeof(double) * N, s), "initial guess");
  const bool mg = w.precond == EB_PRECOND_MG;
  if (mg) {
    st = mg_setup(g, s);
    if (st != EB_OK) return st;
  }
  CUDA_TRY(cudaMemsetAsync(w.conv, 0, sizeof(int), s), "reset");
  double *const part_rz[2] = {w.part + S_RZ0 * w.nb, w.part + S_RZ1 * w.nb};
  double *const rz_of[2] = {mg ? w.part_rz : part_rz[0], mg ? w.part_rz + w.nrz : part_rz[1]};
  const int nrz = mg ? w.nrz : w.nb;   // partial sums of r.z
  float *rf = mg ? w.lev[0].b : nullptr;
  k_init<<<w.nb, PB, 0, s>>>(O, w.x, w.rhs, w.r, rf, w.z, w.p, part_rz[0], w.part + S_RR * w.nb);
  if (mg) {   // z = V(r), p = z
    vcycle(g, w.r, w.z, rz_of[0], s);
    CUDA_TRY(cudaMemcpyAsync(w.p, w.z, sizeof(double) * N, cudaMemcpyDeviceToDevice, s), "search direction");
  }
  cudaError_t e = cudaSuccess;
  const double bb = host_total(g, S_BB, s, e);
  CUDA_TRY(e, "residual norm");
  const double rr0 = host_total(g, S_RR, s, e);
  CUDA_TRY(e, "residual norm");
  const double thr2 = rtol * rtol * bb;
  int it = 0;
  double rr = rr0;
  if (bb > 0.0 && rr0 > thr2) {
    int done = 0;
    for (it = 0; it < maxit; ++it) {
      double *prz = rz_of[it % 2], *prz_next = rz_of[1 - it % 2];
      k_apply<<<w.nb, PB, 0, s>>>(O, w.p, w.q, w.part + S_PQ * w.nb, w.conv);
      if (mg) {
        k_update<false><<<w.nb, PB, 0, s>>>(O, w.x, w.p, w.q, w.r, rf, w.z, w.part + S_PQ * w.nb, prz, nrz, prz_next,
                                            w.part + S_RR * w.nb, w.nb, w.conv);
        vcycle(g, w.r, w.z, prz_next, s);
      } else {
        k_update<true><<<w.nb, PB, 0, s>>>(O, w.x, w.p, w.q, w.r, nullptr, w.z, w.part + S_PQ * w.nb, prz, nrz,
                                           prz_next, w.part + S_RR * w.nb, w.nb, w.conv);
      }
      k_direction<<<w.nb, PB, 0, s>>>(O, w.p, w.z, prz, prz_next, nrz, w.part + S_RR * w.nb, w.nb, thr2, it,
                                      w.conv);
      // the host reads the convergence flag every few iterations (a V-cycle
      // iteration costs far more than a Jacobi one, so it looks sooner)
      if ((it + 1) % (mg ? 4 : 32) == 0 || it + 1 == maxit) {
        CUDA_TRY(cudaMemcpyAsync(&done, w.conv, sizeof(int), cudaMemcpyDeviceToHost, s), "convergence flag");
        CUDA_TRY(cudaStreamSynchronize(s), "convergence flag");
        if (done) break;
      }
    }
    it = done ? done : maxit;
    rr = host_total(g, S_RR, s, e);
    CUDA_TRY(e, "residual norm");
  }
  if (correct) {
    if (g->prec == EB_F64) launch_correct<double>(g, mom, dt, s);
    else launch_correct<float>(g, mom, dt, s);
  }
  if (phi_out) CUDA_TRY(cudaMemcpyAsync(phi_out, w.x, sizeof(double) * N, cudaMemcpyDeviceToDevice, s), "phi");
  CUDA_TRY(cudaGetLastError(), "projection");
  if (iters) *iters = it;
  if (relres) *relres = bb > 0.0 ? sqrt(rr / bb) : 0.0;
  return EB_OK;
}

extern "C" {

eb_status eb_project(eb_geom geom, eb_state *U, double dt, double rtol, int maxit, const double *phi0, double *phi,
                     int *iters, double *relres, void *stream) {
  if (!geom) return fail(EB_ERR_INVALID_ARG, "NULL handle");
  const size_t es = geom->prec == EB_F64 ? 8 : 4;
  if (!state_ok(U, es)) return fail(EB_ERR_INVALID_ARG, "state pointer NULL or misaligned");
  if (!(dt > 0.0) || !isfinite(dt)) return fail(EB_ERR_INVALID_ARG, "dt must be finite and > 0");
  if (!(rtol > 0.0) || !(rtol < 1.0)) return fail(EB_ERR_INVALID_ARG, "rtol must lie in (0, 1)");
  if (maxit < 0) return fail(EB_ERR_INVALID_ARG, "maxit must be >= 0");
  if ((phi0 && ((uintptr_t)phi0 % 8)) || (phi && ((uintptr_t)phi % 8)))
    return fail(EB_ERR_INVALID_ARG, "phi pointer misaligned");
  void **u = state_ptrs(U);
  void *mom[3] = {u[2], u[3], u[4]};
  return eb_project_impl(geom, mom, dt, rtol, maxit, phi0, phi, iters, relres, as_stream(stream), true);
}

eb_status eb_project_set_preconditioner(eb_geom geom, int kind) {
  if (!geom) return fail(EB_ERR_INVALID_ARG, "NULL handle");
  if (kind != EB_PRECOND_JACOBI && kind != EB_PRECOND_MG) return fail(EB_ERR_INVALID_ARG, "unknown preconditioner");
  if (kind == EB_PRECOND_MG) {
    int dims[kMgMaxLevels][3], nlev = 0;
    if (!mg_plan(geom->D, dims, nlev))
      return fail(EB_ERR_INVALID_ARG,
                  "grid cannot be coarsened for multigrid (even sizes needed; coarsest grid <= 32768 cells)");
  }
  geom->pw.precond = kind;
  return EB_OK;
}

eb_status eb_anelastic_step(eb_geom geom, const eb_state *Un, eb_state *Unp1, double dt, int nsteps, double rtol,
                            int maxit, int *iters, void *stream) {
  if (!geom) return fail(EB_ERR_INVALID_ARG, "NULL handle");
  if (!geom->has_ref) return fail(EB_ERR_STATE, "the anelastic step needs a handle built with a reference profile");
  if (geom->src_flags)
    return fail(EB_ERR_STATE, "the anelastic calls take no compressible sources: this handle has them switched on");
  const size_t es = geom->prec == EB_F64 ? 8 : 4;
  if (!state_ok(Un, es) || !state_ok(Unp1, es)) return fail(EB_ERR_INVALID_ARG, "state pointer NULL or misaligned");
  if (!(dt > 0.0) || !isfinite(dt)) return fail(EB_ERR_INVALID_ARG, "dt must be finite and > 0");
  if (nsteps < 1) return fail(EB_ERR_INVALID_ARG, "nsteps must be >= 1");
  if (!(rtol > 0.0) || !(rtol < 1.0)) return fail(EB_ERR_INVALID_ARG, "rtol must lie in (0, 1)");
  if (maxit < 0) return fail(EB_ERR_INVALID_ARG, "maxit must be >= 0");
  void **u0 = state_ptrs(Un), **u1 = state_ptrs(Unp1);
  for (int f = 0; f < 5; ++f)
    for (int e = 0; e < 5; ++e) {
      const char *a = (const char *)u0[f], *b = (const char *)u1[e];
      if (a < b + field_count(geom->D, e) * es && b < a + field_count(geom->D, f) * es)
        return fail(EB_ERR_INVALID_ARG, "Un and Unp1 overlap");
    }
  cudaStream_t s = as_stream(stream);
  // scratch states: C, D alternate between steps, A holds the first stage
  for (int b = 0; b < 3; ++b)
    for (int f = 0; f < 5; ++f)
      if (!geom->scr[b][f]) {
        cudaError_t e = cudaMalloc(&geom->scr[b][f], field_count(geom->D, f) * es);
        if (e != cudaSuccess) return cuda_fail(e, "alloc step scratch");
        geom->allocs.push_back(geom->scr[b][f]);
      }
  void **C = geom->scr[0], **Dd = geom->scr[1], **A = geom->scr[2];
  void **cur = u0;
  for (int n = 0; n < nsteps; ++n) {
    void **dst = (n == nsteps - 1) ? u1 : (cur == C ? Dd : C);
    void **srcs[2] = {cur, A}, **outs[2] = {A, dst};
    const double frac[2] = {0.5, 1.0};
    for (int q = 0; q < 2; ++q) {
      if (geom->prec == EB_F64) stage<double>(geom, srcs[q], cur, outs[q], dt * frac[q], 1, s);
      else stage<float>(geom, srcs[q], cur, outs[q], dt * frac[q], 1, s);
      // the density stays at the reference: perturbation zero
      CUDA_TRY(cudaMemsetAsync(outs[q][0], 0, field_count(geom->D, 0) * es, s), "density");
      void *mom[3] = {outs[q][2], outs[q][3], outs[q][4]};
      int it = 0;
      const eb_status st =
          eb_project_impl(geom, mom, dt * frac[q], rtol, maxit, nullptr, nullptr, &it, nullptr, s, true);
      if (st != EB_OK) return st;
      if (iters) iters[2 * n + q] = it;
    }
    cur = dst;
  }
  CUDA_TRY(cudaGetLastError(), "anelastic step");
  return EB_OK;
}

}  // extern "C"
