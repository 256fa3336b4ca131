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
// Every kernel that forms a dot product writes one partial sum per block; the
// block that finishes last adds them in a fixed order, so the solve is
// deterministic and the next kernel reads one number.  Convergence is
// detected on the device (the kernels of later iterations return at once)
// and read by the host after 32 iterations (4 with the multigrid
// preconditioner) and then where the reduction so far predicts it.
//
// What bounds an iteration of the outer conjugate gradients is FP64 (two
// instructions per clock and SM): nine per cell in the operator and its dot
// product, two each in the update and the direction, conversions from and to
// float counted like arithmetic.  So the operator's constant rows above the
// terrain are formed from sums of opposite neighbours, x is updated with the
// direction (p is read once), floats are widened by integer instructions, and
// nothing is computed for the mask of inactive cells (their r, p and q are
// zero).  192x192x96: a Jacobi iteration 172 -> 147 us (the operator's floor is
// about 47; update and direction 47 and 24 before, 27 and 22 with x moved),
// right-hand side 116 -> 70, correction 114 -> 74, start of the solve 95 -> 30,
// centring 34 -> 25.
#include "eb_handle.cuh"

#include <math.h>

#include <algorithm>

using namespace ebh;

namespace {

constexpr int PB = 256;   // threads per block of every projection kernel

// slots of the scalars (w.scal), their partial sums (w.part) and counters
enum { S_SUM = 0, S_BB = 1, S_PQ = 2, S_RR = 3, S_RZ0 = 4, S_RZ1 = 5, S_CNT = 6, S_SLOTS = 7 };

__device__ inline double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Where a kernel's dot product goes: partial sums (one per block), the total
// and the count of finished blocks (zero before and after).
struct Sum {
  double *part, *total;
  unsigned *done;
};

// sum over the block (PB threads in any shape), in every thread of its first warp
__device__ inline double block_sum(double v) {
  __shared__ double s[PB / 32];
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  v = warp_sum(v);
  __syncthreads();
  if ((tid & 31) == 0) s[tid >> 5] = v;
  __syncthreads();
  double a = 0.0;
  if (tid < 32) {
    a = tid < PB / 32 ? s[tid] : 0.0;
    a = warp_sum(a);
  }
  return a;
}

// Adds v over the grid into *S.total: the last block to finish sums every
// block's partial in the same order whichever block it is.  Every thread of
// every block calls it, once per Sum and launch.
__device__ inline void grid_sum(double v, const Sum &S) {
  __shared__ bool last;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const double a = block_sum(v);
  if (tid == 0) {
    S.part[blockIdx.x] = a;
    __threadfence();
    last = atomicAdd(S.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double t = 0.0;
  for (unsigned q = tid; q < gridDim.x; q += PB) t += __ldcg(S.part + q);
  t = block_sum(t);
  if (tid == 0) {
    *S.total = t;
    *S.done = 0;
  }
}

// The same for two sums of one kernel, with one count of its blocks (A's).
__device__ inline void grid_sum2(double v, const Sum &A, double u, const Sum &B) {
  __shared__ bool last;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const double a = block_sum(v), b = block_sum(u);
  if (tid == 0) {
    A.part[blockIdx.x] = a;
    B.part[blockIdx.x] = b;
    __threadfence();
    last = atomicAdd(A.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double s = 0.0, t = 0.0;
  for (unsigned q = tid; q < gridDim.x; q += PB) {
    s += __ldcg(A.part + q);
    t += __ldcg(B.part + q);
  }
  s = block_sum(s);
  t = block_sum(t);
  if (tid == 0) {
    *A.total = s;
    *B.total = t;
    *A.done = 0;
  }
}

// a float as a double, by integer instructions (FP64 conversions run at the
// FP64 rate); subnormals, infinities and NaN take the conversion
__device__ inline double widen(float f) {
  const unsigned u = __float_as_uint(f), e = u & 0x7f800000u;
  if (e - 0x00800000u >= 0x7f000000u) return (u << 1) ? (double)f : __hiloint2double((int)u, 0);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ inline double widen(double f) { return f; }

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
  const int *kreg;        // per column: every face within two columns open from here up
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

__global__ void k_diag(Op O, double *d, Sum cnt) {
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  double n_act = 0.0;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    const Nbr n = neighbours(D, c);
    const double bzh = n.k + 1 < D.nz ? O.bz[c + D.nxy] : 0.0;
    const double v = (O.bx[c] + O.bx[n.xp]) * O.ix2 + (O.by[c] + O.by[n.yp]) * O.iy2 + (O.bz[c] + bzh) * O.iz2;
    d[c] = v;
    n_act += v > 0.0 ? 1.0 : 0.0;
  }
  grid_sum(n_act, cnt);
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

// The operator's split: the column groups of a plane one after another, 256 to
// a block (no lane idles at ragged rows: 16 x 16 tiles left a third of them
// idle at 130x50), nbx blocks to a plane.  Its FP64 work is what an SM takes time
// for, so the fullest SM decides: its blocks times their levels, and most of a
// level more per block (the planes below and above, the sum); fewer than two
// blocks per SM do not hide their own latency.
inline int apply_blocks(const Dims &D, int V) { return (int)((D.nxy / V + PB - 1) / PB); }
inline Slabs apply_slabs(const Dims &D, int V, int sms) {
  Slabs S{apply_blocks(D, V), 1, 1};
  double best = 0.0;
  for (int n = 1; n <= D.nz && (n == 1 || (long long)S.nbx * n <= 8LL * sms); ++n) {
    const double c = (double)((S.nbx * (long long)n + sms - 1) / sms) * ((D.nz + n - 1) / n + 0.7);
    const bool few = S.nbx * (long long)(n - 1) < 2LL * sms;
    if (few || c <= 1.02 * best) S.nz = n;   // (more blocks where that costs next to nothing)
    best = few ? c : std::min(best, c);
  }
  return S;
}
template <int V>
__device__ inline Cols cols_flat(const Dims &D, const Slabs &S) {
  Cols q;
  const int sl = blockIdx.x / S.nbx, t = (blockIdx.x - sl * S.nbx) * PB + (int)threadIdx.x, g = D.nx / V;
  q.in = t < g * D.ny;
  q.j = q.in ? t / g : 0;
  q.i = q.in ? V * (t - q.j * g) : 0;
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

// rhs = D(m) / dt on the active cells; cx, cy, cz = 1 / (delta dt)
template <typename T>
__global__ void __launch_bounds__(PB) k_rhs(const __grid_constant__ Op O, const __grid_constant__ Slabs SL,
                                            const T *__restrict__ mu, const T *__restrict__ mv,
                                            const T *__restrict__ mw, double cx, double cy, double cz,
                                            double *__restrict__ rhs, Sum total) {
  const Dims &D = O.D;
  const Cols q = cols_of<1>(D, SL);
  double sum = 0.0;
  if (q.in) {
    const int kr = O.kreg[q.c];
    double wl = widen(mw[D.nxy * (long long)q.k0 + q.c]);
#pragma unroll 2
    for (int k = q.k0; k < q.k1; ++k) {
      const long long t = D.nxy * (long long)k, c = t + q.c;
      const double wh = widen(mw[c + D.nxy]);   // rho*w has nz + 1 levels
      const double ul = widen(mu[c]), uh = widen(mu[t + q.xr]), vl = widen(mv[c]), vh = widen(mv[t + q.yp]);
      double v = 0.0;
      if (k >= kr && k > 0 && k < D.nz - 1) {
        v = fma(uh - ul, cx, fma(vh - vl, cy, (wh - wl) * cz));
      } else if (O.d[c] > 0.0) {
        const double bzh = k + 1 < D.nz ? O.bz[c + D.nxy] : 0.0;
        const double bxl = O.bx[c], bxh = O.bx[t + q.xr], byl = O.by[c], byh = O.by[t + q.yp], bzl = O.bz[c];
        const double dx = bxh * uh - bxl * ul, dy = byh * vh - byl * vl, dz = bzh * wh - bzl * wl;
        v = fma(dx, cx, fma(dy, cy, dz * cz));
      }
      rhs[c] = v;
      sum += v;
      wl = wh;
    }
  }
  grid_sum(sum, total);
}

// remove the mean of the right-hand side over the active cells
__global__ void __launch_bounds__(PB) k_center(const __grid_constant__ Op O, double *rhs, const double *sum,
                                               const double *cnt, Sum bb) {
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  const double mean = *sum / fmax(1.0, *cnt);
  double a = 0.0;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    const int k = (int)D.fnxy.div((unsigned)c);
    if (k >= O.kreg[c - D.nxy * (long long)k] || O.d[c] > 0.0) {
      const double v = rhs[c] - mean;
      rhs[c] = v;
      a = fma(v, v, a);
    }
  }
  grid_sum(a, bb);
}

// r = -rhs - A x (x = nullptr: zero) with r.r, and Jacobi: p = z = r / d with r.z
__global__ void __launch_bounds__(PB) k_init(const __grid_constant__ Op O, const double *x, const double *rhs,
                                             double *r, float *rf, double *p, Sum srz, Sum srr) {
  const Dims &D = O.D;
  const long long N = D.nxy * D.nz;
  double rz = 0.0, rr = 0.0;
  for (long long c = blockIdx.x * (long long)PB + threadIdx.x; c < N; c += (long long)gridDim.x * PB) {
    double rv = -rhs[c];   // zero on the inactive cells
    if (x) rv = O.d[c] > 0.0 ? rv - O.apply(x, c, neighbours(D, c)) : 0.0;
    r[c] = rv;
    if (rf) {
      rf[c] = (float)rv;   // the V-cycle's right-hand side
    } else {
      const double zv = rv * O.id[c];
      p[c] = zv;
      rz = fma(rv, zv, rz);
    }
    rr = fma(rv, rv, rr);
  }
  if (!rf) grid_sum(rz, srz);
  grid_sum(rr, srr);
}

// iteration `it` has nothing left to do when an earlier one converged
// (*conv = number of iterations then)
__device__ inline bool finished(const int *conv, int it) {
  const int c = *conv;
  return c != 0 && c <= it;
}

// q = A p and p.q; V = 2 columns per thread where rows hold whole pairs
template <int V>
__global__ void __launch_bounds__(PB) k_apply(const __grid_constant__ Op O, const __grid_constant__ Slabs SL,
                                              const double *__restrict__ p, double *__restrict__ qo, Sum spq,
                                              const int *conv, int it) {
  chain_begin();
  if (finished(conv, it)) return;
  const Dims &D = O.D;
  const Cols q = cols_flat<V>(D, SL);
  const double dreg = 2.0 * (O.ix2 + O.iy2 + O.iz2);
  double pq = 0.0;
  auto ld = [&](const double *s, double (&v)[V]) {
    if constexpr (V == 2) {
      const double2 t = *reinterpret_cast<const double2 *>(s);
      v[0] = t.x, v[1] = t.y;
    } else {
      v[0] = *s;
    }
  };
  if (q.in) {
    int kr = 0;
#pragma unroll
    for (int e = 0; e < V; ++e) kr = max(kr, O.kreg[q.c + e]);
    double xm[V], x0[V], xp[V];
#pragma unroll
    for (int e = 0; e < V; ++e) xm[e] = xp[e] = 0.0;
    if (q.k0 > 0) ld(p + D.nxy * (long long)(q.k0 - 1) + q.c, xm);
    ld(p + D.nxy * (long long)q.k0 + q.c, x0);
#pragma unroll 2
    for (int k = q.k0; k < q.k1; ++k) {
      const long long t = D.nxy * (long long)k, c = t + q.c;
      if (k + 1 < D.nz) ld(p + c + D.nxy, xp);
      double ym[V], yp[V], o[V];
      ld(p + t + q.ym, ym);
      ld(p + t + q.yp, yp);
      const double xl = p[t + q.xl], xr = p[t + q.xr];
      if (k >= kr && k > 0 && k < D.nz - 1) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const double sx = (e ? x0[0] : xl) + (e + 1 < V ? x0[V - 1] : xr);
          o[e] = fma(-O.ix2, sx, fma(-O.iy2, ym[e] + yp[e], fma(-O.iz2, xm[e] + xp[e], dreg * x0[e])));
        }
      } else {
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const long long ce = c + e;
          const double dd = O.d[ce];
          o[e] = 0.0;
          if (__double2hiint(dd) > 0) {   // tests of non-negative doubles by their high words
            const double azl = O.az[ce], azh = k + 1 < D.nz ? O.az[ce + D.nxy] : 0.0;
            double v = dd * x0[e];
            v = fma(-O.ax[ce], e ? x0[0] : xl, v);
            v = fma(-O.ax[e + 1 < V ? ce + 1 : t + q.xr], e + 1 < V ? x0[V - 1] : xr, v);
            v = fma(-O.ay[ce], ym[e], v);
            v = fma(-O.ay[t + q.yp + e], yp[e], v);
            if (__double2hiint(azl) > 0) v = fma(-azl, xm[e], v);
            if (__double2hiint(azh) > 0) v = fma(-azh, xp[e], v);
            o[e] = v;
          }
        }
      }
      if constexpr (V == 2) *reinterpret_cast<double2 *>(qo + c) = make_double2(o[0], o[1]);
      else qo[c] = o[0];
#pragma unroll
      for (int e = 0; e < V; ++e) {
        pq = fma(x0[e], o[e], pq);
        xm[e] = x0[e];
        x0[e] = xp[e];
      }
    }
  }
  grid_sum(pq, spq);
}

// alpha = rz / pq; r -= alpha q, r.r; Jacobi: r.z with z = r / d (the
// multigrid preconditioner forms z and r.z afterwards, from the float copy)
template <bool JAC>
__global__ void __launch_bounds__(PB) k_update(const __grid_constant__ Op O, const double *__restrict__ q,
                                               double *__restrict__ r, float *__restrict__ rf, const double *rz,
                                               const double *pq, Sum srz, Sum srr, const int *conv, int it) {
  chain_begin();
  if (finished(conv, it)) return;
  const long long N = O.D.nxy * O.D.nz, N2 = N & ~1LL;
  const double alpha = *rz / *pq;
  double az = 0.0, rr = 0.0;
  auto one = [&](long long c, double rv, double qv) -> double {
    rv = fma(-alpha, qv, rv);
    if (JAC) az = fma(rv, rv * O.id[c], az);
    rr = fma(rv, rv, rr);
    return rv;
  };
  const long long t0 = 2 * (blockIdx.x * (long long)PB + threadIdx.x), dt = 2LL * gridDim.x * PB;
#pragma unroll 2
  for (long long c = t0; c < N2; c += dt) {
    double2 v = *reinterpret_cast<const double2 *>(r + c);
    const double2 qv = *reinterpret_cast<const double2 *>(q + c);
    v.x = one(c, v.x, qv.x);
    v.y = one(c + 1, v.y, qv.y);
    *reinterpret_cast<double2 *>(r + c) = v;
    if (!JAC) *reinterpret_cast<float2 *>(rf + c) = make_float2((float)v.x, (float)v.y);
  }
  if (t0 == 0 && N2 < N) {   // an odd last cell
    const double v = one(N2, r[N2], q[N2]);
    r[N2] = v;
    if (!JAC) rf[N2] = (float)v;
  }
  if (JAC) grid_sum2(az, srz, rr, srr);
  else grid_sum(rr, srr);
}

// x += alpha p; then, unless r.r meets the threshold (conv is set), p = z +
// (rz_next / rz) p with Jacobi's z = r / d
template <bool JAC>
__global__ void __launch_bounds__(PB) k_direction(const __grid_constant__ Op O, double *__restrict__ x,
                                                  double *__restrict__ p, const double *__restrict__ zr,
                                                  const double *rz, const double *rz_next, const double *pq,
                                                  const double *rr, double thr2, int it, int *conv) {
  chain_begin();
  if (finished(conv, it)) return;
  const long long N = O.D.nxy * O.D.nz, N2 = N & ~1LL;
  const double alpha = *rz / *pq;
  const bool stop = *rr <= thr2;
  if (stop && blockIdx.x == 0 && threadIdx.x == 0) *conv = it + 1;
  const double beta = *rz_next / *rz;
  const long long t0 = 2 * (blockIdx.x * (long long)PB + threadIdx.x), dt = 2LL * gridDim.x * PB;
#pragma unroll 2
  for (long long c = t0; c < N2; c += dt) {
    double2 pv = *reinterpret_cast<const double2 *>(p + c), xv = *reinterpret_cast<const double2 *>(x + c);
    xv.x = fma(alpha, pv.x, xv.x);
    xv.y = fma(alpha, pv.y, xv.y);
    *reinterpret_cast<double2 *>(x + c) = xv;
    if (!stop) {
      double2 z = *reinterpret_cast<const double2 *>(zr + c);
      if (JAC) {
        const double2 i = *reinterpret_cast<const double2 *>(O.id + c);
        z.x *= i.x, z.y *= i.y;
      }
      pv.x = fma(beta, pv.x, z.x);
      pv.y = fma(beta, pv.y, z.y);
      *reinterpret_cast<double2 *>(p + c) = pv;
    }
  }
  if (t0 == 0 && N2 < N) {
    x[N2] = fma(alpha, p[N2], x[N2]);
    if (!stop) p[N2] = fma(beta, p[N2], JAC ? zr[N2] * O.id[N2] : zr[N2]);
  }
}

// m -= dt G(x) on the open faces; cx, cy, cz = dt / delta
template <typename T>
__global__ void __launch_bounds__(PB) k_correct(const __grid_constant__ Op O, const __grid_constant__ Slabs SL,
                                                const double *__restrict__ x, double cx, double cy, double cz,
                                                T *__restrict__ mu, T *__restrict__ mv, T *__restrict__ mw) {
  const Dims &D = O.D;
  const Cols q = cols_of<1>(D, SL);
  if (!q.in) return;
  const int kr = O.kreg[q.c];
  double xm = q.k0 > 0 ? x[D.nxy * (long long)(q.k0 - 1) + q.c] : 0.0;
#pragma unroll 2
  for (int k = q.k0; k < q.k1; ++k) {
    const long long t = D.nxy * (long long)k, c = t + q.c;
    const double x0 = x[c];
    const bool open = k >= kr;
    const T u = mu[c], v = mv[c], w = mw[c];
    if (open || O.bx[c] > 0.0) mu[c] = (T)fma(-cx, x0 - x[t + q.xl], widen(u));
    if (open || O.by[c] > 0.0) mv[c] = (T)fma(-cy, x0 - x[t + q.ym], widen(v));
    if (k >= 1 && (open || O.bz[c] > 0.0)) mw[c] = (T)fma(-cz, x0 - xm, widen(w));
    xm = x0;
  }
}

// ---------------------------------------------------------------------------
// Multigrid preconditioner (EB_PRECOND_MG): z = V(r), one V-cycle in FP32
// (FP64 arithmetic is scarce on this GPU; the outer conjugate gradients stay
// in FP64).  Damped Jacobi with the same weights before and after the coarse
// correction (three sweeps on the finest grid, two on the coarser ones),
// restriction = 1/8 of the transpose of the injection prolongation, and a
// fixed number of Jacobi sweeps from zero on the coarsest grid: up to float
// rounding V is a fixed symmetric positive semi-definite operator, as
// conjugate gradients need.
// ---------------------------------------------------------------------------
// Jacobi sweeps on the coarsest grid (even: the result ends in x).
constexpr int MG_COARSE_SWEEPS = 16;

// Weights of the sweeps: the n sweeps of a smoother are one polynomial in
// D^-1 A, whose eigenvalues lie in [0, 2] (the rows' off-diagonal magnitudes
// sum to the diagonal).  The Chebyshev polynomial of an interval [a, 2]
// damps everything in it to 1 / T_n((2 + a) / (2 - a)) (Saad, "Iterative
// Methods for Sparse Linear Systems", 2003, sec. 12.3): the weights are the
// reciprocals of its roots.  Below a it stays in (0, 1), so the V-cycle, the
// same polynomial before and after the coarse correction, stays definite.
// Three sweeps on [0.4, 2] on the finest grid, two on [0.3, 2] below,
// sixteen on [0.1, 2] on the coarsest (taken in bit-reversed order, which
// keeps the intermediate results small).  Iterations at rtol 1e-10, against
// the weight 0.9 for every sweep: 192x192x96 random terrain 14 -> 11, 44x36x20 14
// -> 9, 160x48x32 50 -> 40.
struct MgWeights {
  float fine[3], coarse[2], coarsest[MG_COARSE_SWEEPS];
  MgWeights() {
    auto weight = [](double a, int q, int n) {
      return (float)(1.0 / (0.5 * (2.0 + a) + 0.5 * (2.0 - a) * cos((2 * q + 1) * M_PI / (2 * n))));
    };
    for (int q = 0; q < 3; ++q) fine[q] = weight(0.4, q, 3);
    for (int q = 0; q < 2; ++q) coarse[q] = weight(0.3, q, 2);
    for (int q = 0; q < MG_COARSE_SWEEPS; ++q) {
      int r = 0;
      for (int b = 1, m = MG_COARSE_SWEEPS / 2; b < MG_COARSE_SWEEPS; b *= 2, m /= 2) r += (q & b) ? m : 0;
      coarsest[q] = weight(0.1, r, MG_COARSE_SWEEPS);
    }
  }
};

// The operator of one level.  From kreg[column] up, every face of the cells
// within two columns is fully open (the terrain lies below), so there, away
// from the floor and the lid, the kernels read no coefficient at all.
struct Op32 {
  Dims D;
  const float *bx, *by, *bz;   // low-face open fractions
  const float *wi;             // 1 / diagonal (0 off the active cells)
  const int *kreg;
  float ix2, iy2, iz2;
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
    wi[c] = d > 0.f ? 1.f / d : 0.f;
  }
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

// One damped Jacobi sweep, xout = (1 - w) x + w (b + S(x)) / d, of
//   FIRST    x = w b / d, the sweep from zero (so two sweeps in one pass),
//   PLAIN    x = xin,
//   PROLONG  x = xin + the parent's coarse correction (injection; inactive
//            cells are never read with a nonzero coefficient).
// FINAL: the finest level's last sweep, which writes the FP64 z and sums r.z.
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
                                                        const float *__restrict__ b, float w0, float w, Sum srz,
                                                        const int *conv) {
  chain_begin();
  if (*conv) return;
  const Dims &D = L.D;
  const Cols q = cols_of<V>(D, SL);
  const float ireg = 1.f / (2.f * (L.ix2 + L.iy2 + L.iz2)), wreg = w * ireg, wfirst = w0 * ireg;
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
        for (int e = 0; e < V; ++e) a.v[e] *= wfirst;
      } else {
        const Vec<V> iv = ldv<V>(L.wi + t);
#pragma unroll
        for (int e = 0; e < V; ++e) a.v[e] *= w0 * iv.v[e];
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
    if constexpr (MODE == FIRST) return b[t] * (reg ? wfirst : w0 * L.wi[t]);
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
          o.v[e] = (1.f - w) * x0.v[e] + wreg * (bv.v[e] + S);
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
          o.v[e] = wi.v[e] > 0.f ? (1.f - w) * x0.v[e] + w * wi.v[e] * (bv.v[e] + S) : 0.f;
        }
      }
      if constexpr (FINAL) {
        double z[V];
#pragma unroll
        for (int e = 0; e < V; ++e) z[e] = widen(o.v[e]);
        if constexpr (V > 1) {
#pragma unroll
          for (int e = 0; e < V; e += 2) {
            const double2 rv = *reinterpret_cast<const double2 *>(r + t + q.c + e);
            *reinterpret_cast<double2 *>(zout + t + q.c + e) = make_double2(z[e], z[e + 1]);
            rz = fma(rv.x, z[e], fma(rv.y, z[e + 1], rz));
          }
        } else {
          zout[t + q.c] = z[0];
          rz = fma(r[t + q.c], z[0], rz);
        }
      } else {
        stv<V>(xout + t + q.c, o);
      }
      xm = x0;
      x0 = xp;
    }
  }
  if constexpr (FINAL) grid_sum(rz, srz);
}

// Coarse right-hand side: the mean of the eight children's residuals b - A x.
// A thread forms V / 2 coarse cells per coarse level from V columns x 2 rows.
// 192x192x96: 11 us (one coarse cell per thread: 25).
template <int V>
__global__ void __launch_bounds__(MBX * MBY) k_mg_restrict(const __grid_constant__ Op32 F, const float *x,
                                                           const float *b, const __grid_constant__ Dims C,
                                                           float *bc, int kper, const int *conv) {
  chain_begin();
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
  float w[2];   // weights of the two sweeps (reversed after the coarse correction)
  float wc[MG_COARSE_SWEEPS];
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
__device__ __forceinline__ void lower_pass(const LowerLevel &L, float om, const float *__restrict__ xin,
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
      else v = (1.f - om) * x0 + om * w * (b[c] + S);
      out[c] = w > 0.f ? v : 0.f;
      xm = x0;
      x0 = xp;
      zl = zh;
    }
  }
  __syncthreads();
}
// the sweep from zero
__device__ __forceinline__ void lower_first(const LowerLevel &L, float om, float *__restrict__ out) {
  const float *__restrict__ wi = L.wi, *__restrict__ b = L.b;
#pragma unroll 4
  for (int c = threadIdx.x; c < L.n; c += blockDim.x) out[c] = om * wi[c] * b[c];
  __syncthreads();
}

template <bool SMEM>
__global__ void __launch_bounds__(1024) k_mg_lower(const __grid_constant__ MgLower M, const int *conv) {
  chain_begin();
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
    lower_first(V, M.w[0], V.t);
    lower_pass<false>(V, M.w[1], V.t, V.x);
    lower_pass<true>(V, 0.f, V.x, V.t);
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
    lower_first(V, M.wc[0], V.t);
    for (int sw = 1; sw < MG_COARSE_SWEEPS; ++sw)   // coarsest sweeps; the result ends in x
      lower_pass<false>(V, M.wc[sw], (sw & 1) ? V.t : V.x, (sw & 1) ? V.x : V.t);
  }
  for (int l = top - 1; l >= lt; --l) {
    const LowerLevel V = lower_level<SMEM>(M, l, lower_smem), W = lower_level<SMEM>(M, l + 1, lower_smem);
    for (int c = threadIdx.x; c < V.n; c += blockDim.x) {   // the parent's correction, as PROLONG
      const int k = (int)V.fnxy.div((unsigned)c), col = c - k * V.nx * V.ny;
      const int j = (int)V.fnx.div((unsigned)col), i = col - j * V.nx;
      V.x[c] += W.x[(i >> 1) + W.nx * ((j >> 1) + W.ny * (k >> 1))];
    }
    __syncthreads();
    lower_pass<false>(V, M.w[1], V.x, V.t);
    lower_pass<false>(V, M.w[0], V.t, V.x);
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
  O.kreg = g->pw.kreg;
  O.ix2 = g->D.idx * g->D.idx;
  O.iy2 = g->D.idy * g->D.idy;
  O.iz2 = g->D.idz * g->D.idz;
  return O;
}

Sum sum_of(eb_geom g, int slot) {
  ProjWork &w = g->pw;
  return Sum{w.part + (long long)slot * w.npart, w.scal + slot, w.done + slot};
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
  w.ncols = D.nx % 2 == 0 ? 2 : 1;
  w.npart = std::max({w.nb, slabs_of(D, 1, sms).blocks(), slabs_of(D, 2, sms).blocks(), slabs_of(D, 4, sms).blocks(),
                      apply_slabs(D, w.ncols, sms).blocks()});
  w.aslabs = apply_slabs(D, w.ncols, sms).nz;
  CUDA_TRY(g->alloc(&w.part, (long long)S_SLOTS * w.npart), "alloc projection work space");
  CUDA_TRY(g->alloc(&w.scal, S_SLOTS), "alloc projection work space");
  CUDA_TRY(g->alloc(&w.done, S_SLOTS), "alloc projection work space");
  CUDA_TRY(cudaMemsetAsync(w.done, 0, sizeof(unsigned) * S_SLOTS, s), "projection work space");
  CUDA_TRY(g->alloc(&w.kreg, D.nxy), "alloc projection work space");
  CUDA_TRY(g->alloc(&w.conv, 1), "alloc projection work space");
  CUDA_TRY(cudaMallocHost(&w.host, sizeof(double) * (S_SLOTS + 1)), "alloc pinned scratch");
  launch_export_geometry(g->h, D, 0, g->G[0], EB_X_BETA_X, w.bx, s);
  launch_export_geometry(g->h, D, 0, g->G[0], EB_X_BETA_Y, w.by, s);
  launch_export_geometry(g->h, D, 0, g->G[0], EB_X_BETA_Z, w.bz, s);
  k_wall<<<(unsigned)((D.nxy + 255) / 256), 256, 0, s>>>(D, w.bz);
  k_scale<<<w.nb, PB, 0, s>>>(N, w.bx, D.idx * D.idx, w.ax);
  k_scale<<<w.nb, PB, 0, s>>>(N, w.by, D.idy * D.idy, w.ay);
  k_scale<<<w.nb, PB, 0, s>>>(N, w.bz, D.idz * D.idz, w.az);
  k_diag<<<w.nb, PB, 0, s>>>(make_op(g), w.d, sum_of(g, S_CNT));
  k_recip<<<w.nb, PB, 0, s>>>(N, w.d, w.id);
  {
    int *top = nullptr;
    CUDA_TRY(cudaMalloc(&top, sizeof(int) * (size_t)D.nxy), "open levels");
    const unsigned nc = (unsigned)((D.nxy + 127) / 128);
    k_open_top<double><<<nc, 128, 0, s>>>(D, w.bx, w.by, w.bz, top);
    k_open_box<<<nc, 128, 0, s>>>(D, top, w.kreg);
    cudaError_t e = cudaMemcpyAsync(w.host, w.scal + S_CNT, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(top);
    CUDA_TRY(e, "count active cells");
  }
  w.nact = (long long)w.host[0];
  w.ready = true;
  return EB_OK;
}

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
  // 1 / diagonal and the open levels of a level whose fractions are set
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
           float w0, float w, const Sum &rz, const int *conv, cudaStream_t s) {
  const int V = level_v(L);
  const Slabs S = slabs_of(L.D, V, ebk_sm_count());
  const Op32 O = level_op(L);
  const Dims C = coarse ? coarse->D : L.D;
  const float *xc = coarse ? coarse->x : nullptr;
  const dim3 blk(MBX, MBY, 1);
  if (V == 4) launch_chained(k_mg_sweep<4, MODE, FINAL>, S.blocks(), blk, 0, s, O, S, xin, xc, C, xout, zout, r, L.b, w0, w, rz, conv);
  else if (V == 2) launch_chained(k_mg_sweep<2, MODE, FINAL>, S.blocks(), blk, 0, s, O, S, xin, xc, C, xout, zout, r, L.b, w0, w, rz, conv);
  else launch_chained(k_mg_sweep<1, MODE, FINAL>, S.blocks(), blk, 0, s, O, S, xin, xc, C, xout, zout, r, L.b, w0, w, rz, conv);
}

// from a level with an even number of columns (it is coarsened)
void restrict_residual(const MgLevel &F, const float *x, const MgLevel &C, const int *conv, cudaStream_t s) {
  const int V = F.D.nx % 4 == 0 ? 4 : 2;
  const long long plane = (long long)(F.D.nx / V) * C.D.ny;
  // two coarse levels per thread where that leaves about a wave of threads
  const int kper = plane * C.D.nz >= 2LL * 2048 * ebk_sm_count() ? 2 : 1;
  const long long n = plane * ((C.D.nz + kper - 1) / kper);
  const unsigned nb = (unsigned)((n + MBX * MBY - 1) / (MBX * MBY));
  if (V == 4) launch_chained(k_mg_restrict<4>, nb, dim3(MBX, MBY, 1), 0, s, level_op(F), x, F.b, C.D, C.b, kper, conv);
  else launch_chained(k_mg_restrict<2>, nb, dim3(MBX, MBY, 1), 0, s, level_op(F), x, F.b, C.D, C.b, kper, conv);
}

// z = V(r) (r in FP64 and, as the finest level's right-hand side, in float)
// and r.z into the slot rz
void vcycle(eb_geom g, const double *r, double *z, int rz, cudaStream_t s) {
  const Sum none{nullptr, nullptr, nullptr};
  ProjWork &w = g->pw;
  static const MgWeights W;
  const MgLevel *L = w.lev;
  const int top = w.nlev - 1;
  // levels lt .. top (at most MG_LOWER_CELLS cells each) run in one block; level 0 never does
  int lt = top;
  while (lt > 1 && L[lt - 1].D.nxy * L[lt - 1].D.nz <= MG_LOWER_CELLS) --lt;
  // sweeps before and after the coarse correction: three on the finest level, two below
  sweep<FIRST, false>(L[0], nullptr, nullptr, L[0].t, nullptr, nullptr, W.fine[0], W.fine[1], none, w.conv, s);
  sweep<PLAIN, false>(L[0], L[0].t, nullptr, L[0].x, nullptr, nullptr, 0.f, W.fine[2], none, w.conv, s);
  restrict_residual(L[0], L[0].x, L[1], w.conv, s);
  for (int l = 1; l < lt; ++l) {
    sweep<FIRST, false>(L[l], nullptr, nullptr, L[l].x, nullptr, nullptr, W.coarse[0], W.coarse[1], none, w.conv, s);
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
    M.w[0] = W.coarse[0], M.w[1] = W.coarse[1];
    for (int q = 0; q < MG_COARSE_SWEEPS; ++q) M.wc[q] = W.coarsest[q];
    M.lt = lt;
    M.top = top;
    static unsigned long long attr = 0;
    ebk_smem_limit(k_mg_lower<true>, MG_LOWER_SMEM, attr);
    if (L[lt].D.nxy * L[lt].D.nz <= MG_LOWER_CELLS) launch_chained(k_mg_lower<true>, 1, 1024, MG_LOWER_SMEM, s, M, w.conv);
    else launch_chained(k_mg_lower<false>, 1, 1024, 0, s, M, w.conv);
  }
  for (int l = lt - 1; l >= 1; --l) {
    sweep<PROLONG, false>(L[l], L[l].x, &L[l + 1], L[l].t, nullptr, nullptr, 0.f, W.coarse[1], none, w.conv, s);
    sweep<PLAIN, false>(L[l], L[l].t, nullptr, L[l].x, nullptr, nullptr, 0.f, W.coarse[0], none, w.conv, s);
  }
  sweep<PROLONG, false>(L[0], L[0].x, &L[1], L[0].t, nullptr, nullptr, 0.f, W.fine[2], none, w.conv, s);
  sweep<PLAIN, false>(L[0], L[0].t, nullptr, L[0].x, nullptr, nullptr, 0.f, W.fine[1], none, w.conv, s);
  sweep<PLAIN, true>(L[0], L[0].x, nullptr, nullptr, z, r, 0.f, W.fine[0], sum_of(g, rz), w.conv, s);
}

// the scalars of slots first .. last on the host (synchronises the stream)
cudaError_t host_scalars(eb_geom g, int first, int last, double *out, cudaStream_t s) {
  ProjWork &w = g->pw;
  const size_t n = sizeof(double) * (size_t)(last - first + 1);
  cudaError_t e = cudaMemcpyAsync(w.host, w.scal + first, n, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  for (int q = 0; q <= last - first; ++q) out[q] = w.host[q];
  return e;
}

// the mean-free right-hand side of the momenta and its square norm (S_BB)
template <typename T>
void launch_rhs(eb_geom g, void *const mom[3], double dt, cudaStream_t s) {
  ProjWork &w = g->pw;
  const Dims &D = g->D;
  const Slabs S = slabs_of(D, 1, ebk_sm_count());
  k_rhs<T><<<S.blocks(), dim3(MBX, MBY, 1), 0, s>>>(make_op(g), S, (const T *)mom[0], (const T *)mom[1],
                                                   (const T *)mom[2], D.idx / dt, D.idy / dt, D.idz / dt, w.rhs,
                                                   sum_of(g, S_SUM));
  k_center<<<w.nb, PB, 0, s>>>(make_op(g), w.rhs, w.scal + S_SUM, w.scal + S_CNT, sum_of(g, S_BB));
}

template <typename T>
void launch_correct(eb_geom g, void *const mom[3], double dt, cudaStream_t s) {
  ProjWork &w = g->pw;
  const Dims &D = g->D;
  const Slabs S = slabs_of(D, 1, ebk_sm_count());
  k_correct<T><<<S.blocks(), dim3(MBX, MBY, 1), 0, s>>>(make_op(g), S, w.x, dt * D.idx, dt * D.idy, dt * D.idz,
                                                       (T *)mom[0], (T *)mom[1], (T *)mom[2]);
}

void launch_apply(eb_geom g, const double *p, double *q, int it, bool chain, cudaStream_t s) {
  ProjWork &w = g->pw;
  const Slabs S{apply_blocks(g->D, w.ncols), 1, w.aslabs};
  if (w.ncols == 2) launch_chained_if(chain, k_apply<2>, S.blocks(), PB, 0, s, make_op(g), S, p, q, sum_of(g, S_PQ), w.conv, it);
  else launch_chained_if(chain, k_apply<1>, S.blocks(), PB, 0, s, make_op(g), S, p, q, sum_of(g, S_PQ), w.conv, it);
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
  double bb = 0.0;
  CUDA_TRY(host_scalars(g, S_BB, S_BB, &bb, s), "right-hand side");
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
  if (phi0) CUDA_TRY(cudaMemcpyAsync(w.x, phi0, sizeof(double) * N, cudaMemcpyDeviceToDevice, s), "initial guess");
  else CUDA_TRY(cudaMemsetAsync(w.x, 0, sizeof(double) * N, s), "initial guess");
  const bool mg = w.precond == EB_PRECOND_MG;
  if (mg) {
    st = mg_setup(g, s);
    if (st != EB_OK) return st;
  }
  CUDA_TRY(cudaMemsetAsync(w.conv, 0, sizeof(int), s), "reset");
  float *rf = mg ? w.lev[0].b : nullptr;
  k_init<<<w.nb, PB, 0, s>>>(O, phi0 ? w.x : nullptr, w.rhs, w.r, rf, w.p, sum_of(g, S_RZ0), sum_of(g, S_RR));
  if (mg) vcycle(g, w.r, w.p, S_RZ0, s);   // p = z = V(r)
  double h[3] = {0.0, 0.0, 0.0};   // S_BB, S_PQ (not yet formed), S_RR
  CUDA_TRY(host_scalars(g, S_BB, S_RR, h, s), "residual norm");
  const double bb = h[0], rr0 = h[2];
  const double thr2 = rtol * rtol * bb;
  int it = 0;
  double rr = rr0;
  if (bb > 0.0 && rr0 > thr2) {
    int done = 0, next = mg ? 4 : 32;
    const int nb = (int)std::max(1LL, std::min<long long>(w.nb, (N / 2 + PB - 1) / PB));   // two cells per thread
    // Kernels of up to two blocks per SM are launched as a chain (launch_chained):
    // 0.79 of the plain time per Jacobi iteration at 24x24x12, 0.90 at 64x64x32.
    // Beside kernels that fill the GPU the waiting blocks cost more than the
    // launches (1.08 at 130x50x26, 1.14 at 192x192x96), but not beside the many
    // short kernels of a V-cycle.
    const bool chain = mg || nb <= 2 * ebk_sm_count();
    for (it = 0; it < maxit; ++it) {
      const int rz = it % 2 ? S_RZ1 : S_RZ0, rz_next = it % 2 ? S_RZ0 : S_RZ1;
      launch_apply(g, w.p, w.q, it, chain, s);
      if (mg) {
        launch_chained(k_update<false>, nb, PB, 0, s, O, w.q, w.r, rf, w.scal + rz, w.scal + S_PQ, sum_of(g, rz_next),
                                            sum_of(g, S_RR), w.conv, it);
        vcycle(g, w.r, w.z, rz_next, s);
        launch_chained(k_direction<false>, nb, PB, 0, s, O, w.x, w.p, w.z, w.scal + rz, w.scal + rz_next, w.scal + S_PQ,
                                               w.scal + S_RR, thr2, it, w.conv);
      } else {
        launch_chained_if(chain, k_update<true>, nb, PB, 0, s, O, w.q, w.r, nullptr, w.scal + rz, w.scal + S_PQ, sum_of(g, rz_next),
                                           sum_of(g, S_RR), w.conv, it);
        launch_chained_if(chain, k_direction<true>, nb, PB, 0, s, O, w.x, w.p, w.r, w.scal + rz, w.scal + rz_next, w.scal + S_PQ,
                                              w.scal + S_RR, thr2, it, w.conv);
      }
      // The host reads the convergence flag after a first few iterations
      // (fewer with V-cycles, which cost far more than Jacobi iterations),
      // and then where the mean reduction so far says the threshold is met.
      if (it + 1 == next || it + 1 == maxit) {
        int *flag = reinterpret_cast<int *>(w.host + S_SLOTS);
        CUDA_TRY(cudaMemcpyAsync(flag, w.conv, sizeof(int), cudaMemcpyDeviceToHost, s), "convergence flag");
        CUDA_TRY(host_scalars(g, S_RR, S_RR, &rr, s), "convergence flag");
        done = *flag;
        if (done) break;
        const double rate = log(rr0 / rr) / (it + 1), left = log(rr / thr2);
        const double more = rate > 0.0 ? ceil(left / rate) : 1.0;
        next = it + 1 + (int)fmin(fmax(more, 1.0), mg ? 8.0 : 64.0);
      }
    }
    it = done ? done : maxit;
    CUDA_TRY(host_scalars(g, S_RR, S_RR, &rr, s), "residual norm");
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
