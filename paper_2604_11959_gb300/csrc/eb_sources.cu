// eb_sources.cu -- the sources of the compressible system (Sec. 2.1, Eq.
// mom-comp) that eb_step adds to the flux divergence of every stage when the
// handle asks for them (eb_geom_set_sources):
//   -grad p' on the momentum grids, p' = p - p0(z) the perturbation pressure,
//            p from the equation of state p = P00 (R rho theta / P00)^gamma;
//   B = -rho' g on rho*w (buoyancy).
// Pressure and density live at cell centres; every momentum CV sits between
// the cell e_d back along its staggering axis d (a) and the cell of the same
// index (b): its source is -(p'_b - p'_a) / dx_d, and on w also
// -g (rho'_a + rho'_b) / 2.  A covered cell takes the other cell's value (no
// pressure force across a wall side).  The source enters the CV's dU as it
// stands, after the flux divergence and before the redistribution.
//
// States hold perturbations about the reference profiles, so
//   p' = p0(k) * expm1(gamma * log1p((rho theta)' / (rho0 theta0)(k)))
// (the deviation form of p - p0: the float path rounds p', not p ~ 1e5 Pa);
// p0(k) and 1 / (rho0 theta0)(k) are per-level tables built in double when
// the sources are switched on.
#include "eb_step.cuh"

#include <algorithm>

namespace {

template <typename T>
struct SourceArgs {
  Dims D;
  const int *kfast;          // from here up a column's cells, and theirs to the low sides, hold fluid
  const uint8_t *cflag;      // dense flags of the c grid (bit 0: holds fluid)
  const uint8_t *gflag[3];   // of the u, v, w grids
  const T *rho, *rt;         // rho', (rho theta)' of the stage's source state
  T *out[3];                 // rho*u, rho*v, rho*w of the stage's output
  const T *p0, *irt0;        // per level: p0, 1 / (rho0 theta0)
  T *pp;                     // double path: p' of every fluid cell (written by k_pressure)
  T dt, gamma, grav, inv[3];
  int pressure, buoyancy;
  int strips, tiles, slabs;  // y strips, x tiles and z slabs of k_sources
  unsigned *status;
};

__device__ inline float log1p_t(float x) { return log1pf(x); }
__device__ inline double log1p_t(double x) { return log1p(x); }
__device__ inline float expm1_t(float x) { return expm1f(x); }
__device__ inline double expm1_t(double x) { return expm1(x); }

template <typename T>
__device__ inline T p_prime(const SourceArgs<T> &S, long long c, int k) {
  return S.p0[k] * expm1_t(S.gamma * log1p_t(S.rt[c] * S.irt0[k]));
}

// double path: p' of every cell that holds fluid, once per stage (FP64
// logarithms and exponentials are what this costs, so none is formed twice)
template <typename T>
__global__ void k_pressure(const __grid_constant__ SourceArgs<T> S) {
  const Dims &D = S.D;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= D.nxy * (long long)D.nz) return;
  if (!(S.cflag[t] & 1)) return;
  S.pp[t] = p_prime(S, t, (int)D.fnxy.div((unsigned)t));
}

// The sources of the u and v CVs of levels 0 .. nz - 1 and the w CVs of face
// levels 1 .. nz - 1.  It reads rho', (rho theta)' and the three momenta and
// writes the momenta, 32 bytes per cell in float, so one pass does all: a block marches a tile of 32 x SR columns up a slab of levels, one
// column per thread.  Each level's p' is formed once per cell into a shared
// plane (two planes, one barrier per level) with the cells beside the tile's
// low x and y sides; the level below stays in registers.  From a column's
// kfast up no flag is read.  Every load of a level precedes its stores, which
// might alias them for all the compiler knows.  256x256x128, float: 80 us (a
// pass that stored p' and one that read it took 40 + 126).  The logarithms and
// exponentials bound it on the float path too: its 268 MB are 40 us.
constexpr int SR = 8;

template <typename T, bool STORED>
__global__ void __launch_bounds__(32 * SR) k_sources(const __grid_constant__ SourceArgs<T> S) {
  const Dims &D = S.D;
  __shared__ T sp[2][SR + 1][33];   // p' at (row, column) = (ty + 1, tx + 1)
  const int tx = threadIdx.x, ty = threadIdx.y;
  int w = blockIdx.x;
  const int slab = w / (S.tiles * S.strips);
  w -= slab * S.tiles * S.strips;
  const int strip = w / S.tiles, i0 = (w - strip * S.tiles) * 32, j0 = strip * SR;
  const int k0 = (int)((long long)D.nz * slab / S.slabs), k1 = (int)((long long)D.nz * (slab + 1) / S.slabs);
  const bool in = i0 + tx < D.nx && j0 + ty < D.ny;
  const int i = min(i0 + tx, D.nx - 1), j = min(j0 + ty, D.ny - 1);
  const int col = i + D.nx * j;
  const int cl = i == 0 ? col + D.nx - 1 : col - 1, cd = j == 0 ? col + D.nx * (D.ny - 1) : col - D.nx;
  const int kf = S.kfast[col];
  // cells beside the tile: row ty == 0 forms those below it, row ty == 1 (its first SR lanes) those left of it
  int hc = -1, hy = 0, hx = 0, hkf = 0;
  if (ty == 0) {
    hc = cd;
    hx = tx + 1;
  } else if (ty == 1 && tx < SR) {
    hc = (i0 == 0 ? D.nx - 1 : i0 - 1) + D.nx * min(j0 + tx, D.ny - 1);
    hy = tx + 1;
  }
  if (hc >= 0) hkf = S.kfast[hc];

  auto value = [&](long long c, int k) -> T {
    if constexpr (STORED) return S.pp[c];
    else return p_prime(S, c, k);
  };
  T pz = T(0), rz = T(0);
  bool fz = false, bad = false;
  if (k0 > 0) {
    const long long c = col + D.nxy * (long long)(k0 - 1);
    fz = k0 - 1 >= kf || (S.cflag[c] & 1);
    if (fz && S.pressure) pz = value(c, k0 - 1);
    rz = S.rho[c];
  }
  for (int k = k0; k < k1; ++k) {
    const long long b = D.nxy * (long long)k, t = col + b;
    const bool all = k >= kf;   // the cells and CVs this column's sources read hold fluid
    const bool own = all || (S.cflag[t] & 1);
    T m[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) m[d] = S.out[d][t];
    const T rho = S.rho[t];
    T p = T(0);
    T(*P)[33] = sp[k & 1];
    if (S.pressure) {
      if (own) p = value(t, k);
      P[ty + 1][tx + 1] = p;
      if (hc >= 0 && (k >= hkf || (S.cflag[hc + b] & 1))) P[hy][hx] = value(hc + b, k);
      __syncthreads();
    }
    if (in) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (d == 2 && k == 0) continue;
        bool fa = true;
        if (!all) {
          fa = d == 2 ? fz : S.cflag[(d == 0 ? cl : cd) + b] & 1;
          if (!(S.gflag[d][t] & 1) || (!fa && !own)) continue;
        }
        T s = T(0);
        if (S.pressure) {
          T pa = d == 0 ? P[ty + 1][tx] : d == 1 ? P[ty][tx + 1] : pz;
          if (!fa) pa = p;
          const T pb = own ? p : pa;
          s -= (pb - pa) * S.inv[d];
        }
        if (S.buoyancy && d == 2) {
          const T ra = fa ? rz : rho;
          const T rb = own ? rho : ra;
          s -= S.grav * T(0.5) * (ra + rb);
        }
        const T v = m[d] + S.dt * s;
        S.out[d][t] = v;
        bad = bad || !isfinite(v);
      }
    }
    pz = p;
    rz = rho;
    fz = own;
  }
  if (bad) atomicOr(S.status, EB_DEV_NUMERIC);
}

}  // namespace

template <typename T>
void launch_sources(const StepArgs<T> &A, int flags, const T *p0, const T *irt0, T *pp, cudaStream_t s) {
  SourceArgs<T> S;
  S.D = A.D;
  S.kfast = A.kfast;
  S.cflag = A.G[0].dflag;
  for (int d = 0; d < 3; ++d) {
    S.gflag[d] = A.G[d + 1].dflag;
    S.out[d] = A.out[d + 2];
  }
  S.rho = A.src.f[0];
  S.rt = A.src.f[1];
  S.p0 = p0;
  S.irt0 = irt0;
  S.pp = pp;
  S.dt = A.dtT;
  S.gamma = (T)(EB_CP / (EB_CP - EB_RD));
  S.grav = (T)EB_GRAV;
  S.inv[0] = (T)A.D.idx;
  S.inv[1] = (T)A.D.idy;
  S.inv[2] = (T)A.D.idz;
  S.pressure = (flags & EB_SOURCE_PRESSURE) ? 1 : 0;
  S.buoyancy = (flags & EB_SOURCE_BUOYANCY) ? 1 : 0;
  S.status = A.status;
  constexpr bool STORED = sizeof(T) == sizeof(double);
  if (STORED && S.pressure) {
    const long long nc = A.D.nxy * (long long)A.D.nz;
    k_pressure<T><<<(unsigned)((nc + 255) / 256), 256, 0, s>>>(S);
  }
  // slabs of at least four levels (each re-forms the level below its first),
  // enough of them for about SOURCE_BLOCKS blocks per SM
  constexpr long long SOURCE_BLOCKS = 16;
  S.tiles = (A.D.nx + 31) / 32;
  S.strips = (A.D.ny + SR - 1) / SR;
  const long long cols = (long long)S.tiles * S.strips;
  S.slabs = (int)std::max(1LL, std::min<long long>(A.D.nz / 4, (SOURCE_BLOCKS * ebk_sm_count() + cols - 1) / cols));
  k_sources<T, STORED><<<(unsigned)(cols * S.slabs), dim3(32, SR, 1), 0, s>>>(S);
}

template void launch_sources<float>(const StepArgs<float> &, int, const float *, const float *, float *,
                                    cudaStream_t);
template void launch_sources<double>(const StepArgs<double> &, int, const double *, const double *, double *,
                                     cudaStream_t);
