// eb_fast.cu -- the bulk kernel (the march itself is in eb_bulk.cuh), the
// pass-through of covered CVs, the work split of the bulk kernel and the
// launchers.
#include "eb_bulk.cuh"

#include <math.h>

#include <algorithm>
#include <functional>
#include <queue>
#include <vector>

namespace {

using namespace bulk;

// One CTA marches the pieces boff[b] .. boff[b+1]-1 of the work split
// (tiles of TYV rows).  The float path is held to EB_BULK_MAXNREG registers
// per thread (96: the fewest without spills), so that beside its two CTAs per
// SM (2 x 256 x 96 of the 65536 registers) the near-EB kernels' blocks still
// find registers on the same SM and run beside the march.
#ifndef EB_BULK_MAXNREG
#define EB_BULK_MAXNREG 96
#endif
template <typename T, int V, int TYV, int TXV>
__global__ void __launch_bounds__(BulkTile<T, TYV, TXV>::NT, (sizeof(T) == 4 ? 2 : 1))
    __maxnreg__(sizeof(T) == 4 ? EB_BULK_MAXNREG : 255) k_fast_tiled(StepArgs<T> A) {
  using P = typename PairOf<T>::type;
  extern __shared__ __align__(16) unsigned char smem_bytes[];
  __shared__ unsigned tm_slot;
  constexpr unsigned NC = BulkTile<T, TYV, TXV>::TMC;
  const unsigned tbase = bulk_tmem_begin<T, bulk_tmem_default<T>(), NC>(&tm_slot);
  P bad = splat(T(0));   // becomes NaN once any written value is not finite
  for (int sgi = A.boff[blockIdx.x]; sgi < A.boff[blockIdx.x + 1]; ++sgi)
    bulk_march<T, V, bulk_tmem_default<T>(), TYV, TXV>(A, A.bseg[sgi], smem_bytes, tbase, bad);
  bulk_tmem_end<T, bulk_tmem_default<T>(), NC>(&tm_slot);
  if (!(isfinite(bad.x) && isfinite(bad.y))) atomicOr(A.status, EB_DEV_NUMERIC);
}

// Pass-through of the CVs no kernel updates (covered CVs and the two wall
// levels of rho*w; zeros when dU itself is written), from per-grid lists
// built at set-up: one thread per listed CV.
// one grid's list per block range (bstart[q] .. bstart[q + 1] - 1); each
// thread copies up to four listed CVs, their loads issued together
struct StaticBlocks {
  unsigned bstart[5];
};
constexpr int STATIC_PER_THREAD = 4;

template <typename T>
__global__ void k_static(StepArgs<T> A, StaticBlocks SB) {
  int q = 0;
  while (q < 3 && blockIdx.x >= SB.bstart[q + 1]) ++q;
  const long long n = A.G[q].nstatic;
  const long long t0 = (long long)(blockIdx.x - SB.bstart[q]) * blockDim.x * STATIC_PER_THREAD + threadIdx.x;
  const unsigned *L = A.G[q].slist;
  const int f0 = q == 0 ? 0 : q + 1, nf = q == 0 ? 2 : 1;
  unsigned c[STATIC_PER_THREAD];
#pragma unroll
  for (int e = 0; e < STATIC_PER_THREAD; ++e) {
    const long long t = t0 + (long long)e * blockDim.x;
    c[e] = t < n ? L[t] : 0xffffffffu;
  }
  for (int f = f0; f < f0 + nf; ++f) {
    T v[STATIC_PER_THREAD];
#pragma unroll
    for (int e = 0; e < STATIC_PER_THREAD; ++e)
      v[e] = (c[e] != 0xffffffffu && A.base[0]) ? A.base[f][c[e]] : T(0);
#pragma unroll
    for (int e = 0; e < STATIC_PER_THREAD; ++e)
      if (c[e] != 0xffffffffu) A.out[f][c[e]] = v[e];
  }
}

template <typename T, int V, int TYV, int TXV>
void set_smem_attr() {
  static unsigned long long done = 0;
  ebk_smem_limit(k_fast_tiled<T, V, TYV, TXV>, (int)BulkTile<T, TYV, TXV>::BYTES, done);
}

template <typename T, int V, int TYV, int TXV = 32>
void launch_bulk(const StepArgs<T> &A, cudaStream_t s) {
  using TL = BulkTile<T, TYV, TXV>;
  if (A.bctas < 1) return;
  set_smem_attr<T, V, TYV, TXV>();
  k_fast_tiled<T, V, TYV, TXV><<<A.bctas, dim3(TL::NPX, TL::TY, 1), TL::BYTES, s>>>(A);
}

template <typename T>
int resident_ctas_per_sm() {
  constexpr int V = 16 / sizeof(T);
  set_smem_attr<T, V, 16, 32>();   // every variant set here, outside any graph capture
  set_smem_attr<T, 1, 16, 32>();
  if constexpr (sizeof(T) == sizeof(float)) {
    set_smem_attr<T, V, 14, 32>();
    set_smem_attr<T, 1, 14, 32>();
  } else {
    set_smem_attr<T, V, 8, 16>();
    set_smem_attr<T, 1, 8, 16>();
  }
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_fast_tiled<T, V, 16, 32>, BulkTile<T>::NT,
                                                    BulkTile<T>::BYTES) != cudaSuccess ||
      n < 1)
    n = 1;
  return n;
}

}  // namespace

namespace {

// Lockstep slabs: every tile is cut at the same levels, and the pieces are
// launched slab by slab from the top, so CTAs of neighbouring tiles march
// the same levels at the same time and read each other's halo from L2; the
// short pieces of the lowest slabs come last.  piece(tile, first, end).
template <typename F>
void for_pieces(const Dims &D, const std::vector<int> &kb, long long Lc, F &&piece) {
  const int nslab = (int)((D.nz + Lc - 1) / Lc);
  for (int sl = nslab - 1; sl >= 0; --sl) {
    const int za = (int)(sl * Lc), zb = (int)std::min<long long>(D.nz, (sl + 1) * Lc);
    for (size_t t = 0; t < kb.size(); ++t) {
      const int a = std::max(za, kb[t]);
      if (a < zb) piece((int)t, a, zb);
    }
  }
}

// lowest kfast of every tile of TX x TY columns
std::vector<int> tile_bottoms(const Dims &D, const int *kfast, int TX, int TY) {
  const int tx = (D.nx + TX - 1) / TX, ty = (D.ny + TY - 1) / TY;
  std::vector<int> kb((size_t)tx * ty, D.nz);
  for (int j = 0; j < D.ny; ++j)
    for (int i = 0; i < D.nx; ++i) {
      int &v = kb[(i / TX) + (size_t)tx * (j / TY)];
      v = std::min(v, kfast[i + (long long)D.nx * j]);
    }
  return kb;
}

// Time of a split on the double path when the pieces start in order on
// `slots` SMs: a piece costs `start` (its two prologue levels, copies and
// fill) plus `level` per level.
double split_time(const Dims &D, const std::vector<int> &kb, long long Lc, int slots, double start, double level) {
  std::vector<double> heap((size_t)slots, 0.0);   // min-heap of the slots' finishing times
  double end = 0.0;
  for_pieces(D, kb, Lc, [&](int, int a, int b) {
    std::pop_heap(heap.begin(), heap.end(), std::greater<double>());
    heap.back() += start + level * (b - a);
    end = std::max(end, heap.back());
    std::push_heap(heap.begin(), heap.end(), std::greater<double>());
  });
  return end;
}

// The float path's march with two CTAs per SM, in units of the time a CTA alone
// on its SM takes per level: a piece costs its levels and three of prologue, and
// of two CTAs on an SM each runs 1.1 times slower.  end: when the last piece is
// done, the pieces starting in order; busy: the SMs' time in it, per SM.
struct MarchTime {
  double end = 0.0, busy = 0.0;
  long long pieces = 0;
};
constexpr int kMarchCtas = 2;   // by registers and shared memory (the occupancy query counts tensor memory and says 1)
constexpr double kMarchShared = 1.1;
// pieces and busy
MarchTime march_work(const Dims &D, const std::vector<int> &kb, long long Lc, int sms) {
  MarchTime M;
  long long levels = 0;
  for_pieces(D, kb, Lc, [&](int, int a, int b) {
    ++M.pieces;
    levels += 3 + (b - a);
  });
  M.busy = (double)levels * kMarchShared / kMarchCtas / sms;
  return M;
}
// end
double march_end(const Dims &D, const std::vector<int> &kb, long long Lc, int sms) {
  std::vector<double> cost;
  for_pieces(D, kb, Lc, [&](int, int a, int b) { cost.push_back(3.0 + (b - a)); });
  struct Sm {
    double left[kMarchCtas], at;   // what its CTAs have left at time at
    int n;
  };
  std::vector<Sm> sm(sms, Sm{{}, 0.0, 0});
  size_t next = 0;
  for (int q = 0; q < kMarchCtas; ++q)
    for (int i = 0; i < sms && next < cost.size(); ++i) sm[i].left[sm[i].n++] = cost[next++];
  using Event = std::pair<double, int>;   // an SM's next finish
  std::priority_queue<Event, std::vector<Event>, std::greater<Event>> events;
  auto slow = [](int n) { return n > 1 ? kMarchShared : 1.0; };
  auto push = [&](int i) {
    const Sm &S = sm[i];
    if (S.n) events.push({S.at + *std::min_element(S.left, S.left + S.n) * slow(S.n), i});
  };
  for (int i = 0; i < sms; ++i) push(i);
  double end = 0.0;
  while (!events.empty()) {
    const auto [t, i] = events.top();
    events.pop();
    Sm &S = sm[i];
    const double done = (t - S.at) / slow(S.n);
    S.at = end = t;
    int n = 0;
    for (int q = 0; q < S.n; ++q)
      if (S.left[q] - done > 1e-9) S.left[n++] = S.left[q] - done;
    while (n < kMarchCtas && next < cost.size()) S.left[n++] = cost[next++];
    S.n = n;
    push(i);
  }
  return end;
}

}  // namespace

cudaError_t bulk_plan(const Dims &D, const int *kfast_host, bool f64, int slab_levels, int tile_rows, bool alone,
                      bool rows_free, long long near_cvs, std::vector<int> &seg, std::vector<int> &off, int &plan_rows) {
  plan_rows = tile_rows;
  std::vector<int> kb = tile_bottoms(D, kfast_host, 32, tile_rows);
  long long W = 0;
  for (int k : kb) W += std::max(0, D.nz - k);
  seg.clear();
  off.assign(1, 0);
  if (W == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  sms = std::max(sms, 1);
  const long long slots = (long long)sms * (f64 ? resident_ctas_per_sm<double>() : resident_ctas_per_sm<float>());
  // Slabs of slab_levels levels, or (0) of at least 16 levels sized for
  // about three waves of CTAs.
  long long Lc = slab_levels > 0 ? (long long)slab_levels : std::max(16LL, (W + 3 * slots - 1) / (3 * slots));
  if (slab_levels == 0 && !f64 && alone) {
    // Float path alone on the GPU: the near-EB kernels run beside the march,
    // so a step ends no sooner than the march by itself (short slabs fill
    // every SM to the end) and than both kinds of work together take the whole
    // GPU (tall slabs have fewer prologues).  The height, of at least eight
    // levels, with the smallest eighth-power mean of the two.  The near-EB and
    // redistribution kernels take 0.025 levels' time per 1000 near-EB CVs, a fifth
    // more where the march has pieces waiting for SMs until late in the step.
    // The constants are the best over 102 domains of 15 thousand to 34 million
    // cells, hills and random terrain, one and three stages: steps take 0.66 to
    // 1.16 times those of slabs of three waves, 0.90 in the mean, and 1.7 % more
    // than with the best height of each.  (A rule of about 1.5 whole CTAs per
    // SM in one wave, or eight levels where that left SMs idle, was 4.7 % above
    // the best in the mean and up to 1.39 times slabs of three waves: 750 us
    // instead of 570 on a 400x400x128 hill, 127 instead of 110 on 320x200x30.)
    const double near = 2.5e-5 * (double)near_cvs / sms * 152;   // in levels, on this GPU's SMs
    double best = 0.0;
    auto consider = [&](long long L) {
      const MarchTime M = march_work(D, kb, L, sms);
      double c = pow(M.busy + near * (M.pieces > (long long)kMarchCtas * sms ? 1.2 : 1.0), 8);
      if (best > 0.0 && c >= best) return;
      c += pow(march_end(D, kb, L, sms), 8);
      if (best == 0.0 || c < best) best = c, Lc = L;
    };
    // heights of 1, 2, ... slabs, at least 15 % apart, and of 16 and 8 levels;
    // splits of more than 16 waves are only taken whole
    const long long tiles = (long long)kb.size(), most = 16LL * kMarchCtas * sms;
    for (long long n = 1; n == 1 || (D.nz / n >= 8 && tiles * n <= most); n = std::max(n + 1, n * 115 / 100))
      consider((D.nz + n - 1) / n);
    for (long long L : {16, 8})
      if (L < D.nz && tiles * ((D.nz + L - 1) / L) <= most) consider(L);
  }
  if (slab_levels == 0 && f64 && alone) {
    // Double path alone on the GPU: the height (and for small domains the
    // 16 x 8 tile) of the shortest estimated time for one CTA per SM: 39 us +
    // 23.7 per level for a 32 x 16 tile; 28 + 13.7 per level for a 16 x 8 tile
    // (four of them per 32 x 16 tile, each cheaper in time but not in FP64
    // instructions: more halo), which is taken only while every piece has an
    // SM of its own, and not where the caller set the rows.  (The constants
    // were measured with a reciprocal that made all four about 6 % shorter.)
    // The kernel alone, 32x32x16 ridge: 364 us with one slab of 32 x 16 tiles,
    // 71 with one level per piece, 46 with 16 x 8 tiles; 64x64x32 hill: 439 in
    // slabs of 16 levels, 97 of two; 256x256x128 hill: 3273 in slabs of 32, 3056
    // of 16.
    double best = split_time(D, kb, Lc, sms, 39.0, 23.7);
    const std::vector<int> ks = tile_bottoms(D, kfast_host, 16, 8);
    for (long long L : {1, 2, 3, 4, 6, 8, 12, 16, 24, 32}) {
      if (L > D.nz) break;
      const double t = split_time(D, kb, L, sms, 39.0, 23.7);
      if (t < best) best = t, Lc = L, plan_rows = tile_rows;
      long long pieces = 0;
      for_pieces(D, ks, L, [&](int, int, int) { ++pieces; });
      if (rows_free && pieces <= sms && 28.0 + 13.7 * L < best) best = 28.0 + 13.7 * L, Lc = L, plan_rows = 8;
    }
    if (plan_rows == 8) kb = ks;
  }
  for_pieces(D, kb, Lc, [&](int t, int a, int zb) {
    seg.push_back(t);
    seg.push_back(a);
    seg.push_back(zb);
    seg.push_back(0);
    off.push_back((int)(seg.size() / 4));
  });
  return cudaGetLastError();
}

template <typename T>
void launch_flux_bulk(const StepArgs<T> &A, cudaStream_t s);

template <typename T>
void launch_static_copy(const StepArgs<T> &A, cudaStream_t s) {
  const Dims &D = A.D;
  if (A.copy_static) {
    StaticBlocks SB;
    SB.bstart[0] = 0;
    for (int q = 0; q < 4; ++q)
      SB.bstart[q + 1] = SB.bstart[q] + (unsigned)((A.G[q].nstatic + 256 * STATIC_PER_THREAD - 1) /
                                                   (256 * STATIC_PER_THREAD));
    if (SB.bstart[4] > 0) k_static<T><<<SB.bstart[4], 256, 0, s>>>(A, SB);
  }
}

template <typename T>
void launch_flux_fast(const StepArgs<T> &A, cudaStream_t s) {
  launch_static_copy(A, s);
  launch_flux_bulk(A, s);
}

template <typename T>
void launch_flux_bulk(const StepArgs<T> &A, cudaStream_t s) {
  const Dims &D = A.D;
  // 16-byte copies and pair stores need every row of every field to start on
  // a 16-byte boundary: nx a multiple of the copy width and aligned pointers
  constexpr int V = 16 / sizeof(T);
  bool vec = D.nx % V == 0;
  for (int f = 0; f < 5; ++f) {
    vec = vec && ((uintptr_t)A.src.f[f] % 16 == 0) && ((uintptr_t)A.out[f] % 16 == 0);
    if (A.base[0]) vec = vec && ((uintptr_t)A.base[f] % 16 == 0);
  }
  if constexpr (sizeof(T) == sizeof(float)) {   // 14-row tiles on the float path only
    if (A.tile_rows == 14) {
      if (vec) launch_bulk<T, V, 14>(A, s);
      else launch_bulk<T, 1, 14>(A, s);
      return;
    }
  } else {   // 16 x 8 tiles on the double path only
    if (A.tile_rows == 8) {
      if (vec) launch_bulk<T, V, 8, 16>(A, s);
      else launch_bulk<T, 1, 8, 16>(A, s);
      return;
    }
  }
  if (vec) launch_bulk<T, V, 16>(A, s);
  else launch_bulk<T, 1, 16>(A, s);
}

template void launch_flux_fast<double>(const StepArgs<double> &, cudaStream_t);
template void launch_flux_fast<float>(const StepArgs<float> &, cudaStream_t);
template void launch_static_copy<double>(const StepArgs<double> &, cudaStream_t);
template void launch_static_copy<float>(const StepArgs<float> &, cudaStream_t);
template void launch_flux_bulk<double>(const StepArgs<double> &, cudaStream_t);
template void launch_flux_bulk<float>(const StepArgs<float> &, cudaStream_t);
