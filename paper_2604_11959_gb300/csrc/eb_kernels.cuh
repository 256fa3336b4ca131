// eb_kernels.cuh -- host-side launch wrappers shared between the library's
// translation units.  Not part of the ABI.
#pragma once

#include "eb_internal.cuh"

#include <vector>

// Compact redistribution tables of one grid (Sec. 5.1) as the set-up builds
// them; only the counts outlive it (the step reads WsrdTab).
struct WsrdDev {
  long long nsmall = 0, naff = 0, nlsq = 0, nw = 0;
  int *sid = nullptr;             // [nrec] small id of a record, -1 if not small
  // per small CV
  long long *s_lin = nullptr;     // state index
  long long *s_rec = nullptr;     // record
  int *s_nmem = nullptr;          // members incl. itself (<= 8)
  int *s_piv = nullptr;           // pivot member of the deviation form
  long long *s_plin = nullptr;    // state index of the pivot member
  long long *s_mlin = nullptr;    // [8 * nsmall] member state indices (slot 0: itself)
  double *s_mw = nullptr;         // [8 * nsmall] Qhat weights (sum 1)
  double *s_me = nullptr;         // [24 * nsmall] member centroid - xhat (limiter points)
  long long *s_loff = nullptr;    // [nsmall + 1] LSQ stencil offsets
  long long *l_lin = nullptr;     // [nlsq] stencil CV state index
  int *l_sid = nullptr;           // [nlsq] small id of the stencil CV or -1
  long long *l_plin = nullptr;    // [nlsq] pivot state index of that small CV, else the CV's own index
  double *l_c = nullptr;          // [3 * nlsq] gradient coefficient rows
  // per affected CV
  long long *a_lin = nullptr;
  int *a_sid = nullptr;           // own small id or -1
  double *a_eself = nullptr;      // [3 * naff] own centroid - own xhat
  long long *a_woff = nullptr;    // [naff + 1]
  int *w_sid = nullptr;           // [nw] small CV r whose neighbourhood holds the CV
  double *w_k = nullptr;          // [nw] kappa_r / N_i
  double *w_e = nullptr;          // [3 * nw] x_i - xhat_r (cell units, relative to r)
};

// The same tables as the step reads them, weights in the state's precision
// T, each component in an array of its own: entry e of small CV s at [e * ns +
// s], the lists of uneven length one after another (several lanes share a
// list, so a warp reads one contiguous run).  Indices are 32 bit (grids hold
// fewer than 2^32 CVs).  A tag holds a small id + 1 (0: none) in its low 28
// bits and a level difference + 8 in the upper 4, which replaces looking up
// the reference profiles at both levels (see WsrdArgs::rdiff).
struct WsrdTab {
  long long ns = 0, na = 0;       // small, affected CVs
  long long nl = 0, nw = 0;       // entries of the two lists
  void *block = nullptr;          // the device memory of all arrays
  unsigned *plin = nullptr;       // [ns] state index of the pivot member
  uint8_t *nmem = nullptr;        // [ns] members incl. itself (<= 8) | pivot member << 4
  unsigned *mlin = nullptr;       // [8][ns] members' state indices
  void *mw = nullptr;             // [8][ns] weights of Qhat
  void *me = nullptr;             // [24][ns] limiter points: member q, direction d at [3 q + d]
  long long *loff = nullptr;      // [ns + 1]
  unsigned *lplin = nullptr;      // [nl] pivot state index of the stencil CV
  unsigned *ltag = nullptr;       // [nl] its small id; level of lplin - level of the CV's own pivot
  void *lc = nullptr;             // [3][nl] gradient coefficients
  unsigned *alin = nullptr;       // [na] state index
  unsigned *atag = nullptr;       // [na] own small id; level of its pivot - own level
  void *es = nullptr;             // [3][na] own centroid - own xhat
  long long *woff = nullptr;      // [na + 1]
  unsigned *wtag = nullptr;       // [nw] small CV r whose neighbourhood holds the CV; level of r's pivot - level of
                                  // the CV's (its own, when it is not small)
  void *wk = nullptr;             // [nw] kappa_r / N_i
  void *we = nullptr;             // [3][nw] x_i - xhat_r
};

// eb_geom.cu
void launch_band_bounds(const double *h, const Dims &D, int g, int *kcov, int *kreg, cudaStream_t s);
void launch_band_top(const Dims &D, int nzg, const int *kcov, const int *kreg, int *kxt, long long *count,
                     cudaStream_t s);
void launch_fluid_level(const Dims &D, const GridDev &G, int *kflu, cudaStream_t s);
void launch_fast_level(const Dims &D, const int *const kreg[4], const int *const kflu[4], int *kfast,
                       cudaStream_t s);
void launch_band_geometry(const double *h, const Dims &D, int g, const GridDev &G, cudaStream_t s);
// two-level refinement (eb_amr.cu): band bounds and geometry records of a
// coarse level (Dc) merged from the c grid of the fine level (Df, Gf), and
// its nodal heights as every other fine node
void launch_coarse_bounds(const Dims &Df, const GridDev &Gf, const Dims &Dc, int g, int *kcov, int *kreg,
                          cudaStream_t s);
void launch_coarse_geometry(const Dims &Df, const GridDev &Gf, const Dims &Dc, int g, const GridDev &Gc,
                            cudaStream_t s);
void launch_subsample_heights(const double *hf, const Dims &Df, double *hc, const Dims &Dc, cudaStream_t s);
void launch_dense_flags(const Dims &D, int g, const GridDev &G, cudaStream_t s);
void launch_band_marks(const Dims &D, int g, const int *kcov, const int *kfast, int kmax, long long *mark,
                       cudaStream_t s);
void launch_band_fill(const Dims &D, int g, const int *kcov, const int *kfast, int kmax, const long long *pos,
                      unsigned *list, cudaStream_t s);
void launch_face_marks(const Dims &D, int g, const GridDev &G, uint8_t *m0, uint8_t *m1, uint8_t *m2, cudaStream_t s);
void launch_marks_to_counts(const uint8_t *m, long long n, long long *cnt, cudaStream_t s);
void launch_marks_fill(const uint8_t *m, long long n, const long long *pos, unsigned *list, cudaStream_t s);
void launch_export_geometry(const double *h, const Dims &D, int g, const GridDev &G, int field, double *dst,
                            cudaStream_t s);

// eb_step.cu: near-EB rows of grid g (CVs with a record), two passes: the
// term count of every (row, direction) segment into cnt[3t + d], then (after
// the scan of cnt and the allocation of G[g].sidx / scoef / scoef_f / stiny)
// the terms themselves at the scanned offsets
void launch_band_rows(const Dims &D, const GridDev G[4], int g, bool fill, long long *cnt, cudaStream_t s);
void launch_rows_to_u32(const long long *src, long long n, unsigned *dst, cudaStream_t s);
// eb_step.cu: availability bits of every listed face into G[q].fmask[d]
void launch_face_masks(const Dims &D, const GridDev G[4], cudaStream_t s);
// eb_step.cu: marks[q][idx] = 1 for every CV of grid q a listed face's
// stencil reads (marks[q] covers levels below G[q].nst)
void launch_stage_marks(const Dims &D, const GridDev G[4], uint8_t *const marks[4], cudaStream_t s);

// eb_fast.cu: split of the bulk kernel's (tile, level) work into lockstep
// slabs of slab_levels levels (0: chosen from the GPU's size); seg holds
// (tile, first level, end level, 0) per piece, off[b] .. off[b+1] the pieces
// of CTA b
// alone: the kernel has the GPU to itself (not one member of an ensemble's step); rows_free: the caller has not set tile_rows;
// near_cvs: near-EB CVs of the four grids (the kernels beside the march); plan_rows: rows of the split's tiles, tile_rows
// or 8 (16 x 8 tiles: double path, automatic height, free rows, small domains)
cudaError_t bulk_plan(const Dims &D, const int *kfast_host, bool f64, int slab_levels, int tile_rows, bool alone,
                      bool rows_free, long long near_cvs, std::vector<int> &seg, std::vector<int> &off, int &plan_rows);

// eb_scan.cu: in-place exclusive scan of n values; total written to *total (device)
void scan_exclusive(long long *data, long long n, long long *total, cudaStream_t s);

// eb_wsrd_setup.cu
struct SetupScratch;
cudaError_t build_wsrd(const Dims &D, int g, GridDev &G, const GridDev *all, double vt, WsrdDev &W,
                       cudaStream_t s, long long *dev_tmp);
void free_wsrd(WsrdDev &W);   // the arrays; the counts stay
// the step's tables from the set-up's (f64: weights in double, else float)
cudaError_t pack_wsrd(const Dims &D, const WsrdDev &W, bool f64, WsrdTab &T, cudaStream_t s);
void free_wsrd_tab(WsrdTab &T);
// sets *far when a CV the redistribution of grid g reads or writes is not a
// near-EB CV (see k_wsrd_reach)
void launch_wsrd_reach(const Dims &D, int g, const WsrdDev &W, const int *kcov, const int *kfast, unsigned *far,
                       cudaStream_t s);

// device allocation helper that tracks every pointer for one release
struct DevArena;
