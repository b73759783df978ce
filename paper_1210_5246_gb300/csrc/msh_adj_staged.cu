// msh_adj_staged.cu -- the reverse steps of a checkpoint segment as grid-wide stages in one
// persistent cooperative launch (the adjoint's counterpart of msh_staged.cuh).
//
// For grids that take the staged step, and segments none of whose steps tagged fallback
// cells.  Per reverse step n (frozen branches, the forward state U^n in seg):
//   R0  per cell: primitive variables of U^n; lam <- lam* = G^T lam^{n+1} (gravity source)
//   A   per cell and direction: the face states lo, hi again (stage A of the step)
//   R2  per face: the HLL flux's adjoint, F^bar = (dt/dx)(lam*_i - lam*_{i-1}); the adjoint
//       of the left face state replaces hi_{i-1}, that of the right one lo_i (only this face
//       reads them)
//   R3  per cell and direction (and per ghost cell of a side that is not periodic): the
//       reconstruction's adjoint; what it gives to the cells before and after replaces lo
//       and hi, what it gives to the cell itself goes to self
//   R4  per cell: the sum of what its own and its neighbours' reconstructions gave to it, and
//       to the ghost cells that are its images, through the conversion to primitives:
//       lam <- lam* + (dW/dU)^T W^bar; then R0 of step n-1
// A face or cell is reversed once, where the pencil kernels reverse 26 of the 32 positions a
// warp holds and fill whole blocks (128^2 FP64, per direction: 96 blocks of 8 warps on 152
// SMs, 120 us, against 48 us of double-precision instructions spread evenly).
#include "msh_adjoint.cuh"
#include "msh_staged.cuh"

namespace msh {

template <typename T> struct StagedAdjArgs {
  StagedArgs<T> a;     // a.seg: states of the segment, a.dts: its time steps, face-state buffers
  T *lam;              // [NV][N]: lam^{n0+len} in, lam^{n0} out
  T *self[3];          // per direction [NV][N]
  T *gself, *gout;     // ghost cells: self and outward parts, [2 ndim][NV][max_pencils] each
  int len;             // reverse steps n0+len-1 .. n0
};

// lam* of cell c to lam, primitive state to W (stage R0).
template <typename T>
__device__ __forceinline__ void reverse_prepare(const StagedAdjArgs<T> &g, const T *U, T dt, size_t N, int c) {
  const StepArgs<T> &s = g.a.s;
  T u[NV], w[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) u[k] = U[k * N + c];
  cons_to_prim(u, w);
#pragma unroll
  for (int k = 0; k < NV; k++) g.a.W[0][k * N + c] = w[k];
  if (s.acc != nullptr) {
    T l[NV], ls[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) l[k] = g.lam[k * N + c];
    const T acc[3] = {s.acc[c], s.acc[N + c], s.acc[2 * N + c]};
    gravity_vjp(acc, dt, l, ls);
#pragma unroll
    for (int k = 0; k < NV; k++) g.lam[k * N + c] = ls[k];
  }
}

// Stage R2 of the lower face of cell `item` along D, or (upper) of the upper boundary face of
// pencil `item`.
template <typename T, int D>
__device__ __forceinline__ void reverse_face(const StagedAdjArgs<T> &g, size_t N, T dtdx, int item, bool upper) {
  const StepArgs<T> &s = g.a.s;
  const int nx = s.nx, ny = s.ny, n = axis_n<D>(s.nx, s.ny, s.nz), st = D == 0 ? 1 : D == 1 ? nx : nx * ny;
  T *lo = g.a.lo + (size_t)D * NV * N, *hi = g.a.hi + (size_t)D * NV * N;
  T *pl, *pr;
  size_t sl = N, sr = N;
  int cl = -1, cr = -1;  // the cells whose lam* enter (a ghost cell is not updated: none)
  if (!upper) {
    if (item >= (int)N) return;
    const int i = coord<D>(item, nx, ny);
    cr = item;
    pr = lo + item;
    if (i > 0 || s.bc[2 * D] == BC_PERIODIC) {
      cl = i > 0 ? item - st : item + (n - 1) * st;
      pl = hi + cl;
    } else {
      pl = g.a.ghost + (size_t)(2 * D) * NV * g.a.max_pencils + pencil_of<D>(item, nx, ny);
      sl = g.a.max_pencils;
    }
  } else {
    if (item >= (int)(N / n)) return;
    cl = pencil_cell<D>(item, nx, ny) + (n - 1) * st;
    pl = hi + cl;
    pr = g.a.ghost + (size_t)(2 * D + 1) * NV * g.a.max_pencils + item;
    sr = g.a.max_pencils;
  }
  T wl[NV], wr[NV], Fb[NV], hb[NV], lb[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) {
    const size_t gk = (size_t)Frame<D>::g(k) * N;
    wl[k] = pl[k * sl];
    wr[k] = pr[k * sr];
    Fb[k] = dtdx * ((cr >= 0 ? g.lam[gk + cr] : T(0)) - (cl >= 0 ? g.lam[gk + cl] : T(0)));
    hb[k] = T(0);
    lb[k] = T(0);
  }
  hll_vjp(wl, wr, Fb, hb, lb);
#pragma unroll
  for (int k = 0; k < NV; k++) {
    pl[k * sl] = hb[k];
    pr[k * sr] = lb[k];
  }
}

// Stage R3 of cell `item` along D, or of the two ghost cells of a pencil (ghost).
template <typename T, int D>
__device__ __forceinline__ void reverse_recon(const StagedAdjArgs<T> &g, size_t N, T nu, int item, bool ghost) {
  const StepArgs<T> &s = g.a.s;
  const int nx = s.nx, ny = s.ny, n = axis_n<D>(s.nx, s.ny, s.nz);
  int c = item, i, j, side = 0, p = 0;
  if (!ghost) {
    if (item >= (int)N) return;
    i = j = coord<D>(item, nx, ny);
  } else {
    const int np = (int)(N / n);
    if (item >= 2 * np) return;
    side = item >= np ? 1 : 0;
    p = item - side * np;
    c = pencil_cell<D>(p, nx, ny);
    i = 0;
    j = side ? n : -1;
  }
  bool mm, m0, mp;
  const int cm = mapped_cell<T, D>(s, c, i, j - 1, mm);
  const int c0 = mapped_cell<T, D>(s, c, i, j, m0);
  const int cp = mapped_cell<T, D>(s, c, i, j + 1, mp);
  T wm[NV], w0[NV], wp[NV], lob[NV], hib[NV], gm[NV], g0[NV], gp[NV];
  const T *W = g.a.W[0];
  load_frame<T, D>(W, N, cm, mm, wm);
  load_frame<T, D>(W, N, c0, m0, w0);
  load_frame<T, D>(W, N, cp, mp, wp);
  T *lo = g.a.lo + (size_t)D * NV * N + item, *hi = g.a.hi + (size_t)D * NV * N + item, *self = g.self[D] + item;
  size_t stride = N;
  if (ghost) {  // lower ghost: only its upper face state has an adjoint; upper ghost: its lower one
    const size_t at = (size_t)(2 * D + side) * NV * g.a.max_pencils + p;
    T *in = g.a.ghost + at;
    stride = g.a.max_pencils;
    lo = side ? in : g.gout + at;  // what goes to the cell before / after: the inward part
    hi = side ? g.gout + at : in;  // replaces the ghost's face state
    self = g.gself + at;
#pragma unroll
    for (int k = 0; k < NV; k++) {
      const T v = in[k * stride];
      lob[k] = side ? v : T(0);
      hib[k] = side ? T(0) : v;
    }
  } else {
#pragma unroll
    for (int k = 0; k < NV; k++) {
      lob[k] = lo[k * stride];
      hib[k] = hi[k * stride];
    }
  }
#pragma unroll
  for (int k = 0; k < NV; k++) gm[k] = g0[k] = gp[k] = T(0);
  reconstruct_vjp(wm, w0, wp, nu, false, false, false, lob, hib, gm, g0, gp);
#pragma unroll
  for (int k = 0; k < NV; k++) {
    lo[k * stride] = gm[k];
    hi[k * stride] = gp[k];
    self[k * stride] = g0[k];
  }
}

// Adds what direction D gives to cell c (stage R4) to Wb (global order): its own part, the
// cells before and after it, and the positions -2, -1, n, n+1 whose images lie in c.
template <typename T, int D>
__device__ __forceinline__ void gather_dir(const StagedAdjArgs<T> &g, size_t N, int c, T (&Wb)[NV]) {
  const StepArgs<T> &s = g.a.s;
  const int nx = s.nx, ny = s.ny, n = axis_n<D>(s.nx, s.ny, s.nz), st = D == 0 ? 1 : D == 1 ? nx : nx * ny;
  const T *lo = g.a.lo + (size_t)D * NV * N, *hi = g.a.hi + (size_t)D * NV * N, *self = g.self[D];
  const int i = coord<D>(c, nx, ny);
  T v[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) v[k] = self[k * N + c];
  auto add = [&](const T *p, size_t stride, bool flip) {
#pragma unroll
    for (int k = 0; k < NV; k++) {
      const T x = p[k * stride];
      v[k] += flip && (k == 1 || k == 5 || k == 6) ? -x : x;
    }
  };
  if (s.bc[2 * D] == BC_PERIODIC) {
    add(lo + (i + 1 < n ? c + st : c - (n - 1) * st), N, false);
    add(hi + (i > 0 ? c - st : c + (n - 1) * st), N, false);
  } else {
    const size_t mp = g.a.max_pencils;
    const int p = pencil_of<D>(c, nx, ny);
    const T *gin[2] = {g.a.ghost + (size_t)(2 * D) * NV * mp + p, g.a.ghost + (size_t)(2 * D + 1) * NV * mp + p};
    const T *gsf[2] = {g.gself + (size_t)(2 * D) * NV * mp + p, g.gself + (size_t)(2 * D + 1) * NV * mp + p};
    const T *got[2] = {g.gout + (size_t)(2 * D) * NV * mp + p, g.gout + (size_t)(2 * D + 1) * NV * mp + p};
    if (i + 1 < n) add(lo + c + st, N, false);
    else add(gin[1], mp, false);  // the upper ghost's part to the cell before it
    if (i > 0) add(hi + c - st, N, false);
    else add(gin[0], mp, false);
    // images: position -1 holds the ghost's own part and what cell 0 gives to the cell before
    // it; position -2 what the ghost gives outward (likewise n and n + 1)
    const int first = c - i * st, last = first + (n - 1) * st;
    const int b0 = s.bc[2 * D], b1 = s.bc[2 * D + 1];
    bool mir;
    if (map_index(-1, n, b0, b1, mir) == i) {
      const bool f = b0 == BC_REFLECT;
      add(gsf[0], mp, f);
      add(lo + first, N, f);
    }
    if (map_index(-2, n, b0, b1, mir) == i) add(got[0], mp, b0 == BC_REFLECT);
    if (map_index(n, n, b0, b1, mir) == i) {
      const bool f = b1 == BC_REFLECT;
      add(gsf[1], mp, f);
      add(hi + last, N, f);
    }
    if (map_index(n + 1, n, b0, b1, mir) == i) add(got[1], mp, b1 == BC_REFLECT);
  }
#pragma unroll
  for (int k = 0; k < NV; k++) Wb[Frame<D>::g(k)] += v[k];
}

template <typename T, int NDIM>
__global__ void __launch_bounds__(kStagedThreads, 1) staged_reverse_kernel(const StagedAdjArgs<T> g) {
  __shared__ int s_dead;
  __shared__ double s_nu[3], s_dtdx[3];
  const StepArgs<T> &s = g.a.s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned nblk = gridDim.x, blk = blockIdx.x;
  const size_t N = (size_t)s.nx * s.ny * s.nz;
  const int ngrp = (int)((N + 31) / 32);
  unsigned epoch = 0;
  if (tid == 0) s_dead = 0;
  const int w0 = warp * (int)nblk + (int)blk, wstep = kStagedWarps * (int)nblk;
  int gh[NDIM], up[NDIM];
  int ngh = 0, nup = 0;
#pragma unroll
  for (int d = 0; d < NDIM; d++) {
    const int n = d == 0 ? s.nx : d == 1 ? s.ny : s.nz;
    const int np = (int)(N / n);
    gh[d] = s.bc[2 * d] == BC_PERIODIC ? 0 : (2 * np + 31) / 32;
    up[d] = s.bc[2 * d] == BC_PERIODIC ? 0 : (np + 31) / 32;
    ngh += gh[d];
    nup += up[d];
  }
  // calls f(direction, first item, extra list) for every group of a stage's list: the cells of
  // each direction, then an extra list (ghost cells or upper faces) of each
  auto deal = [&](const int (&extra)[NDIM], int nextra, auto &&f) {
    for (int q = w0; q < NDIM * ngrp + nextra; q += wstep) {
      const bool ex = q >= NDIM * ngrp;
      int d = 0, it;
      if (!ex) {
        d = q / ngrp;
        it = q - d * ngrp;
      } else {
        it = q - NDIM * ngrp;
#pragma unroll
        for (int e = 0; e + 1 < NDIM; e++)
          if (d == e && it >= extra[e]) {
            it -= extra[e];
            d = e + 1;
          }
      }
      f(d, it * 32 + lane, ex);
    }
  };
  for (int r = g.len - 1; r >= 0; r--) {
    const double dt = g.a.dts[r];
    const T *U = g.a.seg + (size_t)r * NV * N;
    if (r == g.len - 1) {
      for (int q = w0; q < ngrp; q += wstep) {
        const int c = q * 32 + lane;
        if (c < (int)N) reverse_prepare(g, U, (T)dt, N, c);
      }
    }
    if (tid < 3) {
      const double dx = tid == 0 ? s.dx[0] : tid == 1 ? s.dx[1] : s.dx[2];
      s_nu[tid] = 0.5 * dt / dx;
      s_dtdx[tid] = dt / dx;
    }
    if (!grid_barrier(g.a.bar, nblk, epoch, &s_dead)) break;
    deal(gh, ngh, [&](int d, int item, bool ex) {
      if (d == 0) stage_a<T, 0, 0>(g.a, g.a.W[0], N, (T)s_nu[0], item, ex, 0, 0);
      else if (NDIM > 1 && d == 1) stage_a<T, 0, 1>(g.a, g.a.W[0], N, (T)s_nu[1], item, ex, 0, 0);
      else if (NDIM > 2) stage_a<T, 0, 2>(g.a, g.a.W[0], N, (T)s_nu[2], item, ex, 0, 0);
    });
    if (!grid_barrier(g.a.bar, nblk, epoch, &s_dead)) break;
    deal(up, nup, [&](int d, int item, bool ex) {
      if (d == 0) reverse_face<T, 0>(g, N, (T)s_dtdx[0], item, ex);
      else if (NDIM > 1 && d == 1) reverse_face<T, 1>(g, N, (T)s_dtdx[1], item, ex);
      else if (NDIM > 2) reverse_face<T, 2>(g, N, (T)s_dtdx[2], item, ex);
    });
    if (!grid_barrier(g.a.bar, nblk, epoch, &s_dead)) break;
    deal(gh, ngh, [&](int d, int item, bool ex) {
      if (d == 0) reverse_recon<T, 0>(g, N, (T)s_nu[0], item, ex);
      else if (NDIM > 1 && d == 1) reverse_recon<T, 1>(g, N, (T)s_nu[1], item, ex);
      else if (NDIM > 2) reverse_recon<T, 2>(g, N, (T)s_nu[2], item, ex);
    });
    if (!grid_barrier(g.a.bar, nblk, epoch, &s_dead)) break;
    for (int q = w0; q < ngrp; q += wstep) {
      const int c = q * 32 + lane;
      if (c >= (int)N) continue;
      T Wb[NV], u[NV], Ub[NV];
#pragma unroll
      for (int k = 0; k < NV; k++) {
        Wb[k] = T(0);
        u[k] = U[k * N + c];
        Ub[k] = T(0);
      }
      gather_dir<T, 0>(g, N, c, Wb);
      if constexpr (NDIM > 1) gather_dir<T, 1>(g, N, c, Wb);
      if constexpr (NDIM > 2) gather_dir<T, 2>(g, N, c, Wb);
      cons_to_prim_vjp(u, Wb, Ub);
#pragma unroll
      for (int k = 0; k < NV; k++) g.lam[k * N + c] += Ub[k];
      if (r > 0) reverse_prepare(g, g.a.seg + (size_t)(r - 1) * NV * N, (T)g.a.dts[r - 1], N, c);
    }
  }
  __syncthreads();
  if (s_dead != 0 && tid == 0) s.ctrl->status = 5;  // MSH_E_TIMEOUT: the result is void
  grid_leave(g.a.bar, nblk);
}

template <typename T, int NDIM> static cudaError_t launch_reverse_nd(const StagedAdjArgs<T> &a, cudaStream_t s) {
  static std::atomic<int> occ{0};
  int per_sm = occ.load(std::memory_order_relaxed);
  if (per_sm == 0) {
    const cudaError_t e =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, staged_reverse_kernel<T, NDIM>, kStagedThreads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    occ.store(per_sm, std::memory_order_relaxed);
  }
  const int blocks = staged_blocks<NDIM>(a.a.s, per_sm);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kStagedThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, staged_reverse_kernel<T, NDIM>, a);
}

template <typename T>
cudaError_t launch_staged_reverse(const StagedArgs<T> &a, int ndim, T *lam, T *const (&self)[3], T *gself, T *gout,
                                  int len, cudaStream_t s) {
  StagedAdjArgs<T> g;
  g.a = a;
  g.lam = lam;
  for (int d = 0; d < 3; d++) g.self[d] = self[d];
  g.gself = gself;
  g.gout = gout;
  g.len = len;
  if (ndim == 1) return launch_reverse_nd<T, 1>(g, s);
  if (ndim == 2) return launch_reverse_nd<T, 2>(g, s);
  return launch_reverse_nd<T, 3>(g, s);
}
template cudaError_t launch_staged_reverse<float>(const StagedArgs<float> &, int, float *, float *const (&)[3], float *,
                                                  float *, int, cudaStream_t);
template cudaError_t launch_staged_reverse<double>(const StagedArgs<double> &, int, double *, double *const (&)[3],
                                                   double *, double *, int, cudaStream_t);

}  // namespace msh
