// msh_staged.cuh -- the step as grid-wide stages in one persistent cooperative launch.
//
// The streaming kernels of msh_step_kernels.cuh keep everything of a cell in registers and
// shared memory, at the price of halo cells and chunk prologues that are reconstructed
// again.  Two kinds of grids pay too much for that: FP64 grids, where a double-precision
// warp instruction occupies its scheduler's pipe for 64 cycles on GB300 however few of its
// lanes are active (measured: 64.7 cycles for DFMA with 32 lanes or 8), so every repeated
// lane and every idle scheduler is time lost; and small FP32 grids, which cannot fill 608
// schedulers with strips or tiles.  Here the same arithmetic runs as stages over flat lists
// of items, one item per lane, with the intermediate face states in global memory (mostly
// L2):
//   P   primitive variables of U^n (at the start of a launch; later steps get them from C)
//   A   per cell and direction: reconstruction -> lower and upper face state
//   B   per face: flux, left in place of the face state that only this face reads
//   C   per cell: flux divergence, update, source, realizability, signal speed
// Every cell is reconstructed once per direction and every face flux formed once, the items
// of a stage are dealt to all schedulers evenly, and a grid barrier separates the stages.
// The last barrier of a step carries the reduction of the CFL speed: every block reduces
// the blocks' partials and plans the next step itself, so a launch takes many steps without
// the host, and the a-posteriori fallback passes run inside it only when cells were tagged.
// The per-cell arithmetic is that of the streaming kernels (same device functions, same
// order of the flux divergence), and the results agree with theirs bit for bit.
#pragma once
#include "msh_step_kernels.cuh"

namespace msh {

constexpr int kStagedThreads = 256;
constexpr int kStagedWarps = kStagedThreads / 32;

// ------------------------------------------------------------ grid barrier
// Arrivals only grow within a launch; the last block to leave a launch clears them for the
// next.  Waits are bounded: a block that waits longer than 2^33 clocks (about four seconds)
// sets the counter's top bit, every block leaves, and the launch reports MSH_E_TIMEOUT.  One
// release, one polled word: a separate fence, counter and flag cost three trips to L2 (4100
// cycles with 152 blocks on a small grid).
constexpr unsigned kBarDead = 0x80000000u;
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_add(unsigned *p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ bool grid_barrier(GridBar *b, unsigned nblk, unsigned &epoch, int *s_dead) {
  __syncthreads();
  if (nblk == 1) return true;
  epoch += nblk;
  if (threadIdx.x == 0) {
    red_release_add(&b->arrived, 1u);
    unsigned v = ld_acquire_u32(&b->arrived);
    if (v < epoch) {
      const long long t0 = clock64();
      while ((v = ld_acquire_u32(&b->arrived)) < epoch) {  // (a dead counter is above every epoch)
        if (clock64() - t0 > (1ll << 33)) atomicOr(&b->arrived, kBarDead);
      }
    }
    *s_dead = (v & kBarDead) != 0u;
  }
  __syncthreads();
  return *s_dead == 0;
}
__device__ __forceinline__ void grid_leave(GridBar *b, unsigned nblk) {
  if (nblk == 1 || threadIdx.x != 0) return;
  __threadfence();
  if (atomicAdd(&b->left, 1u) == nblk - 1) {  // every block has passed its last barrier
    b->arrived = 0u;
    b->left = 0u;
  }
}

// ------------------------------------------------------------------ helpers
template <int D> __device__ __forceinline__ int axis_n(int nx, int ny, int nz) { return D == 0 ? nx : D == 1 ? ny : nz; }

// Cell index and mirror flag of position j along D (j may be up to two cells outside) on the
// pencil through cell c, whose own coordinate along D is i.
template <typename T, int D>
__device__ __forceinline__ int mapped_cell(const StepArgs<T> &s, int c, int i, int j, bool &mir) {
  const int n = axis_n<D>(s.nx, s.ny, s.nz), st = D == 0 ? 1 : D == 1 ? s.nx : s.nx * s.ny;
  return c + (map_index(j, n, s.bc[2 * D], s.bc[2 * D + 1], mir) - i) * st;
}

// Primitive state of cell c in the local frame of D (mirrored: u_n and P_nt negated).
template <typename T, int D>
__device__ __forceinline__ void load_frame(const T *W, size_t N, int c, bool mir, T (&w)[NV]) {
#pragma unroll
  for (int k = 0; k < NV; k++) w[k] = W[(size_t)Frame<D>::g(k) * N + c];
  if (mir) {
    w[1] = -w[1];
    w[5] = -w[5];
    w[6] = -w[6];
  }
}

template <typename T> __device__ __forceinline__ bool cell_tag(const StepArgs<T> &s, int c, int32_t tag, int level) {
  return tagged(s.flags[c], tag, level);
}

// Stage A of one cell (position j along D on the pencil of cell c; j = -1 and j = n are the
// ghost cells of a side that is not periodic, whose face state the boundary face needs).
template <typename T, int SCH, int D>
__device__ __forceinline__ void stage_a_item(const StagedArgs<T> &a, const T *W, size_t N, T nu, int c, int i, int j,
                                             int32_t tag, int level, T *lo_out, T *hi_out, size_t stride) {
  const StepArgs<T> &s = a.s;
  bool mm, m0, mp;
  const int cm = mapped_cell<T, D>(s, c, i, j - 1, mm);
  const int c0 = mapped_cell<T, D>(s, c, i, j, m0);
  const int cp = mapped_cell<T, D>(s, c, i, j + 1, mp);
  T wm[NV], w0[NV], wp[NV], lo[NV], hi[NV];
  load_frame<T, D>(W, N, cm, mm, wm);
  load_frame<T, D>(W, N, c0, m0, w0);
  load_frame<T, D>(W, N, cp, mp, wp);
  recon<SCH>(wm, w0, wp, nu, lo, hi);
  if (kCharacteristic<SCH> && level > 0)
    first_order_faces(cell_tag(s, cm, tag, level), cell_tag(s, c0, tag, level), cell_tag(s, cp, tag, level), w0, lo, hi);
  if (lo_out != nullptr) {
#pragma unroll
    for (int k = 0; k < NV; k++) lo_out[k * stride] = lo[k];
  }
  if (hi_out != nullptr) {
#pragma unroll
    for (int k = 0; k < NV; k++) hi_out[k * stride] = hi[k];
  }
}

// The pencil of cell c along D, and the first cell of pencil p.
template <int D> __device__ __forceinline__ int pencil_of(int c, int nx, int ny) {
  if (D == 0) return c / nx;
  if (D == 1) {
    const int z = c / (nx * ny);
    return z * nx + (c - z * nx * ny) % nx;
  }
  return c % (nx * ny);
}
template <int D> __device__ __forceinline__ int pencil_cell(int p, int nx, int ny) {
  if (D == 0) return p * nx;
  if (D == 1) {
    const int z = p / nx;
    return z * nx * ny + (p - z * nx);
  }
  return p;
}
template <int D> __device__ __forceinline__ int coord(int c, int nx, int ny) {
  return D == 0 ? c % nx : D == 1 ? (c / nx) % ny : c / (nx * ny);
}

// Face states of direction D are [NV][N] at a.lo / a.hi + D NV N; ghost states of its lower
// and upper side [NV][pencils] at a.ghost + (2 D + side) NV max_pencils.
template <typename T, int SCH, int D>
__device__ __forceinline__ void stage_a(const StagedArgs<T> &a, const T *W, size_t N, T nu, int item, bool ghost,
                                        int32_t tag, int level) {
  const StepArgs<T> &s = a.s;
  const int nx = s.nx, ny = s.ny;
  if (!ghost) {
    if (item >= (int)N) return;
    T *lo = a.lo + (size_t)D * NV * N + item, *hi = a.hi + (size_t)D * NV * N + item;
    const int i = coord<D>(item, nx, ny);
    stage_a_item<T, SCH, D>(a, W, N, nu, item, i, i, tag, level, lo, hi, N);
  } else {  // the two ghost cells of the pencils along a side that is not periodic
    const int n = axis_n<D>(s.nx, s.ny, s.nz), np = (int)(N / n);
    if (item >= 2 * np) return;
    const int side = item >= np ? 1 : 0, p = item - side * np;
    T *g = a.ghost + (size_t)(2 * D + side) * NV * a.max_pencils + p;
    stage_a_item<T, SCH, D>(a, W, N, nu, pencil_cell<D>(p, nx, ny), 0, side ? n : -1, tag, level, side ? g : nullptr,
                            side ? nullptr : g, a.max_pencils);
  }
}

// Stage B: flux through the lower face of cell `item` along D, stored over its lower face
// state; with `upper` the flux through the upper boundary face of pencil `item` (sides that
// are not periodic), stored over the upper face state of the pencil's last cell.
template <typename T, int SCH, int D>
__device__ __forceinline__ void stage_b(const StagedArgs<T> &a, size_t N, int item, bool upper, int32_t tag,
                                        int level) {
  const StepArgs<T> &s = a.s;
  const int nx = s.nx, ny = s.ny, n = axis_n<D>(s.nx, s.ny, s.nz), st = D == 0 ? 1 : D == 1 ? nx : nx * ny;
  T *lo = a.lo + (size_t)D * NV * N, *hi = a.hi + (size_t)D * NV * N;
  const T *pl, *pr;
  size_t sl = N, sr = N;
  T *out;
  int c;
  bool first = false;
  if (!upper) {
    if (item >= (int)N) return;
    c = item;
    const int i = coord<D>(c, nx, ny);
    pr = lo + c;
    out = lo + c;
    if (i > 0 || s.bc[2 * D] == BC_PERIODIC) {
      pl = hi + (i > 0 ? c - st : c + (n - 1) * st);
    } else {
      pl = a.ghost + (size_t)(2 * D) * NV * a.max_pencils + pencil_of<D>(c, nx, ny);
      sl = a.max_pencils;
    }
    if ((SCH == 3 || SCH == 4) && level > 0) {
      bool m;
      first = cell_tag(s, mapped_cell<T, D>(s, c, i, i - 1, m), tag, level) || cell_tag(s, c, tag, level);
    }
  } else {
    if (item >= (int)(N / n)) return;
    c = pencil_cell<D>(item, nx, ny) + (n - 1) * st;
    pl = hi + c;
    out = hi + c;
    pr = a.ghost + (size_t)(2 * D + 1) * NV * a.max_pencils + item;
    sr = a.max_pencils;
    if ((SCH == 3 || SCH == 4) && level > 0) first = cell_tag(s, c, tag, level);  // the ghost cell is its image
  }
  T wl[NV], wr[NV], F[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) {
    wl[k] = pl[k * sl];
    wr[k] = pr[k * sr];
  }
  if constexpr (SCH == 3 || SCH == 4) {
    if (first) hll(wl, wr, F);
    else face_flux<SCH>(wl, wr, F);
  } else {
    face_flux<SCH>(wl, wr, F);
  }
#pragma unroll
  for (int k = 0; k < NV; k++) out[k * N] = F[k];
}

// Lower (fl) and upper (fu) face flux of cell c along D, local frame.
template <typename T, int D>
__device__ __forceinline__ void load_fluxes(const StagedArgs<T> &a, size_t N, int c, T (&fl)[NV], T (&fu)[NV]) {
  const StepArgs<T> &s = a.s;
  const int nx = s.nx, ny = s.ny, n = axis_n<D>(s.nx, s.ny, s.nz), st = D == 0 ? 1 : D == 1 ? nx : nx * ny;
  const T *lo = a.lo + (size_t)D * NV * N;
  const int i = coord<D>(c, nx, ny);
  const T *pu = i + 1 < n ? lo + c + st
                          : (s.bc[2 * D + 1] == BC_PERIODIC ? lo + c - (n - 1) * st : a.hi + (size_t)D * NV * N + c);
#pragma unroll
  for (int k = 0; k < NV; k++) {
    fl[k] = lo[k * N + c];
    fu[k] = pu[k * N];
  }
}

// Flux divergence of cell c in the global component order, the faces added in the order of
// the streaming kernels (1D: x; 2D: lower y, x, upper y; 3D: lower z, x, lower y, upper z,
// upper y), so that the sums round alike.
template <typename T, int NDIM>
__device__ __forceinline__ void divergence(const StagedArgs<T> &a, size_t N, int c, T idx, T idy, T idz, T (&acc)[NV]) {
  // every face flux is requested before the first is used (one wait instead of one per
  // direction: stage C of a 64^3 FP32 grid took longer than the reconstructions)
  T xl[NV], xu[NV], yl[NV], yu[NV], zl[NV], zu[NV], t[NV];
  load_fluxes<T, 0>(a, N, c, xl, xu);
  if constexpr (NDIM > 1) load_fluxes<T, 1>(a, N, c, yl, yu);
  if constexpr (NDIM > 2) load_fluxes<T, 2>(a, N, c, zl, zu);
  if constexpr (NDIM == 1) {
#pragma unroll
    for (int k = 0; k < NV; k++) acc[k] = (xl[k] - xu[k]) * idx;
  } else if constexpr (NDIM == 2) {
#pragma unroll
    for (int k = 0; k < NV; k++) t[Frame<1>::g(k)] = yl[k];
    v_mul(acc, t, idy);
    v_sub(xl, xl, xu);
    v_fma(acc, xl, idx, acc);
#pragma unroll
    for (int k = 0; k < NV; k++) t[Frame<1>::g(k)] = yu[k];
    v_fma(acc, t, -idy, acc);
  } else {
#pragma unroll
    for (int k = 0; k < NV; k++) t[Frame<2>::g(k)] = zl[k];
    v_mul(acc, t, idz);
    v_sub(xl, xl, xu);
    v_fma(acc, xl, idx, acc);
#pragma unroll
    for (int k = 0; k < NV; k++) t[Frame<1>::g(k)] = yl[k];
    v_fma(acc, t, idy, acc);
#pragma unroll
    for (int k = 0; k < NV; k++) t[Frame<2>::g(k)] = zu[k];
    v_fma(acc, t, -idz, acc);
#pragma unroll
    for (int k = 0; k < NV; k++) acc[Frame<1>::g(k)] -= yu[k] * idy;
  }
}

// The time control of a launch, the same in every block (the run's constants are copied from
// the control block once).
struct StagedTime {
  double cfl, t_end, dt_max;
  int64_t max_step, tape_base, tape_len, hist_base, hist_cap;
  double *tape_dt, *hist;
  int32_t *tape_had;
  double t, t_next, dt, dt_last, dt_cfl;
  int64_t step;
  int64_t first_bad;
  double nu[3];  // dt / (2 dx)
  int done, status, realizable, last_tagged, stop, newly, any_tagged;
};

// ------------------------------------------------------------------- kernel
// SCH 0, 3, 4: the characteristic step with its fallback; 1: both stages of the central
// scheme.  a.phase >= 0: only pass a.phase of a phased step (partials for the finalize
// kernel, no time control).  a.seg: recompute a.max_iter states seg[1..] from seg[0] with
// the given time steps.
template <typename T, int NDIM, int SCH>
__global__ void __launch_bounds__(kStagedThreads, sizeof(T) == 4 ? 2 : 1) staged_kernel(const StagedArgs<T> a) {
  constexpr bool kKt = SCH == 1;
  __shared__ StagedTime st;
  __shared__ int s_dead, s_nbad;
  __shared__ double s_red[kStagedWarps][NV];
  __shared__ double s_max[kStagedWarps];
  __shared__ long long s_bad[kStagedWarps];
  __shared__ int s_cnt[kStagedWarps];
  const StepArgs<T> &s = a.s;
  Ctrl *ctrl = s.ctrl;
  if (a.seg == nullptr && ctrl->done) return;  // the same in every block: nothing writes it before the first barrier
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned nblk = gridDim.x, blk = blockIdx.x;
  const size_t N = (size_t)s.nx * s.ny * s.nz;
  const int ngrp = (int)((N + 31) / 32);
  unsigned epoch = 0;
  if (tid == 0) {
    st.cfl = ctrl->cfl;
    st.t_end = ctrl->t_end;
    st.dt_max = ctrl->dt_max;
    st.max_step = ctrl->max_step;
    st.tape_base = ctrl->tape_base;
    st.tape_len = ctrl->tape_len;
    st.tape_dt = ctrl->tape_dt;
    st.tape_had = ctrl->tape_had;
    st.hist = ctrl->hist;
    st.hist_base = ctrl->hist_base;
    st.hist_cap = ctrl->hist_cap;
    st.t = ctrl->t;
    st.t_next = ctrl->t_next;
    st.dt = ctrl->dt;
    st.dt_last = ctrl->dt_last;
    st.dt_cfl = ctrl->dt_cfl;
    st.step = a.seg != nullptr ? a.seg_step : ctrl->step;
    st.done = 0;
    st.status = ctrl->status;
    st.realizable = ctrl->realizable;
    st.first_bad = ctrl->first_bad;
    st.last_tagged = ctrl->last_tagged;
    s_dead = 0;
    s_nbad = 0;
    if (a.seg != nullptr) st.dt = a.dts[0];
  }
  __syncthreads();
  step_factors(s.dx, st.dt, st.nu);
  const T idx = s.rdx[0], idy = s.rdx[1], idz = s.rdx[2];
  // groups of 32 items are dealt out warp by warp, blocks first, so that a short list
  // spreads over the SMs and over the schedulers of each
  const int w0 = warp * (int)nblk + (int)blk, wstep = kStagedWarps * (int)nblk;
  int gh[NDIM], up[NDIM];  // groups of ghost cells and of upper boundary faces per direction
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
  bool alive = true;
  T smax = T(0);
  long long bad = LLONG_MAX;

  auto stages_ab = [&](const T *W, int32_t tag, int level) {
    const T nux = (T)st.nu[0], nuy = (T)st.nu[1], nuz = (T)st.nu[2];
    for (int g = w0; g < NDIM * ngrp + ngh; g += wstep) {
      bool ghost = g >= NDIM * ngrp;
      int d, it;
      if (!ghost) {
        d = g / ngrp;
        it = g - d * ngrp;
      } else {
        it = g - NDIM * ngrp;
        d = 0;
#pragma unroll
        for (int e = 0; e + 1 < NDIM; e++)
          if (d == e && it >= gh[e]) {
            it -= gh[e];
            d = e + 1;
          }
      }
      const int item = it * 32 + lane;
      if (d == 0) stage_a<T, SCH, 0>(a, W, N, nux, item, ghost, tag, level);
      else if (NDIM > 1 && d == 1) stage_a<T, SCH, 1>(a, W, N, nuy, item, ghost, tag, level);
      else if (NDIM > 2) stage_a<T, SCH, 2>(a, W, N, nuz, item, ghost, tag, level);
    }
    alive = alive && grid_barrier(a.bar, nblk, epoch, &s_dead);
    if (!alive) return;
    for (int g = w0; g < NDIM * ngrp + nup; g += wstep) {
      bool upper = g >= NDIM * ngrp;
      int d, it;
      if (!upper) {
        d = g / ngrp;
        it = g - d * ngrp;
      } else {
        it = g - NDIM * ngrp;
        d = 0;
#pragma unroll
        for (int e = 0; e + 1 < NDIM; e++)
          if (d == e && it >= up[e]) {
            it -= up[e];
            d = e + 1;
          }
      }
      const int item = it * 32 + lane;
      if (d == 0) stage_b<T, SCH, 0>(a, N, item, upper, tag, level);
      else if (NDIM > 1 && d == 1) stage_b<T, SCH, 1>(a, N, item, upper, tag, level);
      else if (NDIM > 2) stage_b<T, SCH, 2>(a, N, item, upper, tag, level);
    }
    alive = alive && grid_barrier(a.bar, nblk, epoch, &s_dead);
  };

  // stage C; CS: the scheme finish_cell sees (0 for the characteristic step, 1 and 2 for the
  // stages of the central scheme)
  auto stage_c = [&](auto csc, const T *src, const T *un0, T *dst, T *Wout, double ddt, int32_t tag, int level, T *ck) {
    constexpr int CS = decltype(csc)::value;
    const T dt = (T)ddt;
    Acc<T> none;
    for (int g = w0; g < ngrp; g += wstep) {
      const int c = g * 32 + lane;
      if (c >= (int)N) continue;
      T acc[NV];
      divergence<T, NDIM>(a, N, c, idx, idy, idz, acc);
      finish_cell<T, NDIM, CS, false, false, true>(s, src + c, N, un0 + c, dst, N, (size_t)c, acc, dt, idx, idy, idz, none,
                                                   smax, bad, tag, ck, level, Wout, &s_nbad);
    }
  };

  // the block's CFL speed, first non-realizable cell and newly tagged cells to its partial,
  // then (after the barrier) the grid's in every block
  auto write_part = [&]() {
    smax = warp_max_nonneg(smax);
    if (__any_sync(FULL, bad != LLONG_MAX)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) bad = min(bad, __shfl_xor_sync(FULL, bad, o));
    }
    if (lane == 0) {
      s_max[warp] = (double)smax;
      s_bad[warp] = bad;
    }
    __syncthreads();
    if (tid == 0) {
      double m = s_max[0];
      long long b = s_bad[0];
      for (int w = 1; w < kStagedWarps; w++) {
        m = max_nonneg(m, s_max[w]);
        b = min(b, s_bad[w]);
      }
      Partial *p = s.part + blk;
      p->smax = m;
      p->bad = b;
      a.newly[blk] = s_nbad;
      s_nbad = 0;
    }
    smax = T(0);
    bad = LLONG_MAX;
  };
  // every thread takes a partial, so that all are in flight at once; the result is known to
  // warp 0 (one warp walking over 152 partials waited for L2 five times)
  auto reduce_parts = [&](double &m, long long &b, int &nb) {
    m = 0.0;
    b = LLONG_MAX;
    nb = 0;
    for (unsigned i = tid; i < nblk; i += kStagedThreads) {
      const double pm = __ldcg(&s.part[i].smax);
      const long long pb = __ldcg(&s.part[i].bad);
      nb += __ldcg(&a.newly[i]);
      m = max_nonneg(m, pm);
      b = min(b, pb);
    }
    m = warp_max_nonneg(m);
    nb = __reduce_add_sync(FULL, nb);
    if (__any_sync(FULL, b != LLONG_MAX)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) b = min(b, __shfl_xor_sync(FULL, b, o));
    }
    if (nblk > 32) {
      if (lane == 0) {
        s_max[warp] = m;
        s_bad[warp] = b;
        s_cnt[warp] = nb;
      }
      __syncthreads();
      if (warp == 0) {
        for (int w = 1; w < kStagedWarps; w++) {
          m = max_nonneg(m, s_max[w]);
          b = min(b, s_bad[w]);
          nb += s_cnt[w];
        }
      }
    }
  };

  {  // P
    const T *U = a.seg != nullptr ? a.seg : s.U[st.step & 1];
    T *W = a.W[st.step & 1];
    for (int g = w0; g < ngrp; g += wstep) {
      const int c = g * 32 + lane;
      if (c >= (int)N) continue;
      T u[NV], w[NV];
#pragma unroll
      for (int k = 0; k < NV; k++) u[k] = U[k * N + c];
      cons_to_prim(u, w);
#pragma unroll
      for (int k = 0; k < NV; k++) W[k * N + c] = w[k];
    }
    alive = grid_barrier(a.bar, nblk, epoch, &s_dead);
  }

  int taken = 0;
  while (alive) {
    const int64_t step = st.step;
    const double dt = st.dt;
    const int32_t tag = (int32_t)(step & 0x0fffffff) + 1;
    const T *U0 = a.seg != nullptr ? a.seg + (size_t)taken * NV * N : s.U[step & 1];
    T *Ud = a.seg != nullptr ? a.seg + (size_t)(taken + 1) * NV * N : s.U[(step + 1) & 1];
    const T *W0 = a.W[step & 1];
    T *Wn = a.W[(step + 1) & 1];
    T *const ck = (kKt || a.seg != nullptr) ? nullptr : tape_slot(s, step, N);
    if constexpr (kKt) {
      stages_ab(W0, tag, 0);
      if (!alive) break;
      // the first stage's primitive state goes to the next step's buffer, which the second
      // stage replaces once every face state has been formed from it
      stage_c(std::integral_constant<int, 1>{}, U0, U0, s.U1, Wn, dt, tag, 0, (T *)nullptr);
      alive = grid_barrier(a.bar, nblk, epoch, &s_dead);
      if (!alive) break;
      stages_ab(Wn, tag, 0);
      if (!alive) break;
      stage_c(std::integral_constant<int, 2>{}, s.U1, U0, Ud, Wn, dt, tag, 0, (T *)nullptr);
      write_part();
    } else {
      const int level = a.phase >= 0 ? a.phase : 0;
      stages_ab(W0, tag, level);
      if (!alive) break;
      stage_c(std::integral_constant<int, 0>{}, U0, U0, Ud, Wn, dt, tag, level, level == 0 ? ck : nullptr);
      write_part();
      if (a.phase >= 0) break;
    }
    alive = grid_barrier(a.bar, nblk, epoch, &s_dead);
    if (!alive) break;
    double m;
    long long b;
    int nb;
    reduce_parts(m, b, nb);
    // a-posteriori fallback: passes with first-order faces at the tagged cells, while the
    // pass before tagged new ones
    if (!kKt) {
      if (tid == 0) {
        st.newly = nb;
        st.any_tagged = nb;
      }
      __syncthreads();
      for (int level = 1; level <= kFallbackPasses && st.newly > 0; level++) {
        stages_ab(W0, tag, level);
        if (!alive) break;
        stage_c(std::integral_constant<int, 0>{}, U0, U0, Ud, Wn, dt, tag, level, (T *)nullptr);
        write_part();
        alive = grid_barrier(a.bar, nblk, epoch, &s_dead);
        if (!alive) break;
        reduce_parts(m, b, nb);
        if (tid == 0) st.newly = nb;
        __syncthreads();
      }
      if (!alive) break;
    }
    taken++;
    if (warp == 0) {  // plan the next step, as the finalize kernel does (every lane alike)
      const int any = kKt ? 0 : st.any_tagged;
      double nd;
      bool stop;
      if (a.seg != nullptr) {
        stop = taken >= a.max_iter;
        nd = stop ? dt : a.dts[taken];
        if (lane == 0) {
          st.dt = nd;
          st.step = step + 1;
          if (blk == 0 && a.had != nullptr) a.had[taken - 1] = any > 0;
          if (blk == 0 && any > 0)
            for (int p = 0; p <= kFallbackPasses; p++) ctrl->nbad[p] = 0;
        }
      } else {
        const double t = st.t_next, dt_cfl = st.cfl / m;
        double tn = t + dt_cfl;
        nd = dt_cfl;
        if (nd > st.dt_max) {
          nd = st.dt_max;
          tn = t + nd;
        }
        if (tn >= st.t_end) {
          nd = st.t_end - t;
          tn = st.t_end;
        }
        const bool real = b == LLONG_MAX;
        const bool done = !real || t >= st.t_end || step + 1 >= st.max_step;
        if (done) {
          nd = dt;
          tn = t;
        }
        stop = done || taken >= a.max_iter;
        __syncwarp();  // every lane has read the old state
        if (lane == 0) {
          st.last_tagged = any;
          st.realizable = real;
          st.first_bad = real ? -1 : b;
          st.dt_cfl = dt_cfl;
          if (blk == 0) {
            const int64_t ti = step - st.tape_base, hi_ = step - st.hist_base;
            if (st.tape_dt != nullptr && ti >= 0 && ti < st.tape_len) {
              st.tape_dt[ti] = dt;
              st.tape_had[ti] = any > 0;
            }
            if (st.hist != nullptr && hi_ >= 0 && hi_ < st.hist_cap) st.hist[hi_] = dt;
            if (any > 0)
              for (int p = 0; p <= kFallbackPasses; p++) ctrl->nbad[p] = 0;
          }
          st.dt_last = dt;
          st.t = t;
          st.step = step + 1;
          if (!real) st.status = 4;  // MSH_E_REALIZABILITY
          st.done = done;
          st.dt = nd;
          st.t_next = tn;
        }
      }
      if (lane == 0) st.stop = stop;
      if (lane < 3 && !stop) st.nu[lane] = 0.5 * nd / (lane == 0 ? s.dx[0] : lane == 1 ? s.dx[1] : s.dx[2]);
    }
    __syncthreads();
    if (st.stop) break;
  }
  if (!alive) {  // a barrier gave up: the result is void
    if (tid == 0) {
      ctrl->status = 5;  // MSH_E_TIMEOUT
      if (a.seg == nullptr) ctrl->done = 1;
    }
    grid_leave(a.bar, nblk);
    return;
  }
  if (a.seg == nullptr) {
    // FP64 totals of the state the launch leaves (only the last step's are observable)
    const T *U = s.U[(a.phase >= 0 ? st.step + 1 : st.step) & 1];
    double d[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) d[k] = 0.0;
    for (int g = w0; g < ngrp; g += wstep) {
      const int c = g * 32 + lane;
      if (c >= (int)N) continue;
#pragma unroll
      for (int k = 0; k < NV; k++) d[k] += widen(U[k * N + c]);
    }
    int comp;
    const double x = warp_sum10(d, comp);
    if (comp >= 0 && (lane & 1) == 0) s_red[warp][comp] = x;
    __syncthreads();
    if (tid < NV) {
      double sum = 0.0;
      for (int w = 0; w < kStagedWarps; w++) sum += s_red[w][tid];
      s.part[blk].diag[tid] = sum;
    }
    if (a.phase < 0) {
      __syncthreads();
      alive = grid_barrier(a.bar, nblk, epoch, &s_dead);
      if (blk == 0) {
        if (lane < NV) {
          double sum = 0.0;
          for (unsigned i = warp; i < nblk; i += kStagedWarps) sum += __ldcg(&s.part[i].diag[lane]);
          s_red[warp][lane] = sum;
        }
        __syncthreads();
        if (tid < NV) {
          double sum = 0.0;
          for (int w = 0; w < kStagedWarps; w++) sum += s_red[w][tid];
          ctrl->totals[tid] = sum;
        }
        if (tid == 0) {
          ctrl->t = st.t;
          ctrl->t_next = st.t_next;
          ctrl->dt = st.dt;
          ctrl->dt_last = st.dt_last;
          ctrl->dt_cfl = st.dt_cfl;
          ctrl->step = st.step;
          ctrl->realizable = st.realizable;
          ctrl->first_bad = st.first_bad;
          ctrl->last_tagged = st.last_tagged;
          ctrl->force = 0;
          ctrl->status = alive ? st.status : 5;
          ctrl->done = alive ? st.done : 1;
        }
      }
    }
  }
  grid_leave(a.bar, nblk);
}

// ----------------------------------------------------------------- launcher
// As many blocks as the SMs hold, but no more than give every scheduler one group of 32 items of
// stage A, the ghost cells' included (four groups per block): a second double-precision warp on
// a scheduler doubles a short stage (256 FP64 cells in 1D: stage A 22000 cycles with two blocks).
template <int NDIM, typename T> int staged_blocks(const StepArgs<T> &s, int per_sm) {
  const long long N = (long long)s.nx * s.ny * s.nz;
  long long groups = NDIM * ((N + 31) / 32);
  for (int d = 0; d < NDIM; d++) {
    const long long np = N / (d == 0 ? s.nx : d == 1 ? s.ny : s.nz);
    if (s.bc[2 * d] != BC_PERIODIC) groups += (2 * np + 31) / 32;
  }
  const long long most = std::min<long long>((long long)device_sms() * per_sm, kStagedMaxBlocks);
  return (int)std::max<long long>(1, std::min<long long>(most, (groups + 3) / 4));
}

template <typename T, int NDIM, int SCH> cudaError_t launch_staged_nd(const StagedArgs<T> &a, cudaStream_t s, int *nblk) {
  static std::atomic<int> occ{0};
  int per_sm = occ.load(std::memory_order_relaxed);
  if (per_sm == 0) {
    const cudaError_t e =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, staged_kernel<T, NDIM, SCH>, kStagedThreads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    occ.store(per_sm, std::memory_order_relaxed);
  }
  const int blocks = staged_blocks<NDIM>(a.s, per_sm);
  if (nblk != nullptr) *nblk = blocks;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kStagedThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, staged_kernel<T, NDIM, SCH>, a);
}

template <typename T, int SCH> cudaError_t launch_staged(const StagedArgs<T> &a, int ndim, cudaStream_t s, int *nblk) {
  if (ndim == 1) return launch_staged_nd<T, 1, SCH>(a, s, nblk);
  if (ndim == 2) return launch_staged_nd<T, 2, SCH>(a, s, nblk);
  return launch_staged_nd<T, 3, SCH>(a, s, nblk);
}

}  // namespace msh
