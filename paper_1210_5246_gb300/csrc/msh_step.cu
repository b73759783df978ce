// msh_step.cu -- step launchers of the MUSCL-Hancock scheme and the small kernels of a
// run: scan, gravity field, finalize (fixed-order reduction of the partials, plans the
// next step on the device), run start, conversions.  The step kernels themselves are in
// msh_step_kernels.cuh; the central scheme's stages are instantiated in msh_step_kt.cu.
#include <algorithm>
#include <cfloat>
#include <climits>

#include "msh_step_kernels.cuh"

namespace msh {

// Acceleration a = -grad Phi by central differences from the potential with one ghost
// layer, stored [3][N] in the state's precision.
template <typename T>
__global__ void gravity_field_kernel(const double *__restrict__ phi, T *__restrict__ acc, int ndim, int nx,
                                     int ny, int nz, double dx0, double dx1, double dx2) {
  const size_t N = (size_t)nx * ny * nz;
  const int gy = ndim > 1 ? 1 : 0, gz = ndim > 2 ? 1 : 0;
  const long px = nx + 2, py = ny + 2 * gy;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < N; c += (size_t)gridDim.x * blockDim.x) {
    const long x = (long)(c % nx), y = (long)((c / nx) % ny), z = (long)(c / ((size_t)nx * ny));
    const long ctr = ((z + gz) * py + (y + gy)) * px + (x + 1);
    acc[c] = (T)(-(phi[ctr + 1] - phi[ctr - 1]) / (2.0 * dx0));
    acc[N + c] = ndim > 1 ? (T)(-(phi[ctr + px] - phi[ctr - px]) / (2.0 * dx1)) : T(0);
    acc[2 * N + c] = ndim > 2 ? (T)(-(phi[ctr + px * py] - phi[ctr - px * py]) / (2.0 * dx2)) : T(0);
  }
}

// -------------------------------------------------------- finalize and plan
__device__ void plan(Ctrl *c) {
  if (c->t >= c->t_end || c->step >= c->max_step) {
    c->done = 1;
    return;
  }
  double dt = c->dt_cfl;
  if (dt > c->dt_max) dt = c->dt_max;
  double tn = c->t + dt;
  if (tn >= c->t_end) {
    dt = c->t_end - c->t;
    tn = c->t_end;
  }
  c->dt = dt;
  c->t_next = tn;
}

// mode 0: after a step (advance time, record dt, stop on a non-realizable cell, plan the
// next step); mode 1: after set_state (CFL dt and totals of the state only).  Run by one block
// of kFinalizeThreads threads.
__device__ void finalize_block(Ctrl *ctrl, const Partial *part, int nparts, int mode) {
  constexpr int kWarps = kFinalizeThreads / 32;
  __shared__ double sd[kWarps][NV + 1], stot[NV];
  __shared__ long long sb[kWarps];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  double d[NV];
  for (int k = 0; k < NV; k++) d[k] = 0.0;
  double smax = 0.0;
  long long bad = LLONG_MAX;
  for (int i = t; i < nparts; i += kFinalizeThreads) {
    for (int k = 0; k < NV; k++) d[k] += part[i].diag[k];
    smax = max_nonneg(smax, part[i].smax);
    bad = min(bad, part[i].bad);
  }
  // fixed order: strided sums per thread, warps, then one thread per component over the warps
  int comp;
  const double x = warp_sum10(d, comp);
  smax = warp_max_nonneg(smax);
  for (int o = 16; o > 0; o >>= 1) bad = min(bad, __shfl_xor_sync(FULL, bad, o));
  if (comp >= 0 && (lane & 1) == 0) sd[warp][comp] = x;
  if (lane == 0) {
    sd[warp][NV] = smax;
    sb[warp] = bad;
  }
  __syncthreads();
  if (t < NV) {
    double sum = sd[0][t];
    for (int w = 1; w < kWarps; w++) sum += sd[w][t];
    stot[t] = sum;
  }
  for (int w = 0; w < kWarps; w++) {
    smax = max_nonneg(smax, sd[w][NV]);
    bad = min(bad, sb[w]);
  }
  __syncthreads();
  if (t != 0) return;
  Ctrl *c = ctrl;
  if (mode == 0 && c->stage_timeout) {  // the step kernel gave up waiting for staged data
    c->status = 5;                     // MSH_E_TIMEOUT
    c->done = 1;
    return;
  }
  for (int k = 0; k < NV; k++) c->totals[k] = stot[k];
  const long long b = bad;
  c->realizable = (b == LLONG_MAX);
  c->first_bad = (b == LLONG_MAX) ? -1 : b;
  c->dt_cfl = c->cfl / smax;
  if (mode == 1) {
    c->done = 1;
    return;
  }
  c->last_tagged = c->nbad[0];
  const int64_t ti = c->step - c->tape_base;
  if (c->tape_dt != nullptr && ti >= 0 && ti < c->tape_len) {
    c->tape_dt[ti] = c->dt;
    c->tape_had[ti] = c->nbad[0] > 0;
  }
  for (int p = 0; p <= kFallbackPasses; p++) c->nbad[p] = 0;
  c->force = 0;
  const int64_t hi_ = c->step - c->hist_base;
  if (c->hist != nullptr && hi_ >= 0 && hi_ < c->hist_cap) c->hist[hi_] = c->dt;
  c->dt_last = c->dt;
  c->t = c->t_next;
  c->step += 1;
  if (!c->realizable) {
    c->status = 4;  // MSH_E_REALIZABILITY
    c->done = 1;
    return;
  }
  plan(c);
}

// mode 2: mode 0 unless the step tagged cells (the host then runs the fallback passes and mode
// 0); mode 3: the same in the middle of a run, which stops there with kStatusPending.
// scan_count: a scan counter to clear in any case (nullptr: none)
__global__ void __launch_bounds__(kFinalizeThreads) finalize_kernel(Ctrl *ctrl, const Partial *part, int nparts,
                                                                    int mode, unsigned *scan_count) {
  if (scan_count != nullptr && threadIdx.x == 0) *scan_count = 0u;
  if (mode != 1 && ctrl->done) return;
  if (mode >= 2 && ctrl->nbad[0] != 0 && !ctrl->stage_timeout) {
    if (mode == 3 && threadIdx.x == 0) {
      ctrl->status = kStatusPending;
      ctrl->done = 1;
    }
    return;
  }
  finalize_block(ctrl, part, nparts, mode == 1 ? 1 : 0);
}

// ----------------------------------------------------------------- scan kernel
// One pass over the cells [c0, c1) of a state whose fields are N apart (see launch_scan); every
// block writes its partial, and the last one to finish (a counter) finalizes, which spares a
// launch.  MAXF: the corner-transport-upwind speed (the maximum over the dims instead of the
// sum).  Bound by the FP64 sums of the totals (ten conversions and additions per cell), not by
// the copy: the grid has one block per 256 cells up to four per SM.
template <typename T, int NDIM, bool MAXF>
__global__ void __launch_bounds__(kFinalizeThreads) scan_kernel(const T *src, T *dst, int prim, int32_t *flags,
                                                                size_t N, size_t c0, size_t c1, T idx, T idy, T idz,
                                                                Partial *part, ScanEnd end) {
  double diag[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) diag[k] = 0.0;
  T smax = T(0);
  long long bad = LLONG_MAX;
  for (size_t c = c0 + (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < c1; c += (size_t)gridDim.x * blockDim.x) {
    T Uc[NV], W[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) Uc[k] = src[k * N + c];
    if (prim) {
#pragma unroll
      for (int k = 0; k < NV; k++) W[k] = Uc[k];
      prim_to_cons(W, Uc);
    }
    if (dst != nullptr) {
#pragma unroll
      for (int k = 0; k < NV; k++) dst[k * N + c] = Uc[k];
    }
    if (flags != nullptr) flags[c] = 0;
    cons_to_prim(Uc, W);
    if (!realizable(W)) bad = min(bad, (long long)c);
    smax = max_nonneg(smax, speed_sum<T, NDIM, MAXF>(W, idx, idy, idz));
#pragma unroll
    for (int k = 0; k < NV; k++) diag[k] += widen(Uc[k]);
  }
  block_partial<kFinalizeThreads>(diag, (double)smax, bad, part + blockIdx.x);
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(end.count, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  Ctrl *ctrl = end.ctrl;
  if (threadIdx.x == 0) {
    *end.count = 0u;
    if (end.kind == 1) {
      Ctrl c = {};
      c.cfl = end.cfl;
      c.t_end = INFINITY;
      c.dt_max = INFINITY;
      c.done = 1;
      c.first_bad = -1;
      *ctrl = c;
    }
  }
  __syncthreads();
  finalize_block(ctrl, part, (int)gridDim.x, 1);
  if (end.kind == 1 && threadIdx.x == 0) {
    if (!ctrl->realizable) {  // a non-realizable input is not stepped
      ctrl->status = MSH_E_REALIZABILITY;
    } else {
      ctrl->max_step = 1;
      ctrl->dt_max = end.dt_max;
      ctrl->done = 0;
      double dt = ctrl->dt_cfl;
      if (dt > end.dt_max) dt = end.dt_max;
      ctrl->dt = dt;
      ctrl->t_next = dt;
    }
  }
}

__global__ void accept_kernel(Ctrl *ctrl, const uint2 *src, uint2 *dst, size_t n) {
  if (!ctrl->realizable) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->sg_hist = 0;
  if (n % 2 == 0) {
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
    uint4 *d4 = reinterpret_cast<uint4 *>(dst);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n / 2; i += (size_t)gridDim.x * blockDim.x)
      d4[i] = s4[i];
  } else {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
      dst[i] = src[i];
  }
}

// One step with a given dt: no CFL limit, no end time.
__global__ void set_dt_kernel(Ctrl *c, double dt) {
  c->t_end = INFINITY;
  c->max_step = INT64_MAX;
  c->dt_max = INFINITY;
  c->done = 0;
  c->status = 0;
  c->stage_timeout = 0;
  c->force = 0;
  for (int p = 0; p <= kFallbackPasses; p++) c->nbad[p] = 0;
  c->dt = dt;
  c->t_next = c->t + dt;
}

// A fallback pass that must run even where this grid tagged nothing in the pass before.
__global__ void force_pass_kernel(Ctrl *c, int level) { c->force |= 1 << level; }

// Per cell of [c0, c1): the fallback pass of the current step that tagged it, or -1
// (tags are 8 * (step tag) + pass; a tag of another step is no tag).
__global__ void get_tags_kernel(const Ctrl *ctrl, const int32_t *flags, size_t c0, size_t c1, int32_t *levels) {
  const int32_t tag = (int32_t)(ctrl->step & 0x0fffffff) + 1;
  for (size_t c = c0 + (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < c1; c += (size_t)gridDim.x * blockDim.x) {
    const int32_t f = flags[c];
    levels[c - c0] = (f >> 3) == tag ? (f & 7) : -1;
  }
}

__global__ void set_tags_kernel(const Ctrl *ctrl, int32_t *flags, size_t c0, size_t c1, const int32_t *levels) {
  const int32_t tag = (int32_t)(ctrl->step & 0x0fffffff) + 1;
  for (size_t c = c0 + (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < c1; c += (size_t)gridDim.x * blockDim.x) {
    const int32_t l = levels[c - c0];
    flags[c] = l >= 0 ? tag * 8 + l : 0;
  }
}

// Cells of [c0, c1) tagged by pass `level` of the current step.
__global__ void count_tags_kernel(const Ctrl *ctrl, const int32_t *flags, size_t c0, size_t c1, int level,
                                  unsigned long long *count) {
  const int32_t want = ((int32_t)(ctrl->step & 0x0fffffff) + 1) * 8 + level;
  unsigned long long n = 0;
  for (size_t c = c0 + (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < c1; c += (size_t)gridDim.x * blockDim.x)
    n += flags[c] == want;
  for (int o = 16; o > 0; o >>= 1) n += __shfl_down_sync(0xffffffffu, n, o);
  if ((threadIdx.x & 31) == 0 && n) atomicAdd(count, n);
}

cudaError_t launch_force_pass(Ctrl *ctrl, int level, cudaStream_t s) {
  force_pass_kernel<<<1, 1, 0, s>>>(ctrl, level);
  return cudaGetLastError();
}

cudaError_t launch_tags(Ctrl *ctrl, int32_t *flags, size_t c0, size_t c1, int32_t *levels, bool to_grid,
                        cudaStream_t s) {
  const int blocks = (int)std::min<size_t>((c1 - c0 + 255) / 256 + 1, (size_t)kScanBlocks);
  if (to_grid) set_tags_kernel<<<blocks, 256, 0, s>>>(ctrl, flags, c0, c1, levels);
  else get_tags_kernel<<<blocks, 256, 0, s>>>(ctrl, flags, c0, c1, levels);
  return cudaGetLastError();
}

cudaError_t launch_count_tags(const Ctrl *ctrl, const int32_t *flags, size_t c0, size_t c1, int level,
                              unsigned long long *count, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  const int blocks = (int)std::min<size_t>((c1 - c0 + 255) / 256 + 1, (size_t)kScanBlocks);
  count_tags_kernel<<<blocks, 256, 0, s>>>(ctrl, flags, c0, c1, level, count);
  return cudaGetLastError();
}

__global__ void run_start_kernel(Ctrl *c, double t_end, int64_t max_steps, double dt_max) {
  c->t_end = t_end;
  c->max_step = (max_steps > INT64_MAX - c->step) ? INT64_MAX : c->step + max_steps;
  c->dt_max = dt_max;
  c->done = 0;
  c->status = 0;
  c->stage_timeout = 0;
  c->force = 0;
  for (int p = 0; p <= kFallbackPasses; p++) c->nbad[p] = 0;
  plan(c);
}

// Ensemble runs: after the scan of a new state (finalize mode 1), start it at t = 0 with the
// step counter at step_base (the host knows every state's base, hence its buffer parity and
// fallback tags, without reading the device); a non-realizable input is not stepped and its
// status is MSH_E_REALIZABILITY.  ensemble_end records the status of the state's steps.
__global__ void ensemble_start_kernel(Ctrl *c, int64_t step_base, int64_t nsteps, int32_t *status) {
  c->t = 0.0;
  c->step = step_base;
  c->sg_hist = 0;  // a new state has no previous self-gravity acceleration
  for (int p = 0; p <= kFallbackPasses; p++) c->nbad[p] = 0;
  if (!c->realizable) {
    c->done = 1;
    c->status = 4;  // MSH_E_REALIZABILITY
    *status = 4;
    return;
  }
  *status = 0;
  c->t_end = INFINITY;
  c->max_step = step_base + nsteps;
  c->dt_max = INFINITY;
  c->done = 0;
  c->status = 0;
  c->stage_timeout = 0;
  plan(c);
}

__global__ void ensemble_end_kernel(const Ctrl *c, int32_t *status) {
  if (*status == 0) *status = c->status;
}

cudaError_t launch_ensemble_start(Ctrl *ctrl, int64_t step_base, int64_t nsteps, int32_t *status, cudaStream_t s) {
  ensemble_start_kernel<<<1, 1, 0, s>>>(ctrl, step_base, nsteps, status);
  return cudaGetLastError();
}

cudaError_t launch_ensemble_end(const Ctrl *ctrl, int32_t *status, cudaStream_t s) {
  ensemble_end_kernel<<<1, 1, 0, s>>>(ctrl, status);
  return cudaGetLastError();
}

// ----------------------------------------------------------- default tiling
// Planes a unit of the balanced 3D tiling streams plus p for each of its prologues, at most
// over the units (the same hand-out as step_tile_kernel).
static double balanced_cost(long long ncols, long long nz, long long units, double p) {
  const long long nfull = ncols / units, nrcol = ncols - nfull * units, nrest = nrcol * nz;
  const long long wz = std::max<long long>(1, (nrest + units - 1) / units), nwf = nz / wz, wlast = nz - nwf * wz;
  double worst = 0.0;
  for (long long u = 0; u < units; u++) {
    double cost = (double)nfull * (nz + p);
    long long rp = nrest * u / units;
    const long long rend = nrest * (u + 1) / units;
    while (rp < rend) {
      const long long inwhole = nrcol * wz * nwf;
      const long long left = rp < inwhole ? wz - rp % wz : wlast - (rp - inwhole) % wlast;
      const long long len = std::min(left, rend - rp);
      cost += (double)len + p;
      rp += len;
    }
    worst = std::max(worst, cost);
  }
  return worst;
}

// The shape with the least estimated time.  The estimates are fits to timed sweeps over grid
// sizes (step kernel, GB300):
//   3D FP32  a block of 16 rows takes 5.5 us per plane with one block per SM, one of 8 rows
//            6.3 us with two per SM (corner transport upwind: 10 us and 6.4 us, one per SM);
//            a prologue costs as much as 6 planes.  256^3: 16 rows balanced 1.60 ms against
//            2.14 ms with 8 rows; 160^3: two chunks of 80 planes per column 0.47 ms, balanced
//            0.70 ms (its last windows are 8 planes long); 48^3 CTU: 8 rows in chunks of 6.
//   2D FP32  a row of a strip takes 2.05 us while a scheduler has up to two warps, 2.5 us with
//            three and 2.9 us with four; a chunk's prologue, partial and start cost as much as
//            5.2 rows.  512^2: 4 rows 26.8 us, 8 rows 28.0 us; 1024^2: 16 rows 61.6 us; 700^2: 10 rows
//            43.8 us.
//   FP64     the double-precision pipe is the bound: time goes with the warps per scheduler,
//            a prologue costs about one row or plane.  2D blocks of 16 warps are held to 128
//            registers and spill (780 B), which that pipe hides: 4096^2 29.2 ms in chunks of 50 rows,
//            8 warps in chunks of 16 (the fixed shape before) 29.4, 2500^2 11.0 and 11.4.
Tiling default_tiling(int ndim, const int64_t n[3], int prec, bool ctu) {
  if (ndim == 1) return {8, 1, 0.0};
  const bool f32 = prec == MSH_FP32;
  const long long sms = device_sms();
  Tiling best = {8, ndim == 3 ? 0 : 16, 0.0};
  double best_cost = 1e300;
  auto offer = [&](int rows, int zchunk, double cost) {
    if (cost < 0.995 * best_cost) {  // near ties keep the earlier candidate
      best_cost = cost;
      best = {rows, zchunk, cost};
    }
  };
  if (ndim == 2) {
    const long long strips = (n[0] + kStripX - 1) / kStripX;
    for (int rows : {16, 8, 4})
      for (int c = 1; c <= 64 && c <= n[1]; c++) {
        const long long warps = strips * ((n[1] + c - 1) / c), blocks = (warps + rows - 1) / rows;
        double cost;
        if (f32) {
          const long long slots = sms * (16 / rows), waves = blocks / slots, rest = blocks - waves * slots;
          const double w = (double)((rest + sms - 1) / sms) * rows / 4.0;  // warps per scheduler, last wave
          cost = (c + 5.2) * (2.9 * (double)waves + (rest == 0 ? 0.0 : w <= 2.0 ? 2.05 : w <= 3.0 ? 2.5 : 2.9));
        } else {
          cost = (c + 1.0) * (double)((blocks + sms - 1) / sms) * rows / 4.0;
        }
        offer(rows, c, cost);
      }
    return best;
  }
  const double p = f32 ? 6.0 : 1.0;
  const long long tilesx = (n[0] + kTileX - 1) / kTileX;
  for (int rows : {16, 8}) {
    if (rows == 16 && !f32) continue;
    const long long slots = rows == 8 && f32 && !ctu ? 2 * sms : sms;
    const double plane = !f32 ? 1.0 : ctu ? (rows == 16 ? 10.0 : 6.4) : (rows == 16 ? 5.5 : 6.3);
    const long long ncols = tilesx * ((n[1] + rows - 3) / (rows - 2));
    const long long units = std::max<long long>(1, std::min<long long>(slots, ncols * n[2] / kMinUnitPlanes));
    offer(rows, 0, plane * balanced_cost(ncols, n[2], units, p));
    for (long long m = 1; m <= 64 && m <= n[2]; m++) {
      const long long z = (n[2] + m - 1) / m, u = ncols * ((n[2] + z - 1) / z);
      offer(rows, (int)z, plane * (double)((u + slots - 1) / slots) * ((double)z + p));
    }
  }
  return best;
}

// ------------------------------------------------------------- conversions
template <typename T>
__global__ void convert_kernel(T *U, size_t N, int to_primitive) {
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < N; c += (size_t)gridDim.x * blockDim.x) {
    T a[NV], b[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) a[k] = U[k * N + c];
    if (to_primitive) cons_to_prim(a, b);
    else prim_to_cons(a, b);
#pragma unroll
    for (int k = 0; k < NV; k++) U[k * N + c] = b[k];
  }
}

template <typename T>
cudaError_t launch_step(const StepArgs<T> &a, int ndim, int rows, bool retry, cudaStream_t s, int *nblocks_out) {
  if (nblocks_out) *nblocks_out = step_blocks<T>(ndim, rows, a.nx, a.ny, a.nz, a.zchunk);
  return retry ? launch_step_mode<T, 0, true>(a, ndim, rows, s) : launch_step_mode<T, 0, false>(a, ndim, rows, s);
}

template <typename T>
cudaError_t launch_scan(const T *src, T *dst, bool prim, int32_t *flags, size_t N, int ndim, const double *dx,
                        Partial *part, const ScanEnd &end, cudaStream_t s, size_t c0, size_t c1, bool maxf) {
  static_assert(kFinalizeThreads == 256, "scan blocks finalize");
  const T ix = (T)(1.0 / dx[0]), iy = (T)(1.0 / dx[1]), iz = (T)(1.0 / dx[2]);
  if (c1 == 0) c1 = N;
  const int nb = (int)std::max<size_t>(1, std::min<size_t>((c1 - c0 + 255) / 256, (size_t)kScanBlocks)), p = prim;
  if (ndim == 1) scan_kernel<T, 1, false><<<nb, 256, 0, s>>>(src, dst, p, flags, N, c0, c1, ix, iy, iz, part, end);
  else if (ndim == 2 && maxf)
    scan_kernel<T, 2, true><<<nb, 256, 0, s>>>(src, dst, p, flags, N, c0, c1, ix, iy, iz, part, end);
  else if (ndim == 2) scan_kernel<T, 2, false><<<nb, 256, 0, s>>>(src, dst, p, flags, N, c0, c1, ix, iy, iz, part, end);
  else if (maxf) scan_kernel<T, 3, true><<<nb, 256, 0, s>>>(src, dst, p, flags, N, c0, c1, ix, iy, iz, part, end);
  else scan_kernel<T, 3, false><<<nb, 256, 0, s>>>(src, dst, p, flags, N, c0, c1, ix, iy, iz, part, end);
  return cudaGetLastError();
}

cudaError_t launch_accept(Ctrl *ctrl, const void *src, void *dst, size_t bytes, cudaStream_t s) {
  const size_t n = bytes / 8;
  const int blocks = (int)std::max<size_t>(1, std::min<size_t>((n / 2 + 255) / 256, 8 * (size_t)kScanBlocks));
  accept_kernel<<<blocks, 256, 0, s>>>(ctrl, static_cast<const uint2 *>(src), static_cast<uint2 *>(dst), n);
  return cudaGetLastError();
}

cudaError_t launch_set_dt(Ctrl *ctrl, double dt, cudaStream_t s) {
  set_dt_kernel<<<1, 1, 0, s>>>(ctrl, dt);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gravity_field(const double *phi, T *acc, int ndim, int nx, int ny, int nz, const double *dx,
                                 cudaStream_t s) {
  gravity_field_kernel<T><<<kScanBlocks, 256, 0, s>>>(phi, acc, ndim, nx, ny, nz, dx[0], dx[1], dx[2]);
  return cudaGetLastError();
}

cudaError_t launch_finalize(Ctrl *ctrl, const Partial *part, int nparts, int mode, cudaStream_t s,
                            unsigned *scan_count) {
  finalize_kernel<<<1, kFinalizeThreads, 0, s>>>(ctrl, part, nparts, mode, scan_count);
  return cudaGetLastError();
}

// go on with a run that stopped with kStatusPending
__global__ void resume_kernel(Ctrl *c) {
  c->status = 0;
  c->done = 0;
}

cudaError_t launch_resume(Ctrl *ctrl, cudaStream_t s) {
  resume_kernel<<<1, 1, 0, s>>>(ctrl);
  return cudaGetLastError();
}

cudaError_t launch_run_start(Ctrl *ctrl, double t_end, int64_t max_steps, double dt_max, cudaStream_t s) {
  run_start_kernel<<<1, 1, 0, s>>>(ctrl, t_end, max_steps, dt_max);
  return cudaGetLastError();
}

template <typename T> cudaError_t launch_convert(T *U, size_t N, int to_primitive, cudaStream_t s) {
  const int blocks = (int)((N + 255) / 256 < (size_t)kScanBlocks ? (N + 255) / 256 : kScanBlocks);
  convert_kernel<T><<<blocks > 0 ? blocks : 1, 256, 0, s>>>(U, N, to_primitive);
  return cudaGetLastError();
}

#define MSH_INST(T)                                                                                   \
  template cudaError_t launch_step<T>(const StepArgs<T> &, int, int, bool, cudaStream_t, int *);     \
  template int step_blocks<T>(int, int, int, int, int, int);                                         \
  template size_t step_smem<T>(int, int, bool, bool);                                                    \
  template cudaError_t launch_scan<T>(const T *, T *, bool, int32_t *, size_t, int, const double *, Partial *, \
                                      const ScanEnd &, cudaStream_t, size_t, size_t, bool);           \
  template cudaError_t launch_convert<T>(T *, size_t, int, cudaStream_t);                            \
  template cudaError_t launch_gravity_field<T>(const double *, T *, int, int, int, int, const double *, cudaStream_t);
MSH_INST(float)
MSH_INST(double)

}  // namespace msh
