// msh_batch.cu -- thousands of independent 1D Riemann problems ("tubes") in one
// persistent launch.
//
// Each thread block repeatedly takes the next tube from a device work queue (tubes are
// ordered longest first on the host, since the work of a tube grows as len^2), loads it
// into shared memory and advances it to its own t_end with a block-local CFL reduction;
// the tube never leaves shared memory until it is finished.  In shared memory a tube is held
// in primitive variables W, so the reconstruction reads its three cells without
// conversions; per step every warp sweeps segments of 30 cells on its own (tube_pass) into
// the second tube buffer, and the buffers swap roles, so W^n stays intact for the fallback
// passes without a copy.  A step costs two block barriers; between them one thread plans the
// time step.  Tubes go to the kernel in up to three classes by length, launched side by side:
// long FP32 tubes need a whole SM's shared memory for their two buffers (16 warps, one block per
// SM), shorter ones two or four blocks per SM with 8 or 4 warps each, which hide each other's
// time control and fill the SMs that the long tubes leave.  FP64 tubes: see tube_classes, and
// takes_chunks for their second form of the sweep.
// Bound: instruction issue.  4096 tubes of 128 to 2048 cells to t = 0.1 (7.4e8 cell updates):
// 27.9 ms with one tube per block of 256 threads, three barriers per chunk and every thread
// planning the time step; 19.6 ms now (14.7 + 3.8 + 1.1 for the three classes one after another),
// 0.61 to 0.65 instructions per scheduler and cycle.
// The step is the same as the grid kernels': MUSCL-Hancock on the characteristic
// variables (Sec. 3.3), HLL flux, outflow boundaries by index clamping, CFL time step
// dt = C dx / max(|u| + sqrt(3 P_xx/rho)) with the last step clipped to t_end.
#include <climits>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>
#include <algorithm>
#include <numeric>

#include "../../include/msh.h"
#include "msh_device.cuh"
#include "msh_internal.h"

namespace msh {

template <typename T> struct TubeArgs {
  T *U;                    // [NV][total] conserved, tubes back to back
  const int64_t *off;      // [ntubes] first cell of each tube
  const int32_t *len;      // [ntubes]
  const double *t_end;     // [ntubes]
  const int32_t *order;    // [ntubes] processing order (longest first)
  int32_t *queue;          // work-queue head: tubes order[first + *queue] .. order[last - 1]
  int32_t first, last;
  int64_t *steps;          // [ntubes] out
  double *t_out;           // [ntubes] out
  int32_t *status;         // [ntubes] out: 0 ok, 4 non-realizable, 5 step cap reached
  int64_t *fallback;       // [ntubes] out: steps whose second-order update tagged cells
  int64_t total;
  int32_t cap;             // shared-memory capacity in cells (>= max len)
  double cfl;
  int64_t max_steps;
};

template <typename T> __device__ __forceinline__ void load_w(const T *sW, int cap, int c, int n, T (&W)[NV]) {
  const int cc = min(max(c, 0), n - 1);  // outflow: zero-gradient copy of the edge cell
#pragma unroll
  for (int k = 0; k < NV; k++) W[k] = sW[k * cap + cc];
}

__device__ __forceinline__ float warp_max_speed(float v) {  // v >= 0
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ double warp_max_speed(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max_of(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

template <typename T> __device__ __forceinline__ T tube_speed(const T (&W)[NV], T idx) {
  return signal_speed(W[1], W[4], W[0]) * idx;
}

// One sweep of a tube, segment by segment of kTubeSeg cells, the warps of the block taking
// segments in turn.  Lane l of a warp holds cell first - 1 + l: it reconstructs its cell from
// shared memory, takes the upper face state of its left neighbour and the flux through its
// upper face by warp shuffles, and (lanes 1 .. 30) updates its cell into dst, so no warp waits
// for another within a sweep.  src holds W^n; dst (another buffer) receives W^{n+1}.  With
// FALLBACK, every face that touches a cell tagged by an earlier pass (sFl == 2) takes
// first-order states.  Cells whose update is not realizable and that carry no active tag are
// tagged (sFl = 1) and *s_nbad is set.  Returns the lane's maximum signal speed of the new state.
constexpr int kTubeSeg = 30;
template <typename T, int NT, bool FALLBACK>
__device__ __forceinline__ T tube_pass(const T *src, T *dst, unsigned char *sFl, int n, int cap, T nu, T dtdx, T idx,
                                       int *s_nbad, int *s_any) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T smax = T(0);
  for (int b = warp * kTubeSeg; b < n; b += (NT / 32) * kTubeSeg) {
    const int c = b - 1 + lane;
    T lo[NV], hi[NV], w0[NV], F[NV];
    {
      T wm[NV], wp[NV];
      load_w(src, cap, c - 1, n, wm);
      load_w(src, cap, c, n, w0);
      load_w(src, cap, c + 1, n, wp);
      reconstruct(wm, w0, wp, nu, lo, hi);
      if (FALLBACK) {  // tags of earlier passes (value 2) are active in this pass
        auto f = [&](int i) { return sFl[min(max(i, 0), n - 1)] == 2; };
        first_order_faces(f(c - 1), f(c), f(c + 1), w0, lo, hi);
      }
    }
    {
      T hl[NV];
#pragma unroll
      for (int v = 0; v < NV; v++) hl[v] = __shfl_up_sync(0xffffffffu, hi[v], 1);
      hll(hl, lo, F);  // flux through the lower face (lane 0: not used)
    }
    T U[NV], W[NV];
    prim_to_cons(w0, U);
#pragma unroll
    for (int v = 0; v < NV; v++) U[v] -= dtdx * (__shfl_down_sync(0xffffffffu, F[v], 1) - F[v]);
    if (lane >= 1 && lane <= kTubeSeg && c < n) {
      cons_to_prim(U, W);
#pragma unroll
      for (int v = 0; v < NV; v++) dst[v * cap + c] = W[v];
      if (!realizable(W)) {
        *s_any = 1;
        if (sFl[c] != 2) {  // newly failing cell: tag it for the next pass
          sFl[c] = 1;
          *s_nbad = 1;
        }
      }
      smax = fmax(smax, tube_speed(W, idx));
    }
  }
  return smax;
}

// The same sweep chunk by chunk of NT cells, the face states and fluxes exchanged through shared
// memory (FP64): no cell is reconstructed twice, at three barriers per chunk.  The update of a cell
// runs one chunk position behind its reconstruction, when both its faces are known.
//
// Which of the two sweeps is the faster one follows from the most loaded scheduler: a
// double-precision instruction costs the same at any lane count, and of n cells segments of 30 leave
// it ceil(ceil(n / 30) / 4) groups of 32 lanes, chunks of n + 2 positions ceil((n + 2) / 128).  FP64
// tubes take chunks where that is fewer (n = 121 .. 126, 241 .. 254, 481 .. 510 ...) and segments, which
// need no barriers, otherwise (blocks of 8 warps, one per SM: 64 tubes of 240 to 250 cells take 27 %
// less time by chunks, 152 tubes of 205 to 256 cells, the slowest of them of 256, 5 % more).
__device__ __forceinline__ bool takes_chunks(int n) { return (n + 129) / 128 < (n + 119) / 120; }
template <typename T, int NT, bool FALLBACK>
__device__ __forceinline__ T tube_pass_chunks(const T *src, T *dst, unsigned char *sFl, int n, int cap, T nu, T dtdx,
                                              T idx, T *sF, T *sH, T *sHc, int *s_nbad, int *s_any) {
  const int t = threadIdx.x;
  T smax = T(0);
  for (int b = -1; b <= n; b += NT) {
    const int c = b + t;
    T lo[NV], hi[NV], wm[NV];  // wm: W^n of the cell this thread updates (c - 1)
    if (c <= n) {
      T w0[NV], wp[NV];
      load_w(src, cap, c - 1, n, wm);
      load_w(src, cap, c, n, w0);
      load_w(src, cap, c + 1, n, wp);
      reconstruct(wm, w0, wp, nu, lo, hi);
      if (FALLBACK) {  // tags of earlier passes (value 2) are active in this pass
        auto f = [&](int i) { return sFl[min(max(i, 0), n - 1)] == 2; };
        first_order_faces(f(c - 1), f(c), f(c + 1), w0, lo, hi);
      }
#pragma unroll
      for (int v = 0; v < NV; v++) sH[v * NT + t] = hi[v];
    }
    __syncthreads();
    if (c >= 0 && c <= n) {
      T hl[NV], F[NV];
#pragma unroll
      for (int v = 0; v < NV; v++) hl[v] = (t > 0) ? sH[v * NT + t - 1] : sHc[v];
      hll(hl, lo, F);
#pragma unroll
      for (int v = 0; v < NV; v++) sF[v * (NT + 1) + t + 1] = F[v];
    }
    __syncthreads();
    // the last thread hands its upper face state to the next chunk (read after the next barrier;
    // every read of the current one happened before the barrier above)
    if (t == NT - 1 && c <= n) {
#pragma unroll
      for (int v = 0; v < NV; v++) sHc[v] = hi[v];
    }
    const int cu = c - 1;
    if (cu >= 0 && cu < n) {
      T U[NV], W[NV];
      prim_to_cons(wm, U);
#pragma unroll
      for (int v = 0; v < NV; v++) U[v] -= dtdx * (sF[v * (NT + 1) + t + 1] - sF[v * (NT + 1) + t]);
      cons_to_prim(U, W);
#pragma unroll
      for (int v = 0; v < NV; v++) dst[v * cap + cu] = W[v];
      if (!realizable(W)) {
        *s_any = 1;
        if (sFl[cu] != 2) {
          sFl[cu] = 1;
          *s_nbad = 1;
        }
      }
      smax = fmax(smax, tube_speed(W, idx));
    }
    __syncthreads();
    if (t == 0) {  // the last face of this chunk is the lower face of the next chunk's first update
#pragma unroll
      for (int v = 0; v < NV; v++) sF[v * (NT + 1)] = sF[v * (NT + 1) + NT];
    }
  }
  return smax;
}

// What the block does next with its tube (thread 0 decides between the passes).
enum { TUBE_DONE = 0, TUBE_STEP = 1, TUBE_RETRY = 2 };

template <typename T, int NT>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 512 / NT : 256 / NT) tubes_kernel(TubeArgs<T> a) {
  constexpr bool CHUNKS = sizeof(T) == 8;  // the chunk form too
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int cap = a.cap;
  // two tube buffers (primitive): a step reads W^n from one and writes W^{n+1} to the other
  // (the fallback passes re-read the untouched W^n), then the two swap roles
  T *sU = reinterpret_cast<T *>(smem_raw);  // [NV][cap]
  T *sUo = sU + (size_t)NV * cap;           // [NV][cap]
  // chunk form: [NV][NT+1] fluxes (0: the one carried over), [NV][NT] upper face states, [NV] the
  // one carried over
  T *sF = sUo + (size_t)NV * cap, *sH = sF + (CHUNKS ? NV * (NT + 1) : 0), *sHc = sH + (CHUNKS ? NV * NT : 0);
  unsigned char *sFl = reinterpret_cast<unsigned char *>(sHc + (CHUNKS ? NV : 0));  // [cap] fallback tags
  constexpr int kWarps = NT / 32;
  __shared__ T red[kWarps];
  __shared__ T s_dt;
  __shared__ int s_q, s_act, s_swap, s_clear;
  __shared__ int s_nbad, s_any;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (;;) {
    if (t == 0) s_q = atomicAdd(a.queue, 1);
    __syncthreads();
    const int q = a.first + s_q;
    if (q >= a.last) break;
    const int k = a.order[q];
    const int n = a.len[k];
    const int64_t off = a.off[k];
    const bool chunks = CHUNKS && takes_chunks(n);
    T *cur = sU, *nxt = sUo;  // W^n and W^{n+1} of the current step
    const T idx = (T)n, half_idx = T(0.5) * idx;
    T smax = T(0);  // signal speed of the initial state
    for (int c = t; c < n; c += NT) {
      T U[NV], W[NV];
#pragma unroll
      for (int v = 0; v < NV; v++) U[v] = a.U[v * a.total + off + c];
      cons_to_prim(U, W);
#pragma unroll
      for (int v = 0; v < NV; v++) cur[v * cap + c] = W[v];
      sFl[c] = 0;
      smax = fmax(smax, tube_speed(W, idx));
    }
    // the time control, in thread 0 alone: its FP64 arithmetic (a division, sums, conversions)
    // would hold every scheduler's FP64 pipe for each warp that repeats it
    double tt = 0.0, tn = 0.0;
    const double te = a.t_end[k];
    int64_t steps = 0, fb_steps = 0;
    int status = 0, pass = 0, started = 0;
    if (t == 0) {
      s_nbad = 0;
      s_any = 0;
    }
    for (;;) {
      smax = warp_max_speed(smax);
      if (lane == 0) red[warp] = smax;
      __syncthreads();
      if (t == 0) {
        int act = TUBE_STEP;
        s_swap = 0;
        s_clear = 0;
        if (started) {
          if (pass == 0) fb_steps += s_nbad != 0;
          if (s_nbad && pass < kFallbackPasses) {
            // a-posteriori fallback: redo the step from W^n with first-order faces at every
            // tagged cell; cells still failing are tagged too
            act = TUBE_RETRY;
            pass++;
          } else {  // the step stands
            s_swap = 1;
            s_clear = pass > 0 || s_nbad;
            tt = tn;
            steps++;
            pass = 0;
            if (s_any) {
              status = 4;
              act = TUBE_DONE;
            }
          }
        }
        if (act == TUBE_STEP && !(tt < te)) act = TUBE_DONE;
        if (act == TUBE_STEP && steps >= a.max_steps) {
          status = 5;
          act = TUBE_DONE;
        }
        if (act == TUBE_STEP) {
          T sm = red[0];
          for (int w = 1; w < kWarps; w++) sm = fmax(sm, red[w]);
          double dt = a.cfl / (double)sm;
          tn = tt + dt;
          if (tn >= te) {
            dt = te - tt;
            tn = te;
          }
          s_dt = (T)dt;
        }
        started = 1;
        s_act = act;
        s_nbad = 0;
        s_any = 0;
      }
      __syncthreads();
      const int act = s_act;
      if (s_swap) {
        T *sw = cur;  // W^{n+1} becomes the next step's W^n
        cur = nxt;
        nxt = sw;
      }
      if (s_clear) {
        for (int c = t; c < n; c += NT) sFl[c] = 0;
        __syncthreads();
      }
      if (act == TUBE_DONE) break;
      const T dt = s_dt, nu = dt * half_idx, dtdx = dt * idx;
      if (act == TUBE_RETRY) {
        for (int c = t; c < n; c += NT)
          if (sFl[c] == 1) sFl[c] = 2;  // tags of earlier passes become active
        __syncthreads();
        if (CHUNKS && chunks)
          smax = tube_pass_chunks<T, NT, true>(cur, nxt, sFl, n, cap, nu, dtdx, idx, sF, sH, sHc, &s_nbad, &s_any);
        else smax = tube_pass<T, NT, true>(cur, nxt, sFl, n, cap, nu, dtdx, idx, &s_nbad, &s_any);
      } else {
        if (CHUNKS && chunks)
          smax = tube_pass_chunks<T, NT, false>(cur, nxt, sFl, n, cap, nu, dtdx, idx, sF, sH, sHc, &s_nbad, &s_any);
        else smax = tube_pass<T, NT, false>(cur, nxt, sFl, n, cap, nu, dtdx, idx, &s_nbad, &s_any);
      }
    }
    for (int c = t; c < n; c += NT) {
      T W[NV], U[NV];
#pragma unroll
      for (int v = 0; v < NV; v++) W[v] = cur[v * cap + c];
      prim_to_cons(W, U);
#pragma unroll
      for (int v = 0; v < NV; v++) a.U[v * a.total + off + c] = U[v];
    }
    if (t == 0) {
      a.steps[k] = steps;
      a.t_out[k] = tt;
      a.status[k] = status;
      a.fallback[k] = fb_steps;
    }
    __syncthreads();
  }
}

// FP64 blocks hold the chunk form's buffers too.
template <typename T> size_t tube_smem(int cap, int nt) {
  return sizeof(T) * NV * (2 * (size_t)cap + (sizeof(T) == 8 ? 2 * nt + 2 : 0)) + (size_t)cap;
}

template <typename T, int NT> static cudaError_t launch_tubes_nt(const TubeArgs<T> &a, cudaStream_t s) {
  const size_t smem = tube_smem<T>(a.cap, NT);
  cudaError_t e = cudaFuncSetAttribute(tubes_kernel<T, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int dev = 0, sms = 0, per_sm = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, tubes_kernel<T, NT>, NT, smem);
  if (e != cudaSuccess) return e;
  const int blocks = std::min(sms * std::max(1, per_sm), (int)(a.last - a.first));
  tubes_kernel<T, NT><<<blocks, NT, smem, s>>>(a);
  return cudaGetLastError();
}

template <typename T> cudaError_t launch_tubes(const TubeArgs<T> &a, int nt, cudaStream_t s) {
  if (nt == 64) return launch_tubes_nt<T, 64>(a, s);
  if (nt == 128) return launch_tubes_nt<T, 128>(a, s);
  if (nt == 512) return launch_tubes_nt<T, 512>(a, s);
  return launch_tubes_nt<T, 256>(a, s);
}

}  // namespace msh

// ======================================================================= host
using namespace msh;

namespace {
msh_status bfail(msh_status s, const char *fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  set_error_text(buf);
  return s;
}
#define B_TRY(expr)                                                                             \
  do {                                                                                          \
    cudaError_t e_ = (expr);                                                                    \
    if (e_ != cudaSuccess)                                                                      \
      return bfail(e_ == cudaErrorMemoryAllocation ? MSH_E_NOMEM : MSH_E_CUDA, "%s: %s", #expr, \
                   cudaGetErrorString(e_));                                                     \
  } while (0)
}  // namespace

struct msh_batch {
  int ntubes = 0;
  int prec = MSH_FP32;
  size_t esize = 4;
  double cfl = 0.8;
  int64_t total = 0;
  int cap = 0;
  std::vector<int32_t> order;
  cudaStream_t aux[2] = {nullptr, nullptr};  // side streams of the shorter classes
  cudaEvent_t ev_fork = nullptr, ev_join[2] = {nullptr, nullptr};
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<int32_t> len;
  std::vector<int64_t> off;
  std::vector<double> t_end;
  std::vector<unsigned char> init;  // initial conserved state, host copy for reset
  bool advanced = false;            // the state is no longer the initial one
  bool sized = false;               // a run chose its block sizes itself (threads = 0)
  void *U = nullptr;
  int64_t *d_off = nullptr;
  int32_t *d_len = nullptr, *d_order = nullptr, *d_queue = nullptr, *d_status = nullptr;
  double *d_tend = nullptr, *d_t = nullptr;
  int64_t *d_steps = nullptr;
  int64_t *d_fallback = nullptr;
  std::vector<msh_grid *> grids;  // per-tube grids of the per-launch baseline (lazily built)
};

namespace {

template <typename T> void fill_initial(msh_batch *b, const double *WL, const double *WR) {
  T *h = reinterpret_cast<T *>(b->init.data());
  for (int k = 0; k < b->ntubes; k++) {
    const int n = b->len[k];
    for (int i = 0; i < n; i++) {
      const double x = (i + 0.5) / n;
      const double *w = (x < 0.5) ? WL + 10 * k : WR + 10 * k;
      for (int v = 0; v < NV; v++) h[v * b->total + b->off[k] + i] = (T)w[v];
    }
  }
}

msh_status upload_initial(msh_batch *b) {
  const size_t bytes = (size_t)b->total * NV * b->esize;
  B_TRY(cudaMemcpyAsync(b->U, b->init.data(), bytes, cudaMemcpyHostToDevice, b->stream));
  cudaError_t e = b->prec == MSH_FP32 ? launch_convert<float>((float *)b->U, (size_t)b->total, 0, b->stream)
                                      : launch_convert<double>((double *)b->U, (size_t)b->total, 0, b->stream);
  if (e != cudaSuccess) return bfail(MSH_E_CUDA, "convert: %s", cudaGetErrorString(e));
  B_TRY(cudaMemsetAsync(b->d_steps, 0, sizeof(int64_t) * b->ntubes, b->stream));
  B_TRY(cudaMemsetAsync(b->d_fallback, 0, sizeof(int64_t) * b->ntubes, b->stream));
  B_TRY(cudaMemsetAsync(b->d_t, 0, sizeof(double) * b->ntubes, b->stream));
  B_TRY(cudaMemsetAsync(b->d_status, 0, sizeof(int32_t) * b->ntubes, b->stream));
  B_TRY(cudaStreamSynchronize(b->stream));
  return MSH_OK;
}

// A class of tubes: order[first .. last) on blocks of nt threads.
struct TubeClass {
  int first, last, nt;
};

// threads > 0: every tube on blocks of that size.  0: by length.
// FP32: 16 warps per tube above 1024 cells, 8 above 512, 4 below (each class fills an SM with 16
// warps).  Batches too small to fill the SMs so: a class takes twice the warps, longest first, while
// all its tubes' warps still run at once and have segments to sweep.
// FP64, whose buffers are twice as large and whose pipe two warps per scheduler saturate: 8 warps
// per tube, one tube per SM; many short tubes take blocks of 4 warps (up to 126 cells, whose sweep
// leaves one group of lanes to every scheduler) or 2, two or four per SM.  Times to t = 0.02 with
// 2 / 4 / 8 warps: 220 tubes of 113 to 126 cells 0.64 / 0.46 / 0.44 ms, 600 of them 0.84 / 0.70 / 0.79;
// 300 of 31 to 62 cells 0.28 / 0.19 / 0.21; 600 of 16 to 32 cells 0.146 / 0.144 / 0.20, 2000 of them
// 0.20 / 0.29 / 0.50; 2000 of 31 to 62 cells 0.43 / 0.47 / 0.79.
std::vector<TubeClass> tube_classes(const msh_batch *b, int threads) {
  std::vector<TubeClass> cls;
  if (threads > 0) {
    cls.push_back({0, b->ntubes, threads});
    return cls;
  }
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    (void)cudaGetLastError();
    sms = 1;
  }
  auto longer = [&](int n) {  // tubes of more than n cells
    int i = 0;
    while (i < b->ntubes && b->len[b->order[i]] > n) i++;
    return i;
  };
  const bool f32 = b->prec == MSH_FP32;
  const int tiny = b->ntubes - longer(62) > 12 * sms ? 62 : 30;
  int cut[2] = {longer(f32 ? 1024 : 126), longer(f32 ? 512 : tiny)}, nt[3] = {f32 ? 512 : 256, f32 ? 256 : 128, f32 ? 128 : 64};
  if (!f32) {  // classes of few tubes join the next longer one
    if (b->ntubes - cut[1] <= 2 * sms) cut[1] = b->ntubes;
    if (cut[1] > cut[0] && cut[1] - cut[0] <= (b->len[b->order[cut[0]]] <= 62 ? sms : 2 * sms)) cut[0] = cut[1];
  }
  const int end[4] = {0, cut[0], cut[1], b->ntubes};
  for (int i = 0; i < 3; i++)
    if (end[i + 1] > end[i]) cls.push_back({end[i], end[i + 1], nt[i]});
  if (!f32) return cls;
  long long room = (long long)sms * 16;  // warps that run at once
  for (const TubeClass &c : cls) room -= (long long)(c.last - c.first) * (c.nt / 32);
  for (TubeClass &c : cls)
    while (c.nt < nt[0] && c.nt / 32 * kTubeSeg < b->len[b->order[c.first]] &&
           (long long)(c.last - c.first) * (c.nt / 32) <= room) {
      room -= (long long)(c.last - c.first) * (c.nt / 32);
      c.nt *= 2;
    }
  return cls;
}

template <typename T> cudaError_t launch_class(msh_batch *b, const TubeClass &c, int i, int64_t max_steps, cudaStream_t s) {
  TubeArgs<T> a{(T *)b->U, b->d_off, b->d_len, b->d_tend, b->d_order, b->d_queue + i, c.first, c.last, b->d_steps, b->d_t,
                b->d_status, b->d_fallback, b->total, b->len[b->order[c.first]], b->cfl, max_steps};
  return launch_tubes<T>(a, c.nt, s);
}

msh_status run_once(msh_batch *b, int threads, int64_t max_steps) {
  const std::vector<TubeClass> cls = tube_classes(b, threads);
  B_TRY(cudaMemsetAsync(b->d_queue, 0, 3 * sizeof(int32_t), b->stream));
  if (cls.size() > 1) B_TRY(cudaEventRecord(b->ev_fork, b->stream));
  for (size_t i = 0; i < cls.size(); i++) {
    cudaStream_t s = i == 0 ? b->stream : b->aux[i - 1];
    if (i > 0) B_TRY(cudaStreamWaitEvent(s, b->ev_fork, 0));
    const cudaError_t e = b->prec == MSH_FP32 ? launch_class<float>(b, cls[i], (int)i, max_steps, s)
                                              : launch_class<double>(b, cls[i], (int)i, max_steps, s);
    if (e != cudaSuccess) return bfail(MSH_E_CUDA, "tube kernel launch: %s", cudaGetErrorString(e));
    if (i > 0) {
      B_TRY(cudaEventRecord(b->ev_join[i - 1], s));
      B_TRY(cudaStreamWaitEvent(b->stream, b->ev_join[i - 1], 0));
    }
  }
  return MSH_OK;
}

msh_status check_status(msh_batch *b) {
  std::vector<int32_t> st(b->ntubes);
  B_TRY(cudaMemcpyAsync(st.data(), b->d_status, sizeof(int32_t) * b->ntubes, cudaMemcpyDeviceToHost, b->stream));
  B_TRY(cudaStreamSynchronize(b->stream));
  for (int k = 0; k < b->ntubes; k++) {
    if (st[k] == 4) return bfail(MSH_E_REALIZABILITY, "tube %d became non-realizable", k);
    if (st[k] == 5) return bfail(MSH_E_TIMEOUT, "tube %d reached max_steps before t_end", k);
  }
  return MSH_OK;
}

}  // namespace

extern "C" {

msh_status msh_batch_init(msh_batch **out, int32_t ntubes, const int32_t *len, const double *WL, const double *WR,
                          const double *t_end, int32_t precision, double cfl, void *stream) {
  clear_error();
  if (!out || !len || !WL || !WR || !t_end) return bfail(MSH_E_INVALID_ARG, "null argument");
  if (ntubes < 1) return bfail(MSH_E_INVALID_ARG, "ntubes must be >= 1");
  if (precision != MSH_FP32 && precision != MSH_FP64) return bfail(MSH_E_INVALID_ARG, "bad precision");
  if (!(cfl > 0.0 && cfl <= 1.0)) return bfail(MSH_E_INVALID_ARG, "cfl must be in (0, 1]");
  const int maxlen = precision == MSH_FP32 ? 2048 : 1024;
  int cap = 0;
  for (int k = 0; k < ntubes; k++) {
    if (len[k] < 4 || len[k] > maxlen) return bfail(MSH_E_INVALID_ARG, "len[%d] = %d outside [4, %d]", k, len[k], maxlen);
    if (!(t_end[k] > 0.0) || !std::isfinite(t_end[k])) return bfail(MSH_E_INVALID_ARG, "t_end[%d] must be > 0", k);
    for (int v = 0; v < NV; v++)
      if (!std::isfinite(WL[10 * k + v]) || !std::isfinite(WR[10 * k + v]))
        return bfail(MSH_E_INVALID_ARG, "non-finite state of tube %d", k);
    // realizability of the two input states (rho > 0, P SPD)
    for (const double *w : {WL + 10 * k, WR + 10 * k}) {
      const double m2 = w[4] * w[7] - w[5] * w[5];
      const double m3 = w[4] * (w[7] * w[9] - w[8] * w[8]) - w[5] * (w[5] * w[9] - w[8] * w[6]) +
                        w[6] * (w[5] * w[8] - w[7] * w[6]);
      if (!(w[0] > 0 && w[4] > 0 && m2 > 0 && m3 > 0))
        return bfail(MSH_E_REALIZABILITY, "input state of tube %d not realizable", k);
    }
    cap = std::max(cap, (int)len[k]);
  }
  int dev_count = 0;
  if (cudaGetDeviceCount(&dev_count) != cudaSuccess || dev_count == 0)
    return bfail(MSH_E_CUDA, "no CUDA device available (libmsh has no CPU path)");
  msh_batch *b = new (std::nothrow) msh_batch();
  if (!b) return bfail(MSH_E_NOMEM, "host allocation");
  b->ntubes = ntubes;
  b->prec = precision;
  b->esize = precision == MSH_FP32 ? 4 : 8;
  b->cfl = cfl;
  b->cap = cap;
  b->len.assign(len, len + ntubes);
  b->t_end.assign(t_end, t_end + ntubes);
  b->off.resize(ntubes);
  int64_t acc = 0;
  for (int k = 0; k < ntubes; k++) {
    b->off[k] = acc;
    acc += len[k];
  }
  b->total = acc;
  std::vector<int32_t> &order = b->order;
  order.resize(ntubes);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return len[x] > len[y]; });
  b->init.resize((size_t)b->total * NV * b->esize);
  if (precision == MSH_FP32) fill_initial<float>(b, WL, WR);
  else fill_initial<double>(b, WL, WR);
  auto cleanup = [&](msh_status s) {
    msh_batch_destroy(b);
    return s;
  };
  cudaError_t e = cudaSuccess;
  if (stream) b->stream = (cudaStream_t)stream;
  else {
    e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
    b->own_stream = true;
  }
  for (auto &x : b->aux)
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&x, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming);
  for (auto &x : b->ev_join)
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&x, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaMalloc(&b->U, (size_t)b->total * NV * b->esize);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_off, sizeof(int64_t) * ntubes);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_len, sizeof(int32_t) * ntubes);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_order, sizeof(int32_t) * ntubes);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_queue, 3 * sizeof(int32_t));
  if (e == cudaSuccess) e = cudaMalloc(&b->d_status, sizeof(int32_t) * ntubes);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_tend, sizeof(double) * ntubes);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_t, sizeof(double) * ntubes);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_steps, sizeof(int64_t) * ntubes);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_fallback, sizeof(int64_t) * ntubes);
  if (e != cudaSuccess) return cleanup(bfail(MSH_E_NOMEM, "batch allocation: %s", cudaGetErrorString(e)));
  e = cudaMemcpyAsync(b->d_off, b->off.data(), sizeof(int64_t) * ntubes, cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_len, len, sizeof(int32_t) * ntubes, cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->d_order, order.data(), sizeof(int32_t) * ntubes, cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->d_tend, t_end, sizeof(double) * ntubes, cudaMemcpyHostToDevice, b->stream);
  if (e != cudaSuccess) return cleanup(bfail(MSH_E_CUDA, "batch upload: %s", cudaGetErrorString(e)));
  msh_status st = upload_initial(b);
  if (st) return cleanup(st);
  *out = b;
  return MSH_OK;
}

msh_status msh_batch_reset(msh_batch *b) {
  clear_error();
  if (!b) return bfail(MSH_E_INVALID_ARG, "null batch");
  b->advanced = false;
  return upload_initial(b);
}

msh_status msh_batch_run(msh_batch *b, int32_t threads, int64_t max_steps) {
  msh::NvtxRange nvtx_range("msh_batch_run");
  clear_error();
  if (!b) return bfail(MSH_E_INVALID_ARG, "null batch");
  if (threads != 0 && threads != 128 && threads != 256 && threads != 512)
    return bfail(MSH_E_INVALID_ARG, "threads must be 0, 128, 256 or 512");
  if (max_steps < 1) return bfail(MSH_E_INVALID_ARG, "max_steps must be >= 1");
  const size_t smem = b->prec == MSH_FP32 ? tube_smem<float>(b->cap, threads) : tube_smem<double>(b->cap, threads);
  if (threads > 0 && smem > 227 * 1024)
    return bfail(MSH_E_INVALID_ARG, "tubes too long for %d threads (%zu B shared)", threads, smem);
  // the first run with threads = 0 starts from the initial state, whatever ran before it
  if (threads == 0 && !b->sized && b->advanced) {
    const msh_status st0 = upload_initial(b);
    if (st0) return st0;
  }
  b->sized = b->sized || threads == 0;
  b->advanced = true;
  // one persistent launch per class of lengths, captured in a CUDA graph with the queue reset
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  B_TRY(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
  msh_status st = run_once(b, threads, max_steps);
  cudaError_t e = cudaStreamEndCapture(b->stream, &graph);
  if (st) {
    if (graph) cudaGraphDestroy(graph);
    return st;
  }
  if (e != cudaSuccess) return bfail(MSH_E_CUDA, "capture: %s", cudaGetErrorString(e));
  e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return bfail(MSH_E_CUDA, "instantiate: %s", cudaGetErrorString(e));
  e = cudaGraphLaunch(exec, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  cudaGraphExecDestroy(exec);
  if (e != cudaSuccess) return bfail(MSH_E_CUDA, "tube run: %s", cudaGetErrorString(e));
  return check_status(b);
}

msh_status msh_batch_run_per_tube(msh_batch *b, const int32_t *tubes, int32_t count, int64_t max_steps) {
  msh::NvtxRange nvtx_range("msh_batch_run_per_tube");
  clear_error();
  if (!b) return bfail(MSH_E_INVALID_ARG, "null batch");
  if (tubes && count < 0) return bfail(MSH_E_INVALID_ARG, "bad count");
  const int m = tubes ? count : b->ntubes;
  b->advanced = true;
  if ((int)b->grids.size() < b->ntubes) b->grids.resize(b->ntubes, nullptr);
  for (int i = 0; i < m; i++) {
    const int k = tubes ? tubes[i] : i;
    if (k < 0 || k >= b->ntubes) return bfail(MSH_E_INVALID_ARG, "tube index %d out of range", k);
    if (!b->grids[k]) {
      const int64_t n3[3] = {b->len[k], 1, 1};
      const double lo[3] = {0, 0, 0}, hi[3] = {1, 1, 1};
      const int32_t bc[6] = {MSH_BC_OUTFLOW, MSH_BC_OUTFLOW, 0, 0, 0, 0};
      msh_status st = msh_init_grid(&b->grids[k], 1, n3, lo, hi, bc, b->prec, b->cfl, b->stream);
      if (st) return bfail(st, "per-tube grid: %s", msh_last_error());
    }
    msh_grid *g = b->grids[k];
    const size_t n = (size_t)b->len[k];
    // gather tube k ([10][n]) from the batch state, run it alone, scatter it back
    void *tmp = nullptr;
    B_TRY(cudaMallocAsync(&tmp, n * NV * b->esize, b->stream));
    B_TRY(cudaMemcpy2DAsync(tmp, n * b->esize, (char *)b->U + b->off[k] * b->esize, b->total * b->esize,
                            n * b->esize, NV, cudaMemcpyDeviceToDevice, b->stream));
    msh_status st = msh_set_time(g, 0.0, 0);
    if (!st) st = msh_set_state(g, tmp, MSH_DEVICE, MSH_CONSERVED);
    int64_t steps = 0;
    double tt = 0.0;
    if (!st) st = msh_run(g, b->t_end[k], max_steps, &steps, &tt);
    if (!st) st = msh_get_state(g, tmp, MSH_DEVICE, MSH_CONSERVED);
    if (st) {
      cudaFreeAsync(tmp, b->stream);
      return bfail(st, "tube %d: %s", k, msh_last_error());
    }
    B_TRY(cudaMemcpy2DAsync((char *)b->U + b->off[k] * b->esize, b->total * b->esize, tmp, n * b->esize,
                            n * b->esize, NV, cudaMemcpyDeviceToDevice, b->stream));
    B_TRY(cudaFreeAsync(tmp, b->stream));
    B_TRY(cudaMemcpyAsync(b->d_steps + k, &steps, sizeof(int64_t), cudaMemcpyHostToDevice, b->stream));
    B_TRY(cudaMemcpyAsync(b->d_t + k, &tt, sizeof(double), cudaMemcpyHostToDevice, b->stream));
    B_TRY(cudaStreamSynchronize(b->stream));
  }
  return MSH_OK;
}

msh_status msh_batch_get_state(msh_batch *b, void *U, int32_t where, int32_t kind) {
  clear_error();
  if (!b || !U) return bfail(MSH_E_INVALID_ARG, "null argument");
  if (where != MSH_HOST && where != MSH_DEVICE) return bfail(MSH_E_INVALID_ARG, "bad where");
  if (kind != MSH_CONSERVED && kind != MSH_PRIMITIVE) return bfail(MSH_E_INVALID_ARG, "bad kind");
  const size_t bytes = (size_t)b->total * NV * b->esize;
  const void *src = b->U;
  void *tmp = nullptr;
  if (kind == MSH_PRIMITIVE) {
    B_TRY(cudaMallocAsync(&tmp, bytes, b->stream));
    B_TRY(cudaMemcpyAsync(tmp, b->U, bytes, cudaMemcpyDeviceToDevice, b->stream));
    cudaError_t e = b->prec == MSH_FP32 ? launch_convert<float>((float *)tmp, (size_t)b->total, 1, b->stream)
                                        : launch_convert<double>((double *)tmp, (size_t)b->total, 1, b->stream);
    if (e != cudaSuccess) return bfail(MSH_E_CUDA, "convert: %s", cudaGetErrorString(e));
    src = tmp;
  }
  B_TRY(cudaMemcpyAsync(U, src, bytes, where == MSH_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice,
                        b->stream));
  if (tmp) B_TRY(cudaFreeAsync(tmp, b->stream));
  B_TRY(cudaStreamSynchronize(b->stream));
  return MSH_OK;
}

msh_status msh_batch_info(msh_batch *b, int64_t *steps, double *t, int64_t *cell_updates) {
  clear_error();
  if (!b) return bfail(MSH_E_INVALID_ARG, "null batch");
  std::vector<int64_t> s(b->ntubes);
  std::vector<double> tt(b->ntubes);
  B_TRY(cudaMemcpyAsync(s.data(), b->d_steps, sizeof(int64_t) * b->ntubes, cudaMemcpyDeviceToHost, b->stream));
  B_TRY(cudaMemcpyAsync(tt.data(), b->d_t, sizeof(double) * b->ntubes, cudaMemcpyDeviceToHost, b->stream));
  B_TRY(cudaStreamSynchronize(b->stream));
  if (steps) memcpy(steps, s.data(), sizeof(int64_t) * b->ntubes);
  if (t) memcpy(t, tt.data(), sizeof(double) * b->ntubes);
  if (cell_updates) {
    int64_t cu = 0;
    for (int k = 0; k < b->ntubes; k++) cu += s[k] * b->len[k];
    *cell_updates = cu;
  }
  return MSH_OK;
}

msh_status msh_batch_fallback_steps(msh_batch *b, int64_t *counts) {
  clear_error();
  if (!b || !counts) return bfail(MSH_E_INVALID_ARG, "null argument");
  B_TRY(cudaMemcpyAsync(counts, b->d_fallback, sizeof(int64_t) * b->ntubes, cudaMemcpyDeviceToHost, b->stream));
  B_TRY(cudaStreamSynchronize(b->stream));
  return MSH_OK;
}

msh_status msh_batch_destroy(msh_batch *b) {
  if (!b) return MSH_OK;
  if (b->stream) cudaStreamSynchronize(b->stream);
  for (auto *g : b->grids)
    if (g) msh_destroy(g);
  cudaFree(b->U);
  cudaFree(b->d_off);
  cudaFree(b->d_len);
  cudaFree(b->d_order);
  cudaFree(b->d_queue);
  cudaFree(b->d_status);
  cudaFree(b->d_tend);
  cudaFree(b->d_t);
  cudaFree(b->d_steps);
  cudaFree(b->d_fallback);
  for (auto x : b->aux)
    if (x) cudaStreamDestroy(x);
  if (b->ev_fork) cudaEventDestroy(b->ev_fork);
  for (auto x : b->ev_join)
    if (x) cudaEventDestroy(x);
  if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
  delete b;
  return MSH_OK;
}

}  // extern "C"
