// Total BA cost without any device allocation.
//
// Some callers cannot allocate device memory at the point where they need a cost:
// code running under a fixed memory pool that is already fully handed out, a host
// callback or a real-time thread that must not enter the CUDA allocator (whose calls
// can synchronise the device and take unbounded time), or a process whose device
// memory is owned by another framework.  gpo_ba_cost_noalloc serves them: the caller
// passes its own device buffers for the problem and for the result, and the
// reduction's scratch (one partial sum per CTA and a completion counter) lives in a
// file-scope static device array of fixed size instead of allocated memory.
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>

#include "fp64.cuh"
#include "gpo.h"

namespace {

constexpr int kThreads = 256;
constexpr int kMaxBlocks = 8192;                                    // partials held
constexpr long long kMaxEdges = (long long)kThreads * kMaxBlocks;   // 2,097,152 edges
constexpr int kMaxDevices = 64;

struct Scratch {
  double part[kMaxBlocks];
  unsigned int ticket;
};

// Shared by every call on a device; it keeps the last call's contents.
static __device__ __align__(256) Scratch g_scratch;

std::mutex g_mu;
Scratch* g_addr[kMaxDevices] = {};   // device address of g_scratch, per device

// Rotation matrix (row-major), translation, f, k1, k2 of a camera.
__device__ void camera_block(const double* c, double* o) {
  // R = I + a [w]x + b [w]x^2 (Rodrigues), a = sin t / t, b = (1 - cos t) / t^2
  const double t2 = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
  double a, b;
  if (t2 < 1e-8) {
    a = 1.0 - t2 / 6.0 + t2 * t2 / 120.0;
    b = 0.5 - t2 / 24.0 + t2 * t2 / 720.0;
  } else {
    const double t = sqrt(t2);
    double s, co;
    sincos(t, &s, &co);
    a = s / t;
    b = (1.0 - co) / t2;
  }
  const double x = c[0], y = c[1], z = c[2];
  o[0] = 1.0 + b * (x * x - t2); o[1] = b * x * y - a * z;      o[2] = b * x * z + a * y;
  o[3] = b * x * y + a * z;      o[4] = 1.0 + b * (y * y - t2); o[5] = b * y * z - a * x;
  o[6] = b * x * z - a * y;      o[7] = b * y * z + a * x;      o[8] = 1.0 + b * (z * z - t2);
  for (int i = 0; i < 6; ++i) o[9 + i] = c[3 + i];
}

// rho of an edge (the caller halves the sum).
__device__ double edge_rho(const double* c, const double* X, double2 z, double delta) {
  double P[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) P[i] = fma(c[3 * i], X[0], fma(c[3 * i + 1], X[1], fma(c[3 * i + 2], X[2], c[9 + i])));
  const double iz = -gpo::rcp_newton(P[2]), p0 = P[0] * iz, p1 = P[1] * iz;
  const double r2 = fma(p0, p0, p1 * p1), fd = c[12] * fma(r2, fma(r2, c[14], c[13]), 1.0);
  const double r0 = fma(fd, p0, -z.x), r1 = fma(fd, p1, -z.y);
  return gpo::huber_value(fma(r0, r0, r1 * r1), delta);
}

// The rotation of an edge's camera costs several times the edge's own FP64 work (a sine, a
// cosine, a square root, three divisions), and observations usually come in runs of one
// camera, so a CTA forms it once per run: a thread whose edge starts a run writes the camera's
// block to shared memory, and the run's edges read it there.  Edges in no order make every
// thread its own run.  FP64-bound: 400 cameras, 1.01 million edges in camera order 248 ->
// 113 us, in point order or none (a camera block per edge) 248 -> 227; RMS error over 16
// scenes 6.3e-16 -> 5.7e-16.
__global__ void __launch_bounds__(kThreads) k_cost_noalloc(const double* cams, const double* pts, const int* ci,
                                                          const int* pi, const double* obs, long long n, double delta,
                                                          double* out, Scratch* scr) {
  constexpr int CW = 15;   // an odd count of 8-byte words: the runs' blocks start in different banks
  __shared__ double red[kThreads];
  __shared__ double cam_s[kThreads * CW];
  __shared__ int warp_runs[kThreads / 32];
  __shared__ bool last;
  const long long e = (long long)blockIdx.x * kThreads + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = e < n ? ci[e] : -1;
  const bool head = e < n && (threadIdx.x == 0 || ci[e - 1] != c);
  double X[3] = {0.0, 0.0, 0.0};
  double2 z = make_double2(0.0, 0.0);
  if (e < n) {
    const double* Xp = pts + 3 * (size_t)pi[e];
    X[0] = Xp[0]; X[1] = Xp[1]; X[2] = Xp[2];
    z = make_double2(obs[2 * e], obs[2 * e + 1]);
  }
  const unsigned heads = __ballot_sync(0xffffffffu, head);
  if (lane == 0) warp_runs[warp] = __popc(heads);
  __syncthreads();
  int before = 0, runs = 0;
  for (int w = 0; w < kThreads / 32; ++w) {
    if (w < warp) before += warp_runs[w];
    runs += warp_runs[w];
  }
  const int run = before + __popc(heads & (0xffffffffu >> (31 - lane))) - 1;   // the edge's run
  // the runs' cameras, dealt to consecutive threads
  int* run_cam = reinterpret_cast<int*>(red);
  if (head) run_cam[run] = c;
  __syncthreads();
  const int mine = (int)threadIdx.x < runs ? run_cam[threadIdx.x] : -1;
  if (mine >= 0) camera_block(cams + 9 * (size_t)mine, cam_s + threadIdx.x * CW);
  __syncthreads();
  double v = 0.0;
  if (e < n) v = edge_rho(cam_s + run * CW, X, z, delta);
  red[threadIdx.x] = v;
  __syncthreads();
  for (int s = kThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    scr->part[blockIdx.x] = 0.5 * red[0];
    __threadfence();
    last = atomicAdd(&scr->ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double acc = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += kThreads) acc += scr->part[b];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = kThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

}  // namespace

extern "C" gpo_status gpo_ba_cost_noalloc(int32_t device, void* cuda_stream, const double* cams,
                                          const double* points, const int32_t* cam_idx, const int32_t* pt_idx,
                                          const double* obs, int64_t n_edges, double huber_delta,
                                          double* cost_out) {
  if (n_edges < 0 || n_edges > kMaxEdges || !cost_out || device < 0 || device >= kMaxDevices)
    return GPO_ERR_ARG;   // n_edges beyond 2,097,152 exceeds the static scratch
  if (n_edges > 0 && (!cams || !points || !cam_idx || !pt_idx || !obs)) return GPO_ERR_ARG;
  int prev = 0;
  if (cudaGetDevice(&prev) != cudaSuccess) return GPO_ERR_CUDA;
  if (cudaSetDevice(device) != cudaSuccess) return GPO_ERR_CUDA;
  gpo_status st = GPO_OK;
  Scratch* scr = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_addr[device]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess) st = GPO_ERR_CUDA;
      else g_addr[device] = static_cast<Scratch*>(p);
    }
    scr = g_addr[device];
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  if (st == GPO_OK) {
    const int blocks = n_edges > 0 ? (int)((n_edges + kThreads - 1) / kThreads) : 1;
    // the completion counter must start at zero; the partials are overwritten
    if (cudaMemsetAsync(&scr->ticket, 0, sizeof(unsigned int), s) != cudaSuccess) st = GPO_ERR_CUDA;
    if (st == GPO_OK) {
      k_cost_noalloc<<<blocks, kThreads, 0, s>>>(cams, points, cam_idx, pt_idx, obs, n_edges, huber_delta, cost_out,
                                                scr);
      if (cudaGetLastError() != cudaSuccess) st = GPO_ERR_CUDA;
    }
  }
  cudaSetDevice(prev);
  return st;
}
