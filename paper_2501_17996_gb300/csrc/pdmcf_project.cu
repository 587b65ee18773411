// pdmcf_project.cu — the capped-simplex projection Pi (Zhang & Boyd, Sec. 2.3) as a
// standalone C ABI operation on device arrays (mcf_project_capped_simplex).
//
// The kernels run the edge phase's projection (warm-started Newton on
// phi(mu) = sum (q - mu)_+ - c with exact active-set finish) on caller-provided columns.
// Per-column FP64 squared distances, where the caller wants them, go to scratch memory and are
// summed in a fixed order, so the reported distance does not depend on the launch grid.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <string>

#include "pdmcf_internal.h"
#include "pdmcf_kernels.h"
#include "pdmcf_sub.cuh"

namespace pdmcf {

// pdmcf_solver.cu
cudaMemPool_t state_pool(int device);
cudaError_t pool_alloc(void** p, size_t bytes, cudaMemPool_t pool, cudaStream_t st);

// Fixed-order sum of x[0..count) into *out by one block of 1024 threads: thread t adds x[t],
// x[t + 1024], ... (coalesced; a segment per thread took 20 us at 30 000 columns), then a tree.
__global__ void __launch_bounds__(1024) fixed_order_sum_kernel(const double* x, long long count,
                                                               double* out) {
  __shared__ double sh[1024];
  double s = 0.0;
#pragma unroll 8
  for (long long b = threadIdx.x; b < count; b += 1024) s += x[b];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int off = 512; off > 0; off >>= 1) {
    if (threadIdx.x < off) sh[threadIdx.x] += sh[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

// m columns given as rows of Qt (edge-major, ld >= n floats per row): Ft row l = (q_l - mu_l)_+,
// mu in/out (warm start in, multipliers out), and, if col_d2 is not NULL, the per-column squared
// distance ||Pi(q_l) - q_l||^2. Entries n..ld-1 of Qt are ignored; those of Ft are written as zero.
struct ProjArgs {
  int n, m, ld;
  const float* Qt;
  const float* cap;
  float* Ft;
  float* mu;
  double* col_d2;
};

// Short columns: L lanes per column, 32 / L columns per warp (project_mu_lanes).
template <int L, int VPT, int BLOCK, int MINB>
__global__ void __launch_bounds__(BLOCK, MINB)
project_lanes_kernel(ProjArgs a) {
  constexpr int VW = 4;
  constexpr int ROWS = BLOCK / L;
  const int hl = threadIdx.x % L;
  const int nchunks = a.ld / VW;
  for (int base = blockIdx.x * ROWS; base < a.m; base += gridDim.x * ROWS) {
    const bool live = base + (int)(threadIdx.x / L) < a.m;
    const int e = live ? base + (int)(threadIdx.x / L) : a.m - 1;
    const float* qr = a.Qt + (size_t)e * a.ld;
    const float mu0 = a.mu[e], c = a.cap[e];
    float q[VPT][VW];
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int ci = v * L + hl;
      ld_stream<float, VW>(qr + min(ci, nchunks - 1) * VW, q[v]);
#pragma unroll
      for (int u = 0; u < VW; ++u)
        if (ci * VW + u >= a.n) q[v][u] = 0.f;         // pads never enter the active set
    }
    const float mu = project_mu_lanes<L, VPT * VW>([&](int i) { return q[i / VW][i % VW]; }, c,
                                                   mu0 > 0.f ? mu0 : 0.f, 0.f);
    float dloc = 0.f;
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int ci = v * L + hl;
      float out[VW];
#pragma unroll
      for (int u = 0; u < VW; ++u) {
        out[u] = q[v][u] > mu ? q[v][u] - mu : 0.f;
        const float d = out[u] - q[v][u];
        dloc = fmaf(d, d, dloc);
      }
      if (live && ci < nchunks) st_stream<float, VW>(a.Ft + (size_t)e * a.ld + ci * VW, out);
    }
    if (a.col_d2) {
      const double d2 = lanes_reduce<L>((double)dloc, [](double x, double y) { return x + y; });
      if (live && hl == 0) a.col_d2[e] = d2;
    }
    if (live && hl == 0) a.mu[e] = mu;
  }
}

// Multiplier from a guess that may be far off: project_mu_n, but where the first Newton step is
// not certified its iteration continues on the first SUB chunks per lane with their share of
// the capacity, and the whole column goes on from the multiplier found there. With columns in no
// particular order that lands near the root, and the passes on the way cost SUB / VPT of a pass;
// any start is valid (one step from the right of the root lands on its left).
template <int GROUP, int VPT, int SUB>
__device__ __forceinline__ float project_mu_far(const float (&q)[VPT][4], float c, float mu0, float share,
                                                GroupScratch<GROUP>& sh, int& phase) {
  float mu = mu0 > 0.f ? mu0 : 0.f, s, amin, imax = 0.f;
  int n;
  auto eval = [&](auto want_imax, auto chunks) {
    constexpr bool IM = decltype(want_imax)::value;
    float ls = 0.f, am = INFINITY, im = -INFINITY;
    int lc = 0;
#pragma unroll
    for (int v = 0; v < decltype(chunks)::value; ++v)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float x = q[v][u];
        if (x > mu) { ls += x; ++lc; am = fminf(am, x); }
        else if constexpr (IM) im = fmaxf(im, x);
      }
    group_stats<GROUP, IM, float>(ls, lc, am, im, sh, phase);
    s = ls; n = lc; amin = am;
    if constexpr (IM) imax = im;
  };
  using with_imax = std::true_type;
  using without_imax = std::false_type;
  using all = std::integral_constant<int, VPT>;
  using some = std::integral_constant<int, SUB>;
  eval(with_imax{}, all{});
  float phi = s - (float)n * mu - c;
  if (phi <= 0.f && (mu == 0.f || phi == 0.f)) return mu;   // at the floor, or at the root
  float left = 0.f;                                         // known not to be right of the root
  if (phi > 0.f) {
    left = (s - c) / (float)n;
    if (!(left > mu)) return mu;
    if (left < amin) return left;                           // no active entry leaves: the root
    mu = left;
#pragma unroll 1
    for (int it = 0; it < 16; ++it) {
      eval(without_imax{}, some{});
      const float next = n > 0 ? (s - c * share) / (float)n : mu;
      if (!(next > mu * 1.002f)) break;
      mu = next;
    }
    eval(with_imax{}, all{});
    phi = s - (float)n * mu - c;
    if (phi == 0.f) return mu;
  }
  if (phi <= 0.f) {                                         // Newton step from the right
    const float next = n > 0 ? (s - c) / (float)n : left;
    if (next <= left) {
      mu = left;
      eval(without_imax{}, all{});
      if (left == 0.f && s - c <= 0.f) return 0.f;
    } else {
      if (n > 0 && next >= imax) return next;               // no inactive entry joins: the root
      mu = next;
      eval(without_imax{}, all{});
    }
  }
#pragma unroll 1
  for (int it = 0; it < 64; ++it) {
    if (n == 0) break;
    const float next = (s - c) / (float)n;
    if (!(next > mu)) break;
    mu = next;
    if (next < amin) break;                                 // no active entry leaves: the root
    eval(without_imax{}, all{});
  }
  return mu;
}

// Longer columns: GROUP threads per column, the next column on its way to L2 meanwhile.
template <int VPT, int GROUP, int BLOCK, int MINB, int SUB>
__global__ void __launch_bounds__(BLOCK, MINB)
project_row_kernel(ProjArgs a) {
  constexpr int VW = 4;
  constexpr int GPB = BLOCK / GROUP;
  __shared__ GroupScratch<GROUP> sh_all[GPB];
  GroupScratch<GROUP>& sh = sh_all[threadIdx.x / GROUP];
  int phase = 0;
  const int lane = threadIdx.x % GROUP;
  const int gid = blockIdx.x * GPB + threadIdx.x / GROUP;
  const int ngroups = gridDim.x * GPB;
  const int nchunks = a.ld / VW;
  for (int e = gid; e < a.m; e += ngroups) {
    const float* qr = a.Qt + (size_t)e * a.ld;
    if (lane == 0 && e + ngroups < a.m)
      prefetch_l2(a.Qt + (size_t)(e + ngroups) * a.ld, (uint32_t)a.ld * 4u);
    const float mu0 = a.mu[e], c = a.cap[e];
    float q[VPT][VW];
#pragma unroll
    for (int v = 0; v < VPT; ++v) {   // unconditional, so that all loads are in flight
      const int ci = v * GROUP + lane;
      ld_stream<float, VW>(qr + min(ci, nchunks - 1) * VW, q[v]);
#pragma unroll
      for (int u = 0; u < VW; ++u)
        if (ci * VW + u >= a.n) q[v][u] = 0.f;         // pads never enter the active set
    }
    float mu;
    if constexpr (SUB > 0) mu = project_mu_far<GROUP, VPT, SUB>(q, c, mu0, (float)(SUB * GROUP) / (float)nchunks, sh, phase);
    else mu = project_mu<GROUP, VPT, VW, float>(q, c, mu0 > 0.f ? mu0 : 0.f, 0.f, sh, phase);
    float dloc = 0.f;
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int ci = v * GROUP + lane;
      if (ci < nchunks) {
        float out[VW];
#pragma unroll
        for (int u = 0; u < VW; ++u) {
          out[u] = q[v][u] > mu ? q[v][u] - mu : 0.f;
          const float d = out[u] - q[v][u];
          dloc = fmaf(d, d, dloc);
        }
        st_stream<float, VW>(a.Ft + (size_t)e * a.ld + ci * VW, out);
      }
    }
    if (a.col_d2) {
      const double d2 = group_sum_double<GROUP>((double)dloc, sh, phase);
      if (lane == 0) a.col_d2[e] = d2;
    }
    if (lane == 0) a.mu[e] = mu;
  }
}

// Variants by column length, for launches with several columns per SM. Measured against one
// group of the solver's shapes per column (GB300, 3e8 entries or 1e6 columns, normal columns, a
// guess far below the multiplier): n = 100 428 -> 225 us, n = 200 612 -> 483, n = 400 708 -> 600,
// n = 1000 673 -> 493, n = 3000 734 -> 571, n = 10 000 1081 -> 565 (4.3 TB/s; the rest is the
// passes' arithmetic). Below `few` columns a group per column from the first (a pass of some 12 us
// with its launch and events): shapes / variant in us, n = 400: 4096 columns 13.8 / 15.1, 8192 18.4 / 18.9,
// 16 384 20.5 / 20.8; n = 1000: 2048 13.8 / 15.0, 4096 17.7 / 18.1; n = 3000: 512 14.0 / 16.0, 1024
// 17.1 / 18.5, 2048 20.5 / 20.8; up to 200 entries both take 11.5 to 14 us below 16 384 columns.
using ProjKernel = void (*)(ProjArgs);
struct ProjVariant {
  ProjKernel fn;
  int chunks, rows, block, few;   // longest column, columns per CTA; `few`: fewer columns keep the shapes
};
static const ProjVariant kProj[] = {
    {project_lanes_kernel<4, 2, 128, 12>, 8, 32, 128, 16384},
    {project_lanes_kernel<4, 4, 128, 12>, 16, 32, 128, 16384},
    {project_lanes_kernel<4, 7, 128, 10>, 28, 32, 128, 16384},
    {project_lanes_kernel<8, 8, 128, 8>, 64, 16, 128, 16384},
    {project_lanes_kernel<8, 13, 128, 6>, 104, 16, 128, 16384},
    {project_row_kernel<4, 32, 256, 6, 1>, 128, 8, 256, 4096},
    {project_row_kernel<8, 32, 256, 4, 1>, 256, 8, 256, 4096},
    {project_row_kernel<16, 32, 128, 4, 0>, 512, 4, 128, 4096},
    {project_row_kernel<24, 32, 128, 3, 0>, 768, 4, 128, 4096},
    {project_row_kernel<8, 128, 128, 7, 1>, 1024, 1, 128, 1024},
    {project_row_kernel<12, 128, 128, 6, 2>, 1536, 1, 128, 1024},
    {project_row_kernel<20, 128, 128, 4, 2>, 2560, 1, 128, 1024},
    {project_row_kernel<16, 256, 256, 2, 2>, 4096, 1, 256, 1024},
    {project_row_kernel<16, 512, 512, 1, 2>, 8192, 1, 512, 512},
};
constexpr int NUM_PROJ = (int)(sizeof(kProj) / sizeof(kProj[0]));

template <int IDX>
static ProjVariant shape_proj() {
  constexpr ShapeDesc d = kShapes[IDX];
  constexpr int MB = min_blocks<float, d.vpt, 4, d.block>();
  return {project_row_kernel<d.vpt, d.group, d.block, MB, 0>, d.group * d.vpt, d.block / d.group, d.block, 0};
}
static const ProjVariant* shape_table() {
  static const ProjVariant t[NUM_SHAPES] = {
      shape_proj<0>(), shape_proj<1>(), shape_proj<2>(), shape_proj<3>(), shape_proj<4>(), shape_proj<5>(),
      shape_proj<6>(), shape_proj<7>(), shape_proj<8>(), shape_proj<9>(), shape_proj<10>(), shape_proj<11>(),
      shape_proj<12>(), shape_proj<13>()};
  return t;
}

// Resident CTAs of a variant on a device (the occupancy query costs as much as a launch, so its
// answer is kept; 0 = not asked yet).
static int resident_ctas(int dev, int slot, const ProjVariant& v, cudaError_t* e) {
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices][NUM_PROJ + NUM_SHAPES];
  const bool keep = dev >= 0 && dev < kDevices;
  if (keep) {
    const int c = known[dev][slot].load(std::memory_order_relaxed);
    if (c > 0) return c;
  }
  int sms = 0, occ = 0;
  *e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (*e == cudaSuccess) *e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void*)v.fn, v.block, 0);
  const int c = (occ > 0 ? occ : 1) * (sms > 0 ? sms : 1);
  if (*e == cudaSuccess && keep) known[dev][slot].store(c, std::memory_order_relaxed);
  return c;
}

// Launches the projection and, if dist2 is not NULL, the fixed-order sum into scratch[m] and its
// copy to *dist2. scratch must then hold m + 1 doubles; arguments already validated.
int project_launch(int32_t n, int32_t m, int32_t ld, const float* Qt, const float* cap,
                   float* Ft, float* mu, double* dist2, cudaStream_t st, double* scratch) {
  const int nchunks = ld / 4;
  int slot = 0;
  while (slot < NUM_PROJ && kProj[slot].chunks < nchunks) ++slot;
  const ProjVariant* v = slot < NUM_PROJ && m >= kProj[slot].few ? &kProj[slot] : nullptr;
  if (!v) {
    const int shape = pick_shape(nchunks);
    slot = NUM_PROJ + shape;
    v = shape_table() + shape;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  const int ctas = e == cudaSuccess ? resident_ctas(dev, slot, *v, &e) : 0;
  if (e != cudaSuccess) {
    set_error(std::string("CUDA error ") + cudaGetErrorString(e));
    return MCF_ERR_CUDA;
  }
  const int need = (m + v->rows - 1) / v->rows;
  const int grid = need < ctas ? need : ctas;
  ProjArgs a{n, m, ld, Qt, cap, Ft, mu, dist2 ? scratch : nullptr};
  void* kargs[] = {&a};
  e = cudaLaunchKernel((const void*)v->fn, dim3(grid > 0 ? grid : 1), dim3(v->block), kargs, 0, st);
  if (e == cudaSuccess && dist2) {
    fixed_order_sum_kernel<<<1, 1024, 0, st>>>(scratch, (long long)m, scratch + m);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(dist2, scratch + m, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e != cudaSuccess) {
    set_error(std::string("CUDA error ") + cudaGetErrorString(e));
    return MCF_ERR_CUDA;
  }
  return MCF_OK;
}

int project_validate(int32_t n, int32_t m, int32_t ld, const float* Qt, const float* cap,
                     const float* Ft, const float* mu) {
  if (n < 1 || m < 0 || ld < n || (ld % 4) != 0) {
    set_error("need n >= 1, m >= 0, ld >= n and ld a multiple of 4");
    return MCF_ERR_INVALID;
  }
  if (m > 0 && (!Qt || !cap || !Ft || !mu)) {
    set_error("Qt, cap, Ft and mu must be device pointers");
    return MCF_ERR_INVALID;
  }
  if (((uintptr_t)Qt | (uintptr_t)Ft) % 16 != 0) {
    set_error("Qt and Ft must be 16-byte aligned");
    return MCF_ERR_INVALID;
  }
  if (pick_shape(ld / 4) < 0) {
    set_error("ld too large (at most 32768 floats per column)");
    return MCF_ERR_INVALID;
  }
  return MCF_OK;
}

}  // namespace pdmcf

using namespace pdmcf;

extern "C" int mcf_project_capped_simplex(int32_t n, int32_t m, int32_t ld, const float* Qt,
                                          const float* cap, float* Ft, float* mu,
                                          double* dist2, void* stream) {
  int rc = project_validate(n, m, ld, Qt, cap, Ft, mu);
  if (rc != MCF_OK) return rc;
  if (m == 0) {
    if (dist2) *dist2 = 0.0;
    return MCF_OK;
  }
  cudaStream_t st = (cudaStream_t)stream;
  // the scratch comes from the device's pool of freed memory in the order of the caller's
  // stream: cudaMalloc and cudaFree took as long as the kernel at 30 000 columns of 10 000
  double* scratch = nullptr;
  cudaMemPool_t pool = nullptr;
  if (dist2) {
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) pool = state_pool(dev);
    const size_t bytes = ((size_t)m + 1) * sizeof(double);
    const cudaError_t ea = pool ? pool_alloc((void**)&scratch, bytes, pool, st) : cudaMalloc((void**)&scratch, bytes);
    if (ea != cudaSuccess) {
      cudaGetLastError();
      set_error("device allocation of the projection scratch failed");
      return MCF_ERR_OOM;
    }
  }
  rc = project_launch(n, m, ld, Qt, cap, Ft, mu, dist2, st, scratch);
  if (scratch && pool) cudaFreeAsync(scratch, st);
  cudaError_t e = cudaStreamSynchronize(st);
  if (scratch && !pool) cudaFree(scratch);
  if (rc == MCF_OK && e != cudaSuccess) {
    set_error(std::string("CUDA error ") + cudaGetErrorString(e));
    rc = MCF_ERR_CUDA;
  }
  return rc;
}
