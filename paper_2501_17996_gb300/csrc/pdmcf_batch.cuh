// pdmcf_batch.cuh — batched PDMCF iteration: many independent instances of different sizes
// advanced together (Algorithm 2.1, step 2, for every resident instance).
//
// A launch walks a global work list (edges, or pieces of the nodes' columns) in short runs dealt
// out to the warps in turn (batch_walk). What bounds it is latency: an item is a chain of loads
// (edge, rows) and warp reductions or root searches, and its length differs several times over
// between instances. 64 networks of 50 to 400 nodes (edge phase 97 k rows of 50 to 400 entries,
// 89 us; node phase 10 k columns, 98 us): 231 us per iteration with a launch per shape and phase,
// one item at a time per group, and sums in every iteration; 201 with a contiguous range of the
// list per warp, which gave the longest rows to neighbouring warps of one SM; 184 dealt out.
// Twelve networks of 100 to 1000 nodes: 198, 112 and 117 us.
// Each instance keeps its scalars (k, parity, alpha, beta, omega, stop state) on the device,
// so kernels decide on their own whether an iteration is a check iteration and whether the
// instance is still active; a captured iteration therefore replays for any mix.
// Reductions are per work item (one FP64 value per edge and per piece, summed in a fixed
// order by the instance's own scalar block, in iterations whose scalar tail uses them), so an
// instance's iterates are bit-identical whether it runs alone or with others.
#pragma once

#include "pdmcf_device.cuh"
#include "pdmcf_resident.cuh"

namespace pdmcf {

struct BatchScalars {
  DevScalars s;            // shared fields (step sizes, k, check results, ...)
  int parity;              // F[parity], Y[parity] hold F^{k-1/2}, Y^k
  int active;              // 1 while the instance iterates
  int done;                // set by the scalar kernel when the stop rule holds
  int stop_mode;           // MCF_STOP_*
  long long max_iters;
  long long k_check;
  double eps;
  int stall_checks;        // stall rule (see mcf_options.stall_checks)
  int stall_count;
  int stalled;
  double stall_best;
  int stall_frozen;        // omega had stopped adapting when the count last restarted
};

struct BatchInst {
  int n, m, ld, kind;
  float gamma, rho;
  const int32_t* e_tail;
  const int32_t* e_head;
  const int32_t* in_ptr;
  const int32_t* out_ptr;
  const int32_t* out_idx;
  const float* cap;
  const float* W;
  const float* Gm;
  float* F[2];
  float* Y[2];
  __nv_bfloat16* Ylo[2];   // compensated-dual tails (nullptr: plain Y)
  float* Pm;
  float* mu;               // projection multipliers, hi/lo pair
  float* mu_lo;
  float* That;
  float* Uprime;
  float* Yhat;
  double* pe;              // [m] per-edge ||dF||^2 parts
  int per;                 // pieces per node (batch_pieces_per)
  double* pn;              // [n * per * NODE_PARTS] parts per piece
  double* pc;              // [m * CHECK_PARTS] per-edge check parts
  BatchScalars* sc;
};

// Entries per lane of the node phase's pieces. Two per lane: 174 instead of 184 us per iteration
// for the 64 networks above (their columns leave lanes idle at four), 128 instead of 117 us for
// the twelve. Both, by column length, in one kernel: 200 and 124 us (it no longer fits the
// instruction cache).
constexpr int BATCH_N = 4;
inline int batch_pieces_per(int ld) { return (ld + 32 * BATCH_N - 1) / (32 * BATCH_N); }

struct BatchClassDev {
  const int* count;        // number of instances in the class (device, so graphs replay)
  const int* inst;         // [count] indices into the instance table
  const long long* eoff;   // [count + 1] edge prefix sums
  const long long* noff;   // [count + 1] prefix sums of the node phase's pieces
};

__device__ __forceinline__ int batch_find(const long long* off, int count, long long g) {
  int lo = 0, hi = count - 1;            // largest b with off[b] <= g
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= g) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Calls fn(instance, first, last + 1) for the warp's runs of RUN consecutive items: run r of the
// list goes to warp r mod (number of warps), numbered across the CTAs first, so that every SM gets
// its share of each instance. RUN 4 for edges (a run shares its instance's fields; 8: 119 to 127 us
// for the twelve networks above, 2: 203 us for the 64) and 1 for pieces (2: 194, 4: 202 us).
template <int RUN, typename Fn>
__device__ __forceinline__ void batch_walk(const BatchInst* __restrict__ insts, const BatchClassDev& cls,
                                           const long long* __restrict__ off, Fn fn) {
  const int count = *cls.count;
  if (count == 0) return;
  const long long total = off[count];
  const int per_cta = blockDim.x >> 5;
  const long long w = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x, nw = (long long)gridDim.x * per_cta;
  if (w * RUN >= total) return;
  int b = batch_find(off, count, w * RUN);
#pragma unroll 1
  for (long long r = w * RUN; r < total; r += nw * RUN) {
    long long g = r;
    const long long g1 = min(total, r + RUN);
#pragma unroll 1
    while (g < g1) {
      while (off[b + 1] <= g) ++b;
      const long long base = off[b], end = min(g1, off[b + 1]);
      const BatchInst& I = insts[cls.inst[b]];
      if (I.sc->active) fn(I, (int)(g - base), (int)(end - base));
      g = end;
    }
  }
}

__device__ __forceinline__ bool batch_is_check(const BatchScalars* sc) {
  const long long k1 = sc->s.k + 1;
  return (k1 % sc->k_check) == 0 || k1 >= sc->max_iters;
}

// Warp sums of K values a lane (K a power of two, at most 32): lane l gets the sum of value
// l / (32 / K). Halving the values with the lanes takes K - 1 + log2(32 / K) additions a lane
// instead of 5 K, on an FP64 unit that runs at 1/64 of FP32.
template <int K>
__device__ __forceinline__ double warp_sums(double (&v)[K]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16, k = K; o > 0; o >>= 1) {
    if (k > 1) {
      k >>= 1;
#pragma unroll
      for (int i = 0; i < k; ++i) {
        const double send = lane & o ? v[i] : v[i + k], keep = lane & o ? v[i + k] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  return v[0];
}

// Iterations whose scalar tail uses the reductions: a multiple of k_adapt, or a stop test.
__device__ __forceinline__ bool batch_reduces(const BatchScalars* sc) {
  return batch_is_check(sc) || sc->s.k % sc->s.k_adapt == 0;
}

// ------------------------------------------------------------------ edge phase, short rows
// A warp per edge, V chunks of 4 entries per lane. The instance's fields are read once per run. (The
// next edge's rows loaded ahead cost registers and spills: 316 instead of 231 us per iteration.)
template <int V>
__device__ __forceinline__ void batch_edges(const BatchInst& I, int e, int e1) {
  constexpr int VW = 4;
  const BatchScalars* sc = I.sc;
  const int lane = threadIdx.x & 31;
  const int ld = I.ld, nchunks = ld / VW;
  const int par = sc->parity;
  const bool reduce = batch_reduces(sc);
  const float alpha = (float)sc->s.alpha, rho = I.rho;
  const float* F0 = I.F[par];
  float* F1 = I.F[par ^ 1];
  const float* Y = I.Y[par];
  const __nv_bfloat16* ylo = I.Ylo[par];
  const int32_t *e_head = I.e_head, *e_tail = I.e_tail;
  const float* cap = I.cap;
  float *mu_hi = I.mu, *mu_lo = I.mu_lo;
  bool finite = true;
  auto tails = [](unsigned w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); };
#pragma unroll 1
  for (; e < e1; ++e) {
    const size_t fo = (size_t)e * ld, ho = (size_t)e_head[e] * ld, to = (size_t)e_tail[e] * ld;
    const float mc = cap[e], m0 = mu_hi[e], m0l = mu_lo[e];
    const float floor = shifted_floor<float>(m0, m0l);
    float q[V][VW], f[V][VW];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int ci = v * 32 + lane, co = min(ci, nchunks - 1) * VW;   // loads past the row repeat its end
      float yh[VW], yt[VW];
      uint2 lh = make_uint2(0u, 0u), lt = lh;
      ld_plain<float, VW>(F0 + fo + co, f[v]);
      ld_plain<float, VW>(Y + ho + co, yh);
      ld_plain<float, VW>(Y + to + co, yt);
      if (ylo) {
        lh = *reinterpret_cast<const uint2*>(ylo + ho + co);
        lt = *reinterpret_cast<const uint2*>(ylo + to + co);
      }
#pragma unroll
      for (int u = 0; u < VW; u += 2) {
        const float2 qq = shifted_q2(make_float2(f[v][u], f[v][u + 1]), make_float2(yh[u], yh[u + 1]),
                                     make_float2(yt[u], yt[u + 1]),
                                     p2_sub(tails(u ? lh.y : lh.x), tails(u ? lt.y : lt.x)),
                                     p2(alpha), p2(-m0), p2(-m0l));
        q[v][u] = ci < nchunks ? qq.x : floor;
        q[v][u + 1] = ci < nchunks ? qq.y : floor;
      }
    }
    GroupScratch<32> none;   // warp groups reduce without scratch memory
    int phase = 0;
    const float mu = project_mu<32, V, VW, float>(q, mc, 0.f, floor, none, phase);
    float dloc = 0.f;
    float* fn = F1 + (size_t)e * ld;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int ci = v * 32 + lane;
      if (ci < nchunks) {
        float out[VW];
        float2 sq = p2(0.f);   // (f^ - f)^2, the step itself (not the rounded difference)
#pragma unroll
        for (int u = 0; u < VW; u += 2) {
          const float2 ff = make_float2(f[v][u], f[v][u + 1]);
          const float2 t2 = p2_add(make_float2(q[v][u], q[v][u + 1]), p2(-mu));
          const float2 st = p2_sub(make_float2(fmaxf(t2.x, 0.f), fmaxf(t2.y, 0.f)), ff);
          const float2 fnew = p2_fma(p2(rho), st, ff);   // rho f^ + (1 - rho) f
          sq = p2_fma(st, st, sq);
          out[u] = fnew.x;
          out[u + 1] = fnew.y;
        }
        dloc += rho * rho * (sq.x + sq.y);
        st_plain<float, VW>(fn + ci * VW, out);
      }
    }
    if (reduce) {
      double d2 = (double)dloc;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) d2 += __shfl_xor_sync(0xffffffffu, d2, o);
      if (lane == 0) I.pe[e] = d2;
    } else {
      finite = finite && isfinite(dloc);
    }
    if (lane == 0) {
      float hi, lo;
      shifted_mu<float>(m0, m0l, mu, hi, lo);
      mu_hi[e] = hi;
      mu_lo[e] = lo;
    }
  }
  if (!finite) I.sc->s.numeric_error = 1;   // as the scalar tail would report
}

// LONG: rows of up to 1024 entries, else up to 512 (one launch serves every row length of its
// range: instances of all sizes fill the GPU together).
template <bool LONG, int BLOCK, int MINB>
__global__ void __launch_bounds__(BLOCK, MINB)
batch_edge_warp_kernel(const BatchInst* __restrict__ insts, BatchClassDev cls) {
  batch_walk<4>(insts, cls, cls.eoff, [](const BatchInst& I, int e, int e1) {
    if constexpr (LONG) {
      batch_edges<8>(I, e, e1);
    } else {
      const int nchunks = I.ld / 4;
      if (nchunks <= 32) batch_edges<1>(I, e, e1);
      else if (nchunks <= 64) batch_edges<2>(I, e, e1);
      else batch_edges<4>(I, e, e1);
    }
  });
}

// ------------------------------------------------------------------ edge phase, longer rows

template <int VPT, int GROUP, int BLOCK, int MINB>
__global__ void __launch_bounds__(BLOCK, MINB)
batch_edge_kernel(const BatchInst* __restrict__ insts, BatchClassDev cls) {
  using P = float;
  constexpr int VW = 4;
  constexpr int GPB = BLOCK / GROUP;
  __shared__ GroupScratch<GROUP> sh_all[GPB];
  GroupScratch<GROUP>& sh = sh_all[threadIdx.x / GROUP];
  int phase = 0;
  const int lane = threadIdx.x % GROUP;
  const int gid = blockIdx.x * GPB + threadIdx.x / GROUP;
  const int ngroups = gridDim.x * GPB;
  const int count = *cls.count;
  if (count == 0) return;
  const long long total = cls.eoff[count];
  for (long long g = gid; g < total; g += ngroups) {
    const int b = batch_find(cls.eoff, count, g);
    const BatchInst& I = insts[cls.inst[b]];
    const BatchScalars* sc = I.sc;
    if (!sc->active) continue;
    const int e = (int)(g - cls.eoff[b]);
    const int par = sc->parity;
    const P alpha = (P)sc->s.alpha;
    const P rho = I.rho;
    const int nchunks = I.ld / VW;
    const int h = I.e_head[e], t = I.e_tail[e];
    const P mu0 = I.mu[e], mu0l = I.mu_lo[e];
    const float* fo = I.F[par] + (size_t)e * I.ld;
    const float* yh = I.Y[par] + (size_t)h * I.ld;
    const float* yt = I.Y[par] + (size_t)t * I.ld;
    P q[VPT][VW], f[VPT][VW];
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int ci = v * GROUP + lane;
      if (ci < nchunks) {
        P a1[VW], a2[VW], dl[VW];
        ld_plain<P, VW>(fo + ci * VW, f[v]);
        ld_plain<P, VW>(yh + ci * VW, a1);
        ld_plain<P, VW>(yt + ci * VW, a2);
#pragma unroll
        for (int u = 0; u < VW; ++u) dl[u] = P(0);
        if (I.Ylo[par]) {
          float l1[VW], l2[VW];
          ld_lo<VW>(I.Ylo[par] + (size_t)h * I.ld + ci * VW, l1);
          ld_lo<VW>(I.Ylo[par] + (size_t)t * I.ld + ci * VW, l2);
#pragma unroll
          for (int u = 0; u < VW; ++u) dl[u] = l1[u] - l2[u];
        }
#pragma unroll
        for (int u = 0; u < VW; u += 2) {   // packed pairs, the same rounding as shifted_q
          const float2 qq = shifted_q2(make_float2(f[v][u], f[v][u + 1]),
                                       make_float2(a1[u], a1[u + 1]), make_float2(a2[u], a2[u + 1]),
                                       make_float2(dl[u], dl[u + 1]), p2(alpha), p2(-mu0), p2(-mu0l));
          q[v][u] = qq.x;
          q[v][u + 1] = qq.y;
        }
      } else {
#pragma unroll
        for (int u = 0; u < VW; ++u) { f[v][u] = P(0); q[v][u] = shifted_floor<P>(mu0, mu0l); }
      }
    }
    const P mu = project_mu<GROUP, VPT, VW, P>(q, I.cap[e], P(0), shifted_floor<P>(mu0, mu0l), sh, phase);
    P dloc = P(0);
    float* fn = I.F[par ^ 1] + (size_t)e * I.ld;
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int ci = v * GROUP + lane;
      if (ci < nchunks) {
        P out[VW];
        float2 sq = p2(0.f);   // (f^ - f)^2, the step itself (not the rounded difference)
#pragma unroll
        for (int u = 0; u < VW; u += 2) {
          const float2 ff = make_float2(f[v][u], f[v][u + 1]);
          const float2 t2 = p2_add(make_float2(q[v][u], q[v][u + 1]), p2(-mu));
          const float2 st = p2_sub(make_float2(fmaxf(t2.x, 0.f), fmaxf(t2.y, 0.f)), ff);
          const float2 fnew = p2_fma(p2(rho), st, ff);   // rho f^ + (1 - rho) f
          sq = p2_fma(st, st, sq);
          out[u] = fnew.x;
          out[u + 1] = fnew.y;
        }
        dloc += rho * rho * (sq.x + sq.y);
        st_plain<P, VW>(fn + ci * VW, out);
      }
    }
    if (batch_reduces(sc)) {
      const double d2 = group_sum_double<GROUP>((double)dloc, sh, phase);
      if (lane == 0) I.pe[e] = d2;
    } else if (!isfinite(dloc)) {
      I.sc->s.numeric_error = 1;   // as the scalar tail would report
    }
    if (lane == 0) {
      P hi, lo;
      shifted_mu<P>(mu0, mu0l, mu, hi, lo);
      I.mu[e] = hi;
      I.mu_lo[e] = lo;
    }
  }
}

// ------------------------------------------------------------------ node phase
// A warp per piece of a node's column (node_gather and node_update
// of the resident iteration); the sums per piece are written where the scalar tail uses them.
template <bool CHECK>
__device__ __forceinline__ void batch_piece(const BatchInst& I, int p) {
  using P = float;
  constexpr int N = BATCH_N;
  const BatchScalars* sc = I.sc;
  const int par = sc->parity;
  const int lane = threadIdx.x & 31, per = I.per;
  IterArgs<float, float> a;   // the fields that the node phase uses; old state in slot 0, new in 1
  a.n = I.n;
  a.ld = I.ld;
  a.in_ptr = I.in_ptr;
  a.out_ptr = I.out_ptr;
  a.out_idx = I.out_idx;
  a.F[0] = nullptr;
  a.F[1] = I.F[par ^ 1];
  a.Y[0] = I.Y[par];
  a.Y[1] = I.Y[par ^ 1];
  a.Ylo[0] = I.Ylo[par];
  a.Ylo[1] = I.Ylo[par ^ 1];
  a.Pm = I.Pm;
  a.W = I.W;
  a.Gm = I.Gm;
  a.gamma = I.gamma;
  a.kind = I.kind;
  a.rho = I.rho;
  if constexpr (CHECK) {
    a.That = I.That;
    a.Uprime = I.Uprime;
    a.Yhat = I.Yhat;
  }
  NodePiece q;
  NodeItem<P, N> x;
  P s[N], loc[NODE_PARTS];
#pragma unroll
  for (int k = 0; k < NODE_PARTS; ++k) loc[k] = P(0);
  q.j = p / per;
  q.c = (p - q.j * per) * 32 + lane;
  q.ib = a.in_ptr[q.j];
  q.nin = a.in_ptr[q.j + 1] - q.ib;
  q.ob = a.out_ptr[q.j];
  q.deg = q.nin + a.out_ptr[q.j + 1] - q.ob;
  q.edge = node_edge(a, q, lane);
  node_state<P, float, N>(a, 0, q, x);
  node_data<P, float, N>(a, q, x);
  node_gather<P, float, N, false>(a, a.F[1], q, s);
  node_update<P, float, N, CHECK>(a, 0, q, s, x, (float)sc->s.beta, loc);
  if constexpr (CHECK) {
    double d[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) d[k] = k < NODE_PARTS ? (double)loc[k] : 0.0;
    const double sum = warp_sums<8>(d);
    if ((lane & 3) == 0 && lane / 4 < NODE_PARTS) I.pn[(size_t)p * NODE_PARTS + lane / 4] = sum;
  } else if (batch_reduces(sc)) {
    double d[1] = {(double)loc[0]};
    const double sum = warp_sums<1>(d);
    if (lane == 0) I.pn[(size_t)p * NODE_PARTS] = sum;
  } else if (!isfinite(loc[0])) {
    I.sc->s.numeric_error = 1;   // as the scalar tail would report
  }
}

// One launch for the instances of all classes. CHECK: the kernel of iterations in which some
// instance takes a stop test (each instance still decides for itself).
// That kernel's sums and logarithms leave it bound by latency: three blocks per SM, although registers
// spill, take 251 us against 267 with two (n = 3000; n = 10^4, m = 40 000: 2.18 against 2.45 ms).
template <bool CHECK>
__global__ void __launch_bounds__(256, CHECK ? 3 : 2)
batch_node_kernel(const BatchInst* __restrict__ insts, BatchClassDev all) {
  batch_walk<1>(insts, all, all.noff, [](const BatchInst& I, int p, int) {
    if (CHECK && batch_is_check(I.sc)) batch_piece<true>(I, p);
    else batch_piece<false>(I, p);
  });
}

// ------------------------------------------------------------------ check phase
// A warp per edge of the instances that take a stop test (see check_kernel). Bound by the latency of
// the gathered rows, so four blocks per SM: n = 3000, m = 24 000, 219 us (292 with three).
static __global__ void __launch_bounds__(256, 4)
batch_check_kernel(const BatchInst* __restrict__ insts, BatchClassDev all) {
  using P = float;
  constexpr int VW = 4;
  const int lane = threadIdx.x & 31;
  batch_walk<4>(insts, all, all.eoff, [lane](const BatchInst& I, int e, int e1) {
    const BatchScalars* sc = I.sc;
    if (batch_is_check(sc)) {
      const int par = sc->parity, n = I.n, nchunks = I.ld / VW;
      const size_t ld = (size_t)I.ld;
      const P alpha = (P)sc->s.alpha;
      const float *F = I.F[par], *Y = I.Y[par];
      const __nv_bfloat16* ylo = I.Ylo[par];
      for (; e < e1; ++e) {
        const P mu = I.mu[e];
        const size_t fo = (size_t)e * ld, ho = (size_t)I.e_head[e] * ld, to = (size_t)I.e_tail[e] * ld;
        P ymax = -INFINITY, lg2 = P(0), lgd = P(0), ld2 = P(0);
#pragma unroll 1
        for (int ci = lane; ci < nchunks; ci += 32) {
          P fs[VW], y1[VW], y2[VW], g1v[VW], g2v[VW], z1[VW], z2[VW], dl[VW];
          ld_plain<P, VW>(F + fo + ci * VW, fs);
          ld_plain<P, VW>(Y + ho + ci * VW, y1);
          ld_plain<P, VW>(Y + to + ci * VW, y2);
          ld_plain<P, VW>(I.Uprime + ho + ci * VW, g1v);
          ld_plain<P, VW>(I.Uprime + to + ci * VW, g2v);
          ld_plain<P, VW>(I.Yhat + ho + ci * VW, z1);
          ld_plain<P, VW>(I.Yhat + to + ci * VW, z2);
#pragma unroll
          for (int u = 0; u < VW; ++u) dl[u] = P(0);
          if (ylo) {
            float l1[VW], l2[VW];
            ld_lo<VW>(ylo + ho + ci * VW, l1);
            ld_lo<VW>(ylo + to + ci * VW, l2);
#pragma unroll
            for (int u = 0; u < VW; ++u) dl[u] = l1[u] - l2[u];
          }
#pragma unroll
          for (int u = 0; u < VW; ++u) {
            if (ci * VW + u >= n) continue;
            const P q = fs[u] + alpha * ((y1[u] - y2[u]) + dl[u]);
            const P fh = q > mu ? q - mu : P(0);
            const P d = fh - q, gg = g1v[u] - g2v[u];
            lg2 = fma(gg, gg, lg2);
            lgd = fma(gg, d, lgd);
            ld2 = fma(d, d, ld2);
            ymax = fmax(ymax, z1[u] - z2[u]);
          }
        }
        double v[4] = {(double)lg2, (double)lgd, (double)ld2, 0.0};
        const double sum = warp_sums<4>(v);
        ymax = warp_max(ymax);
        double* pc = I.pc + (size_t)e * CHECK_PARTS;
        if ((lane & 7) == 0 && lane < 24) pc[lane / 8] = sum;
        if (lane == 24) pc[3] = ymax > P(0) ? (double)I.cap[e] * (double)ymax : 0.0;
      }
    }
  });
  // A node's pieces summed into its first one, so that the instance's scalar block has n sets to add
  // instead of n * per (24 n at n = 3000).
  batch_walk<1>(insts, all, all.noff, [lane](const BatchInst& I, int p, int) {
    const int per = I.per, j = p / per;
    if (per == 1 || j * per != p || !batch_is_check(I.sc)) return;
    double* first = I.pn + (size_t)p * NODE_PARTS;
    double d[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) d[k] = 0.0;
    for (int q = lane; q < per; q += 32)
#pragma unroll
      for (int k = 0; k < NODE_PARTS; ++k) d[k] += first[(size_t)q * NODE_PARTS + k];
    const double sum = warp_sums<8>(d);
    if ((lane & 3) == 0 && lane / 4 < NODE_PARTS) first[lane / 4] = sum;
  });
}

}  // namespace pdmcf
