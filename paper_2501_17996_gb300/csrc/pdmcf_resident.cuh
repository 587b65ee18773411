// pdmcf_resident.cuh — resident iteration (Zhang & Boyd, Algorithm 2.1): one cooperative
// launch runs many iterations of a network whose rows fit a warp's registers.
//
// On short rows an iteration is a few microseconds of dependent loads, so the launches of the
// three kernels of pdmcf_device.cuh and the one-block scalar kernel between them were most of
// its time. Here all CTAs stay resident and meet at a grid barrier after the edge phase and
// after the node phase; the scalar tail runs only in iterations whose result depends on it (a
// multiple of k_adapt, or a stop test). What does not depend on the other phase (a row of F,
// the incidence, P, Y and w) is loaded before the barrier is waited for.
//
// Data that another SM wrote in this launch is read after the barrier's acquire, which drops
// the SM's L1 lines, with plain loads: warps of one CTA that read the same dual row share it
// in L1 until the next barrier.
//
// What bounds it (n = 100, m = 1000, 10 400 cycles per iteration at 2.06 GHz, stamps of one CTA):
// the two barriers 4400 (each a store flush, an atomic and a poll through L2, and the skew
// between CTAs), the edge phase's chain of one L2 read and the projection's warp reductions
// 1700, the node phase's row reads and root search 3300. At n = 1000 it is issue and latency at
// four warps per scheduler (a row of q fills 128 registers).
#pragma once

#include "pdmcf_resident.h"

namespace pdmcf {

// ------------------------------------------------------------------ loads and stores of N entries

template <typename T, int N>
__device__ __forceinline__ void ld_words(const T* p, T (&v)[N]) {
  constexpr int BYTES = N * (int)sizeof(T);
  if constexpr (BYTES == 2) {
    unsigned short u = *reinterpret_cast<const unsigned short*>(p);
    memcpy(&v[0], &u, 2);
  } else if constexpr (BYTES == 4) {
    unsigned u = *reinterpret_cast<const unsigned*>(p);
    memcpy(&v[0], &u, 4);
  } else {
    ld_plain<T, N>(p, v);
  }
}
template <int N>
__device__ __forceinline__ void ld_tail(const __nv_bfloat16* p, float (&v)[N]) {
  __nv_bfloat16 b[N];
  ld_words<__nv_bfloat16, N>(p, b);
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = __bfloat162float(b[k]);
}
template <typename T, int N>
__device__ __forceinline__ void ld_const(const T* p, T (&v)[N]) {
  if constexpr (N * sizeof(T) < 8) {
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = __ldg(p + k);
  } else {
    ld_keep<T, N>(p, v);
  }
}
template <typename T, int N>
__device__ __forceinline__ void st_words(T* p, const T (&v)[N]) {
  if constexpr (N * sizeof(T) < 8) {
#pragma unroll
    for (int k = 0; k < N; ++k) p[k] = v[k];
  } else {
    st_plain<T, N>(p, v);
  }
}
template <int N>
__device__ __forceinline__ void st_tail(__nv_bfloat16* p, const float (&v)[N]) {
  if constexpr (N == 1) p[0] = __float2bfloat16_rn(v[0]);
  else st_lo<N>(p, v);
}

// ------------------------------------------------------------------ grid barrier
// Counter barrier over the CTAs of a cooperative launch, split in arrive and wait. The waits
// are bounded (2^22 polls, 0.9 s; an iteration of the largest network that comes here, 1024 nodes
// with every edge, takes 5 ms in FP32 and 65 ms in FP64): a CTA that gives up records
// wait_timeout and leaves, the others run out of polls the same way, the launches queued behind
// this one return at once (resident_start), and the solve reports MCF_ERR_CUDA.
struct GridBarrier {
  unsigned* arrived;
  DevScalars* sc;
  int* failed;        // shared memory, 0 at the start
  unsigned target;
  __device__ __forceinline__ void arrive() {
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0)
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrived) : "memory");
  }
  __device__ __forceinline__ bool wait() {
    if (threadIdx.x == 0) {
      unsigned v = 0;
      bool ok = false;
      for (int it = 0; it < (1 << 22) && !ok; ++it) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arrived) : "memory");
        ok = (int)(v - target) >= 0;
      }
      if (!ok) {
        sc->wait_timeout = 1;
        *failed = 1;
      }
    }
    __syncthreads();
    return *failed == 0;
  }
};

// ------------------------------------------------------------------ utility prox

// Approximate root of t^(c1+1) (t + y) = k (prox_pow) in FP32 with the special-function power:
// the same bounds and monotone Newton search, to about 1e-5.
__device__ __forceinline__ float prox_pow_start(float y, float k, float c1) {
  const float tlo = fmaxf(-y, 0.f);
  const float b1 = __powf(k, __fdividef(1.f, c1 + 2.f));
  float t;
  if (y >= 0.f) t = fminf(b1, __powf(__fdividef(k, y), __fdividef(1.f, c1 + 1.f)));
  else t = tlo + fminf(b1, __fdividef(k, __powf(tlo, c1 + 1.f)));
#pragma unroll 1
  for (int it = 0; it < 20; ++it) {
    const float p = __powf(t, c1);
    const float h = p * t * (t + y) - k;
    const float dh = p * ((c1 + 2.f) * t + (c1 + 1.f) * y);
    const float tn = fmaxf(t - __fdividef(h, dh), tlo);
    if (!(tn < t * (1.f - 1e-5f))) break;
    t = tn;
  }
  return t;
}

// How far off the start of prox_pow_traffic may be, times c1 + 1. What the correction leaves grows as
// ((c1 + 1) d)^4 for two steps (FP64: at most 8.6e-17 of the root and 1.0e-16 of the traffic at the
// limit, exponents 0.05 to 0.95) and as ((c1 + 1) d)^2 for one (FP32: 4e-8): below half a last place.
template <typename P> __device__ constexpr P prox_reach() { return sizeof(P) == 8 ? P(1e-4) : P(2e-4); }

// prox of the power utility and the traffic t = T(Y^) = (w gamma / -Y^)^(1/(1-gamma)) of its
// result, given wg = (w gamma)^(1/(1-gamma)). With c1 + 1 = 1/(1-gamma) the root equation of
// prox_pow is t^(c1+1) (t + y) = beta wg (its constant c1 (1/gamma - 1) is 1), and the traffic
// is wg / t^(c1+1). One full-precision power serves the whole search: the FP32 start is good to
// about 1e-5, one Newton step leaves the square of that, and for the second the power at the
// moved point follows from the binomial series (1 + d)^c1 up to its third order. (The search of
// prox_pow takes about eight powers, each some hundred FP64 instructions on a unit that runs at
// 1/64 of FP32.) A start that turns out farther off than prox_reach, or out of FP32's range, takes
// the full search.
template <typename P>
__device__ __forceinline__ P prox_pow_traffic(P y, P beta, P w, P wg, P gamma, P& traffic) {
  if (gamma == P(0.5)) {
    const P z = prox_pow<P>(y, beta, w, gamma);
    traffic = util_traffic<P>(1, z, w, gamma);
    return z;
  }
  const P tlo = y < P(0) ? -y : P(0);
  const P c1 = gamma / (P(1) - gamma);
  const P k = beta * wg;
  const float kf = (float)k, yf = (float)y;
  if (kf > 1e-25f && kf < 1e25f && fabsf(yf) < 1e8f && fabsf(yf) > 1e-8f && c1 < P(20)) {
    const P t0 = fmax((P)prox_pow_start(yf, kf, (float)c1), tlo);
    const P p0 = pow(t0, c1);
    const P a = c1 + P(2), b = (c1 + P(1)) * y;
    const P t1 = fmax(t0 - (p0 * t0 * (t0 + y) - k) / (p0 * (a * t0 + b)), tlo);
    const P d = (t1 - t0) / t0;
    if (fabs(d) * (c1 + P(1)) < prox_reach<P>()) {
      const P p1 = p0 * (P(1) + c1 * d * (P(1) + (c1 - P(1)) * P(0.5) * d *
                                                   (P(1) + (c1 - P(2)) * P(1.0 / 3.0) * d)));
      P t = t1, p = p1;
      if constexpr (std::is_same<P, double>::value) {
        t = fmax(t1 - (p1 * t1 * (t1 + y) - k) / (p1 * (a * t1 + b)), tlo);
        p = p1 * (P(1) + c1 * ((t - t1) / t1));
      }
      traffic = wg / (p * t);
      return -t;
    }
  }
  const P z = prox_pow<P>(y, beta, w, gamma);
  traffic = util_traffic<P>(1, z, w, gamma);
  return z;
}

// ------------------------------------------------------------------ node phase on N entries

// A warp's piece of a node's column: 32 x N consecutive entries. `edge` holds the incident
// edges, lane l the l-th (in-edges first): the rows' addresses come from a shuffle instead of
// a chain of index loads.
struct NodePiece {
  int j = -1, c = 0;           // node; this lane's group of N entries
  int nin = 0, deg = 0, ib = 0, ob = 0;
  int edge = 0;
};

template <typename P, typename S>
__device__ __forceinline__ int node_edge(const IterArgs<P, S>& a, const NodePiece& q, int l) {
  if (l >= q.deg) l = q.deg - 1;   // a row that is read anyway
  return l < q.nin ? q.ib + l : __ldg(a.out_idx + q.ob + l - q.nin);
}

// Piece `p` of the n x per pieces, node index fastest; the edges are loaded by node_edge.
template <typename P, typename S, int N>
__device__ __forceinline__ void node_place(const IterArgs<P, S>& a, unsigned p, NodePiece& q) {
  const unsigned c = p / (unsigned)a.n;
  q.j = (int)(p - c * (unsigned)a.n);
  q.c = (int)c * 32 + (int)(threadIdx.x & 31);
  q.ib = __ldg(a.in_ptr + q.j);
  q.nin = __ldg(a.in_ptr + q.j + 1) - q.ib;
  q.ob = __ldg(a.out_ptr + q.j);
  q.deg = q.nin + __ldg(a.out_ptr + q.j + 1) - q.ob;
}

// What does not depend on the edge phase: data (constant) and state of a piece.
template <typename P, int N>
struct NodeItem {
  P wv[N], gv[N], wg[N];
  P po[N], yo[N], yl[N];
};

// The utility; BF16-stored F comes here with log utility only (setup_resident, setup_flat).
template <typename P, typename S>
__device__ __forceinline__ int node_kind(const IterArgs<P, S>& a) { return sizeof(S) == 2 ? 0 : a.kind; }

template <typename P, typename S, int N>
__device__ __forceinline__ void node_data(const IterArgs<P, S>& a, const NodePiece& q, NodeItem<P, N>& x) {
  if (q.c * N >= a.ld) return;
  const size_t o = (size_t)q.j * a.ld + (size_t)q.c * N;
  ld_const<P, N>(a.W + o, x.wv);
  if (a.Gm) ld_const<P, N>(a.Gm + o, x.gv);
  else {
#pragma unroll
    for (int u = 0; u < N; ++u) x.gv[u] = a.gamma;
  }
  if (node_kind(a) == 1) {
#pragma unroll
    for (int u = 0; u < N; ++u)
      x.wg[u] = x.gv[u] == P(0.5) ? P(0) : pow(x.wv[u] * x.gv[u], P(1) / (P(1) - x.gv[u]));
  }
}

template <typename P, typename S, int N>
__device__ __forceinline__ void node_state(const IterArgs<P, S>& a, int par, const NodePiece& q,
                                           NodeItem<P, N>& x) {
  if (q.c * N >= a.ld) return;
  const size_t o = (size_t)q.j * a.ld + (size_t)q.c * N;
  ld_words<P, N>(a.Pm + o, x.po);
  ld_words<P, N>(a.Y[par] + o, x.yo);
#pragma unroll
  for (int u = 0; u < N; ++u) x.yl[u] = P(0);
  if constexpr (std::is_same<P, float>::value) {
    if (a.Ylo[par]) ld_tail<N>(a.Ylo[par] + o, x.yl);
  }
}

// R of the node's rows, k.. of the 32 whose edges the lanes hold, added to s with their signs.
// The loads are unconditional (rows past the last repeat it with weight 0), so that all R are in
// flight at once.
// PAIRS: rounded as node_kernel rounds it, consecutive rows added as pairs; else one row after the
// other (the batched engine's order).
template <typename P, typename S, int N, int R, bool PAIRS>
__device__ __forceinline__ void node_rows(const S* __restrict__ f0, size_t ld, int edge, int k, int nin, int deg,
                                          P (&s)[N]) {
  S f[R][N];
#pragma unroll
  for (int r = 0; r < R; ++r)
    ld_words<S, N>(f0 + (size_t)__shfl_sync(0xffffffffu, edge, k + r) * ld, f[r]);
#pragma unroll
  for (int r = 0; r < R; r += 2) {
    const P s0 = k + r < nin ? P(1) : k + r < deg ? P(-1) : P(0);
    const P s1 = k + r + 1 < nin ? P(1) : k + r + 1 < deg ? P(-1) : P(0);
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const P x0 = to_p<P>(f[r][u]), x1 = to_p<P>(f[r + 1][u]);
      if constexpr (PAIRS) s[u] += fma(s0, x0, s1 * x1);
      else s[u] = fma(s1, x1, fma(s0, x0, s[u]));
    }
  }
}

// s = sum_{in(j)} f - sum_{out(j)} f over the lane's N entries.
template <typename P, typename S, int N, bool PAIRS = true>
__device__ __forceinline__ void node_gather(const IterArgs<P, S>& a, const S* __restrict__ Fn,
                                            const NodePiece& q, P (&s)[N]) {
  const S* f0 = Fn + (q.c * N < a.ld ? (size_t)q.c * N : 0);
#pragma unroll
  for (int u = 0; u < N; ++u) s[u] = P(0);
  int edge = q.edge;
#pragma unroll 1
  for (int b = 0; b < q.deg; b += 32) {
    if (b) edge = node_edge(a, q, b + (int)(threadIdx.x & 31));
    const int nin = q.nin - b, deg = q.deg - b, cnt = min(32, deg);
    int k = 0;
    if (N == 1 && cnt > 16) {
      node_rows<P, S, N, 24, PAIRS>(f0, a.ld, edge, 0, nin, deg, s);
      k = 24;
    } else if (N <= 2 && cnt > 12) {
      node_rows<P, S, N, 16, PAIRS>(f0, a.ld, edge, 0, nin, deg, s);
      k = 16;
    }
    if constexpr (N > 2) {
#pragma unroll 1
      for (; k + 6 < cnt; k += 8) node_rows<P, S, N, 8, PAIRS>(f0, a.ld, edge, k, nin, deg, s);
    }
#pragma unroll 1
    for (; k < cnt; k += 4) node_rows<P, S, N, 4, PAIRS>(f0, a.ld, edge, k, nin, deg, s);
  }
}

template <typename P, typename S, int N, bool CHECK>
__device__ __forceinline__ void node_update(const IterArgs<P, S>& a, int par, const NodePiece& q, const P (&s)[N],
                                            NodeItem<P, N>& x, P beta, P (&loc)[NODE_PARTS]) {
  if (q.c * N >= a.ld) return;
  const int j = q.j, c = q.c;
  const P rho = a.rho, inv_rho = P(1) / rho;
  const size_t o = (size_t)j * a.ld + (size_t)c * N;
  const int kind = node_kind(a);
  P yn[N], th_v[N], up_v[N], yh_v[N];
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const int i = c * N + u;
    const P fhat_at = (s[u] - (P(1) - rho) * x.po[u]) * inv_rho;   // (F^ A^T)_{ij}
    const P fplus_at = P(2) * fhat_at - x.po[u];                   // (F^{k+1} A^T)_{ij}
    const bool live = (i < a.n) && (i != j);
    // Y^ - Y = -beta (F^{k+1}A^T + t), t = T(Y^) (Moreau); Y^ = 0 on the diagonal and in pads
    P delta, tr = P(0);
    if (live) {
      const P vv = x.yo[u] + (x.yl[u] - beta * fplus_at);
      if (kind == 0) tr = prox_traffic<P>(0, vv, beta, x.wv[u], x.gv[u]);
      else prox_pow_traffic<P>(vv, beta, x.wv[u], x.wg[u], x.gv[u], tr);
      delta = -beta * (fplus_at + tr);
    } else {
      delta = -(x.yo[u] + x.yl[u]);
    }
    const P yhat = live ? (x.yo[u] + (x.yl[u] + delta)) : P(0);
    P hi = x.yo[u], lo = x.yl[u];
    add_split(hi, lo, rho * delta);
    yn[u] = hi;
    x.yl[u] = lo;
    const P dy = rho * delta;
    loc[0] = fma(dy, dy, loc[0]);
    if constexpr (CHECK) {
      const P th = -fhat_at;
      th_v[u] = i < a.n ? th : P(0);
      yh_v[u] = yhat;
      up_v[u] = P(0);
      if (live) {
        if (!(th > P(0))) loc[1] += P(1);
        else {
          loc[2] += util_value<P>(kind, th, x.wv[u], x.gv[u]);
          up_v[u] = util_grad<P>(kind, th, x.wv[u], x.gv[u]);
        }
        if (yhat < P(0)) {
          loc[3] += util_conj_neg<P>(kind, yhat, x.wv[u], x.gv[u]);
          const P dt = tr - th;
          loc[4] = fma(dt, dt, loc[4]);
        } else {
          loc[6] += P(1);
        }
        loc[5] = fma(th, th, loc[5]);
      }
    }
  }
  if constexpr (std::is_same<P, float>::value) {
    if (a.Ylo[par ^ 1]) st_tail<N>(a.Ylo[par ^ 1] + o, x.yl);
  }
  st_words<P, N>(a.Y[par ^ 1] + o, yn);
  st_words<P, N>(a.Pm + o, s);
  if constexpr (CHECK) {
    st_words<P, N>(a.That + o, th_v);
    st_words<P, N>(a.Uprime + o, up_v);
    st_words<P, N>(a.Yhat + o, yh_v);
  }
}

// The node phase. Every warp of the grid has about as many pieces (a warp per node left 5 of 6
// SMs idle at n = 200), and a thread's serial chain is N root searches instead of a whole row's.
// Pieces go column block by column block over all nodes, so that the rows of a block that nodes
// gather (each row by its head and by its tail) are in L2 together: F is read from HBM once
// where it does not fit L2. The next piece's edges and data are loaded while this one's rows
// arrive.
template <typename P, typename S, int N, bool CHECK>
__device__ __forceinline__ void node_pieces(const IterArgs<P, S>& a, int par, unsigned p0, unsigned p1,
                                            unsigned step, NodePiece& q, NodeItem<P, N>& x, P beta,
                                            double (&acc)[NODE_PARTS]) {
  const S* Fn = a.F[par ^ 1];
#pragma unroll 1
  for (unsigned pc = p0; pc < p1; pc += step) {
    P s[N], loc[NODE_PARTS];
#pragma unroll
    for (int k = 0; k < NODE_PARTS; ++k) loc[k] = P(0);
    const bool more = pc + step < p1;
    NodePiece qn;
    if (more) node_place<P, S, N>(a, pc + step, qn);
    node_gather<P, S, N>(a, Fn, q, s);
    if (more) qn.edge = node_edge(a, qn, (int)(threadIdx.x & 31));
    node_update<P, S, N, CHECK>(a, par, q, s, x, beta, loc);
#pragma unroll
    for (int k = 0; k < (CHECK ? NODE_PARTS : 1); ++k) acc[k] += (double)loc[k];
    if (more) {
      q = qn;
      node_data<P, S, N>(a, q, x);
      node_state<P, S, N>(a, par, q, x);
    }
  }
}

// Residual check (Eq. e-res and the dual bound; see check_kernel), a warp per edge.
template <typename P, typename S>
__device__ __forceinline__ void check_phase(const IterArgs<P, S>& a, int par, P alpha, int warp, int nwarps,
                                            double (&acc)[CHECK_PARTS]) {
  constexpr int VW = StoreTraits<S>::VW;
  const int lane = threadIdx.x & 31;
  const int nchunks = a.ld / VW;
  const S* Fo = a.F[par];
  const P* Y = a.Y[par];
  const __nv_bfloat16* ylo = a.Ylo[par];
#pragma unroll
  for (int q = 0; q < CHECK_PARTS; ++q) acc[q] = 0.0;
#pragma unroll 1
  for (int e = warp; e < a.m; e += nwarps) {
    const int hh = __ldg(a.e_head + e), tt = __ldg(a.e_tail + e);
    const P mu = __ldcg(a.mu + e);
    const size_t fo = (size_t)e * a.ld, ho = (size_t)hh * a.ld, to = (size_t)tt * a.ld;
    P ymax = -INFINITY, lg2 = P(0), lgd = P(0), ld2 = P(0);
#pragma unroll 1
    for (int ci = lane; ci < nchunks; ci += 32) {
      S fv[VW];
      P y1[VW], y2[VW], g1[VW], g2[VW], z1[VW], z2[VW], dl[VW];
      ld_words<S, VW>(Fo + fo + ci * VW, fv);
      ld_words<P, VW>(Y + ho + ci * VW, y1);
      ld_words<P, VW>(Y + to + ci * VW, y2);
      ld_words<P, VW>(a.Uprime + ho + ci * VW, g1);
      ld_words<P, VW>(a.Uprime + to + ci * VW, g2);
      ld_words<P, VW>(a.Yhat + ho + ci * VW, z1);
      ld_words<P, VW>(a.Yhat + to + ci * VW, z2);
#pragma unroll
      for (int u = 0; u < VW; ++u) dl[u] = P(0);
      if constexpr (std::is_same<P, float>::value) {
        if (ylo) {
          float l1[VW], l2[VW];
          ld_tail<VW>(ylo + ho + ci * VW, l1);
          ld_tail<VW>(ylo + to + ci * VW, l2);
#pragma unroll
          for (int u = 0; u < VW; ++u) dl[u] = l1[u] - l2[u];
        }
      }
#pragma unroll
      for (int u = 0; u < VW; ++u) {
        if (ci * VW + u >= a.n) continue;
        const P q = to_p<P>(fv[u]) + alpha * ((y1[u] - y2[u]) + dl[u]);
        const P fh = q > mu ? q - mu : P(0);
        const P d = fh - q, g = g1[u] - g2[u];
        lg2 = fma(g, g, lg2);
        lgd = fma(g, d, lgd);
        ld2 = fma(d, d, ld2);
        ymax = fmax(ymax, z1[u] - z2[u]);
      }
    }
    acc[0] += (double)lg2;
    acc[1] += (double)lgd;
    acc[2] += (double)ld2;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ymax = fmax(ymax, __shfl_xor_sync(0xffffffffu, ymax, o));
    if (lane == 0 && ymax > P(0)) acc[3] += (double)__ldg(a.cap + e) * (double)ymax;
  }
}

// ------------------------------------------------------------------ scalar tail

// Scalar tail in block 0: a warp per field sums the shares' FP64 partials in a fixed order, then
// one thread updates the scalars and evaluates the stop test.
template <typename P, typename S, int BLOCK>
__device__ __forceinline__ void scalar_phase(const IterArgs<P, S>& a, const ResidentArgs& ra, long long k,
                                          bool check) {
  constexpr int FIELDS = 1 + NODE_PARTS + CHECK_PARTS;
  __shared__ double field[FIELDS];
  const int lane = threadIdx.x & 31;
  const int nf = check ? FIELDS : 2;
  for (int f = threadIdx.x >> 5; f < nf; f += BLOCK / 32) {
    const double* base = f == 0 ? a.part_edge : f <= NODE_PARTS ? a.part_node + (f - 1)
                                              : a.part_check + (f - 1 - NODE_PARTS);
    const int stride = f == 0 ? 1 : f <= NODE_PARTS ? NODE_PARTS : CHECK_PARTS;
    double s = 0.0;
    for (int b = lane; b < ra.ctas; b += 32) s += __ldcg(base + (size_t)b * stride);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) field[f] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a.sc->k = k;
    scalar_update(a.sc, field[0], field[1], field + 1, field + 1 + NODE_PARTS, check);
    if (check) ra.ctl->stop.verdict = stop_test(*a.sc, ra.rule, ra.ctl->stop);
  }
}

// FP64 projection of a warp's row: project_mu_n with the comparisons, minima and maxima on
// order-preserving 64-bit integers, since the FP64 unit runs at 1/64 of FP32 and a pass
// is otherwise four FP64 operations per entry. Entries equal to -0 do not occur (see
// shifted_q; the floor is made +0), so the integer order is the numeric one.
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double order_value(long long k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}
template <int VPT, int VW>
__device__ __forceinline__ double project_mu64(const double (&q)[VPT][VW], double c, double lo) {
  const long long kInf = 0x7fffffffffffffffll;
  auto eval = [&](double mu, double& s, int& cnt, double& amin, double& imax) {
    const long long km = order_key(mu);
    double ls = 0.0;
    long long am = kInf, im = -kInf;
    int lc = 0;
#pragma unroll
    for (int v = 0; v < VPT; ++v)
#pragma unroll
      for (int u = 0; u < VW; ++u) {
        const long long kx = order_key(q[v][u]);
        const bool act = kx > km;
        if (__any_sync(0xffffffffu, act)) ls += act ? q[v][u] : 0.0;
        lc += act;
        am = act && kx < am ? kx : am;
        im = !act && kx > im ? kx : im;
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ls += __shfl_xor_sync(0xffffffffu, ls, o);
      const long long a2 = __shfl_xor_sync(0xffffffffu, am, o), i2 = __shfl_xor_sync(0xffffffffu, im, o);
      am = a2 < am ? a2 : am;
      im = i2 > im ? i2 : im;
    }
    s = ls;
    cnt = __reduce_add_sync(0xffffffffu, lc);
    amin = am == kInf ? INFINITY : order_value(am);
    imax = im == -kInf ? -INFINITY : order_value(im);
  };
  double mu = lo < 0.0 ? 0.0 : lo, s, amin, imax;
  int cnt;
  eval(mu, s, cnt, amin, imax);
  const double phi = s - (double)cnt * mu - c;
  if (phi <= 0.0) {
    if (mu == lo || phi == 0.0) return mu;
    double mn = cnt > 0 ? (s - c) / (double)cnt : lo;
    if (mn <= lo) {
      mu = lo;
      eval(mu, s, cnt, amin, imax);
      if (s - (double)cnt * lo - c <= 0.0) return lo;
    } else {
      if (cnt > 0 && mn >= imax) return mn;
      mu = mn + 0.0;
      eval(mu, s, cnt, amin, imax);
    }
  }
#pragma unroll 1
  for (int it = 0; it < 64; ++it) {
    if (cnt == 0) break;
    const double mn = (s - c) / (double)cnt;
    if (!(mn > mu)) break;
    if (mn < amin) return mn;
    mu = mn + 0.0;
    eval(mu, s, cnt, amin, imax);
  }
  return mu;
}

// ------------------------------------------------------------------ edge phase

// Edges [e0, e1) of the CTA, a warp each (e starts at the warp's first): q, the projection and
// the relaxation as in edge_kernel; returns this thread's ||dF||^2. The first row of F is loaded
// before the barrier (`pending`) is waited for.
template <typename P, typename S, int VPT, int NW>
__device__ __forceinline__ P edge_phase(const IterArgs<P, S>& a, int par, P alpha, int e, int e1,
                                        GridBarrier& bar, bool pending, bool& ok) {
  constexpr int VW = StoreTraits<S>::VW;
  // long rows keep only q in registers through the projection and read f again (from L1)
  constexpr bool KEEP_F = VPT * VW * (int)sizeof(P) <= 64;
  const int lane = threadIdx.x & 31;
  const int nchunks = a.ld / VW;
  const P rho = a.rho;
  const S* Fo = a.F[par];
  S* Fn = a.F[par ^ 1];
  const P* Y = a.Y[par];
  const __nv_bfloat16* ylo = a.Ylo[par];
  P dsum = P(0);
  S fs[VPT][VW];
  int h = 0, t = 0;
  P cap = P(0), mu0 = P(0), mu0l = P(0);
  auto load_row = [&](int x) {
    h = __ldg(a.e_head + x);
    t = __ldg(a.e_tail + x);
    cap = __ldg(a.cap + x);
    mu0 = a.mu[x];
    mu0l = a.mu_lo[x];
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int ci = v * 32 + lane;
      if (ci < nchunks) ld_words<S, VW>(Fo + (size_t)x * a.ld + ci * VW, fs[v]);
    }
  };
  if (e < e1) load_row(e);
  ok = !pending || bar.wait();
  if (!ok) return dsum;
#pragma unroll 1
  while (e < e1) {
    P q[VPT][VW];
    const P* yh = Y + (size_t)h * a.ld;
    const P* yt = Y + (size_t)t * a.ld;
    const P floor = shifted_floor<P>(mu0, mu0l) + P(0);
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int ci = v * 32 + lane;
      if (ci < nchunks) {
        P a1[VW], a2[VW];
        ld_words<P, VW>(yh + ci * VW, a1);
        ld_words<P, VW>(yt + ci * VW, a2);
        if constexpr (std::is_same<P, float>::value) {
          float dl[VW];
#pragma unroll
          for (int u = 0; u < VW; ++u) dl[u] = 0.f;
          if (ylo) {
            float l1[VW], l2[VW];
            ld_tail<VW>(ylo + (size_t)h * a.ld + ci * VW, l1);
            ld_tail<VW>(ylo + (size_t)t * a.ld + ci * VW, l2);
#pragma unroll
            for (int u = 0; u < VW; ++u) dl[u] = l1[u] - l2[u];
          }
#pragma unroll
          for (int u = 0; u < VW; u += 2) {
            const float2 ff = make_float2(to_p<P>(fs[v][u]), to_p<P>(fs[v][u + 1]));
            const float2 qq = shifted_q2(ff, make_float2(a1[u], a1[u + 1]), make_float2(a2[u], a2[u + 1]),
                                         make_float2(dl[u], dl[u + 1]), p2(alpha), p2(-mu0), p2(-mu0l));
            q[v][u] = qq.x;
            q[v][u + 1] = qq.y;
          }
        } else {
#pragma unroll
          for (int u = 0; u < VW; ++u)
            q[v][u] = shifted_q<P>(to_p<P>(fs[v][u]), a1[u], a2[u], P(0), alpha, mu0, mu0l);
        }
      } else {
#pragma unroll
        for (int u = 0; u < VW; ++u) q[v][u] = floor;
      }
    }
    P mu;
    if constexpr (std::is_same<P, double>::value) {
      mu = project_mu64<VPT, VW>(q, cap, floor);
    } else {
      GroupScratch<32> none;   // warp groups reduce without scratch memory
      int phase = 0;
      mu = project_mu<32, VPT, VW, P>(q, cap, P(0), floor, none, phase);
    }
    P dloc = P(0);
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int ci = v * 32 + lane;
      if (ci < nchunks) {
        S out[VW];
        if constexpr (!KEEP_F) ld_words<S, VW>(Fo + (size_t)e * a.ld + ci * VW, fs[v]);
        if constexpr (std::is_same<P, float>::value) {
          float2 sq = p2(0.f);
#pragma unroll
          for (int u = 0; u < VW; u += 2) {
            const float2 ff = make_float2(to_p<P>(fs[v][u]), to_p<P>(fs[v][u + 1]));
            const float2 t2 = p2_add(make_float2(q[v][u], q[v][u + 1]), p2(-mu));
            const float2 st = p2_sub(make_float2(fmaxf(t2.x, 0.f), fmaxf(t2.y, 0.f)), ff);
            const float2 fnew = p2_fma(p2(rho), st, ff);
            sq = p2_fma(st, st, sq);
            out[u] = from_p<S, P>(fnew.x);
            out[u + 1] = from_p<S, P>(fnew.y);
          }
          dloc += rho * rho * (sq.x + sq.y);
        } else {
#pragma unroll
          for (int u = 0; u < VW; ++u) {
            const P ff = to_p<P>(fs[v][u]);
            const P fh = q[v][u] > mu ? q[v][u] - mu : P(0);
            out[u] = from_p<S, P>(rho * fh + (P(1) - rho) * ff);
            const P d = rho * (fh - ff);   // the step itself (see edge_kernel)
            dloc = fma(d, d, dloc);
          }
        }
        st_plain<S, VW>(Fn + (size_t)e * a.ld + ci * VW, out);
      }
    }
    dsum += dloc;
    if (lane == 0) {
      P hi, lo;
      shifted_mu<P>(mu0, mu0l, mu, hi, lo);
      a.mu[e] = hi;
      a.mu_lo[e] = lo;
    }
    e += NW;
    if (e < e1) load_row(e);
  }
  return dsum;
}

// ------------------------------------------------------------------ the kernels

// The work of a phase is dealt to `ctas` CTAs; this warp's part as one of CTA `cta`.
struct ResidentPlace {
  int e0, e1, warp, nwarps;
  unsigned pieces;   // of the node phase: this warp takes warp, warp + nwarps, ...
};

template <int NW>
__device__ __forceinline__ ResidentPlace resident_place(int n, int m, int ld, int N, int cta, int ctas) {
  ResidentPlace w;
  // numbered across the CTAs first, so that few pieces spread over all SMs
  w.warp = (threadIdx.x >> 5) * ctas + cta;
  w.nwarps = ctas * NW;
  // consecutive edges per CTA (their heads' dual rows are shared in L1)
  w.e0 = (int)((long long)m * cta / ctas) + (threadIdx.x >> 5);
  w.e1 = (int)((long long)m * (cta + 1) / ctas);
  w.pieces = (unsigned)n * ((unsigned)(ld + 32 * N - 1) / (32 * N));
  return w;
}

// Start of a launch, in thread 0 and before a barrier of the CTA: whether a wait of an earlier launch
// of the group has run out. That launch left the count of arrivals short, so every barrier behind
// it would run out of polls as well.
template <typename P, typename S>
__device__ __forceinline__ void resident_start(const IterArgs<P, S>& a, int& failed) {
  if (threadIdx.x == 0) failed = __ldcg(&a.sc->wait_timeout);
}

// Iterations without a scalar tail. No function call and no spilled register is in the loop: a
// spilled register would be read back through L2, since every barrier drops the L1.
template <typename P, typename S, int VPT, int N, int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1)
resident_kernel(const __grid_constant__ IterArgs<P, S> a, const __grid_constant__ ResidentArgs ra) {
  constexpr int NW = BLOCK / 32;
  __shared__ int failed;
  if (__ldcg(&ra.ctl->stop.verdict) != STOP_NO) return;
  const ResidentPlace w = resident_place<NW>(a.n, a.m, a.ld, N, blockIdx.x, gridDim.x);
  const P alpha = (P)__ldcg(&a.sc->alpha), beta = (P)__ldcg(&a.sc->beta);
  NodePiece piece;
  NodeItem<P, N> x;      // data of the first piece: stays in registers when it is the only one
  const bool any = (unsigned)w.warp < w.pieces, one = (unsigned)(w.warp + w.nwarps) >= w.pieces;
  if (any) {
    node_place<P, S, N>(a, w.warp, piece);
    piece.edge = node_edge(a, piece, (int)(threadIdx.x & 31));
    node_data<P, S, N>(a, piece, x);
  }
  resident_start(a, failed);
  __syncthreads();
  if (failed) return;
  GridBarrier bar{&ra.ctl->arrived, a.sc, &failed, ra.arrived};
  int par = a.parity;
#pragma unroll 1
  for (int i = 0; i < ra.count; ++i, par ^= 1) {
    bool ok;
    const P dsum = edge_phase<P, S, VPT, NW>(a, par, alpha, w.e0, w.e1, bar, i > 0, ok);
    if (!ok) return;
    bar.arrive();
    if (any) {
      if (!one) {
        node_place<P, S, N>(a, w.warp, piece);
        piece.edge = node_edge(a, piece, (int)(threadIdx.x & 31));
        node_data<P, S, N>(a, piece, x);
      }
      node_state<P, S, N>(a, par, piece, x);
    }
    if (!bar.wait()) return;
    double acc[NODE_PARTS] = {0.0};
    node_pieces<P, S, N, false>(a, par, w.warp, w.pieces, w.nwarps, piece, x, beta, acc);
    // a sum that is not finite here is reported as the scalar tail would
    if (!isfinite(dsum) || !isfinite(acc[0])) a.sc->numeric_error = 1;
    if (i + 1 < ra.count) bar.arrive();
  }
}

// Iterations with a scalar tail (a multiple of k_adapt, or a stop test), usually one or two. The work
// is split into the shares of ra.ctas CTAs whatever the grid: CTA b of a smaller one takes the shares b,
// b + gridDim.x, ... one after the other. So the sums, and with them the iterates, do not depend on
// the grid, and solves under way at the same time can run on a part of the SMs each (ResidentTurn).
template <typename P, typename S, int VPT, int N, int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1)
resident_special_kernel(const __grid_constant__ IterArgs<P, S> a, const __grid_constant__ ResidentArgs ra) {
  constexpr int NW = BLOCK / 32;
  __shared__ int failed;
  if (__ldcg(&ra.ctl->stop.verdict) != STOP_NO) return;
  resident_start(a, failed);
  __syncthreads();
  if (failed) return;
  GridBarrier bar{&ra.ctl->arrived, a.sc, &failed, ra.arrived};
  int par = a.parity;
#pragma unroll 1
  for (int i = 0; i < ra.count; ++i, par ^= 1) {
    const long long k = ra.k + i;
    const bool check = (k + 1) % ra.k_check == 0 || k + 1 >= ra.max_iters;
    const P alpha = (P)__ldcg(&a.sc->alpha), beta = (P)__ldcg(&a.sc->beta);
#pragma unroll 1
    for (int share = blockIdx.x; share < ra.ctas; share += gridDim.x) {
      const ResidentPlace w = resident_place<NW>(a.n, a.m, a.ld, N, share, ra.ctas);
      bool ok;
      double v1[1] = {(double)edge_phase<P, S, VPT, NW>(a, par, alpha, w.e0, w.e1, bar, false, ok)};
      block_sum_write<BLOCK, 1>(v1, a.part_edge + share);
      __syncthreads();   // its scratch is used again
    }
    bar.arrive();
    if (!bar.wait()) return;
#pragma unroll 1
    for (int share = blockIdx.x; share < ra.ctas; share += gridDim.x) {
      const ResidentPlace w = resident_place<NW>(a.n, a.m, a.ld, N, share, ra.ctas);
      double acc[NODE_PARTS];
#pragma unroll
      for (int q = 0; q < NODE_PARTS; ++q) acc[q] = 0.0;
      NodePiece piece;
      NodeItem<P, N> x;
      if ((unsigned)w.warp < w.pieces) {
        node_place<P, S, N>(a, w.warp, piece);
        piece.edge = node_edge(a, piece, (int)(threadIdx.x & 31));
        node_data<P, S, N>(a, piece, x);
        node_state<P, S, N>(a, par, piece, x);
      }
      if (check) node_pieces<P, S, N, true>(a, par, w.warp, w.pieces, w.nwarps, piece, x, beta, acc);
      else node_pieces<P, S, N, false>(a, par, w.warp, w.pieces, w.nwarps, piece, x, beta, acc);
      block_sum_write<BLOCK, NODE_PARTS>(acc, a.part_node + (size_t)share * NODE_PARTS);
      __syncthreads();
    }
    bar.arrive();
    if (!bar.wait()) return;
    if (check) {
#pragma unroll 1
      for (int share = blockIdx.x; share < ra.ctas; share += gridDim.x) {
        double cacc[CHECK_PARTS];
        check_phase<P, S>(a, par, alpha, (threadIdx.x >> 5) * ra.ctas + share, ra.ctas * NW, cacc);
        block_sum_write<BLOCK, CHECK_PARTS>(cacc, a.part_check + (size_t)share * CHECK_PARTS);
        __syncthreads();
      }
      bar.arrive();
      if (!bar.wait()) return;
    }
    if (blockIdx.x == 0) scalar_phase<P, S, BLOCK>(a, ra, k, check);
    if (i + 1 == ra.count) return;
    bar.arrive();
    if (!bar.wait()) return;
    if (check && __ldcg(&ra.ctl->stop.verdict) != STOP_NO) return;
  }
}

template <typename P, typename S, int IDX>
void fill_resident(ResidentTable<P, S>& t) {
  constexpr ResidentVariant v = resident_variant<P, S>(IDX);
  if constexpr (32 * v.vpt * StoreTraits<S>::VW <= 1024) {
    t.plain[IDX] = resident_kernel<P, S, v.vpt, v.entries, RESIDENT_BLOCK>;
    t.special[IDX] = resident_special_kernel<P, S, v.vpt, v.entries, RESIDENT_BLOCK>;
  }
}
template <typename P, typename S>
ResidentTable<P, S> make_resident_table() {
  ResidentTable<P, S> t{};
  fill_resident<P, S, 0>(t);
  fill_resident<P, S, 1>(t);
  fill_resident<P, S, 2>(t);
  fill_resident<P, S, 3>(t);
  return t;
}

}  // namespace pdmcf
