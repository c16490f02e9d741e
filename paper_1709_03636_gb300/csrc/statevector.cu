// Full-Hilbert-space reference on the GPU (the comparison method of Section 5:
// simulate the whole 2^n state).  QAOA Max-Cut of Section 4.1: |+>^n, then per
// layer the diagonal phase exp(-i gamma/2 sum_e z_a z_b) and exp(-i beta X) on
// every qubit; finally <C> = sum_x |psi_x|^2 cut(x) (Eqs. 9-10) and, on request,
// <Z_a Z_b> per edge.
//
// Layout: qubit q is bit q of the element index.  A pass moves tiles of 2^tb
// elements (64 KB: 2^13 complex64 or 2^12 complex128, two CTAs per SM) through
// registers.  Pass 0 of a layer holds qubits 0..tb-1 (contiguous tiles) and
// applies the layer's phase on load; every further pass mixes its own group of
// qubits and carries as many low qubits along (unmixed) as fill the tile, so
// tiles stay full and rows contiguous.  The qubits above pass 0 are split evenly
// over the fewest passes.  A state smaller than a tile is held in shared memory
// by one CTA (sv_small_kernel).
// The last pass of the last layer accumulates |psi|^2 cut(x).
//
// The rotation [[c, -i s], [-i s, c]] (c = cos beta, s = sin beta) is applied
// without its larger factor f (c when |c| >= |s|, else s): x0' = x0 - i t x1
// with t = s / c, or x0' = u x0 - i x1 with u = c / s, two fused multiply-adds
// per element and qubit instead of four.  A layer therefore leaves the state
// divided by F = f^n; the next layer's phase table carries F (applied with the
// phase), and the last layer's F scales the stored state and F^2 the sum for
// <C>.  |f| >= 1/sqrt(2), so the stored amplitudes stay within
// 2^(-n/2) .. 1 of the unit-norm state's scale.
//
// The phase and rotation values are computed once per launch (FP64 angles).
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "exec_common.cuh"
#include "sv_launch.h"

namespace qtc {

constexpr int kSvThreads = 512;
constexpr int kSvMaxEdges = 512;

template <typename T> struct RealOf;
template <> struct RealOf<float2> { using type = float; };
template <> struct RealOf<double2> { using type = double; };

int sv_tile_bits(int dtype) { return dtype == 0 ? 12 : 13; }

int sv_passes(int n, int tmax, int* lo, int* len, int* rl) {
  lo[0] = 0;
  len[0] = n < tmax ? n : tmax;
  rl[0] = 0;
  const int rest = n - len[0];
  if (rest <= 0) return 1;
  const int per = tmax - 4;                    // at least 4 carried qubits per pass
  const int k = (rest + per - 1) / per;
  int q = len[0];
  for (int i = 0; i < k; ++i) {
    const int l = rest / k + (i < rest % k ? 1 : 0);
    lo[1 + i] = q;
    len[1 + i] = l;
    rl[1 + i] = tmax - l;
    q += l;
  }
  return 1 + k;
}

std::vector<uint16_t> sv_cut_table(const std::vector<uint32_t>& adj) {
  const int n = (int)adj.size();
  std::vector<uint16_t> w((size_t)1 << n);
  for (uint32_t t = 0; t < (1u << n); ++t) {
    int c = 0;
    for (int v = 0; v < n; ++v)
      if ((t >> v) & 1u) c += __builtin_popcount(adj[v] & ~t);
    w[t] = (uint16_t)c;
  }
  return w;
}

struct SvArgs {
  void* psi;
  int n, m;
  const uint32_t* adj;       // per qubit: bit mask of its neighbours (n <= 32)
  const void* phase;         // per layer m + 1 values exp(-i gamma (m - 2c) / 2)
  const void* rot;           // per layer (cos beta, sin beta)
  const uint16_t* wcut;      // cut(x) of every x (states smaller than a tile), else null
  int layer;
  int lo, len, rl;           // pass: tile bits 0..len-1 (lo = 0) or 0..rl-1 and lo..lo+len-1
  int first;                 // 1: the state is |+>, do not read it
  int last;                  // 1: accumulate <C> after this pass
  int store;                 // 0: the pass's result is not needed in memory (last pass, no
                             // per-edge values): it is only reduced into <C>
  const double2* scale;      // (F, F^2) of the last layer (see the rotation above)
  double* acc;               // [<C>, <ZZ> per edge]
};

template <typename T>
__device__ __forceinline__ uint64_t sv_gidx(const SvArgs& a, uint64_t blk, uint32_t t) {
  if (a.lo == 0) return (blk << a.len) | t;
  const int rl = a.rl;
  const uint64_t low = t & ((1u << rl) - 1u), mid = t >> rl;
  const uint64_t below = blk & ((1ull << (a.lo - rl)) - 1);  // bits rl..lo-1
  const uint64_t above = blk >> (a.lo - rl);                   // bits lo+len..
  return low | (below << rl) | (mid << a.lo) | (above << (a.lo + a.len));
}

// Sets up the tables of an evaluation, one CTA per layer: phase[layer][c] (times
// the previous layer's F), rot[layer] = (t or u, 1 when the cos form) and scale =
// (F, F^2) of the last layer; clears the sums.  Bound by the latency of one FP64
// sincos: the CTA's last warp takes the previous and this layer's rotation (lanes
// 0 and 1) while the others take a phase each, and F = f^n is raised by squaring.
// With both sincos and n multiplications in each thread, and a memset for the sums,
// it took 7.6 us of the 119 us of a p=3 n=21 evaluation (115 us now).
template <typename T>
__global__ void __launch_bounds__(kSvMaxEdges + 64)
sv_setup_kernel(const double* params, int n, int p, int m, T* phase, T* rot, double2* scale,
                double* acc) {
  __shared__ double s_before;   // F of the previous layer
  const int layer = blockIdx.x, c = threadIdx.x, last = (int)blockDim.x - 32;
  double sn = 0.0, cs = 0.0;
  if (c <= m) {
    sincos(-0.5 * params[layer] * (double)(m - 2 * c), &sn, &cs);
  } else if (c == last || c == last + 1) {
    const int l = layer - 1 + (c - last);
    double F = 1.0;
    if (l >= 0) {
      sincos(params[p + l], &sn, &cs);
      const bool kc = fabs(cs) >= fabs(sn);
      double f = kc ? cs : sn;
      for (int e = n; e > 0; e >>= 1, f *= f)
        if (e & 1) F *= f;
      if (l == layer) {
        rot[layer] = from_d2<T>(make_double2(kc ? sn / cs : cs / sn, kc ? 1.0 : 0.0));
        if (layer == p - 1) *scale = make_double2(F, F * F);
      }
    }
    if (c == last) s_before = F;
  }
  for (int i = layer * (int)blockDim.x + c; i <= m; i += p * (int)blockDim.x) acc[i] = 0.0;
  __syncthreads();
  if (c <= m)
    phase[(size_t)layer * (m + 1) + c] = from_d2<T>(make_double2(s_before * cs, s_before * sn));
}

// exp(-i beta X) on the pair (x0, x1) = amplitudes with the qubit at 0 and 1,
// without the factor f: KC: x0' = x0 - i t x1; else x0' = u x0 - i x1 (r = t
// or u; the same on both sides of the pair).
template <bool KC, typename T, typename R>
__device__ __forceinline__ void rxs_pair(T& x0, T& x1, R r) {
  const T a = x0, b = x1;
  if (KC) {
    x0.x = a.x + r * b.y;
    x0.y = a.y - r * b.x;
    x1.x = b.x + r * a.y;
    x1.y = b.y - r * a.x;
  } else {
    x0.x = r * a.x + b.y;
    x0.y = r * a.y - b.x;
    x1.x = r * b.x + a.y;
    x1.y = r * b.y - a.x;
  }
}

// The same with the partner amplitude in another lane (bit q of the lane).
template <bool KC, typename T, typename R>
__device__ __forceinline__ void rxs_shfl(T& v, R r, int q) {
  const R px = __shfl_xor_sync(0xffffffffu, v.x, 1u << q);
  const R py = __shfl_xor_sync(0xffffffffu, v.y, 1u << q);
  if (KC) {
    v.x = v.x + r * py;
    v.y = v.y - r * px;
  } else {
    v.x = r * v.x + py;
    v.y = r * v.y - px;
  }
}

// The rotation on k = 1..3 consecutive qubit bits of 2^k amplitudes in registers.
template <int K, bool KC, typename T, typename R>
__device__ __forceinline__ void rx_bits(T (&v)[8], R r) {
#pragma unroll
  for (int q = 0; q < K; ++q)
#pragma unroll
    for (int i = 0; i < (1 << K); ++i)
      if (!((i >> q) & 1)) rxs_pair<KC>(v[i], v[i | (1 << q)], r);
}

// One mixer round on tile bits b..b+K-1: groups of 2^K amplitudes.
template <int K, bool KC, typename T, typename R>
__device__ __forceinline__ void rx_round(T* tile, uint32_t tsize, int b, R r) {
  const uint32_t ngroups = tsize >> K;
  const uint32_t lowm = (1u << b) - 1u;
  for (uint32_t g = threadIdx.x; g < ngroups; g += blockDim.x) {
    const uint32_t base = (g & lowm) | ((g & ~lowm) << K);
    T v[8];
#pragma unroll
    for (int i = 0; i < (1 << K); ++i) v[i] = tile[base | ((uint32_t)i << b)];
    rx_bits<K, KC>(v, r);
#pragma unroll
    for (int i = 0; i < (1 << K); ++i) tile[base | ((uint32_t)i << b)] = v[i];
  }
}

// A layer of a state smaller than a tile: one CTA, the state in shared memory.
template <typename T>
__global__ void __launch_bounds__(kSvThreads) sv_small_kernel(const SvArgs a) {
  using R = typename RealOf<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tile = reinterpret_cast<T*>(smem_raw);
  __shared__ T s_phase[kSvMaxEdges + 1];
  __shared__ double s_red[kSvThreads / 32];
  const int n = a.n, tb = n;
  const uint32_t tsize = 1u << tb;
  const T* phase = reinterpret_cast<const T*>(a.phase) + (size_t)a.layer * (a.m + 1);
  for (int c = threadIdx.x; c <= a.m; c += blockDim.x) s_phase[c] = phase[c];
  __syncthreads();
  const T rot = reinterpret_cast<const T*>(a.rot)[a.layer];
  const R rr = rot.x;
  const bool kc = rot.y != (R)0;
  auto cut = [&](uint32_t t) { return (int)__ldg(a.wcut + t); };
  T* psi = reinterpret_cast<T*>(a.psi);
  const R amp0 = (R)exp2(-0.5 * n);

  // Load.  With at least one element per thread, lanes hold consecutive tile
  // elements (coalesced loads, conflict-free stores) and qubits 0..4 are
  // mixed with shuffles (the partner of lane l for qubit q is l ^ 2^q:
  // x' = c x - i s partner, the same on both sides of the pair).
  const bool full_warps = tsize >= (uint32_t)blockDim.x;
  const int shuffled = full_warps ? (tb < 5 ? tb : 5) : 0;
  constexpr int kBatch = 8;
  for (uint32_t t0 = 0; t0 < tsize; t0 += kBatch * blockDim.x) {
    T v[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const uint32_t t = t0 + k * blockDim.x + threadIdx.x;
      if (t < tsize) {
        if (a.first) {
          v[k].x = amp0;
          v[k].y = 0;
        } else {
          v[k] = psi[t];
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const uint32_t t = t0 + k * blockDim.x + threadIdx.x;
      if (t < tsize) {
        const T ph = s_phase[cut(t)];
        const T x = v[k];
        v[k].x = x.x * ph.x - x.y * ph.y;
        v[k].y = x.x * ph.y + x.y * ph.x;
      }
      if (t0 + k * blockDim.x < tsize)  // uniform: whole warps
        for (int q = 0; q < shuffled; ++q) {
          if (kc) rxs_shfl<true>(v[k], rr, q);
          else rxs_shfl<false>(v[k], rr, q);
        }
      if (t < tsize) tile[t] = v[k];
    }
  }
  // the remaining qubits, three at a time
  for (int b = shuffled; b < tb; b += 3) {
    __syncthreads();
    const int k = tb - b < 3 ? tb - b : 3;
    if (kc) {
      if (k == 3) rx_round<3, true>(tile, tsize, b, rr);
      else if (k == 2) rx_round<2, true>(tile, tsize, b, rr);
      else rx_round<1, true>(tile, tsize, b, rr);
    } else {
      if (k == 3) rx_round<3, false>(tile, tsize, b, rr);
      else if (k == 2) rx_round<2, false>(tile, tsize, b, rr);
      else rx_round<1, false>(tile, tsize, b, rr);
    }
  }
  __syncthreads();
  R part = 0;
  const R fin = a.last ? (R)a.scale->x : (R)1;
  for (uint32_t t = threadIdx.x; t < tsize; t += blockDim.x) {
    T v = tile[t];
    if (a.last) {
      part += (v.x * v.x + v.y * v.y) * (R)cut(t);
      v.x *= fin;
      v.y *= fin;
    }
    if (a.store) psi[t] = v;
  }
  if (!a.last) return;
  for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = (double)part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += s_red[w];
    atomicAdd(&a.acc[0], sum * a.scale->y);
  }
}

// A full tile of 2^(K + 8) elements with 2^K per thread in registers (K = 5 for
// complex64, 4 for complex128; 256 threads, two CTAs per SM, so that each thread
// has 2^K loads in flight).  Two layouts of the tile index:
//  * top: registers on the top K bits; lanes on bits 0..4, except that the last
//    `sh` (at most two) lane bits take tile bits 8 - sh .. 7 when these are the
//    only mixed bits below the registers: they are mixed by shuffles, and the
//    pass needs no shared memory;
//  * low: registers on bits 8 - K .. 7, lanes on the bits below and the first
//    ones above, reached by one exchange through shared memory (pass 0, and
//    passes that mix more than two bits below the top ones).
// The mixer's shuffles and shared-memory round trips share one pipe, which bounds
// passes that compute cut(x): per amplitude pass 0 took ten shuffles, a table
// lookup and an exchange with 16 elements per thread; with 32 it takes six and an
// exchange (p=1 n=26 complex64 675 -> 508 us; p=3 n=21 149 -> 119 us).  cut(x) of a thread's elements comes from the adjacency masks by bit
// counts: cut(x | r) = cut(x) + sum_{k in r} c_k - 2 e(r), c_k = degree of
// register bit k's vertex - 2 popc(its neighbours in x), e(r) the edges among the
// register bits of r (one table per CTA).
constexpr int kSvWideThreads = 256;

template <int K, bool KC, typename T, typename R>
__device__ __forceinline__ void rx_reg_bits(T (&v)[1 << K], int r0, int lo, R r) {
#pragma unroll
  for (int q = 0; q < K; ++q)
    if (r0 + q >= lo)
#pragma unroll
      for (int i = 0; i < (1 << K); ++i)
        if (!((i >> q) & 1)) rxs_pair<KC>(v[i], v[i | (1 << q)], r);
}

// Register r's part of an index whose register bits have the offsets g.
template <int K>
__device__ __forceinline__ uint32_t reg_offset(const uint32_t (&g)[K], int r) {
  uint32_t o = 0;
#pragma unroll
  for (int k = 0; k < K; ++k)
    if ((r >> k) & 1) o |= g[k];
  return o;
}

template <typename T, int K, bool pass0>
__global__ void __launch_bounds__(kSvWideThreads, 2) sv_wide_kernel(const SvArgs a) {
  using R = typename RealOf<T>::type;
  constexpr int NR = 1 << K, TB = K + 8, NB = 8 - K;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tile = reinterpret_cast<T*>(smem_raw);
  __shared__ T s_phase[kSvMaxEdges + 1];
  __shared__ uint32_t s_adj[32];
  __shared__ int s_inner[2][NR];   // -2 e(r) of the top and of the low layout
  __shared__ double s_red[2 * kSvWideThreads / 32];
  const int n = a.n, rl = a.rl, lo = a.lo;
  const int mix_lo = pass0 ? 0 : rl;
  const int below = mix_lo < 8 ? 8 - mix_lo : 0;   // mixed bits below the top registers
  const bool exchange = pass0 || below > 2;
  const int sh = exchange ? 0 : below;
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  auto vertex = [&](int j) { return pass0 || j < rl ? j : lo + j - rl; };
  // tile index of a thread (registers zero) in each layout, register offsets
  const uint32_t top_base = (lane & ((1u << (5 - sh)) - 1u)) | (w << (5 - sh)) |
                            ((lane >> (5 - sh)) << (8 - sh));
  const uint32_t low_base = (lane & ((1u << NB) - 1u)) |
                            (((lane >> NB) | (w << (5 - NB))) << 8);
  uint32_t g_top[K], g_low[K];
  if (threadIdx.x < 32) s_adj[threadIdx.x] = (int)threadIdx.x < n ? a.adj[threadIdx.x] : 0u;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    g_top[k] = 1u << vertex(8 + k);
    g_low[k] = 1u << vertex(NB + k);
  }
  if (threadIdx.x < 2 * NR) {
    const int r = threadIdx.x & (NR - 1);
    const bool low = threadIdx.x >= NR;
    const uint32_t o = low ? reg_offset<K>(g_low, r) : reg_offset<K>(g_top, r);
    int e = 0;
#pragma unroll
    for (int k = 0; k < K; ++k)
      if ((r >> k) & 1) e += __popc(s_adj[vertex((low ? NB : 8) + k)] & o);
    s_inner[low][r] = -e;          // each inner edge counted from both ends: 2 e(r)
  }
  if (pass0) {
    const T* ph = reinterpret_cast<const T*>(a.phase) + (size_t)a.layer * (a.m + 1);
    for (int c = threadIdx.x; c <= a.m; c += kSvWideThreads) s_phase[c] = ph[c];
  }
  const T rot = reinterpret_cast<const T*>(a.rot)[a.layer];
  const R rr = rot.x;
  const bool kc = rot.y != (R)0;   // the form of the layer's rotation (uniform)
  T* psi = reinterpret_cast<T*>(a.psi);
  const R fin = a.last ? (R)a.scale->x : (R)1;
  // <C>: two sums per thread, of one half of its registers each, so that a chain of
  // single-precision additions is 16 terms per tile (complex64)
  R part[2] = {0, 0};
  __syncthreads();
  // f(r, cut) for the registers of a layout (first register bit j0), x their index
  // with registers zero; registers in Gray code order, one addition apart
  auto each_cut = [&](uint32_t x, int j0, const int* inner, auto&& f) {
    int c = 0, ck[K];
    for (int q = 0; q < n; ++q) c += (x >> q) & 1u ? __popc(s_adj[q] & ~x) : 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t m = s_adj[vertex(j0 + k)];
      ck[k] = __popc(m) - 2 * __popc(m & x);
    }
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      const int r = i ^ (i >> 1), was = i ? (i - 1) ^ ((i - 1) >> 1) : 0;
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (((r ^ was) >> k) & 1) c += (r >> k) & 1 ? ck[k] : -ck[k];
      f(r, c + inner[r]);
    }
  };
  const uint32_t n_tiles = (uint32_t)(1ull << (n - TB));
  for (uint32_t blk = blockIdx.x; blk < n_tiles; blk += gridDim.x) {
    uint32_t x = (uint32_t)sv_gidx<T>(a, blk, top_base);
    T v[NR];
    if (pass0 && a.first) {
      const R amp0 = (R)exp2(-0.5 * n);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        v[r].x = amp0;
        v[r].y = 0;
      }
    } else {
#pragma unroll
      for (int r = 0; r < NR; ++r) v[r] = psi[x | reg_offset<K>(g_top, r)];
    }
    if (pass0) {
      each_cut(x, 8, s_inner[0], [&](int r, int c) {
        const T ph = s_phase[c], y = v[r];
        v[r].x = y.x * ph.x - y.y * ph.y;
        v[r].y = y.x * ph.y + y.y * ph.x;
      });
    }
    if (kc) rx_reg_bits<K, true>(v, 8, mix_lo, rr);
    else rx_reg_bits<K, false>(v, 8, mix_lo, rr);
    for (int q = 5 - sh; q < 5; ++q)
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if (kc) rxs_shfl<true>(v[r], rr, q);
        else rxs_shfl<false>(v[r], rr, q);
      }
    if (exchange) {
      // (bit 3 flipped by bit 8: the reads of a half warp, bits 0..2 and 8, then
      // fall into distinct banks; 16-byte elements need no flip)
      auto at = [](uint32_t i) { return sizeof(T) == 8 ? i ^ ((i >> 5) & 8u) : i; };
      __syncthreads();   // earlier readers of the tile are done
#pragma unroll
      for (int r = 0; r < NR; ++r) tile[at(top_base | ((uint32_t)r << 8))] = v[r];
      __syncthreads();
#pragma unroll
      for (int r = 0; r < NR; ++r) v[r] = tile[at(low_base | ((uint32_t)r << NB))];
      x = (uint32_t)sv_gidx<T>(a, blk, low_base);
      if (kc) rx_reg_bits<K, true>(v, NB, mix_lo, rr);
      else rx_reg_bits<K, false>(v, NB, mix_lo, rr);
      for (int q = mix_lo; q < NB; ++q)
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          if (kc) rxs_shfl<true>(v[r], rr, q);
          else rxs_shfl<false>(v[r], rr, q);
        }
    }
    if (a.last) {
      auto add = [&](int r, int c) {
        part[r >> (K - 1)] += (v[r].x * v[r].x + v[r].y * v[r].y) * (R)c;
        v[r].x *= fin;
        v[r].y *= fin;
      };
      if (exchange) each_cut(x, NB, s_inner[1], add);
      else each_cut(x, 8, s_inner[0], add);
    }
    if (!a.store) continue;
    if (exchange) {
#pragma unroll
      for (int r = 0; r < NR; ++r) psi[x | reg_offset<K>(g_low, r)] = v[r];
    } else {
#pragma unroll
      for (int r = 0; r < NR; ++r) psi[x | reg_offset<K>(g_top, r)] = v[r];
    }
  }
  if (!a.last) return;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    for (int off = 16; off > 0; off >>= 1) part[h] += __shfl_xor_sync(0xffffffffu, part[h], off);
    if (lane == 0) s_red[2 * w + h] = (double)part[h];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int i = 0; i < 2 * kSvWideThreads / 32; ++i) sum += s_red[i];
    atomicAdd(&a.acc[0], sum * a.scale->y);
  }
}

// ---- <Z_a Z_b> of every edge in one pass over the state ----------------------
//
// Signed sums of p(x) = |psi_x|^2.  A tile is 2^12 consecutive amplitudes: lanes
// are bits 0..4, a thread's 16 registers bits 5..8, its warp bits 9..11.  A
// thread forms the signed sums of its 16 values over every subset of at most two
// register bits (a pruned Walsh-Hadamard transform); an edge inside the tile
// bits is one of these with the signs of its lane and warp bits, so they are
// accumulated over all tiles and signed once per CTA.  An edge with one end
// above the tile bits needs that end's sign per tile: a tile's 12 one-bit sums
// and its total are left in the first amplitudes of the tile itself (read for
// the last time here; the state is internal), and a second launch adds them up
// per edge.
//
// Probabilities and sums are FP64 for both element types.  GB300's FP64 pipe does two
// operations per clock and SM, and that bounds the kernel at about ten operations per
// amplitude for all edges (it bound the former one at sixteen per amplitude and launch,
// m / 16 launches): n = 21 with 63 edges, depth 3, 654 -> 150 us in all.  (Sums in pairs
// of floats took 113 us, but held 48 bits: 1e-16 rms off the FP64 sums of the same
// state, twice to four times what FP64 is.)
constexpr int kZzBits = 12, kZzThreads = 256;

__device__ __forceinline__ double zprob(double2 v) { return v.x * v.x + v.y * v.y; }

template <typename T>
__global__ void __launch_bounds__(kZzThreads) sv_zz_kernel(T* psi, int n, int m, const int2* edges,
                                                           double* acc) {
  // sums over subsets of register bits: none, {i}, {i, j} (i < j)
  constexpr int kSums = 11;
  __shared__ double s_sum[kSums][kZzThreads];
  __shared__ double s_warp[kZzThreads / 32][10];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint64_t n_tiles = 1ull << (n - kZzBits);
  double total[kSums];
#pragma unroll
  for (int k = 0; k < kSums; ++k) total[k] = 0.0;
  for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    T* at = psi + (tile << kZzBits);
    double p[16];
    {
      T v[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = at[(warp << 9) | (r << 5) | lane];
#pragma unroll
      for (int r = 0; r < 16; ++r) p[r] = zprob(to_d2(v[r]));
    }
    // one[i] = sum of p signed by register bit i, two[] by pairs of bits; each
    // step folds the lowest remaining bit away
    double one[4], two[6];
    int k2 = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int half = 8 >> i;
      double d[8];
#pragma unroll
      for (int r = 0; r < half; ++r) {
        d[r] = p[2 * r] - p[2 * r + 1];
        p[r] = p[2 * r] + p[2 * r + 1];
      }
      // the differences folded further: signed by bit i and by one later bit
      int rest = half;
#pragma unroll
      for (int j = i + 1; j < 4; ++j) {
        double t = d[0] - d[1];
#pragma unroll
        for (int r = 1; r < 4; ++r)
          if (2 * r < rest) t += d[2 * r] - d[2 * r + 1];
        two[k2++] = t;
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (2 * r < rest) d[r] = d[2 * r] + d[2 * r + 1];
        rest >>= 1;
      }
      one[i] = d[0];
    }
    total[0] += p[0];
#pragma unroll
    for (int i = 0; i < 4; ++i) total[1 + i] += one[i];
#pragma unroll
    for (int k = 0; k < 6; ++k) total[5 + k] += two[k];
    // the tile's one-bit sums and total (only edges above the tile bits use
    // them): p[0] over the lanes as a Walsh-Hadamard transform, lane l ending
    // with the sum signed by subset l of the lane bits
    if (n > kZzBits) {
      double w = p[0];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const double o = __shfl_xor_sync(0xffffffffu, w, 1 << q);
        w = ((lane >> q) & 1u) ? o - w : w + o;
#pragma unroll
        for (int i = 0; i < 4; ++i) one[i] += __shfl_xor_sync(0xffffffffu, one[i], 1 << q);
      }
      const int slot = lane == 0 ? 0 : (lane & (lane - 1)) == 0 ? 32 - __clz(lane) : -1;
      __syncthreads();   // every thread has read the tile; s_warp is free
      if (slot >= 0) s_warp[warp][slot] = w;   // total, lane bits 0..4
      if (lane < 4) {
        const double o = lane == 0 ? one[0] : lane == 1 ? one[1] : lane == 2 ? one[2] : one[3];
        s_warp[warp][6 + lane] = o;
      }
      __syncthreads();
      if (threadIdx.x < 13) {
        // 0: total; 1 + a: signed by tile bit a
        const int a = (int)threadIdx.x - 1;
        double s = 0.0;
        for (int u = 0; u < kZzThreads / 32; ++u) {
          const double v = s_warp[u][a < 5 ? a + 1 : a < 9 ? a + 1 : 0];
          s += a >= 9 && ((u >> (a - 9)) & 1) ? -v : v;
        }
        reinterpret_cast<double*>(at)[threadIdx.x] = s;
      }
    }
  }
  // edges inside the tile bits
#pragma unroll
  for (int k = 0; k < kSums; ++k) s_sum[k][threadIdx.x] = total[k];
  __syncthreads();
  for (int e = warp; e < m; e += kZzThreads / 32) {
    const int2 ed = edges[e];
    if (ed.x >= kZzBits || ed.y >= kZzBits) continue;
    const uint32_t mask = (1u << ed.x) | (1u << ed.y), reg = (mask >> 5) & 15u;
    const uint32_t thr = (mask & 31u) | ((mask >> 9) << 5);   // thread index bits in the sign
    int k = 0;
    if (reg) {
      const int i = __ffs(reg) - 1, j = 31 - __clz(reg);
      // {i} -> 1 + i; {i, j}: pairs (0,1) (0,2) (0,3) (1,2) (1,3) (2,3) -> 5..10
      k = i == j ? 1 + i : 5 + (i == 0 ? j - 1 : i == 1 ? j + 1 : 5);
    }
    double s = 0.0;
    for (uint32_t t = lane; t < kZzThreads; t += 32) {
      const double v = s_sum[k][t];
      s += (__popc(t & thr) & 1) ? -v : v;
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) atomicAdd(&acc[1 + e], s);
  }
}

// Edges with an end above the tile bits: one CTA per edge adds the tiles' sums
// with that end's sign (both ends above: the totals).
template <typename T>
__global__ void __launch_bounds__(kZzThreads) sv_zz_tiles_kernel(const T* psi, int n,
                                                                 const int2* edges, double* acc) {
  __shared__ double s_part[kZzThreads / 32];
  const int2 ed = edges[blockIdx.x];
  const int lo = min(ed.x, ed.y), hi = max(ed.x, ed.y);
  if (hi < kZzBits) return;
  const uint64_t n_tiles = 1ull << (n - kZzBits);
  const uint64_t sign = (1ull << (hi - kZzBits)) | (lo >= kZzBits ? 1ull << (lo - kZzBits) : 0ull);
  const int slot = lo >= kZzBits ? 0 : 1 + lo;
  double s = 0.0;
  for (uint64_t t = threadIdx.x; t < n_tiles; t += kZzThreads) {
    const double v = reinterpret_cast<const double*>(psi + (t << kZzBits))[slot];
    s += (__popcll(t & sign) & 1) ? -v : v;
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kZzThreads / 32; ++w) s += s_part[w];
    acc[1 + blockIdx.x] = s;
  }
}

// <Z_a Z_b> for edges [e0, e0 + 16) of a state of fewer than 2^12 amplitudes.
template <typename T>
__global__ void __launch_bounds__(256) sv_edge_kernel(void* psi_v, int n, int m,
                                                      const int2* edges, double* acc, int e0) {
  __shared__ double s_red[16][256 / 32];
  const T* psi = reinterpret_cast<const T*>(psi_v);
  const int ne = min(16, m - e0);
  double sums[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) sums[k] = 0.0;
  int2 ed[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) ed[k] = k < ne ? edges[e0 + k] : make_int2(0, 0);
  const uint64_t total = 1ull << n;
  for (uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total;
       x += (uint64_t)gridDim.x * blockDim.x) {
    const double2 d = to_d2(psi[x]);
    const double pr = d.x * d.x + d.y * d.y;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const uint32_t diff = ((x >> ed[k].x) ^ (x >> ed[k].y)) & 1u;
      sums[k] += diff ? -pr : pr;
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    double v = sums[k];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) s_red[k][warp] = v;
  }
  __syncthreads();
  if (threadIdx.x < ne) {
    double v = 0.0;
    for (int w = 0; w < 256 / 32; ++w) v += s_red[threadIdx.x][w];
    atomicAdd(&acc[1 + e0 + threadIdx.x], v);
  }
}

template <typename T>
static cudaError_t sv_launch_t(void* psi, int n, int m, const uint32_t* adj_dev,
                               const int2* edges_dev, const double* params_dev, int p,
                               const SvTables& tabs, double* acc_dev, int per_edge,
                               cudaStream_t stream, int* launches) {
  int lo[16], len[16], rl[16];
  const int tmax = sv_tile_bits(sizeof(T) == 16 ? 0 : 1);
  int dev = 0, sms = 0;
  cudaError_t aerr = cudaGetDevice(&dev);
  if (aerr == cudaSuccess) aerr = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (aerr != cudaSuccess) return aerr;
  if (sms < 1) sms = 1;
  const int passes = sv_passes(n, tmax, lo, len, rl);
  *launches = 0;
  T* phase = reinterpret_cast<T*>(tabs.scratch);
  T* rot = phase + (size_t)p * (m + 1);
  double2* scale = reinterpret_cast<double2*>(
      (reinterpret_cast<uintptr_t>(rot + p) + 15) & ~static_cast<uintptr_t>(15));
  const int setup_threads = (m + 32) / 32 * 32 + 32;   // m + 1 phases and a warp, at most 576
  sv_setup_kernel<T><<<p, setup_threads, 0, stream>>>(params_dev, n, p, m, phase, rot, scale,
                                                      acc_dev);
  ++*launches;
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  for (int layer = 0; layer < p; ++layer)
    for (int k = 0; k < passes; ++k) {
      SvArgs a{};
      a.psi = psi;
      a.n = n;
      a.m = m;
      a.adj = adj_dev;
      a.phase = phase;
      a.rot = rot;
      a.layer = layer;
      a.lo = lo[k];
      a.len = len[k];
      a.rl = rl[k];
      a.first = layer == 0 && k == 0;
      a.last = layer == p - 1 && k == passes - 1;
      a.wcut = tabs.wcut;
      a.store = !(a.last && !per_edge);
      a.scale = scale;
      a.acc = acc_dev;
      const int tb = k == 0 ? len[k] : rl[k] + len[k];
      const size_t smem = sizeof(T) << tb;
      const unsigned blocks = (unsigned)(1ull << (n - tb));
      if (tb == tmax) {
        // full tiles: 2^K elements per thread in registers (K + 8 = tb); one CTA per
        // resident slot (two per SM), each walking tiles
        constexpr int K = sizeof(T) == 16 ? 4 : 5;
        const unsigned grid = std::min<unsigned>(blocks, 2u * (unsigned)sms);
        auto run = [&](auto kernel) {
          cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
          kernel<<<grid, kSvWideThreads, smem, stream>>>(a);
        };
        if (k == 0) run(sv_wide_kernel<T, K, true>);
        else run(sv_wide_kernel<T, K, false>);
      } else {
        cudaFuncSetAttribute(sv_small_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
        sv_small_kernel<T><<<1, kSvThreads, smem, stream>>>(a);
      }
      ++*launches;
      err = cudaGetLastError();
      if (err != cudaSuccess) return err;
    }
  if (per_edge && n >= kZzBits) {
    const unsigned tiles = (unsigned)(1ull << (n - kZzBits));
    // two CTAs per SM: each thread has 16 loads in flight
    sv_zz_kernel<T><<<std::min<unsigned>(tiles, 2u * (unsigned)sms), kZzThreads, 0, stream>>>(
        reinterpret_cast<T*>(psi), n, m, edges_dev, acc_dev);
    ++*launches;
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    if (n > kZzBits) {
      sv_zz_tiles_kernel<T><<<m, kZzThreads, 0, stream>>>(reinterpret_cast<const T*>(psi), n,
                                                          edges_dev, acc_dev);
      ++*launches;
      err = cudaGetLastError();
      if (err != cudaSuccess) return err;
    }
  } else if (per_edge)
    for (int e0 = 0; e0 < m; e0 += 16) {
      sv_edge_kernel<T><<<1, 256, 0, stream>>>(psi, n, m, edges_dev, acc_dev, e0);
      ++*launches;
      err = cudaGetLastError();
      if (err != cudaSuccess) return err;
    }
  return cudaSuccess;
}

cudaError_t sv_qaoa_launch(int dtype, void* psi, int n, int m, const uint32_t* adj_dev,
                           const int2* edges_dev, const double* params_dev, int p,
                           const SvTables& tabs, double* acc_dev, int per_edge,
                           cudaStream_t stream, int* launches) {
  if (dtype == 0)
    return sv_launch_t<double2>(psi, n, m, adj_dev, edges_dev, params_dev, p, tabs, acc_dev,
                                per_edge, stream, launches);
  return sv_launch_t<float2>(psi, n, m, adj_dev, edges_dev, params_dev, p, tabs, acc_dev,
                             per_edge, stream, launches);
}

}  // namespace qtc
