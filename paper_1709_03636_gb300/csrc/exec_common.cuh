// Device helpers shared by the executors: complex arithmetic, gate tensors,
// execution teams and the bit-map contraction of one op (Eq. 1 with batch
// indices).
#pragma once

#include <cuda_runtime.h>

#include "device_program.h"

namespace qtc {

constexpr int kMaxParams = 64;

__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 acc) {
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(-a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(a.y, b.x, acc.y);
  return acc;
}
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 acc) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
  return acc;
}
template <typename T> __device__ __forceinline__ T czero();
template <> __device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }
template <> __device__ __forceinline__ double2 czero<double2>() { return make_double2(0.0, 0.0); }
template <typename T> __device__ __forceinline__ T from_d2(double2 v);
template <> __device__ __forceinline__ float2 from_d2<float2>(double2 v) {
  return make_float2((float)v.x, (float)v.y);
}
template <> __device__ __forceinline__ double2 from_d2<double2>(double2 v) { return v; }
__device__ __forceinline__ double2 to_d2(float2 v) { return make_double2(v.x, v.y); }
__device__ __forceinline__ double2 to_d2(double2 v) { return v; }

__device__ __forceinline__ void sincos_r(float x, float* s, float* c) { sincosf(x, s, c); }
__device__ __forceinline__ void sincos_r(double x, double* s, double* c) { sincos(x, s, c); }

// Values (and derivatives with respect to params[slot]) of one gate table
// entry, element index bit k = label k (see LeafKind), written straight into
// val and der (der may be null: no derivative wanted).  The angle is formed in
// FP64; sine and cosine are taken in the element precision (FP32 for
// complex64: GB300's FP64 pipe is slow, and the tensor is stored in FP32).
template <typename T>
__device__ inline void gate_tensor(const GateSpec& s, const double* params, T* val, T* der_out) {
  T scratch[16];
  T* der = der_out ? der_out : scratch;
  using R = decltype(T::x);
  const double theta = s.constant + (s.slot >= 0 ? s.coeff * params[s.slot] : 0.0);
  const R dth = s.slot >= 0 ? (R)s.coeff : R(0);  // d theta / d param
  const int rank = leaf_rank_of(s.kind);
  const int n = 1 << rank;
  for (int i = 0; i < n; ++i) {
    val[i] = T{R(0), R(0)};
    der[i] = T{R(0), R(0)};
  }
  const R r = R(0.70710678118654752440);
  const R half = R(0.5);
  R sh, ch;
  sincos_r((R)(0.5 * theta), &sh, &ch);
  switch (s.kind) {
    case LK_ZERO: case LK_PROJ0: val[0].x = R(1); break;
    case LK_PROJ1: val[1].x = R(1); break;
    case LK_PLUS: val[0].x = r; val[1].x = r; break;
    case LK_ZDIAG: val[0].x = R(1); val[1].x = R(-1); break;
    case LK_H:
      for (int i = 0; i < 4; ++i) val[i].x = (i == 3) ? -r : r;
      break;
    case LK_X: case LK_OBS_X: val[2].x = R(1); val[1].x = R(1); break;
    case LK_Y: case LK_OBS_Y:
      val[2].y = R(-1);  // [0][1] = -i  (index out=0 | in=1 << 1)
      val[1].y = R(1);   // [1][0] = +i
      break;
    case LK_Z: case LK_OBS_Z: val[0].x = R(1); val[3].x = R(-1); break;
    case LK_RX:  // cos(t/2) I - i sin(t/2) X, [out, in]
      val[0].x = ch; val[3].x = ch; val[1].y = -sh; val[2].y = -sh;
      der[0].x = -half * sh * dth; der[3].x = -half * sh * dth;
      der[1].y = -half * ch * dth; der[2].y = -half * ch * dth;
      break;
    case LK_RZ: case LK_RZDIAG: {
      // diag(exp(-i t/2), exp(+i t/2)); dense form at [0][0] and [1][1]
      const int i1 = s.kind == LK_RZ ? 3 : 1;
      val[0] = T{ch, -sh};
      val[i1] = T{ch, sh};
      der[0] = T{-half * sh * dth, -half * ch * dth};
      der[i1] = T{-half * sh * dth, half * ch * dth};
      break;
    }
    case LK_ZZDIAG: case LK_ZZ:
      for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b) {
          const R zz = (a == b) ? R(1) : R(-1);  // z_a z_b
          const int idx = s.kind == LK_ZZDIAG ? (a | b << 1) : (a | b << 1 | a << 2 | b << 3);
          val[idx] = T{ch, -zz * sh};  // exp(-i zz t/2)
          // d/dt = -i zz/2 * value
          der[idx] = T{-half * sh * dth, -half * zz * ch * dth};
        }
      break;
    case LK_CNOT:
      for (int c = 0; c < 2; ++c)
        for (int t = 0; t < 2; ++t) val[c | (t ^ c) << 1 | c << 2 | t << 3].x = R(1);
      break;
    case LK_OBS_I: val[0].x = R(1); val[3].x = R(1); break;
    case LK_ONES: val[0].x = R(1); val[1].x = R(1); break;
    case LK_OBS_P0: val[0].x = R(1); break;
    case LK_OBS_P1: val[3].x = R(1); break;
    case LK_CNOTX:  // [t_out, c, t_in]: 1 where t_out = t_in xor c
      for (int i = 0; i < 8; ++i) val[i].x = ((i & 1) == (((i >> 1) ^ (i >> 2)) & 1)) ? R(1) : R(0);
      break;
    case LK_DEPOL: case LK_DEPHASE: case LK_AMPDAMP: {
      // sum_k K[ko][ki] conj(K[bo][bi]) at index ko | bo<<1 | ki<<2 | bi<<3, in
      // closed form (all real): depolarizing (1-s) I(x)I + s/3 (XX* + YY* + ZZ*),
      // dephasing (1-s) I(x)I + s ZZ*, amplitude damping K0 K0* + K1 K1*
      const R st = (R)s.constant;
      for (int i = 0; i < 16; ++i) {
        const int ko = i & 1, bo = (i >> 1) & 1, ki = (i >> 2) & 1, bi = (i >> 3) & 1;
        const bool keep = ko == ki && bo == bi;
        const R zz = (ko ^ bo) ? R(-1) : R(1);   // Z[ko][ko] Z[bo][bo]
        R v = R(0);
        if (s.kind == LK_DEPOL) {
          if (keep) v = (R(1) - st) + st / R(3) * zz;
          else if (ko != ki && bo != bi && ko == bo) v = R(2) * st / R(3);  // XX* + YY*
        } else if (s.kind == LK_DEPHASE) {
          if (keep) v = (R(1) - st) + st * zz;
        } else {
          if (keep) v = (ko ? sqrt(R(1) - st) : R(1)) * (bo ? sqrt(R(1) - st) : R(1));
          else if (ko == 0 && bo == 0 && ki == 1 && bi == 1) v = st;
        }
        val[i].x = v;
      }
      break;
    }
    default:
      break;
  }
  if (s.conj)
    for (int i = 0; i < n; ++i) {
      val[i].y = -val[i].y;
      der[i].y = -der[i].y;
    }
}

// Writes every gate table entry (values, and derivatives for parameterised
// entries) into the table at the start of shared memory; all threads of the
// CTA take part.
template <typename T>
__device__ __forceinline__ void build_gate_table(const GateEntryDev* gates, int n_gates,
                                                 const double* params, T* table,
                                                 const GateEntryDev* inline_gates = nullptr,
                                                 int n_inline = 0) {
  for (int e = threadIdx.x; e < n_gates; e += blockDim.x) {
    const GateEntryDev g = e < n_inline ? inline_gates[e] : gates[e];
    gate_tensor<T>(g.spec, params, table + g.val_off,
                   g.spec.slot >= 0 ? table + g.der_off : nullptr);
  }
}

// Sum of v over aligned groups of `width` lanes (a power of two <= 32); every
// lane of the group receives it.
template <typename T>
__device__ __forceinline__ T warp_csum(T v, uint32_t width) {
  for (uint32_t off = 1; off < width; off <<= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
  }
  return v;
}

// One warp: grad[2 slot], grad[2 slot + 1] += sum_j g[j] * d[j] over cnt
// terms (at most 16 for a leaf), in the element precision.  grad holds one
// network's partial derivatives; the sums over networks are taken in FP64.
template <typename T, typename G>
__device__ __forceinline__ void warp_leaf_dot(const T* g, const T* d, uint32_t cnt,
                                              uint32_t lane, G* grad, uint32_t slot) {
  T acc = czero<T>();
  for (uint32_t j = lane; j < cnt; j += 32) acc = cfma(g[j], d[j], acc);
  acc = warp_csum(acc, cnt < 32 ? cnt : 32u);
  if (lane == 0) {
    grad[2 * slot] += (G)acc.x;
    grad[2 * slot + 1] += (G)acc.y;
  }
}

// Explicit shared-memory accesses on 32-bit shared addresses (the warp
// program loop addresses its operands this way, never through generic
// pointers).  Ordered with respect to barriers and each other.
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint4 lds_u4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
template <typename T> __device__ __forceinline__ T lds_c(uint32_t a);
template <> __device__ __forceinline__ float2 lds_c<float2>(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
template <> __device__ __forceinline__ double2 lds_c<double2>(uint32_t a) {
  double2 v;
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_c(uint32_t a, float2 v) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void sts_c(uint32_t a, double2 v) {
  asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}

// 16-byte asynchronous global -> shared copy (L2 only) and the wait for all
// of this thread's outstanding copies.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Adds one to a counter with acquire-release semantics at GPU scope and
// returns the old value.  Called by one thread after a CTA barrier, it
// publishes the writes of the whole CTA (the barrier orders them before it)
// and, for the CTA that sees the last count, makes every other CTA's
// published writes visible.
__device__ __forceinline__ unsigned atomic_add_acq_rel(unsigned* p, unsigned v) {
  unsigned old;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v)
               : "memory");
  return old;
}

constexpr int kReduceThreads = 128;   // threads of the final reduction

// Final reduction of the last CTA (threads < kReduceThreads take part; all
// threads of the CTA must call it): <C> = sum_e w_e (1 - Re s_e)/2 and
// d<C>/dparam_q = -1/2 sum_e w_e Re ds_e/dparam_q (Section 4.1), in FP64, one
// pass over the per-network rows (stride 2 + 2P: s_e, then ds_e/dparam as
// complex pairs).  out = [<C>, gradient (P), Re s_e per network (N)].
// s_part holds (1 + P) * kReduceThreads / 32 doubles.
__device__ inline void reduce_network_rows(const volatile double* res, const double* weights,
                                           int N, int P, bool qaoa_reduce, double* out,
                                           double* s_part) {
  constexpr int kW = kReduceThreads / 32;
  const int stride = 2 + 2 * P;
  const int nq = 1 + P;
  const int tid = threadIdx.x;
  if (tid < kReduceThreads) {
    for (int q0 = 0; q0 < nq; q0 += 8) {
      double part[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) part[i] = 0.0;
      for (int e = tid; e < N; e += kReduceThreads) {
        const double w = weights[e];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int q = q0 + i;
          if (q == 0)
            part[i] += w * 0.5 * (1.0 - res[(size_t)e * stride]);
          else if (q < nq)
            part[i] += -0.5 * w * res[(size_t)e * stride + 2 + 2 * (q - 1)];
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (q0 + i >= nq) break;
        double v = part[i];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if ((tid & 31) == 0) s_part[(q0 + i) * kW + tid / 32] = v;
      }
    }
    for (int e = tid; e < N; e += kReduceThreads) out[1 + P + e] = res[(size_t)e * stride];
  }
  __syncthreads();
  for (int q = tid; q < nq; q += blockDim.x) {
    double t = 0.0;
    for (int w = 0; w < kW; ++w) t += s_part[q * kW + w];
    out[q] = qaoa_reduce ? t : 0.0;
  }
}

// A team is one warp (small networks, kWarp) or the whole CTA.
template <bool kWarp>
struct Team {
  int tid, size, id;
  __device__ Team() {
    if (kWarp) {
      tid = threadIdx.x & 31;
      size = 32;
      id = threadIdx.x >> 5;
    } else {
      tid = threadIdx.x;
      size = blockDim.x;
      id = 0;
    }
  }
  __device__ __forceinline__ void sync() const {
    if (kWarp)
      __syncwarp();
    else
      __syncthreads();
  }
};

// Element pointer of an op offset: gate table below table_elems, else the
// team's own arena.
template <typename T>
__device__ __forceinline__ T* resolve(uint32_t off, T* table, T* arena, uint32_t table_elems) {
  return off < table_elems ? table + off : arena + (off - table_elems);
}

// v << n, zero for n >= 32 (PTX clamps; an absent label's position is 255).
__device__ __forceinline__ uint32_t shl_clamped(uint32_t v, uint32_t n) {
  uint32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
  return r;
}

// Bit positions of one map of an op (16 bytes) held in registers.
struct BitMap {
  uint32_t w[4];
  __device__ explicit BitMap(const uint8_t* p) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    w[0] = v.x;
    w[1] = v.y;
    w[2] = v.z;
    w[3] = v.w;
  }
  // position of bit i (i known at compile time after unrolling)
  __device__ __forceinline__ uint32_t at(int i) const { return (w[i >> 2] >> (8 * (i & 3))) & 0xffu; }
};

// Deposits bits 0..N-1 of v at the positions of map bits first..first+N-1.
template <int N>
__device__ __forceinline__ uint32_t deposit_bits(const BitMap& m, int first, uint32_t v) {
  uint32_t off = 0;
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (first + i < 16) off |= shl_clamped((v >> i) & 1u, m.at(first + i));
  return off;
}

// Deposit of an arbitrary index from bit `first` up (uniform, rarely more than
// a few bits).
__device__ __forceinline__ uint32_t deposit_from(const uint8_t* pos, int first, uint32_t v) {
  uint32_t off = 0;
  for (int i = first; v; ++i, v >>= 1) off |= shl_clamped(v & 1u, pos[i]);
  return off;
}

// Sums of G outputs over the op's 2^ry summed values, in order of the summed
// index (y_lane: this lane's packed operand offsets of summed value `lane`; the
// values beyond 32 add the high bits' offsets).  All loads of a pass issue
// before its multiply-adds.
template <typename T, int G>
__device__ __forceinline__ void sum_outputs(const SOp& op, const T* a, const T* b,
                                            const uint32_t (&oa)[G], const uint32_t (&ob)[G],
                                            uint32_t y_lane, T (&acc)[G]) {
  constexpr int Y = G == 1 ? 4 : 2;
  const uint32_t ny = 1u << op.ry;
#pragma unroll
  for (int g = 0; g < G; ++g) acc[g] = czero<T>();
  if (ny == 1) {
#pragma unroll
    for (int g = 0; g < G; ++g) acc[g] = cfma(a[oa[g]], b[ob[g]], acc[g]);
    return;
  }
  for (uint32_t y0 = 0; y0 < ny; y0 += 32) {
    const uint32_t ha = y0 ? deposit_from(op.y1, 5, y0 >> 5) : 0u;
    const uint32_t hb = y0 ? deposit_from(op.y2, 5, y0 >> 5) : 0u;
    const uint32_t n = ny - y0 < 32u ? ny - y0 : 32u;   // 2, 4, ..., 32
    for (uint32_t y = 0; y < n; y += Y) {
      T av[Y][G], bv[Y][G];
#pragma unroll
      for (int u = 0; u < Y; ++u) {
        // (two summed values only: the pass of four reads them twice)
        const uint32_t e = __shfl_sync(0xffffffffu, y_lane, (y + u) & (n - 1u));
        const uint32_t ea = (e & 0xffffu) | ha, eb = (e >> 16) | hb;
#pragma unroll
        for (int g = 0; g < G; ++g) {
          av[u][g] = a[oa[g] | ea];
          bv[u][g] = b[ob[g] | eb];
        }
      }
#pragma unroll
      for (int u = 0; u < Y; ++u)
        if (y + u < n) {
#pragma unroll
          for (int g = 0; g < G; ++g) acc[g] = cfma(av[u][g], bv[u][g], acc[g]);
        }
    }
  }
}

// One contraction by 2^kLog threads (the team, or one warp: kLog = 5), thread t
// computing outputs c = t + k 2^kLog, up to four at a time.  The offsets of a
// thread's own index bits and of the lane's summed value are formed once from
// the op's bit maps held in registers; a pass then costs one shuffle per summed
// value and the operands' loads.  Sums run in order of the summed index.  Bound
// by latency: programs are chains of levels of a few small ops.  Against one
// barrier per op with the maps walked bit by bit for every operand element, the
// p=2 n=100 gradient launch on CTA teams went from 495 to 209 us, the dense
// one's graph launch from 1.83 to 1.47 ms.
template <typename T, int kLog>
__device__ __forceinline__ void contract_by(const SOp& op, T* out, const T* a, const T* b,
                                         uint32_t t) {
  const uint32_t nout = 1u << op.rc, lane = t & 31u;
  if ((t & ~31u) >= nout) return;   // whole warps
  const BitMap p1(op.p1), p2(op.p2);
  uint32_t y_lane = 0;
  if (op.ry) {
    const BitMap y1(op.y1), y2(op.y2);
    y_lane = deposit_bits<5>(y1, 0, lane) | deposit_bits<5>(y2, 0, lane) << 16;
  }
  const bool active = t < nout;     // only a warp of fewer than 32 outputs has idle lanes
  const uint32_t a0 = deposit_bits<kLog>(p1, 0, active ? t : 0u);
  const uint32_t b0 = deposit_bits<kLog>(p2, 0, active ? t : 0u);
  const uint32_t nk = op.rc > kLog ? nout >> kLog : 1u;
  if (nk >= 4) {
    const uint32_t k1a = shl_clamped(1u, op.p1[kLog]), k1b = shl_clamped(1u, op.p2[kLog]);
    const uint32_t k2a = shl_clamped(1u, op.p1[kLog + 1]), k2b = shl_clamped(1u, op.p2[kLog + 1]);
    for (uint32_t k = 0; k < nk; k += 4) {
      const uint32_t ha = a0 | deposit_from(op.p1, kLog + 2, k >> 2);
      const uint32_t hb = b0 | deposit_from(op.p2, kLog + 2, k >> 2);
      const uint32_t oa[4] = {ha, ha | k1a, ha | k2a, ha | k1a | k2a};
      const uint32_t ob[4] = {hb, hb | k1b, hb | k2b, hb | k1b | k2b};
      T acc[4];
      sum_outputs<T, 4>(op, a, b, oa, ob, y_lane, acc);
#pragma unroll
      for (int g = 0; g < 4; ++g) out[t + ((k + g) << kLog)] = acc[g];
    }
  } else if (nk == 2) {
    const uint32_t oa[2] = {a0, a0 | shl_clamped(1u, op.p1[kLog])};
    const uint32_t ob[2] = {b0, b0 | shl_clamped(1u, op.p2[kLog])};
    T acc[2];
    sum_outputs<T, 2>(op, a, b, oa, ob, y_lane, acc);
    out[t] = acc[0];
    out[t + (1u << kLog)] = acc[1];
  } else {
    const uint32_t oa[1] = {a0}, ob[1] = {b0};
    T acc[1];
    sum_outputs<T, 1>(op, a, b, oa, ob, y_lane, acc);
    if (active) out[t] = acc[0];
  }
}

// A narrow adjoint op (at most 32 outputs) by one warp: with SOPF_LANES the
// lanes take the summed values lane, lane + 32, ... of each output in turn and
// are added by shuffles (long sums over few outputs); else lane c sums output
// c.  With SOPF_LEAFDOT the outputs are dS/dleaf: their dot with the leaf's
// derivative `der` goes to the gradient slot (one warp owns a slot, so the order
// of its terms is fixed).
template <typename T, typename G>
__device__ __forceinline__ void adjoint_by_warp(const SOp& op, T* out, const T* a, const T* b,
                                             const T* der, G* grad, uint32_t lane) {
  const uint32_t nout = 1u << op.rc, ny = 1u << op.ry;
  const BitMap p1(op.p1), p2(op.p2), y1(op.y1), y2(op.y2);
  T mine = czero<T>();   // output `lane`
  if (op.flags & SOPF_LANES) {
    const uint32_t la = deposit_bits<5>(y1, 0, lane), lb = deposit_bits<5>(y2, 0, lane);
    for (uint32_t c = 0; c < nout; ++c) {
      const uint32_t oa = deposit_bits<5>(p1, 0, c) | la, ob = deposit_bits<5>(p2, 0, c) | lb;
      T acc = czero<T>();
      for (uint32_t y = 0; y < ny; y += 128) {
        T av[4], bv[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
          const uint32_t yy = y + 32 * u < ny ? y + 32 * u : y;
          av[u] = a[oa | deposit_from(op.y1, 5, yy >> 5)];
          bv[u] = b[ob | deposit_from(op.y2, 5, yy >> 5)];
        }
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
          if (y + 32 * u < ny) acc = cfma(av[u], bv[u], acc);
      }
      acc = warp_csum(acc, 32u);
      if (lane == c) mine = acc;
    }
  } else {
    const uint32_t y_lane = deposit_bits<5>(y1, 0, lane) | deposit_bits<5>(y2, 0, lane) << 16;
    const uint32_t c = lane < nout ? lane : 0u;
    const uint32_t oa[1] = {deposit_bits<5>(p1, 0, c)}, ob[1] = {deposit_bits<5>(p2, 0, c)};
    T acc[1];
    sum_outputs<T, 1>(op, a, b, oa, ob, y_lane, acc);
    mine = acc[0];
  }
  if (!(op.flags & SOPF_LEAFDOT)) {
    if (lane < nout) out[lane] = mine;
    return;
  }
  T v = czero<T>();
  if (lane < nout) v = cfma(mine, der[lane], v);
  v = warp_csum(v, 16u);
  if (lane == 0) {
    const uint32_t slot = op.p1[kLeafSlotByte];
    grad[2 * slot] += (G)v.x;
    grad[2 * slot + 1] += (G)v.y;
  }
}

// One staged op of a task, called by the whole team (kLog = log2 of its
// threads); `at` resolves an operand offset, `result` takes the scalar.
template <typename T, int kLog, typename TeamT, typename At, typename G, typename Result>
__device__ __forceinline__ void run_op(const SOp& op, const TeamT& team, const At& at,
                                       const T* table, G* grad, const Result& result) {
  const uint32_t tid = team.tid, lane = tid & 31u;
  const uint4 head = *reinterpret_cast<const uint4*>(&op);
  const uint32_t code = head.x & 15u, flags = head.x >> 24;
  if (!(flags & SOPF_NARROW)) {
    contract_by<T, kLog>(op, at(head.y, flags & SOPF_OUT_GLOBAL), at(head.z, flags & SOPF_IN1_GLOBAL),
                         at(head.w, flags & SOPF_IN2_GLOBAL), tid);
  } else if ((tid >> 5) == ((head.x >> 4) & 15u)) {
    if (code == SOP_CONTRACT) {
      const T* a = at(head.z, flags & SOPF_IN1_GLOBAL);
      const T* b = at(head.w, flags & SOPF_IN2_GLOBAL);
      if (flags & SOPF_LEAFDOT)
        adjoint_by_warp<T>(op, (T*)nullptr, a, b, table + head.y, grad, lane);
      else if (flags & SOPF_LANES)
        adjoint_by_warp<T>(op, at(head.y, flags & SOPF_OUT_GLOBAL), a, b, (const T*)nullptr, grad,
                           lane);
      else
        contract_by<T, 5>(op, at(head.y, flags & SOPF_OUT_GLOBAL), a, b, lane);
    } else if (code == SOP_LEAFGRAD) {
      warp_leaf_dot<T>(at(head.z, 0u), at(head.w, 0u), 1u << op.rc, lane, grad, head.y);
    } else if (lane == 0) {
      if (code == SOP_RESULT) result(*at(head.z, flags & SOPF_IN1_GLOBAL));
      else if (code == SOP_SEED)
        *at(head.y, flags & SOPF_OUT_GLOBAL) = from_d2<T>(make_double2(1.0, 0.0));
    }
  }
  if (flags & SOPF_SYNC) team.sync();
}

// One term of a leaf's dot into its accumulator: in the element type (as the
// networks that run in shared memory alone keep their slots), or in FP64 (the graph
// executor's).
template <typename T>
__device__ __forceinline__ void add_dot(T& sum, T v, T d) {
  sum = cfma(v, d, sum);
}
__device__ __forceinline__ void add_dot(double2& sum, float2 v, float2 d) {
  const float2 t = cfma(v, d, czero<float2>());
  sum.x += (double)t.x;
  sum.y += (double)t.y;
}

// A team's program (see CLane): runs the stream's batches, each copied into one
// half of `stage` while the other half's records run.  `lacc`: accumulators of
// lane leaf dots (n_dots parameters x 32 lanes), or null.  Every record of a
// level ends in the same barrier; the next record's header and this thread's
// lane are read before it, so a level of lanes costs about one round trip
// through shared memory and the barrier (an op run from its record forms its
// offsets first, 100 instructions or so).  The p=2 n=100 gradient launch (250
// networks of about 485 ops in 163 levels): 209 -> 105 us.
template <typename T, int kLog, typename TeamT, typename At, typename A, typename G,
          typename Result>
__device__ __forceinline__ void run_stream(const uint4* src, uint32_t batches, uint4* stage,
                                           uint32_t half, const TeamT& team, const At& at,
                                           T* table, A* lacc, int n_dots, G* grad,
                                           const Result& result) {
  const uint32_t tid = team.tid, lane = tid & 31u, warp = tid >> 5;
  constexpr uint32_t kWarps = 1u << (kLog - 5);
  uint32_t units = batches & 0xffffu, next_units = batches >> 16;
  if (lacc)
    for (int q = (int)warp; q < n_dots; q += (int)kWarps) lacc[q * 32 + lane] = czero<A>();
  for (uint32_t u = tid; u < units; u += 1u << kLog) cp_async16(stage + u, src + u);
  uint4* cur = stage;
  uint4* other = stage + half;
  for (uint32_t head_units = 0; units; head_units = 1) {
    cp_async_wait_all();
    team.sync();
    if (head_units) next_units = cur[0].y;
    src += units;
    for (uint32_t u = tid; u < next_units; u += 1u << kLog) cp_async16(other + u, src + u);
    const uint4* rec = cur + head_units;
    const uint4* end = cur + units;
    uint4 head = rec[0], L = make_uint4(0, 0, 0, 0);
    bool have = (head.x & 15u) == SOP_LANES && tid < head.y;
    if (have) L = rec[1 + tid];
    while (rec < end) {
      if ((head.x & 15u) != SOP_LANES) {
        run_op<T, kLog>(*reinterpret_cast<const SOp*>(rec), team, at, (const T*)table, grad, result);
        rec += kSOpUnits;
        if (rec < end) {
          head = rec[0];
          have = (head.x & 15u) == SOP_LANES && tid < head.y;
          if (have) L = rec[1 + tid];
        }
        continue;
      }
      const uint32_t n = head.y;
      const bool sync = (head.x >> 24) & SOPF_SYNC;
      const uint4* next = rec + 1 + n;
      for (uint32_t i = tid;;) {
        if (have) {
          const uint32_t flags = (L.y >> 16) & 0xffu;
          const T* a = at(L.x >> 16, 0u);
          const T* b = at(L.y & 0xffffu, 0u);
          const uint32_t ya1 = L.z & 0xffffu, yb1 = L.z >> 16;
          const uint32_t ya2 = L.w & 0xffffu, yb2 = L.w >> 16;
          const T a0 = a[0], b0 = b[0], a1 = a[ya1], b1 = b[yb1];
          T acc = cfma(a0, b0, czero<T>());
          if (flags & 3u) acc = cfma(a1, b1, acc);
          if (flags & 2u) {
            const T a2 = a[ya2], b2 = b[yb2], a3 = a[ya1 | ya2], b3 = b[yb1 | yb2];
            acc = cfma(a2, b2, acc);
            acc = cfma(a3, b3, acc);
          }
          if (flags & CLF_STORE) *at(L.x & 0xffffu, 0u) = acc;
          if (flags & CLF_DOT) {
            add_dot(lacc[(L.y >> 24) * 32u + lane], acc, table[L.x & 0xffffu]);
          }
        }
        i += 1u << kLog;
        if ((i & ~31u) >= n) break;   // (uniform in a warp)
        have = i < n;
        if (have) L = rec[1 + i];
      }
      rec = next;
      have = false;
      if (rec < end) {
        head = rec[0];
        have = (head.x & 15u) == SOP_LANES && tid < head.y;
        if (have) L = rec[1 + tid];
      }
      if (sync) team.sync();
    }
    units = next_units;
    uint4* t = cur;
    cur = other;
    other = t;
  }
  team.sync();
  if (lacc) {
    for (int q = (int)warp; q < n_dots; q += (int)kWarps) {
      const A v = warp_csum(lacc[q * 32 + lane], 32u);
      if (lane == 0) {
        grad[2 * q] += (G)v.x;
        grad[2 * q + 1] += (G)v.y;
      }
    }
    team.sync();
  }
}

}  // namespace qtc
