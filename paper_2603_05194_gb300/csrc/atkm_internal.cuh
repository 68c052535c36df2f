// Internal declarations of the GB300 PCG-ATKM library: complex helpers, the
// batched line-FFT engine, the plan structure and the launchers shared by the
// translation units.  Not part of the public interface (see include/atkm.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/atkm.h"
#include "i64.cuh"

namespace atkm {

// ---------------------------------------------------------------- complex
template <typename R> struct CT;
template <> struct CT<float> { using c = float2; };
template <typename R> using cx = typename CT<R>::c;

template <typename R> __host__ __device__ __forceinline__ cx<R> mk(R a, R b) {
  cx<R> z; z.x = a; z.y = b; return z;
}
// binary64 <-> binary32 conversions on the integer pipe from the IEEE-754 bit
// layouts (the hardware conversion instructions share the slow FP64 pipe on
// this part; each FP32 pass uses these, the hardware or a mix, whichever was
// measured faster for it: see from64 in ops.cuh).  binary64 -> binary32 rounds the 29
// dropped mantissa bits half-up (a mantissa carry moves into the exponent),
// flushes results below the binary32 normal range to signed zero and
// saturates to infinity (a NaN becomes an infinity); binary32 -> binary64 is
// exact for normal numbers and flushes binary32 subnormals to signed zero.
__device__ __forceinline__ float d2f_bits(double d) {
  const unsigned int hi = (unsigned int)__double2hiint(d), lo = (unsigned int)__double2loint(d);
  // the high word with the exponent rebased to binary32: (e32 << 20) | the
  // top 20 mantissa bits; e32 <= 0 flushes, e32 >= 255 saturates (a NaN
  // becomes an infinity)
  int a = (int)(hi & 0x7fffffffu) - 0x38000000;
  const bool tiny = a < 0x00100000;
  a = min(a, 0x0ff00000);
  // (a:lo) + 2^28 rounds the 29 dropped bits half-up; bits 29..60 are the result
  const unsigned int lr = lo + 0x10000000u;
  const unsigned int ar = (unsigned int)a + (lr < lo ? 1u : 0u);
  unsigned int bits = min(__funnelshift_r(lr, ar, 29), 0x7f800000u);
  bits = tiny ? 0u : bits;
  return __uint_as_float(bits | (hi & 0x80000000u));
}
__device__ __forceinline__ double f2d_bits(float f) {
  const unsigned int u = __float_as_uint(f);
  const unsigned int sign = u & 0x80000000u;
  const unsigned int e = (u >> 23) & 0xffu;
  const unsigned int m = u & 0x7fffffu;
  unsigned int hi, lo;
  if (e == 0u) { hi = sign; lo = 0u; }
  else if (e == 255u) { hi = sign | 0x7ff00000u | (m >> 3); lo = (m & 7u) << 29; }
  else { hi = sign | ((e + 896u) << 20) | (m >> 3); lo = (m & 7u) << 29; }
  return __longlong_as_double((long long)(((unsigned long long)hi << 32) | lo));
}
template <typename R> __device__ __forceinline__ R tor(double v);
template <> __device__ __forceinline__ double tor<double>(double v) { return v; }
template <> __device__ __forceinline__ float tor<float>(double v) { return d2f_bits(v); }
template <typename R> __device__ __forceinline__ double tod(R v);
template <> __device__ __forceinline__ double tod<double>(double v) { return v; }
template <> __device__ __forceinline__ double tod<float>(float v) { return f2d_bits(v); }
template <typename R> __device__ __forceinline__ cx<R> add(cx<R> a, cx<R> b) {
  return mk<R>(a.x + b.x, a.y + b.y);
}
template <typename R> __device__ __forceinline__ cx<R> sub(cx<R> a, cx<R> b) {
  return mk<R>(a.x - b.x, a.y - b.y);
}
template <typename R> __device__ __forceinline__ cx<R> scl(cx<R> a, R s) {
  return mk<R>(a.x * s, a.y * s);
}
// a * b
template <typename R> __device__ __forceinline__ cx<R> cmul(cx<R> a, cx<R> b) {
  return mk<R>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
template <typename R> __device__ __forceinline__ cx<R> cmulc(cx<R> a, cx<R> b) {
  return mk<R>(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
// s * i * a  (s = +1 or -1)
template <typename R, int S> __device__ __forceinline__ cx<R> mul_si(cx<R> a) {
  return S > 0 ? mk<R>(-a.y, a.x) : mk<R>(a.y, -a.x);
}

// Number of SMs of the current device, queried once per device ordinal and
// cached; 0 when the query fails (callers then size their grids without it).
inline int device_sm_count() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return 0;
  }
  int v = cache[dev].load(std::memory_order_relaxed);
  if (v > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
    cudaGetLastError();
    return 0;
  }
  cache[dev].store(v, std::memory_order_relaxed);
  return v;
}

// p + i strides, the stride in bytes: one 32 x 32 -> 64 multiply-add
template <typename T> __device__ __forceinline__ T* step(T* p, int i, int stride) {
  return (T*)((const char*)p + (long long)i * stride);
}

// Programmatic dependent launch: a kernel started by launch_pdl may be resident
// before its predecessor in the stream has ended, which hides the launch gap
// (1 to 2 us, as long as a small pass itself).  It calls pdl_trigger() at its
// start (its own successor may be placed as soon as all its CTAs are) and
// pdl_wait() before its first access to memory that an earlier kernel reads or
// writes: the wait ends when the predecessor has completed, which had itself
// waited for its own.  Tables written at plan creation may be read before it.
// Everything else is read by plain loads: a load through the read-only path
// (__ldg, const __restrict__) may be moved ahead of the wait, or find a line
// cached before it.  Kernels that read that way are launched in the ordinary
// way (no wait needed) and may still trigger.  Both calls are without effect
// in an ordinary launch.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ------------------------------------------------------------- FFT engine
// A CTA transforms T lines of length L held in shared memory.  Stockham
// auto-sort formulation (Govindaraju et al., "High performance discrete
// Fourier transforms on graphics processors", SC'08): stage s with radix R
// reads element j + r L/R, applies the twiddle w^{(j mod Ns) r} with
// w = e^{sign 2 pi i/(Ns R)}, does an R-point DFT in registers and writes
// element (j - j mod Ns) R + j mod Ns + r Ns.  All butterflies of a stage are
// read into registers before any is written (one shared buffer).
constexpr int kThreads = 256;      // threads per FFT CTA
constexpr int kMaxElems = 4096;    // complex elements per CTA tile (upper bound)
// 16 complex floats per thread keep a stage's butterflies in registers
// without spilling.
template <typename R> struct TileElems;
template <> struct TileElems<float> { static constexpr int value = 4096; };
constexpr int kMaxStages = 12;
constexpr int kMaxLen = 2048;     // longest (padded) line

struct FftLen {
  int L;
  int nstages;
  int radix[kMaxStages];
  const float2* tw32;  // e^{-2 pi i m / L}, m = 0..L-1
  const float2* tws;   // the same by stage, for the power-of-two register engine (k_fast_twiddles)
};

template <typename R> __host__ __device__ __forceinline__ const cx<R>* tw_table(const FftLen& f);
template <> __host__ __device__ __forceinline__ const float2* tw_table<float>(const FftLen& f) { return f.tw32; }
template <typename R> inline const cx<R>* tw_table_host(const FftLen& f) { return tw_table<R>(f); }

// Exact trigonometric constants of the small DFTs (closed forms in radicals).
#define ATKM_SQRT1_2 0.70710678118654752440084436210485
#define ATKM_SIN60 0.86602540378443864676372317075294
#define ATKM_C72 0.30901699437494742410229341718282    /* cos(2pi/5) = (sqrt5-1)/4 */
#define ATKM_C144 (-0.80901699437494742410229341718282) /* cos(4pi/5) = -(sqrt5+1)/4 */
#define ATKM_S72 0.95105651629515357211643933337938    /* sin(2pi/5) */
#define ATKM_S144 0.58778525229247312916870595463907   /* sin(4pi/5) */

// In-register R-point DFT, X_q = sum_r v_r e^{S 2 pi i r q / R}.
template <typename R, int RAD, int S> struct Dft;

// run: the full DFT.  run_zu: inputs in the upper half are zero (the zero
// padding of a forward transform) and are not read.  run_lo: only outputs in
// the lower half are formed (the crop after an inverse transform); the others
// are left unspecified.
template <typename R, int S> struct Dft<R, 2, S> {
  static __device__ __forceinline__ void run(cx<R>* v) {
    cx<R> a = v[0], b = v[1];
    v[0] = add<R>(a, b); v[1] = sub<R>(a, b);
  }
  static __device__ __forceinline__ void run_lo(cx<R>* v) { v[0] = add<R>(v[0], v[1]); }
};
template <typename R, int S> struct Dft<R, 4, S> {
  static __device__ __forceinline__ void run(cx<R>* v) {
    cx<R> a = add<R>(v[0], v[2]), b = sub<R>(v[0], v[2]);
    cx<R> c = add<R>(v[1], v[3]), d = mul_si<R, S>(sub<R>(v[1], v[3]));
    v[0] = add<R>(a, c); v[2] = sub<R>(a, c);
    v[1] = add<R>(b, d); v[3] = sub<R>(b, d);
  }
  static __device__ __forceinline__ void run_zu(cx<R>* v) {  // v[2] = v[3] = 0
    const cx<R> a = v[0], c = v[1], d = mul_si<R, S>(v[1]);
    v[0] = add<R>(a, c); v[2] = sub<R>(a, c);
    v[1] = add<R>(a, d); v[3] = sub<R>(a, d);
  }
  static __device__ __forceinline__ void run_lo(cx<R>* v) {  // v[0], v[1] only
    cx<R> a = add<R>(v[0], v[2]), b = sub<R>(v[0], v[2]);
    cx<R> c = add<R>(v[1], v[3]), d = mul_si<R, S>(sub<R>(v[1], v[3]));
    v[0] = add<R>(a, c); v[1] = add<R>(b, d);
  }
};
template <typename R, int S> struct Dft<R, 8, S> {
  template <bool ZU, bool LO>
  static __device__ __forceinline__ void go(cx<R>* v) {
    cx<R> e[4] = {v[0], v[2], v[4], v[6]};
    cx<R> o[4] = {v[1], v[3], v[5], v[7]};
    if (ZU) {
      Dft<R, 4, S>::run_zu(e);
      Dft<R, 4, S>::run_zu(o);
    } else {
      Dft<R, 4, S>::run(e);
      Dft<R, 4, S>::run(o);
    }
    const R c = (R)ATKM_SQRT1_2;
    // o_q *= e^{S i pi q / 4}
    cx<R> o1 = mk<R>(c * (o[1].x - S * o[1].y), c * (o[1].y + S * o[1].x));
    cx<R> o2 = mul_si<R, S>(o[2]);
    cx<R> o3 = mk<R>(-c * (o[3].x + S * o[3].y), c * (S * o[3].x - o[3].y));
    v[0] = add<R>(e[0], o[0]);
    v[1] = add<R>(e[1], o1);
    v[2] = add<R>(e[2], o2);
    v[3] = add<R>(e[3], o3);
    if (!LO) {
      v[4] = sub<R>(e[0], o[0]);
      v[5] = sub<R>(e[1], o1);
      v[6] = sub<R>(e[2], o2);
      v[7] = sub<R>(e[3], o3);
    }
  }
  static __device__ __forceinline__ void run(cx<R>* v) { go<false, false>(v); }
  static __device__ __forceinline__ void run_zu(cx<R>* v) { go<true, false>(v); }
  static __device__ __forceinline__ void run_lo(cx<R>* v) { go<false, true>(v); }
};
template <typename R, int S> struct Dft<R, 3, S> {
  static __device__ __forceinline__ void run(cx<R>* v) {
    cx<R> t1 = add<R>(v[1], v[2]);
    cx<R> t2 = mul_si<R, S>(scl<R>(sub<R>(v[1], v[2]), (R)ATKM_SIN60));
    cx<R> m = sub<R>(v[0], scl<R>(t1, (R)0.5));
    v[0] = add<R>(v[0], t1);
    v[1] = add<R>(m, t2);
    v[2] = sub<R>(m, t2);
  }
};
template <typename R, int S> struct Dft<R, 5, S> {
  static __device__ __forceinline__ void run(cx<R>* v) {
    cx<R> a1 = add<R>(v[1], v[4]), b1 = sub<R>(v[1], v[4]);
    cx<R> a2 = add<R>(v[2], v[3]), b2 = sub<R>(v[2], v[3]);
    const R c1 = (R)ATKM_C72, c2 = (R)ATKM_C144, s1 = (R)ATKM_S72, s2 = (R)ATKM_S144;
    cx<R> m1 = mk<R>(v[0].x + c1 * a1.x + c2 * a2.x, v[0].y + c1 * a1.y + c2 * a2.y);
    cx<R> m2 = mk<R>(v[0].x + c2 * a1.x + c1 * a2.x, v[0].y + c2 * a1.y + c1 * a2.y);
    cx<R> n1 = mul_si<R, S>(mk<R>(s1 * b1.x + s2 * b2.x, s1 * b1.y + s2 * b2.y));
    cx<R> n2 = mul_si<R, S>(mk<R>(s2 * b1.x - s1 * b2.x, s2 * b1.y - s1 * b2.y));
    v[0] = mk<R>(v[0].x + a1.x + a2.x, v[0].y + a1.y + a2.y);
    v[1] = add<R>(m1, n1); v[4] = sub<R>(m1, n1);
    v[2] = add<R>(m2, n2); v[3] = sub<R>(m2, n2);
  }
};

// Element (t, j) of the tile: line-major tiles keep lines contiguous (x
// lines), column tiles keep the T columns of one position contiguous.
template <bool LM> __device__ __forceinline__ int tix(int t, int j, int T, int L) {
  return LM ? t * L + j : j * T + t;
}

template <typename R, int RAD, int S, bool LM>
__device__ __forceinline__ void fft_stage(cx<R>* buf, const cx<R>* tw, int L, int T, int Ns) {
  constexpr int NB = (TileElems<R>::value + RAD * kThreads - 1) / (RAD * kThreads);
  const int nb = L / RAD;
  const int total = nb * T;
  const int tws = L / (Ns * RAD);
  cx<R> v[NB][RAD];
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int b = threadIdx.x + i * kThreads;
    if (b < total) {
      int t, j;
      if (LM) { t = b / nb; j = b - t * nb; } else { j = b / T; t = b - j * T; }
#pragma unroll
      for (int r = 0; r < RAD; ++r) v[i][r] = buf[tix<LM>(t, j + r * nb, T, L)];
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int b = threadIdx.x + i * kThreads;
    if (b < total) {
      int t, j;
      if (LM) { t = b / nb; j = b - t * nb; } else { j = b / T; t = b - j * T; }
      const int k = j % Ns;
      if (Ns > 1) {
#pragma unroll
        for (int r = 1; r < RAD; ++r) {
          cx<R> w = tw[k * r * tws];
          v[i][r] = (S < 0) ? cmul<R>(v[i][r], w) : cmulc<R>(v[i][r], w);
        }
      }
      Dft<R, RAD, S>::run(v[i]);
      const int base = (j - k) * RAD + k;
#pragma unroll
      for (int r = 0; r < RAD; ++r) buf[tix<LM>(t, base + r * Ns, T, L)] = v[i][r];
    }
  }
  __syncthreads();
}

// Transforms all T lines of the tile (forward S = -1, inverse S = +1,
// unnormalised).  Caller has synchronised after filling the tile; returns
// synchronised.
template <typename R, int S, bool LM>
__device__ __forceinline__ void fft_tile(cx<R>* buf, const cx<R>* tw, const FftLen& f, int T) {
  int Ns = 1;
  for (int s = 0; s < f.nstages; ++s) {
    const int rad = f.radix[s];
    switch (rad) {
      case 8: fft_stage<R, 8, S, LM>(buf, tw, f.L, T, Ns); break;
      case 4: fft_stage<R, 4, S, LM>(buf, tw, f.L, T, Ns); break;
      case 2: fft_stage<R, 2, S, LM>(buf, tw, f.L, T, Ns); break;
      case 3: fft_stage<R, 3, S, LM>(buf, tw, f.L, T, Ns); break;
      default: fft_stage<R, 5, S, LM>(buf, tw, f.L, T, Ns); break;
    }
    Ns *= rad;
  }
}

// Copies the twiddle table of f into shared memory (no sync).
template <typename R> __device__ __forceinline__ void load_tw(cx<R>* dst, const FftLen& f) {
  const cx<R>* src = tw_table<R>(f);
  for (int i = threadIdx.x; i < f.L; i += kThreads) dst[i] = src[i];
}

// Block-wide sum of NS doubles; thread 0 writes part[s * stride + slot].
template <int NS>
__device__ __forceinline__ void block_reduce_store(double (&acc)[NS], double* part, int stride, int slot) {
  __shared__ double red[NS][kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    double v = acc[s];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[s][warp] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      double v = 0.0;
      for (int w = 0; w < kThreads / 32; ++w) v += red[s][w];
      part[s * stride + slot] = v;
    }
  }
}

// The same for FP32 per-thread partials: the warp stage shuffles and adds in
// FP32 (a 32-term sum, about 5 roundings), each warp's sum is widened once,
// and the block stage adds in FP64 -- so no per-thread FP64 work is done in
// FP32 kernels (the FP64 pipe is slow on this part).
template <int NS>
__device__ __forceinline__ void block_reduce_store_f32(float (&acc)[NS], double* part, int stride, int slot) {
  __shared__ double red[NS][kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    float v = acc[s];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[s][warp] = tod<float>(v);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      double v = 0.0;
      for (int w = 0; w < kThreads / 32; ++w) v += red[s][w];
      part[s * stride + slot] = v;
    }
  }
}

// The last block of a grid to arrive here (every thread of the block calls it;
// `wrote`: the threads that wrote the block's partial results): true in that
// block only, whose threads then see every block's partial results (read them
// with __ldcg).  It leaves *cnt at zero for the next kernel of the stream.  A
// reduction finished this way needs no second launch.  Only the writers fence:
// the block's other stores need not have arrived.
__device__ __forceinline__ bool last_block(unsigned* cnt, bool wrote) {
  __shared__ int last;
  if (wrote) __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned n = gridDim.x * gridDim.y;
    last = atomicAdd(cnt, 1u) == n - 1u;
    if (last) {
      *cnt = 0u;
      __threadfence();
    }
  }
  __syncthreads();
  return last != 0;
}
// Grid sums of the block sums part[s * nblocks + i], s < NS, by one block of
// 256 threads in a fixed order: thread t adds i = t, t + 256, ..., then a tree
// over the threads (pairs 128, 64, 32, ... apart).  All NS sums go through it
// together (one after another they took about 2 us each).
template <int NS> __device__ __forceinline__ void finalize_sums(const double* part, int nblocks, double* out) {
  static_assert(NS <= 8, "one warp a sum");
  __shared__ double fsh[NS][256];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  double acc[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s] = 0.0;
#pragma unroll 2
  for (int i = t; i < nblocks; i += 256) {
#pragma unroll
    for (int s = 0; s < NS; ++s) acc[s] += __ldcg(part + (size_t)s * nblocks + i);
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) fsh[s][t] = acc[s];
  __syncthreads();
#pragma unroll
  for (int w = 128; w > 16; w >>= 1) {
    if (t < w) {
#pragma unroll
      for (int s = 0; s < NS; ++s) fsh[s][t] += fsh[s][t + w];
    }
    __syncthreads();
  }
  if (warp < NS) {
    double v = fsh[warp][lane];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) out[warp] = v;
  }
}
// The same by a block of nw warps, one value a warp.
__device__ __forceinline__ void finalize_sums_warps(const double* part, int nblocks, int ns, double* out, int nw) {
  const int lane = threadIdx.x & 31;
  for (int s = threadIdx.x >> 5; s < ns; s += nw) {
    double acc = 0.0;
#pragma unroll 4
    for (int i = lane; i < nblocks; i += 32) acc += __ldcg(part + (size_t)s * nblocks + i);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) out[s] = acc;
  }
}

// A line length of the integer passes: its stages with the multiplicative
// inverses of their divisors, and the stages' twiddles.  Stage s > 0 of radix R
// after Ns = product of the earlier radices has (R - 1) Ns entries
// e^{-2 pi i k r / (Ns R)} = (c.h, c.l, s.h, s.l) at w[off[s] + (r - 1) Ns + k]
// in units 2^(stage_shift(R) - 64): a thread's R - 1 twiddles lie at fixed
// distances, and those of neighbouring k next to each other.
// wm, wr: the same tables for the orders of the engine k_imix (its list and the
// reversed one), where the length is one of int_radices.
struct IntLen {
  int L, nst, shift;  // shift: the exponent that a transform adds
  int rad[kMaxStages], off[kMaxStages];
  unsigned mns[kMaxStages], mnb[kMaxStages];
  const int4* w;
  const int4* wm;
  const int4* wr;
};

// Per-axis tables of a plan (binary64, length N_a each): nu_k / N_a,
// (nu_k^2 / 2) / N_a, nu_k^2 / 2, and half the square of the coordinate
// -L_a + i h_a.
struct AxT {
  const double* nuN;
  const double* kinN;
  const double* hnu2;
  const double* hxc2;
};

// ---------------------------------------------------------------- plan
struct Geo {
  int Nx, Ny, Nz, Mx, My, Mz;
  int Xh;  // Nx + 1: x-frequencies 0..Nx kept by the real-data ATKM transform
  int XS;  // row stride of the half-spectrum workspaces (Xh rounded up to 16)
  double Lx, Ly, Lz, hx, hy, hz;
};

struct Phys {  // physical parameters passed by value to kernels
  double gx2, gy2, gz2;  // gamma^2
  double beta, lambda, Omega;
};

struct PcgBuffers;  // defined in pcg.cu
struct Profiler;    // defined in plan.cu

// One choice of the FFT-tile autotuner (tune.cu): for the arithmetic r (0
// binary64, 1 FP32, 2 the DF32 form), the line length L and the layout lm (1:
// line-major x pass, 0: strided pass), the engine (mix = 1: in FP32 the
// mixed-radix register engine, in binary64 and the DF32 form the engine of
// compile-time lengths, k_imix; else the arithmetic's generic shared-memory
// engine with its default tile width shifted right by `shift`), with the timed
// operator set's milliseconds under the default rule and under this choice.
struct TuneEntry {
  int r, L, lm, mix, shift;
  double ms_default, ms_best;
};
constexpr int kMaxTune = 48;

}  // namespace atkm

// Scalar slots in plan->scal (device) and their host mirror.
enum {
  SC_ALPHA = 0,
  SC_RED = 8,     // reduction outputs start here
  SC_COUNT = 128
};

struct atkm_plan {
  atkm::Geo g;
  double n[3];
  unsigned flags;
  double hvol;
  atkm::FftLen fN[3];  // unpadded lengths N_x, N_y, N_z
  atkm::FftLen fM[3];  // padded lengths 2N_x, 2N_y, 2N_z
  float2* tw32;        // twiddle pool (by index, then by stage)
  atkm::IntLen iN[3];  // the same lengths for the integer passes
  atkm::IntLen iM[3];
  int4* twi;           // integer twiddle pool
  const int4* tw_x;    // e^{-2 pi i k / Mx}, k < Nx, in units 2^-61 (the real-data post-twist)
  double* U0;          // octant (Nz+1)(Ny+1)(Nx+1)
  float* U0f;          // FP32 copy of U0 (FP32 workspaces only)
  long long* Kz;       // z-pass multiplier K_sym / (2 Mx My Mz), [Mz][My][XS] half spectrum, integers
  int k_midbits, k_midshift;  // scale of the z pass around that multiplier (k_multiplier_half)
  double* axtab;       // per-axis tables (AxT): for a = x, y, z four arrays of N_a doubles
  double* Pw;          // [Nz][Ny][Nx] preconditioner weights, binary64 passes
  atkm::c64* W1;       // [Nz][Ny][XS] half spectrum in x
  atkm::c64* W2;       // [Nz][My][XS]
  atkm::c64* T1;       // [Nz][Ny][Nx]
  atkm::c64* T2;       // [Nz][Ny][Nx], the y part of H; W2 itself where memory is short (share_T2)
  int* ex[5];          // tile exponents of the integer arrays (ATKM and P: 0..2, H: 3, 4)
  float2* W1f;
  float2* W2f;
  float2* T1f;
  double* partials;    // reduction partials
  int partials_cap;    // doubles
  double* scal;        // device scalars
  unsigned* cnt;       // arrival counter of last_block
  double* scal_host;   // pinned mirror
  atkm::PcgBuffers* pcg;
  atkm::TuneEntry tune[atkm::kMaxTune];  // autotuned engine choices (n_tune of them)
  int n_tune;
  atkm::Profiler* prof;  // non-null while profiling is on
  atkm::Profiler* prof_stopped_;  // last record after profiling was switched off
  unsigned long long bytes;
  std::string err;
};

namespace atkm {

// H's y part has a workspace of its own so that H p and the ATKM of Re(conj(phi) p)
// can run side by side.  Where the device has no room for it (16 bytes a point of
// about 130 for a plan, 300 with a solve's vectors) it lies in W2, and the two run
// one after the other.
inline bool T2_shared(const atkm_plan* p) { return p->T2 == p->W2; }
void share_T2(atkm_plan* p);

// Lengths for which a plan's passes and its tuner may take k_imix (the powers of
// two among them on small grids only, see ipass_grid).
inline bool imix_ok(const atkm_plan* p, int L) { return int_radices(L).n > 0 && !(p->flags & ATKM_PLAN_GENERIC_FFT); }

extern thread_local std::string g_last_error;

int fail(atkm_plan* p, int code, const std::string& msg);
int cuda_fail(atkm_plan* p, cudaError_t e, const char* where);
cudaError_t dev_alloc(atkm_plan* p, void** ptr, size_t bytes);

// Process-wide count of kernel launches issued by the library.
void count_launches(int n);

// Profiling hooks: no-ops unless profiling is on.  `name` must be a literal.
void prof_begin(atkm_plan* p, const char* name, double bytes, double flops, cudaStream_t st);
void prof_end(atkm_plan* p, cudaStream_t st);

// Event pair of one pass launch recorded into a captured CUDA graph; every
// replay re-records the same events.  The owner destroys the events.
struct ProfRec {
  const char* name;
  double bytes, flops;
  cudaEvent_t a, b;
};
// While a sink is set, prof_begin/prof_end record into it with fresh events
// (for graph capture) instead of the plan's eager record.
void prof_set_sink(atkm_plan* p, std::vector<ProfRec>* sink);
// Adds the elapsed times of a replayed graph's records to the plan's totals
// (call after the replay has completed).
void prof_accumulate(atkm_plan* p, const std::vector<ProfRec>& recs);

// Launchers of the FP32 passes (passes_impl.cuh).  All enqueue on `st`.
enum AtkmSrc { SRC_RHO = 0, SRC_PSI = 1, SRC_PAIR = 2 };
template <typename R>
cudaError_t launch_atkm(atkm_plan* p, int mode, const double* a, const double* b, double* phi,
                        cudaStream_t st);
// H f; if red_slot >= 0 the energy sums go to scal[red_slot .. red_slot + 9].
template <typename R>
cudaError_t launch_H(atkm_plan* p, const Phys& ph, const double* f, const double* phi,
                     const double* Phi, double* Hf, int red_slot, cudaStream_t st);
template <typename R>
cudaError_t launch_precond(atkm_plan* p, const Phys& ph, const double* alpha_dev, const double* r,
                           const double* phi, const double* Phi, double* Pr, cudaStream_t st);


// Launchers of the binary64 passes (ipasses_*.cu).  dw: called for the
// double-word form (the same arithmetic; the profiler's and the tuner's name).
cudaError_t launch_atkm64(atkm_plan* p, bool dw, int mode, const double* a, const double* b, double* phi,
                          cudaStream_t st);
cudaError_t launch_H64(atkm_plan* p, bool dw, const Phys& ph, const double* f, const double* phi, const double* Phi,
                       double* Hf, int red_slot, cudaStream_t st);
cudaError_t launch_precond64(atkm_plan* p, const Phys& ph, const double* alpha_dev, const double* r, const double* phi,
                             const double* Phi, double* Pr, cudaStream_t st);
// In-place unnormalised 3D complex FFT (sign S) of buf on the plan's grid.
cudaError_t launch_cfft3(atkm_plan* p, double2* buf, int sign, cudaStream_t st);

Phys make_phys(const atkm_params* prm);

}  // namespace atkm
