// The binary64 passes of the spectral operators in 64-bit block floating
// point (i64.cuh).  As in ops.cuh a pass is an op (load, spectral step, store,
// fused sums) run by a line-FFT engine, with T adjacent lines per CTA:
//   * k_ifast: power-of-two lengths 16 ... 1024, 8 elements a thread in
//     registers, radix-8 stages (plus one radix-2/4 stage) exchanged through
//     shared memory;
//   * k_imix: the composite lengths of int_radices, one butterfly a thread in
//     every stage;
//   * k_igen: every other {2,3,5}-smooth length up to 2048, radix-8/6/5/4/3/2
//     stages between two shared-memory tiles.
// A pass whose input is binary64 finds its tile's largest exponent (H: each
// line's) and turns the elements into integers; between passes the spectra stay integers in the
// workspaces, each tile (line) with its exponent in a small table, so only the first
// and the last pass of an operator convert.  Between a forward and an inverse
// transform the tile is scaled up again to its actual size.
#pragma once

#include <math.h>

#include <atomic>
#include <type_traits>

#include "atkm_internal.cuh"
#include "i64.cuh"

namespace atkm {

__device__ __forceinline__ int ikfreq(int m, int M) { return m < (M >> 1) ? m : m - M; }

// Exponents of an integer array written by one pass: element (row, col) of
// the array belongs to the tile (row >> rs, col >> cs).
struct ExpTab {
  int* e;
  int rs, cs, nc;
  __device__ __forceinline__ int at_ro(int row, int col) const { return __ldg(step(e + (col >> cs), row >> rs, nc * 4)); }
  __device__ __forceinline__ int at(int row, int col) const { return *step(e + (col >> cs), row >> rs, nc * 4); }
};

constexpr int kInBits = 59;  // components of a transform's input stay below 2^59

// A real multiplier m 2^(ex - 1084): |m| in [2^61, 2^62), to within 2^-22 of it
// at either end; ex = 0 stands for 0, ex = 4095 for infinity and NaN.
struct Mult {
  long long m;
  int ex;
};
__device__ __forceinline__ Mult mult_of(double d) {
  const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
  const long long m = (long long)(((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32 | l) << 9);
  const int ex = (int)((h >> 20) & 0x7ffu);
  return Mult{(int)h < 0 ? -m : m, ex + ((ex + 1) & 0x800)};
}

enum ISrc { kSrcF64 = 0, kSrcInt = 1 };

template <int S1, bool SECOND, int NRED, bool LM, int SRC> struct IOpBase {
  static constexpr int kSign1 = S1;
  static constexpr bool kSecond = SECOND;   // inverse transform after the spectral step
  static constexpr int kRed = NRED;         // fused sums (binary64 per thread)
  static constexpr bool kLM = LM;           // line-major (x) pass
  static constexpr int kSrc = SRC;
  static constexpr bool kMirror = false;    // post-processing needs the frequency L - k
  static constexpr bool kTwin = false;      // the input is formed from the elements k and L - k
  static constexpr bool kZeroUpper = false; // positions >= L/2 of the input are zero
  static constexpr bool kHalfOut = false;   // only positions < L/2 of the output are used
  static constexpr bool kNyqTail = false;   // column pass over columns 0..Nx (see ipass_place)
  static constexpr bool kMul = false;       // the spectral step is mul_tile
  static constexpr bool kLineExp = false;   // (kMul) every line has an exponent of its own, not the tile one
  // launched by launch_pdl, inputs read by plain loads; an op whose loads should
  // be moved ahead of its own stores reads by __ldg and is launched normally
  static constexpr bool kPdl = true;
  static constexpr bool kPre = false;       // the spectral step's 8-byte table entries are prefetched (op.table)
  double* part = nullptr;
  int pstride = 0;
  double* sums_out = nullptr;  // where the last block leaves the grid sums
  unsigned* cnt = nullptr;
  // bits the tile is scaled to before the spectral step, and the exponent
  // that the step adds
  __device__ __forceinline__ int midbits() const { return 62; }
  __device__ __forceinline__ int midshift() const { return 0; }
  struct Acc { int e; };
  __device__ __forceinline__ c64 spectral(int, int, int, c64 v, Acc&, const long long*) const { return v; }
  __device__ __forceinline__ double mline(int, int) const { return 0.0; }
  __device__ __forceinline__ Mult mult(double, int) const { return Mult{1ll << 61, 1023}; }
};

// ------------------------------------------------------------ geometry
// The line (o, x) and first position j of a thread: element r of a thread is
// position j + P r of its line.
struct Line {
  int t, j, o, x;
  bool ok;
};

// The line of a thread with l->t set; true: the CTA has none.
template <class Op> __device__ __forceinline__ bool ipass_place(const Op& op, int T, Line* l) {
  if (Op::kLM) {
    l->o = blockIdx.x * T + l->t;
    l->x = 0;
    l->ok = op.valid(l->o, 0);
    return false;
  }
  l->o = blockIdx.y;
  l->x = blockIdx.x * T + l->t;
  if constexpr (Op::kNyqTail) {
    // Half-spectrum column passes (columns 0..Nx): when T divides Nx the last
    // block column would carry column Nx alone; it takes column Nx of T
    // consecutive rows instead, so that no CTA transforms idle columns.
    if (blockIdx.x == gridDim.x - 1 && op.Nx % T == 0) {
      l->x = op.Nx;
      l->o = blockIdx.y * T + l->t;
      l->ok = l->o < (int)gridDim.y && op.valid(l->o, l->x);
      return blockIdx.y * T >= gridDim.y;
    }
  }
  l->ok = op.valid(l->o, l->x);
  return false;
}
template <class Op> __device__ __forceinline__ bool ipass_line(const Op& op, int T, int P, Line* l) {
  if (Op::kLM) {
    l->t = threadIdx.x / P;
    l->j = threadIdx.x - l->t * P;
  } else {
    l->j = threadIdx.x / T;
    l->t = threadIdx.x - l->j * T;
  }
  return ipass_place(op, T, l);
}

// Scratch of the tile-wide reductions, one slot per use so that no barrier is
// needed between a slot's readers and the next use.
struct TileRedBase {
  unsigned m[4][16];
  int nan[128];
};
template <class Op> struct TileRedT : TileRedBase {
  c64 last[Op::kTwin ? 128 : 1];               // element L of each line (load_twin)
  unsigned line[Op::kLineExp ? 3 : 1][128];    // line_max: size of the input, of the spectrum, of the products
};

// Over a CTA of NW warps.
template <int NW> __device__ __forceinline__ unsigned tile_or(unsigned v, unsigned* slot) {
  v = __reduce_or_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) slot[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned r = 0;
#pragma unroll
  for (int i = 0; i < NW; ++i) r |= slot[i];
  return r;
}
template <int NW> __device__ __forceinline__ unsigned tile_max(unsigned v, unsigned* slot) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) slot[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned r = 0;
#pragma unroll
  for (int i = 0; i < NW; ++i) r = max(r, slot[i]);
  return r;
}
template <int NW> __device__ __forceinline__ int tile_max_s(int v, unsigned* slot) {
  return (int)(tile_max<NW>((unsigned)v ^ 0x80000000u, slot) ^ 0x80000000u);
}

// The same over each line of a tile, into slot[t].  Lanes LO, 2 LO, ... HI apart
// hold elements of the same line; lanes of the group's first LO (column tiles) or
// first one (line-major) write.  All slots are zero on entry (init_lines) and hold
// the maxima after the barrier.
template <int LO, int HI> __device__ __forceinline__ void line_max(unsigned v, unsigned* slot, int t) {
#pragma unroll
  for (int o = HI; o >= LO; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (HI < LO || (threadIdx.x & (2 * HI - LO)) == 0) atomicMax(slot + t, v);
  __syncthreads();
}
// Lane distances of a tile's lines: LM: P consecutive threads a line (grouped
// where P is a power of two); else T lines side by side.
template <bool LM, int T, int P> struct LineLanes {
  static constexpr bool pow2 = LM ? (P & (P - 1)) == 0 : (T & (T - 1)) == 0;
  static constexpr int LO = pow2 ? (LM ? 1 : T) : 32, HI = pow2 && (LM ? P > 1 : T < 32) ? (LM ? (P < 32 ? P / 2 : 16) : 16) : 0;
};
template <class TR> __device__ __forceinline__ void init_lines(TR& tr) {
  for (int i = threadIdx.x; i < 3 * 128; i += blockDim.x) tr.line[0][i] = 0u;
}

__device__ __forceinline__ unsigned dmag(double2 z) {
  return (unsigned)max(__double2hiint(z.x) & 0x7fffffff, __double2hiint(z.y) & 0x7fffffff);
}

// ------------------------------------------------------------ tile loads
// State of a tile: its exponent, whether this thread's line holds a NaN or an
// infinity (its values are then zero here), whether any line of the tile does.
struct Tile {
  int e;
  bool bad, anybad;
};

// The exponent that a tile or line of largest |hi word| M < 0x7ff00000 gets.
template <int B> __device__ __forceinline__ int load_exp(unsigned M) { return (int)(M >> 20) - 1023 - (B - 1); }

// Loads a thread's E elements (guarded by pos < L) as integers of the tile's (of
// the line's with kLineExp) common exponent, components below 2^59 (2^60 when the
// first stage sees a zero upper half, unless the post-twist needs the room).
template <int E, bool FULL, int NW, class LL, class Op, class TR>
__device__ __forceinline__ Tile load_tile(const Op& op, const Line& l, int P, int L, c64 (&v)[E], TR& tr) {
  constexpr int EL = Op::kZeroUpper ? (E + 1) / 2 : E;  // elements that can lie below L/2 (P E >= L)
  const int lim = Op::kZeroUpper ? L / 2 : L;
  constexpr int B = (Op::kZeroUpper && !Op::kMirror) ? kInBits + 1 : kInBits;
  if constexpr (Op::kSrc == kSrcF64) {
    double2 d[EL];
    unsigned m = 0;
#pragma unroll
    for (int r = 0; r < EL; ++r) {
      const int pos = l.j + P * r;
      d[r] = (l.ok && (FULL || pos < lim)) ? op.load(l.o, l.x, pos) : make_double2(0.0, 0.0);
      m = max(m, dmag(d[r]));
    }
    unsigned M;
    bool bad = false, any = false;
    if constexpr (Op::kLineExp) {
      __syncthreads();  // init_lines
      line_max<LL::LO, LL::HI>(m, tr.line[0], l.t);
      M = tr.line[0][l.t];
      if (M >= 0x7ff00000u) {  // the line holds a NaN or an infinity
        bad = true;
        M = 0;
#pragma unroll
        for (int r = 0; r < EL; ++r) d[r] = make_double2(0.0, 0.0);
      }
    } else {
      M = tile_max<NW>(m, tr.m[0]);
      if (M >= 0x7ff00000u) {  // a NaN or an infinity: the lines that hold one are left out of the tile's size
        if (threadIdx.x < 128) tr.nan[threadIdx.x] = 0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < EL; ++r) bad |= dmag(d[r]) >= 0x7ff00000u;
        if (bad) tr.nan[l.t] = 1;
        __syncthreads();
        bad = tr.nan[l.t] != 0;
        any = true;
        m = 0;
#pragma unroll
        for (int r = 0; r < EL; ++r) {
          if (bad) d[r] = make_double2(0.0, 0.0);
          m = max(m, dmag(d[r]));
        }
        M = tile_max<NW>(m, tr.m[1]);
      }
    }
    int ex = (int)(M >> 20);
    // d2i takes zeros and subnormals for 2^-1023: such a tile or line into its range
    // first (with a branch of each thread the potential took 1% more)
    if (__any_sync(0xffffffffu, ex < 64)) {
      const double up = ex < 64 ? 0x1p512 : 1.0;
      ex += ex < 64 ? 512 : 0;
#pragma unroll
      for (int r = 0; r < EL; ++r) d[r].x *= up, d[r].y *= up;
    }
    const int base = 64 - B + ex;
#pragma unroll
    for (int r = 0; r < E; ++r) v[r] = r < EL ? c64{d2i(d[r < EL ? r : 0].x, base), d2i(d[r < EL ? r : 0].y, base)} : cz();
    return Tile{load_exp<B>(M), bad, any};
  } else {
    int ee[EL];
    int em = -0x40000000;
#pragma unroll
    for (int r = 0; r < EL; ++r) {
      const int pos = l.j + P * r;
      const bool in = l.ok && (FULL || pos < lim);
      v[r] = in ? op.load(l.o, l.x, pos) : cz();
      ee[r] = in ? op.lexp(l.o, l.x, pos) : -0x40000000;
      em = max(em, ee[r]);
    }
    em = tile_max_s<NW>(em, tr.m[0]);
    if (em >= kExpNaN / 2) {  // uniform in the CTA
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = cz();
      return Tile{kExpNaN, true, true};
    }
    unsigned m = 0;
#pragma unroll
    for (int r = 0; r < EL; ++r) {
      const int d = min(em - ee[r], 64);
      v[r].x = shr_clamp(v[r].x, d);
      v[r].y = shr_clamp(v[r].y, d);
      m |= mag(v[r]);
    }
    const int sh = B - mag_bits(tile_or<NW>(m, tr.m[1]));
#pragma unroll
    for (int r = 0; r < E; ++r) v[r] = r < EL ? cshift(v[r], sh) : cz();
    return Tile{em - sh, false, false};
  }
}

// The same for an op that forms its input from the elements k and L - k of
// the stored half spectrum (op.combine): loads the elements, and element L
// into *last for the threads of position 0, scaled to 60 bits.
template <int E, bool FULL, int NW, class Op>
__device__ __forceinline__ Tile load_twin(const Op& op, const Line& l, int P, int L, c64 (&v)[E], c64* last, TileRedBase& tr) {
  int ev[E], el = -0x40000000;
  *last = cz();
  if (l.ok && l.j == 0) {
    *last = op.load(l.o, L);
    el = op.lexp(l.o, L);
  }
  int em = el;
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int pos = l.j + P * r;
    const bool in = l.ok && (FULL || pos < L);
    v[r] = in ? op.load(l.o, pos) : cz();
    ev[r] = in ? op.lexp(l.o, pos) : -0x40000000;
    em = max(em, ev[r]);
  }
  em = tile_max_s<NW>(em, tr.m[0]);
  if (em >= kExpNaN / 2) {
#pragma unroll
    for (int r = 0; r < E; ++r) v[r] = cz();
    *last = cz();
    return Tile{kExpNaN, true, true};
  }
  const int dl = min(em - el, 64);
  *last = c64{shr_clamp(last->x, dl), shr_clamp(last->y, dl)};
  unsigned m = mag(*last);
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int d = min(em - ev[r], 64);
    v[r] = c64{shr_clamp(v[r].x, d), shr_clamp(v[r].y, d)};
    m |= mag(v[r]);
  }
  const int sh = 60 - mag_bits(tile_or<NW>(m, tr.m[1]));
  *last = cshift(*last, sh);
#pragma unroll
  for (int r = 0; r < E; ++r) v[r] = cshift(v[r], sh);
  return Tile{em - sh + 3, false, false};  // combine() divides by 8
}

// Scales the tile up to BITS = op.midbits() bits and applies the op's
// spectral step to every element.
template <int E, bool FULL, int NW, class Op>
__device__ __forceinline__ void mid_tile(const Op& op, const Line& l, int P, int L, c64 (&v)[E], int* e,
                                         typename Op::Acc& acc, unsigned* slot, const long long* pre) {
  unsigned m = 0;
#pragma unroll
  for (int r = 0; r < E; ++r) m |= mag(v[r]);
  const int sh = op.midbits() - mag_bits(tile_or<NW>(m, slot));
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int pos = l.j + P * r;
    if (l.ok && (FULL || pos < L)) v[r] = op.spectral(l.o, l.x, pos, cshift(v[r], sh), acc, Op::kPre && pre ? pre + r * (NW * 32) : nullptr);
  }
  *e -= sh;
  acc.e = *e;
  *e += op.midshift();
}

// mul_tile's shift up, from the largest mag of the tile or line, and what it does
// to the exponent: an element of multiplier 2^(ex - 1023) f, f in [1, 2), is held as
// v f 2^61 / 2^64.
__device__ __forceinline__ int mul_shift(unsigned m) { return 62 - mag_bits(m); }
__device__ __forceinline__ void mul_exp(Tile& tl, int sh, int M) {
  tl.e += M - sh + 64 - 1084 - (kInBits - 32);
  if (M >= 4095) {  // an infinite or NaN multiplier (a finite one: at most 2046 + 31)
    tl.e = kExpNaN;
    tl.bad = tl.anybad = true;
  }
}

// The same for an op with real multipliers of any size (kMul; op.mult(c, k), c =
// op.mline(o, x) the line's part, formed once a thread: left to the compiler, H x
// formed it at every element, 3 of its 4 binary64 operations, 86 against 77 us at
// 256x256x64): an element times the mantissa of its multiplier keeps the element's bits, and the products are then aligned to
// the tile's largest one.  (With the multiplier in fixed point, nu^2 / 2 of
// the low frequencies, 2^-18 of the largest at length 1024, would leave the
// product 2^18 fewer units.)
template <int E, bool FULL, int NW, class LL, class Op, class TR>
__device__ __forceinline__ void mul_tile(const Op& op, const Line& l, int P, int L, c64 (&v)[E], Tile& tl,
                                         typename Op::Acc& acc, TR& tr) {
  unsigned m = 0;
#pragma unroll
  for (int r = 0; r < E; ++r) m |= mag(v[r]);
  int sh;
  if constexpr (Op::kLineExp) {
    line_max<LL::LO, LL::HI>(m, tr.line[1], l.t);
    sh = mul_shift(tr.line[1][l.t]);
  } else {
    sh = mul_shift(tile_or<NW>(m, tr.m[2]));
  }
  acc.e = tl.e - sh;
  const double c = op.mline(l.o, l.x);
  int ex[E];
  int eb = -0x40000000;
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int pos = l.j + P * r;
    ex[r] = 0;
    if (l.ok && (FULL || pos < L)) {
      const c64 u = cshift(v[r], sh);
      const Limbs x = limbs(u.x), y = limbs(u.y);
      op.tally(l.o, l.x, pos, x, y, acc);
      const Mult d = op.mult(c, pos);
      ex[r] = d.ex;
      const Limbs w = limbs(d.m);
      v[r] = c64{mul64(x, w), mul64(y, w)};
      eb = max(eb, 32 - __clz((int)mag(v[r])) + ex[r]);  // bits of the aligned product, less 32
    }
  }
  int M;
  if constexpr (Op::kLineExp) {
    line_max<LL::LO, LL::HI>((unsigned)eb ^ 0x80000000u, tr.line[2], l.t);
    M = (int)(tr.line[2][l.t] ^ 0x80000000u);
  } else {
    M = tile_max_s<NW>(eb, tr.m[3]);
  }
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int s = kInBits - 32 - M + ex[r], lf = max(s, 0), rt = min(max(-s, 0), 62);
    v[r].x = shr_rnd((long long)((unsigned long long)v[r].x << lf), rt);
    v[r].y = shr_rnd((long long)((unsigned long long)v[r].y << lf), rt);
  }
  mul_exp(tl, sh, M);
}

// Block sums of the threads' NR values through shared memory (NR NW 256 bytes,
// free of other use), one warp a value: each lane adds NW values and the warp
// shuffles once, 12 binary64 additions a warp and value at 8 warps (a shuffle
// tree in every warp took 40).
template <int NR, int NW>
__device__ __forceinline__ void ireduce_out(double (&acc)[NR], double* sh, double* part, int pstride, double* out,
                                            unsigned* cnt) {
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NR; ++i) sh[i * (NW * 32) + threadIdx.x] = acc[i];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x >> 5; i < NR; i += NW) {
    double v = sh[i * (NW * 32) + lane];
    for (int w = 1; w < NW; ++w) v += sh[i * (NW * 32) + w * 32 + lane];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) part[i * pstride + blockIdx.y * gridDim.x + blockIdx.x] = v;
  }
  if (last_block(cnt, lane == 0)) finalize_sums_warps(part, pstride, NR, out, NW);
}

// ------------------------------------------------------------ k_ifast
// Bound by instruction issue (52-62% of the slots; ALU and integer multiplier
// half busy each; DRAM a quarter or less).  Three CTAs an SM at 80 registers: two
// cost 10-15% (H 318 against 276 us at 256x256x64), four, at 64, gained 2% in the
// forward passes and lost 7% in the inverse ones.  At 256x256x64, against radix-8
// transforms in FP64 instructions (FP64 pipe 88-93% busy): ATKM x, y, z, y, x 246,
// 336, 1063, 357, 238 -> 51, 71, 231, 76, 60 us; H x, y, z 351, 369, 344 -> 84, 85,
// 115 (77, 80, 110 with one exponent a tile); P x, y, z, y, x 298, 168, 336, 168,
// 183 -> 108, 42, 70, 42, 61.
constexpr int kIElems = 2048;  // elements per CTA (256 threads x 8)

template <int L> struct IFast {
  static constexpr int TPL = L / 8;
  static constexpr int T = kIElems / L;
  static constexpr int A = (L >= 512) ? 3 : (L >= 64 ? 2 : 1);  // radix-8 stages
  static constexpr int REM = L / (A == 3 ? 512 : (A == 2 ? 64 : 8));
  static constexpr int SHIFT = 3 * (A - 1) + (REM > 1 ? 2 : 0);  // exponent gained by a transform
  // Shared-memory index of element (t, pos): line-major tiles with one pad
  // element every 8 positions, column tiles [pos][t] with a pad row every 8
  // positions where a row is less than 128 bytes.  Both keep the 16-byte
  // accesses of a quarter warp in distinct banks, and both are affine in the
  // stage's inner index, so that an exchange computes two addresses.
  template <bool LM> static constexpr bool kPad = LM || T < 8;
  template <bool LM> static constexpr int kRow = LM ? 1 : T;  // index step of one position
  template <bool LM> __device__ static __forceinline__ int at(int t, int pos) {
    if (LM) return t * (L + L / 8) + pos + (pos >> 3);
    return (kPad<LM> ? pos + (pos >> 3) : pos) * T + t;
  }
  // index step of n positions, n a multiple of 8 (or less than 8 within an aligned 8)
  template <bool LM> static constexpr int span(int n) { return (kPad<LM> ? n + n / 8 : n) * kRow<LM>; }
  template <bool LM> static constexpr size_t bytes() {
    return (size_t)(kPad<LM> ? kIElems + kIElems / 8 : kIElems) * sizeof(c64);
  }
};

// Transforms the register elements v[r] = line[j + TPL r] in place; on return
// v[r] holds frequency j + TPL r.  The caller's last barrier frees b.  One
// buffer and two barriers an exchange: with two buffers a CTA more per SM
// would not fit.
template <int L, int S, bool LM, bool ZU, bool LO>
__device__ __forceinline__ void ifast_fft(c64 (&v)[8], c64* b, const int4* __restrict__ w, int t, int j) {
  using C = IFast<L>;
  int Ns = 1;
#pragma unroll
  for (int s = 0; s < C::A; ++s) {
    const int k = j & (Ns - 1);
    const bool last = (s == C::A - 1) && (C::REM == 1);
    if (s > 0) {
      const int4* wk = w + (s == 2 ? 56 : 0) + k;  // the tables of the stages before: 7 Ns entries each
      v[0] = crsh<3>(v[0]);
#pragma unroll
      for (int r = 1; r < 8; ++r) v[r] = tmul<S>(v[r], __ldg(wk + (r - 1) * Ns));
    }
    if (ZU && s == 0) IDft<8, S>::template go<true, false>(v);
    else if (LO && last) IDft<8, S>::template go<false, true>(v);
    else IDft<8, S>::template go<false, false>(v);
    if (!last) {
      if (s > 0) __syncthreads();
      c64* p = b + C::template at<LM>(t, (j - k) * 8 + k);
#pragma unroll
      for (int r = 0; r < 8; ++r) p[C::template span<LM>(r * Ns)] = v[r];
      __syncthreads();
      if constexpr (C::TPL >= 8) {
        const c64* q = b + C::template at<LM>(t, j);
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = q[C::template span<LM>(C::TPL * r)];
      } else {
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = b[C::template at<LM>(t, j + C::TPL * r)];
      }
    }
    Ns *= 8;
  }
  if constexpr (C::REM > 1) {
    constexpr int Q = C::REM, M = 8 / C::REM, NsQ = L / Q;
    const int4* wk = w + (C::A == 3 ? 504 : (C::A == 2 ? 56 : 0)) + j;
#pragma unroll
    for (int m = 0; m < M; ++m) {
      c64 u[Q];
      u[0] = crsh<2>(v[m]);
#pragma unroll
      for (int q = 1; q < Q; ++q) u[q] = tmul<S>(v[m + M * q], __ldg(wk + (q - 1) * NsQ + C::TPL * m));
      IDft<Q, S>::template go<false, LO>(u);
#pragma unroll
      for (int q = 0; q < (LO ? Q / 2 : Q); ++q) v[m + M * q] = u[q];
    }
  }
}

__device__ __forceinline__ void icp_async8(void* smem_dst, const void* gsrc) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gsrc) : "memory");
}

template <int L, class Op>
__global__ void __launch_bounds__(kThreads, 3) k_ifast(Op op, const int4* __restrict__ w) {
  using C = IFast<L>;
  extern __shared__ __align__(16) unsigned char ism[];
  __shared__ __align__(16) TileRedT<Op> tr;
  c64* b0 = reinterpret_cast<c64*>(ism);
  // [r][thread]: this thread's table entries
  long long* pre = reinterpret_cast<long long*>(ism + C::template bytes<Op::kLM>()) + threadIdx.x;
  Line l;
  using LL = LineLanes<Op::kLM, C::T, C::TPL>;
  pdl_trigger();
  if (ipass_line(op, C::T, C::TPL, &l)) return;  // the whole CTA
  if constexpr (Op::kLineExp) init_lines(tr);
  if constexpr (Op::kPre) {
    if (l.ok) {
#pragma unroll
      for (int r = 0; r < 8; ++r) icp_async8(pre + r * kThreads, op.table(l.o, l.x, l.j + C::TPL * r));
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  if constexpr (Op::kPdl) pdl_wait();
  c64 v[8];
  Tile tl;
  if constexpr (Op::kTwin) {
    c64 last;
    tl = load_twin<8, true, 8>(op, l, C::TPL, L, v, &last, tr);
#pragma unroll
    for (int r = 0; r < 8; ++r) b0[C::template at<Op::kLM>(l.t, l.j + C::TPL * r)] = v[r];
    if (l.j == 0) tr.last[l.t] = last;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int pos = l.j + C::TPL * r;
      v[r] = op.combine(pos, v[r], pos == 0 ? tr.last[l.t] : b0[C::template at<Op::kLM>(l.t, L - pos)]);
    }
    __syncthreads();
  } else {
    tl = load_tile<8, true, 8, LL>(op, l, C::TPL, L, v, tr);
  }
  typename Op::Acc acc{};
  constexpr bool kLo1 = Op::kHalfOut && !Op::kSecond && !Op::kMirror;
  ifast_fft<L, Op::kSign1, Op::kLM, Op::kZeroUpper, kLo1>(v, b0, w, l.t, l.j);
  tl.e += C::SHIFT;
  if constexpr (Op::kMirror) {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; ++r) b0[C::template at<Op::kLM>(l.t, l.j + C::TPL * r)] = v[r];
    __syncthreads();
    if (l.ok) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int k = l.j + C::TPL * r;
        op.post(l.o, k, v[r], b0[C::template at<Op::kLM>(l.t, (L - k) & (L - 1))]);
      }
    }
  } else {
    if constexpr (Op::kSecond) {
      if constexpr (Op::kPre) asm volatile("cp.async.wait_all;\n" ::: "memory");
      // its barrier also frees b0
      if constexpr (Op::kMul) mul_tile<8, true, 8, LL>(op, l, C::TPL, L, v, tl, acc, tr);
      else mid_tile<8, true, 8>(op, l, C::TPL, L, v, &tl.e, acc, tr.m[2], pre);
      ifast_fft<L, -Op::kSign1, Op::kLM, false, Op::kHalfOut>(v, b0, w, l.t, l.j);
      tl.e += C::SHIFT;
    }
    if (l.ok) {
#pragma unroll
      for (int r = 0; r < (Op::kHalfOut ? 4 : 8); ++r) op.store(l.o, l.x, l.j + C::TPL * r, v[r], tl, acc);
    }
  }
  op.put_exp(l, tl);
  if constexpr (Op::kRed > 0) {
    double a[Op::kRed];
    op.sums(l, acc, tl, a);
    ireduce_out<Op::kRed, 8>(a, reinterpret_cast<double*>(ism), op.part, op.pstride, op.sums_out, op.cnt);
  }
}

// ------------------------------------------------------------ k_igen
constexpr int kGenMax = 2560;  // elements per CTA at most (256 threads x 10)
constexpr int kGenE = 10;

__device__ __forceinline__ int fdiv(int n, unsigned magic, int d) { return d == 1 ? n : (int)__umulhi((unsigned)n, magic); }

// Shared-memory index of element (t, pos): as in IFast, one pad element (a pad
// row where a row is less than 128 bytes) every 8 positions.
struct GenTile {
  int T, tsh, ps, LP;
  __device__ __forceinline__ GenTile(int T, int tsh, int L) : T(T), tsh(tsh), ps(tsh < 3 ? 3 : 31), LP(L + L / 8 + 1) {}
  template <bool LM> __device__ __forceinline__ int at(int t, int pos) const {
    return LM ? t * LP + pos + (pos >> 3) : ((pos + (pos >> ps)) << tsh) + t;
  }
};

template <int RAD, int S, bool LM>
__device__ __forceinline__ void igen_stage(const c64* __restrict__ src, c64* __restrict__ dst, const IntLen& f, int st,
                                           int Ns, const GenTile& g) {
  const int L = f.L, nb = L / RAD, total = nb * g.T;
  const int4* __restrict__ w = f.w + f.off[st];
  for (int b = threadIdx.x; b < total; b += kThreads) {
    int t, j;
    if (LM) {
      t = fdiv(b, f.mnb[st], nb);
      j = b - t * nb;
    } else {
      j = b >> g.tsh;
      t = b - (j << g.tsh);
    }
    const int k = j - fdiv(j, f.mns[st], Ns) * Ns;
    c64 v[RAD];
#pragma unroll
    for (int r = 0; r < RAD; ++r) v[r] = src[g.template at<LM>(t, j + r * nb)];
    if (Ns > 1) {
      v[0] = crsh<stage_shift(RAD)>(v[0]);
#pragma unroll
      for (int r = 1; r < RAD; ++r) v[r] = tmul<S>(v[r], __ldg(w + k + (r - 1) * Ns));
    }
    IDft<RAD, S>::template go<false, false>(v);
    const int base = (j - k) * RAD + k;
#pragma unroll
    for (int r = 0; r < RAD; ++r) dst[g.template at<LM>(t, base + r * Ns)] = v[r];
  }
  __syncthreads();
}

// Transforms the tile in *a (filled, synchronised) through *b; the result is
// in *a on return.
template <int S, bool LM>
__device__ __forceinline__ void igen_fft(c64** a, c64** b, const IntLen& f, const GenTile& g) {
  int Ns = 1;
  for (int s = 0; s < f.nst; ++s) {
    const int rad = f.rad[s];
    switch (rad) {
      case 8: igen_stage<8, S, LM>(*a, *b, f, s, Ns, g); break;
      case 6: igen_stage<6, S, LM>(*a, *b, f, s, Ns, g); break;
      case 5: igen_stage<5, S, LM>(*a, *b, f, s, Ns, g); break;
      case 4: igen_stage<4, S, LM>(*a, *b, f, s, Ns, g); break;
      case 3: igen_stage<3, S, LM>(*a, *b, f, s, Ns, g); break;
      default: igen_stage<2, S, LM>(*a, *b, f, s, Ns, g); break;
    }
    Ns *= rad;
    c64* x = *a;
    *a = *b;
    *b = x;
  }
}

template <class Op> __global__ void __launch_bounds__(kThreads, 2) k_igen(Op op, IntLen f, int T, int tsh) {
  extern __shared__ __align__(16) unsigned char ism[];
  __shared__ __align__(16) TileRedT<Op> tr;
  const int L = f.L, P = kThreads >> tsh;
  c64* a = reinterpret_cast<c64*>(ism);
  const GenTile g(T, tsh, L);
  c64* b = a + T * g.LP;
  Line l;
  using LL = LineLanes<false, 32, 1>;
  pdl_trigger();
  if (ipass_line(op, T, P, &l)) return;  // the whole CTA
  if constexpr (Op::kLineExp) init_lines(tr);
  if constexpr (Op::kPdl) pdl_wait();
  c64 v[kGenE];
  Tile tl;
  if constexpr (Op::kTwin) {
    c64 last;
    tl = load_twin<kGenE, false, 8>(op, l, P, L, v, &last, tr);
#pragma unroll
    for (int r = 0; r < kGenE; ++r) {
      const int pos = l.j + P * r;
      if (pos < L) b[g.template at<Op::kLM>(l.t, pos)] = v[r];
    }
    if (l.j == 0) tr.last[l.t] = last;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kGenE; ++r) {
      const int pos = l.j + P * r;
      if (pos < L) v[r] = op.combine(pos, v[r], pos == 0 ? tr.last[l.t] : b[g.template at<Op::kLM>(l.t, L - pos)]);
    }
  } else {
    tl = load_tile<kGenE, false, 8, LL>(op, l, P, L, v, tr);
  }
  typename Op::Acc acc{};
#pragma unroll
  for (int r = 0; r < kGenE; ++r) {
    const int pos = l.j + P * r;
    if (pos < L) a[g.template at<Op::kLM>(l.t, pos)] = v[r];
  }
  __syncthreads();
  igen_fft<Op::kSign1, Op::kLM>(&a, &b, f, g);
  tl.e += f.shift;
  if constexpr (Op::kMirror) {
    if (l.ok) {
      for (int pos = l.j; pos < L; pos += P)
        op.post(l.o, pos, a[g.template at<true>(l.t, pos)], a[g.template at<true>(l.t, pos == 0 ? 0 : L - pos)]);
    }
  } else {
#pragma unroll
    for (int r = 0; r < kGenE; ++r) {
      const int pos = l.j + P * r;
      v[r] = pos < L ? a[g.template at<Op::kLM>(l.t, pos)] : cz();
    }
    if constexpr (Op::kSecond) {
      // its barrier also frees the tile
      if constexpr (Op::kMul) mul_tile<kGenE, false, 8, LL>(op, l, P, L, v, tl, acc, tr);
      else mid_tile<kGenE, false, 8>(op, l, P, L, v, &tl.e, acc, tr.m[2], nullptr);
#pragma unroll
      for (int r = 0; r < kGenE; ++r) {
        const int pos = l.j + P * r;
        if (pos < L) a[g.template at<Op::kLM>(l.t, pos)] = v[r];
      }
      __syncthreads();
      igen_fft<-Op::kSign1, Op::kLM>(&a, &b, f, g);
      tl.e += f.shift;
#pragma unroll
      for (int r = 0; r < kGenE; ++r) {
        const int pos = l.j + P * r;
        v[r] = pos < L ? a[g.template at<Op::kLM>(l.t, pos)] : cz();
      }
    }
    if (l.ok) {
#pragma unroll
      for (int r = 0; r < (Op::kHalfOut ? kGenE / 2 : kGenE); ++r) {
        const int pos = l.j + P * r;
        if (pos < (Op::kHalfOut ? L / 2 : L)) op.store(l.o, l.x, pos, v[r], tl, acc);
      }
    }
  }
  op.put_exp(l, tl);
  if constexpr (Op::kRed > 0) {
    double s[Op::kRed];
    op.sums(l, acc, tl, s);
    ireduce_out<Op::kRed, 8>(s, reinterpret_cast<double*>(ism), op.part, op.pstride, op.sums_out, op.cnt);
  }
}

// ------------------------------------------------------------ k_imix
// Composite lengths known at compile time (int_radices): radices in ascending
// order, one butterfly a thread in every stage.  A line has M = L / R0 threads;
// in a stage of radix R the first L / R of them work (in a column tile whole
// warps then idle; a line-major tile deals its butterflies out anew each
// stage).  The inputs of the first stage and the outputs of the last one stay
// in registers, and the inverse transform takes the radices in the opposite
// order, so that its first stage finds its inputs in the registers where the
// forward transform left them.  All passes of an ATKM, an H and a P against
// k_igen: 561 -> 351 us at 144x144x36, 656 -> 473 at 160x160x40, 234 -> 151 at
// 96x96x24.  Bound by instruction issue, as k_ifast.
template <int L> struct IMix {
  static constexpr RadList R = int_radices(L);
  static constexpr int n = R.n, R0 = R.r[0], RL = R.r[R.n - 1];
  static constexpr int M = L / R0, ML = L / RL;
  static constexpr int T = imix_tile(L);
  static constexpr int NW = (T * M + 31) / 32;
  static constexpr int LP = L + L / 8 + 1;
  static constexpr int fshift() {
    int v = 0;
    for (int s = 1; s < n; ++s) v += stage_shift(R.r[s]);
    return v;
  }
  static constexpr int rshift() {
    int v = 0;
    for (int s = 0; s < n - 1; ++s) v += stage_shift(R.r[s]);
    return v;
  }
  // one pad element every 8 positions in a line-major tile; a column tile's
  // rows have at least 128 bytes
  template <bool LM> __device__ static __forceinline__ int at(int t, int pos) {
    return LM ? t * LP + pos + (pos >> 3) : pos * T + t;
  }
  template <class Op> static constexpr size_t bytes() {
    const size_t tile = (size_t)T * (Op::kLM ? LP : L) * sizeof(c64), red = (size_t)Op::kRed * NW * 32 * sizeof(double);
    return tile > red ? tile : red;
  }
  // CTAs per SM: 768 threads at up to 85 registers
  static constexpr int kMinB = 768 / (NW * 32) > 0 ? 768 / (NW * 32) : 1;
};

// The (t, j) of a thread in a stage with nb butterflies a line; false: none.
template <int L, bool LM> __device__ __forceinline__ bool imix_map(int nb, int* t, int* j) {
  constexpr int T = IMix<L>::T;
  if (LM) {
    *t = threadIdx.x / nb;
    *j = threadIdx.x - *t * nb;
  } else {
    *j = threadIdx.x / T;
    *t = threadIdx.x - *j * T;
  }
  return threadIdx.x < T * nb;
}

template <int L, int RAD, bool LM> __device__ __forceinline__ void imix_read(c64 (&v)[RAD], const c64* b, int t, int j) {
  constexpr int nb = L / RAD;
  if constexpr (!LM || nb % 8 == 0) {
    const c64* p = b + IMix<L>::template at<LM>(t, j);
#pragma unroll
    for (int r = 0; r < RAD; ++r) v[r] = p[LM ? r * (nb + nb / 8) : r * nb * IMix<L>::T];
  } else {
#pragma unroll
    for (int r = 0; r < RAD; ++r) v[r] = b[IMix<L>::template at<LM>(t, j + r * nb)];
  }
}
template <int L, int RAD, int NS, bool LM> __device__ __forceinline__ void imix_write(const c64 (&v)[RAD], c64* b, int t, int j) {
  const int k = j % NS, base = (j - k) * RAD + k;
#pragma unroll
  for (int r = 0; r < RAD; ++r) b[IMix<L>::template at<LM>(t, base + r * NS)] = v[r];
}

// Stage i > 0 of the order (REV: the opposite order) up to its DFT.
template <int L, int S, bool LM, bool REV, int I> struct IStage {
  using C = IMix<L>;
  static constexpr int rad(int i) { return C::R.r[REV ? C::n - 1 - i : i]; }
  static constexpr int ns(int i) {
    int v = 1;
    for (int q = 0; q < i; ++q) v *= rad(q);
    return v;
  }
  static constexpr int off(int i) {  // of the stage's twiddles
    int o = 0;
    for (int q = 1; q < i; ++q) o += (rad(q) - 1) * ns(q);
    return o;
  }
  static constexpr int RAD = rad(I), NS = ns(I);
  template <bool LO> static __device__ __forceinline__ void go(c64 (&v)[RAD], const c64* b, const int4* __restrict__ w, int t, int j) {
    imix_read<L, RAD, LM>(v, b, t, j);
    const int4* wk = w + off(I) + j % NS;
    v[0] = crsh<stage_shift(RAD)>(v[0]);
#pragma unroll
    for (int r = 1; r < RAD; ++r) v[r] = tmul<S>(v[r], __ldg(wk + (r - 1) * NS));
    IDft<RAD, S>::template go<false, LO>(v);
  }
};
// Stages 1 ... n - 2 in shared memory (entered and left synchronised).
template <int L, int S, bool LM, bool REV, int I> __device__ __forceinline__ void imix_middle(c64* b, const int4* __restrict__ w) {
  using C = IMix<L>;
  if constexpr (I < C::n - 1) {
    using St = IStage<L, S, LM, REV, I>;
    c64 v[St::RAD];
    int t, j;
    const bool on = imix_map<L, LM>(L / St::RAD, &t, &j);
    if (on) St::template go<false>(v, b, w, t, j);
    __syncthreads();
    if (on) imix_write<L, St::RAD, St::NS, LM>(v, b, t, j);
    __syncthreads();
    imix_middle<L, S, LM, REV, I + 1>(b, w);
  }
}

template <int L, class Op>
__global__ void __launch_bounds__(IMix<L>::NW * 32, IMix<L>::kMinB)
k_imix(Op op, const int4* __restrict__ wf, const int4* __restrict__ wr) {
  using C = IMix<L>;
  constexpr bool LM = Op::kLM;
  extern __shared__ __align__(16) unsigned char ism[];
  __shared__ __align__(16) TileRedT<Op> tr;
  c64* b = reinterpret_cast<c64*>(ism);
  // la: this thread's line and elements j + M r; lb: those of the last stage, j + ML r
  Line la, lb;
  const bool ona = imix_map<L, LM>(C::M, &la.t, &la.j), onb = imix_map<L, LM>(C::ML, &lb.t, &lb.j);
  pdl_trigger();
  if (ipass_place(op, C::T, &la)) return;  // the whole CTA
  ipass_place(op, C::T, &lb);
  la.ok = la.ok && ona;
  lb.ok = lb.ok && onb;
  if (!ona) la.t = 0, la.j = 1;
  if (!onb) lb.t = 0, lb.j = 1;
  using LA = LineLanes<LM, C::T, C::M>;
  using LB = LineLanes<LM, C::T, C::ML>;
  if constexpr (Op::kLineExp) init_lines(tr);
  if constexpr (Op::kPdl) pdl_wait();
  c64 v[C::R0];
  Tile tl;
  if constexpr (Op::kTwin) {
    c64 last;
    tl = load_twin<C::R0, true, C::NW>(op, la, C::M, L, v, &last, tr);
    if (ona) {
#pragma unroll
      for (int r = 0; r < C::R0; ++r) b[C::template at<LM>(la.t, la.j + C::M * r)] = v[r];
      if (la.j == 0) tr.last[la.t] = last;
    }
    __syncthreads();
    if (ona) {
#pragma unroll
      for (int r = 0; r < C::R0; ++r) {
        const int pos = la.j + C::M * r;
        v[r] = op.combine(pos, v[r], pos == 0 ? tr.last[la.t] : b[C::template at<LM>(la.t, L - pos)]);
      }
    }
    __syncthreads();
  } else {
    // positions from L / 2 on are zero for kZeroUpper: with an odd radix they begin inside an element's range
    tl = load_tile<C::R0, !Op::kZeroUpper || C::R0 % 2 == 0, C::NW, LA>(op, la, C::M, L, v, tr);
  }
  typename Op::Acc acc{};
  constexpr bool kZU = Op::kZeroUpper && (C::R0 == 4 || C::R0 == 8);
  IDft<C::R0, Op::kSign1>::template go<kZU, false>(v);
  if (ona) imix_write<L, C::R0, 1, LM>(v, b, la.t, la.j);
  __syncthreads();
  imix_middle<L, Op::kSign1, LM, false, 1>(b, wf);
  c64 u[C::RL];
  constexpr bool kLO = Op::kHalfOut && C::RL % 2 == 0;
  if (onb) IStage<L, Op::kSign1, LM, false, C::n - 1>::template go<kLO && !Op::kSecond && !Op::kMirror>(u, b, wf, lb.t, lb.j);
  tl.e += C::fshift();
  Tile tb = tl;  // of the line lb
  if constexpr (Op::kLineExp && LM) {
    const unsigned M = tr.line[0][lb.t];
    tb.bad = M >= 0x7ff00000u;
    tb.e = load_exp<kInBits>(tb.bad ? 0u : M) + C::fshift();
  }
  if constexpr (Op::kMirror) {
    __syncthreads();
    if (onb) {
#pragma unroll
      for (int r = 0; r < C::RL; ++r) b[C::template at<LM>(lb.t, lb.j + C::ML * r)] = u[r];
    }
    __syncthreads();
    if (lb.ok) {
#pragma unroll
      for (int r = 0; r < C::RL; ++r) {
        const int k = lb.j + C::ML * r;
        op.post(lb.o, k, u[r], b[C::template at<LM>(lb.t, k == 0 ? 0 : L - k)]);
      }
    }
  } else if constexpr (Op::kSecond) {
    if (!onb) {
#pragma unroll
      for (int r = 0; r < C::RL; ++r) u[r] = cz();
    }
    // its barriers also free the tile
    if constexpr (Op::kMul) {
      mul_tile<C::RL, true, C::NW, LB>(op, lb, C::ML, L, u, tb, acc, tr);
      // (the threads of la include some that lb leaves idle)
      if constexpr (Op::kLineExp) mul_exp(tl, mul_shift(tr.line[1][la.t]), (int)(tr.line[2][la.t] ^ 0x80000000u));
      else tl = tb;
    } else mid_tile<C::RL, true, C::NW>(op, lb, C::ML, L, u, &tl.e, acc, tr.m[2], nullptr);
    IDft<C::RL, -Op::kSign1>::template go<false, false>(u);
    if (onb) imix_write<L, C::RL, 1, LM>(u, b, lb.t, lb.j);
    __syncthreads();
    imix_middle<L, -Op::kSign1, LM, true, 1>(b, wr);
    if (la.ok) {
      IStage<L, -Op::kSign1, LM, true, C::n - 1>::template go<Op::kHalfOut && C::R0 % 2 == 0>(v, b, wr, la.t, la.j);
      tl.e += C::rshift();
#pragma unroll
      for (int r = 0; r < (Op::kHalfOut ? (C::R0 + 1) / 2 : C::R0); ++r) {
        const int pos = la.j + C::M * r;
        if (!Op::kHalfOut || C::R0 % 2 == 0 || pos < L / 2) op.store(la.o, la.x, pos, v[r], tl, acc);
      }
    }
  } else {
    if (lb.ok) {
#pragma unroll
      for (int r = 0; r < (Op::kHalfOut ? (C::RL + 1) / 2 : C::RL); ++r) {
        const int pos = lb.j + C::ML * r;
        if (!Op::kHalfOut || C::RL % 2 == 0 || pos < L / 2) op.store(lb.o, lb.x, pos, u[r], tl, acc);
      }
    }
  }
  op.put_exp(la, tl);
  if constexpr (Op::kRed > 0) {
    double a[Op::kRed];
    op.sums(lb, acc, tb, a);
    ireduce_out<Op::kRed, C::NW>(a, reinterpret_cast<double*>(ism), op.part, op.pstride, op.sums_out, op.cnt);
  }
}

// ------------------------------------------------------------ dispatch
struct IPassGrid {
  dim3 grid;
  int T, tsh;
  bool fast, mix;
};

inline int ilog2(int v) {
  int s = 0;
  while ((1 << (s + 1)) <= v) ++s;
  return s;
}

// LM passes: `lines` lines; column passes: X columns x `outer` outer indices.
// The tiles of the generic engine are powers of two, narrowed until the pass
// has two CTAs per SM (a column tile not below 8, which keeps its accesses in
// whole 128-byte lines).  An autotuned plan's entry decides instead (the DF32
// form runs these passes too, on the binary64 entries).
inline IPassGrid ipass_grid(const atkm_plan* p, int L, bool LM, long lines, int X, int outer, bool mix = true) {
  IPassGrid pg;
  pg.fast = L >= 16 && L <= 1024 && (L & (L - 1)) == 0;
  const TuneEntry* te = nullptr;
  for (int i = 0; i < p->n_tune; ++i)
    if (p->tune[i].r == 0 && p->tune[i].L == L && p->tune[i].lm == (LM ? 1 : 0)) te = p->tune + i;
  pg.mix = mix && !pg.fast && imix_ok(p, L) && (!te || te->mix);
  // Power-of-two lengths up to 256 where the register engine's CTAs (2048
  // elements, 8 a thread) would not give every SM one: k_imix has half the
  // elements a thread and a CTA, so twice the warps share the work.  All passes
  // of an ATKM, an H and a P: 148 -> 124 us at 64x64x16, 139 -> 119 at 32x32x16;
  // at two CTAs per SM the line would cost 226 -> 243 us at 128x128x32.
  if (pg.fast && mix && int_radices(L).n > 0) {
    const int T = kIElems / L;
    const long ctas = LM ? (lines + T - 1) / T : (long)std::max(X / T, 1) * outer;
    if (ctas < (long)device_sm_count()) {
      pg.fast = false;
      pg.mix = true;
    }
  }
  if (pg.fast) {
    pg.T = kIElems / L;
  } else if (pg.mix) {
    pg.T = imix_tile(L);
  } else {
    int T = 1 << ilog2(std::min(128, std::max(1, kGenMax / L)));
    const long want = 2L * device_sm_count();
    if (LM) {
      while (T > 1 && (lines + T - 1) / T < want) T >>= 1;
    } else {
      while (T > 1 && T / 2 >= X) T >>= 1;
      while (T > 8 && (long)((X + T - 1) / T) * outer < want) T >>= 1;
    }
    if (te && !te->mix) T = std::max(T >> te->shift, 1);
    pg.T = T;
  }
  pg.tsh = ilog2(pg.T);
  pg.grid = LM ? dim3((unsigned)((lines + pg.T - 1) / pg.T), 1, 1) : dim3((X + pg.T - 1) / pg.T, outer, 1);
  return pg;
}

// Dynamic shared memory above the default is opted into once per kernel and
// device; `done` holds one bit per device already prepared.
template <typename K>
inline cudaError_t iprepare(std::atomic<unsigned long long>& done, K kernel, size_t bytes) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_acq_rel);
  return e;
}

template <int L, class Op>
inline cudaError_t launch_ifast(const Op& op, const IntLen& f, const IPassGrid& pg, cudaStream_t st) {
  static std::atomic<unsigned long long> prepared{0};
  constexpr size_t sm = IFast<L>::template bytes<Op::kLM>() + (Op::kPre ? (size_t)8 * 8 * kThreads : 0);
  cudaError_t e = iprepare(prepared, k_ifast<L, Op>, sm);
  if (e != cudaSuccess) return e;
  if constexpr (Op::kPdl) return launch_pdl(k_ifast<L, Op>, pg.grid, kThreads, sm, st, op, f.w);
  k_ifast<L, Op><<<pg.grid, kThreads, sm, st>>>(op, f.w);
  return cudaGetLastError();
}

template <int L, class Op>
inline cudaError_t launch_imix(const Op& op, const IntLen& f, const IPassGrid& pg, cudaStream_t st) {
  static std::atomic<unsigned long long> prepared{0};
  constexpr size_t sm = IMix<L>::template bytes<Op>();
  cudaError_t e = iprepare(prepared, k_imix<L, Op>, sm);
  if (e != cudaSuccess) return e;
  if constexpr (Op::kPdl) return launch_pdl(k_imix<L, Op>, pg.grid, IMix<L>::NW * 32, sm, st, op, f.wm, f.wr);
  k_imix<L, Op><<<pg.grid, IMix<L>::NW * 32, sm, st>>>(op, f.wm, f.wr);
  return cudaGetLastError();
}

template <bool MIX, class Op> inline cudaError_t irun(const Op& op, const IntLen& f, const IPassGrid& pg, cudaStream_t st) {
  if constexpr (MIX) {
    if (pg.mix) switch (f.L) {
#define ATKM_IMIX_CASE(L) \
  case L: return launch_imix<L>(op, f, pg, st);
      ATKM_IMIX_LENGTHS(ATKM_IMIX_CASE)
#undef ATKM_IMIX_CASE
      default: return cudaErrorInvalidValue;
    }
  }
  if (pg.fast) {
    switch (f.L) {
      case 16: return launch_ifast<16>(op, f, pg, st);
      case 32: return launch_ifast<32>(op, f, pg, st);
      case 64: return launch_ifast<64>(op, f, pg, st);
      case 128: return launch_ifast<128>(op, f, pg, st);
      case 256: return launch_ifast<256>(op, f, pg, st);
      case 512: return launch_ifast<512>(op, f, pg, st);
      case 1024: return launch_ifast<1024>(op, f, pg, st);
      default: return cudaErrorInvalidValue;
    }
  }
  static std::atomic<unsigned long long> prepared{0};
  // T (L + L / 8 + 1) elements a buffer, T L <= kGenMax, T <= 128
  constexpr size_t most = (size_t)2 * (kGenMax + kGenMax / 8 + 128) * sizeof(c64);
  cudaError_t e = iprepare(prepared, k_igen<Op>, most);
  if (e != cudaSuccess) return e;
  const size_t sm = std::max((size_t)2 * pg.T * (f.L + f.L / 8 + 1) * sizeof(c64), (size_t)Op::kRed * kThreads * sizeof(double));
  if constexpr (Op::kPdl) return launch_pdl(k_igen<Op>, pg.grid, kThreads, sm, st, op, f, pg.T, pg.tsh);
  k_igen<Op><<<pg.grid, kThreads, sm, st>>>(op, f, pg.T, pg.tsh);
  return cudaGetLastError();
}

// ================================================================ ops
// Writes the tile's exponent (every line of the tile writes the same value).
__device__ __forceinline__ void put_exp_at(const ExpTab& x, int row, int col, const Line& l, int e) {
  if (l.j == 0 && l.ok) x.e[(row >> x.rs) * x.nc + (col >> x.cs)] = e;
}

__device__ __forceinline__ c64 ldc(const c64* p) {
  const longlong2 t = *reinterpret_cast<const longlong2*>(p);
  return c64{t.x, t.y};
}
__device__ __forceinline__ c64 ldc_ro(const c64* p) {
  const longlong2 t = __ldg(reinterpret_cast<const longlong2*>(p));
  return c64{t.x, t.y};
}
__device__ __forceinline__ void stc(c64* p, c64 v) { *reinterpret_cast<longlong2*>(p) = make_longlong2(v.x, v.y); }

// ---- ATKM (twofold-padded grid, real-data form).  The density is real, so
// the x transform of each padded line (length Mx = 2 Nx, upper half zero) is
// a complex FFT of length Nx of z_m = rho_{2m} + i rho_{2m+1} with the exact
// post-twist X_k = (Z_k + conj Z_{Nx-k})/2 - (i/2) e^{-2 pi i k/Mx}
// (Z_k - conj Z_{Nx-k}), k = 0..Nx (Hermitian symmetry gives the rest); the y
// and z passes then run on the Nx + 1 half-spectrum columns only, and the
// inverse x transform rebuilds the real output from that half.  With a real
// density this equals the real part of the full complex convolution once K is
// symmetrised on the padded Nyquist planes (k_multiplier_half).  W1:
// [Nz][Ny][XS], W2: [Nz][My][XS], columns 0..Nx used; W1 and W2 hold 2 X
// (the post-twist's 1/2 sits in the z pass's exponent).
template <int MODE> struct IAtkmXF : IOpBase<-1, false, 0, true, kSrcF64> {
  static constexpr bool kMirror = true;
  static constexpr bool kZeroUpper = true;
  const double* a;
  const double* b;
  c64* W1;
  const int4* wM;
  ExpTab ex;
  int Nx, nl, XS;
  __device__ __forceinline__ double dens(size_t i) const {
    if (MODE == SRC_RHO) return a[i];
    const double2 u = reinterpret_cast<const double2*>(a)[i];
    const double2 w = MODE == SRC_PSI ? u : reinterpret_cast<const double2*>(b)[i];
    return u.x * w.x + u.y * w.y;
  }
  __device__ __forceinline__ bool valid(int o, int) const { return o < nl; }
  __device__ __forceinline__ double2 load(int o, int, int m) const {  // m < Nx / 2
    const size_t i = (size_t)o * Nx + 2 * m;
    return make_double2(dens(i), dens(i + 1));
  }
  // 2 X_k / 8 = (Z_k + conj Z_{Nx-k}) / 8 - i w (Z_k - conj Z_{Nx-k}) / 8.
  // With the zero upper half the moduli stay below 2^61.5 here, so the sums fit.
  __device__ __forceinline__ void post(int o, int k, c64 z, c64 m) const {
    const c64 s = crsh<3>(c64{z.x + m.x, z.y - m.y});
    const c64 d = tmul<-1>(c64{z.x - m.x, z.y + m.y}, __ldg(wM + k));
    stc(W1 + (size_t)o * XS + k, c64{s.x + d.y, s.y - d.x});
    if (k == 0) stc(W1 + (size_t)o * XS + Nx, c64{rsh<2>(z.x - z.y), 0});
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const {
    put_exp_at(ex, l.o, 0, l, t.anybad ? kExpNaN : t.e + 3);
  }
};

// y forward: o = z, x = kx in [0, Nx]; rows y < Ny of W1, zero beyond.
struct IAtkmYF : IOpBase<-1, false, 0, false, kSrcInt> {
  static constexpr bool kZeroUpper = true;
  static constexpr bool kNyqTail = true;
  const c64* W1;
  c64* W2;
  ExpTab in, ex;
  int Nx, Ny, My, XS;
  __device__ __forceinline__ bool valid(int, int x) const { return x <= Nx; }
  __device__ __forceinline__ c64 load(int o, int x, int pos) const { return ldc(step(W1 + (size_t)o * Ny * XS + x, pos, XS * 16)); }
  __device__ __forceinline__ int lexp(int o, int x, int pos) const { return in.at(o * Ny + pos, x); }
  __device__ __forceinline__ void store(int o, int x, int pos, c64 v, const Tile&, Acc&) const {
    stc(step(W2 + (size_t)o * My * XS + x, pos, XS * 16), v);
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const { put_exp_at(ex, l.o, l.x, l, t.e); }
};

// z forward * K_sym * inverse: o = ky, x = kx in [0, Nx]; rows z < Nz.  The
// multiplier is the plan's integer table in the layout of W2 (k_multiplier_half).
struct IAtkmZ : IOpBase<-1, true, 0, false, kSrcInt> {
  static constexpr bool kZeroUpper = true;
  static constexpr bool kHalfOut = true;
  static constexpr bool kNyqTail = true;
  c64* W2;
  const long long* K;
  ExpTab in, ex;
  int Nx, Nz, My, XS, mb, ms;
  __device__ __forceinline__ int midbits() const { return mb; }
  __device__ __forceinline__ int midshift() const { return ms; }
  __device__ __forceinline__ bool valid(int, int x) const { return x <= Nx; }
  __device__ __forceinline__ c64 load(int o, int x, int pos) const { return ldc(step(W2 + (size_t)o * XS + x, pos, My * XS * 16)); }
  __device__ __forceinline__ int lexp(int, int x, int pos) const { return in.at(pos, x); }
  static constexpr bool kPre = true;
  __device__ __forceinline__ const long long* table(int o, int x, int k) const {
    return step(K + (size_t)o * XS + x, k, My * XS * 8);
  }
  // pre: the prefetched entry (null in the generic engine)
  __device__ __forceinline__ c64 spectral(int o, int x, int k, c64 v, Acc&, const long long* pre) const {
    const Limbs m = limbs(pre ? *pre : __ldg(table(o, x, k)));
    return c64{mul64(limbs(v.x), m), mul64(limbs(v.y), m)};
  }
  __device__ __forceinline__ void store(int o, int x, int pos, c64 v, const Tile&, Acc&) const {
    stc(step(W2 + (size_t)o * XS + x, pos, My * XS * 16), v);
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const { put_exp_at(ex, l.o, l.x, l, t.e); }
};

// y inverse: o = z, x = kx in [0, Nx]; output rows y < Ny into W1.
struct IAtkmYI : IOpBase<1, false, 0, false, kSrcInt> {
  static constexpr bool kHalfOut = true;
  static constexpr bool kNyqTail = true;
  const c64* W2;
  c64* W1;
  ExpTab in, ex;
  int Nx, Ny, My, XS;
  __device__ __forceinline__ bool valid(int, int x) const { return x <= Nx; }
  __device__ __forceinline__ c64 load(int o, int x, int pos) const { return ldc(step(W2 + (size_t)o * My * XS + x, pos, XS * 16)); }
  __device__ __forceinline__ int lexp(int, int x, int pos) const { return in.at(pos, x); }
  __device__ __forceinline__ void store(int o, int x, int pos, c64 v, const Tile&, Acc&) const {
    stc(step(W1 + (size_t)o * Ny * XS + x, pos, XS * 16), v);
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const { put_exp_at(ex, l.o, l.x, l, t.e); }
};

// x inverse: Z_k = (X_k + conj X_{Nx-k}) + i e^{2 pi i k/Mx} (X_k - conj
// X_{Nx-k}), k < Nx, then an inverse FFT of length Nx gives z_m = Phi_{2m} +
// i Phi_{2m+1}; kept for 2m < Nx (the crop).
struct IAtkmXI : IOpBase<1, false, 0, true, kSrcInt> {
  static constexpr bool kTwin = true;
  static constexpr bool kHalfOut = true;
  const c64* W1;
  double* phi;
  const int4* wM;
  ExpTab in;
  int Nx, Ny, nl, XS;
  __device__ __forceinline__ bool valid(int o, int) const { return o < nl; }
  __device__ __forceinline__ c64 load(int o, int k) const { return ldc(W1 + (size_t)o * XS + k); }
  __device__ __forceinline__ int lexp(int o, int k) const { return in.at(o / Ny, k); }
  __device__ __forceinline__ c64 combine(int k, c64 a, c64 b) const {  // Z_k / 8
    const c64 s = crsh<3>(c64{a.x + b.x, a.y - b.y});
    const c64 d = tmul<1>(c64{a.x - b.x, a.y + b.y}, __ldg(wM + k));
    return c64{s.x - d.y, s.y + d.x};
  }
  __device__ __forceinline__ void store(int o, int, int m, c64 v, const Tile& t, Acc&) const {
    double2 d;
    if (i2d_ok(t.e)) d = make_double2(i2d(v.x, t.e + 1085), i2d(v.y, t.e + 1085));
    else d = make_double2(i2d_any(v.x, t.e), i2d_any(v.y, t.e));
    *reinterpret_cast<double2*>(phi + (size_t)o * Nx + 2 * m) = d;
  }
  __device__ __forceinline__ void put_exp(const Line&, const Tile&) const {}
};

// ---- H_phi f (unpadded grid).  A line's multiplier is (nu_k^2 / 2 + c nu_k) / N
// with c = Omega y on x lines, -Omega x on y lines, from the axis's tables.
// H f at a point depends on its three lines only, so every line has its own
// exponent (kLineExp): a quiet line beside a loud one keeps its 59 bits.  The
// passes of the other operators mix all three axes, so that their error follows
// the loudest line in any arithmetic, and one exponent a tile is enough.
// Sums of k^2 |v|^2 and k |v|^2 over a thread's elements, exact but for the
// last step: |v|^2 / 2^64 = A + F 2^-31 (v below 2^62 a component; the 31
// fraction bits matter because k^2 reaches 2^18 where |v|^2 is small), each
// of A's two limbs and F multiplied by the integer k or k^2 and summed in 64
// bits.
struct KinAcc {
  int e;  // exponent of v
  long long h2, l2, f2, h1, l1, f1;
  __device__ __forceinline__ void add(int k, Limbs x, Limbs y) {
    const unsigned long long ll = (unsigned long long)mulw(x.l, x.l) + (unsigned long long)mulw(y.l, y.l);
    const long long t = mulw(x.h, x.l) + mulw(y.h, y.l) + (long long)((unsigned)(ll >> 32) >> 1);
    const Limbs a = limbs((t >> 31) + mulw(x.h, x.h) + mulw(y.h, y.h));
    const int f = (int)t & 0x7fffffff, kk = k * k;
    h2 += mulw(kk, a.h);
    l2 += mulw(kk, a.l);
    f2 += mulw(kk, f);
    h1 += mulw(k, a.h);
    l1 += mulw(k, a.l);
    f1 += mulw(k, f);
  }
  // the sums of k^2 |v|^2 and k |v|^2 in binary64
  __device__ __forceinline__ double2 get() const {
    const double s = pow2d(2 * e + 64), q = 4.656612873077392578125e-10;  // 2^-31
    const double a = fma((double)h2, 4294967296.0, (double)l2) + (double)f2 * q;
    const double b = fma((double)h1, 4294967296.0, (double)l1) + (double)f1 * q;
    if (2 * e + 64 < -1022) {  // v below 2^-480: the scale alone is no normal value, the sums may be
      const double t = pow2d(e + 32);
      return make_double2(a * t * t, b * t * t);
    }
    return make_double2(a * s, b * s);
  }
};

// Marks an element of a line that holds a NaN or an infinity.
constexpr long long kBadElem = (long long)0x8000000000000000ull;

template <bool RED> struct IHX : IOpBase<-1, true, RED ? 2 : 0, true, kSrcF64> {
  const double2* f;
  c64* A;
  ExpTab ex;
  const double* kin;  // (nu_k^2 / 2) / N
  const double* nu;   // nu_k / N
  int Nx, Ny, nl;
  double Om, Ly, hy;
  double ck, cr;       // nu^2 / (2 N) = ck k'^2, Omega nu / N = cr k', k' the signed index
  static constexpr bool kMul = true, kLineExp = true;
  struct Acc : KinAcc {};
  __device__ __forceinline__ bool valid(int o, int) const { return o < nl; }
  __device__ __forceinline__ double yc(int o) const { return -Ly + (double)(o % Ny) * hy; }
  __device__ __forceinline__ double2 load(int o, int, int pos) const { return f[(size_t)o * Nx + pos]; }
  __device__ __forceinline__ void tally(int, int, int k, Limbs x, Limbs y, Acc& a) const {
    if (RED) a.add(ikfreq(k, Nx), x, y);
  }
  __device__ __forceinline__ double mline(int o, int) const { return Om * yc(o); }
  __device__ __forceinline__ Mult mult(double c, int k) const { return mult_of(fma(c, __ldg(nu + k), __ldg(kin + k))); }
  __device__ __forceinline__ void store(int o, int, int pos, c64 v, const Tile& t, Acc&) const {
    if (t.bad) v.x = kBadElem;
    stc(A + (size_t)o * Nx + pos, v);
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const { put_exp_at(ex, l.o, 0, l, t.e); }
  __device__ __forceinline__ void sums(const Line& l, const Acc& a, const Tile& t, double* s) const {
    const double2 k = a.get();
    s[0] = l.ok ? ck * k.x : 0.0;
    s[1] = l.ok ? cr * yc(l.o) * k.y : 0.0;
    if (t.bad) s[0] = s[1] = __longlong_as_double(0x7ff8000000000000ll);
  }
};

template <bool RED> struct IHY : IOpBase<-1, true, RED ? 2 : 0, false, kSrcF64> {
  const double2* f;
  c64* A;
  ExpTab ex;
  const double* kin;
  const double* nu;
  int Nx, Ny;
  double Om, Lx, hx;
  double ck, cr;
  static constexpr bool kMul = true, kLineExp = true;
  struct Acc : KinAcc {};
  __device__ __forceinline__ bool valid(int, int x) const { return x < Nx; }
  __device__ __forceinline__ double xc(int x) const { return -Lx + (double)x * hx; }
  __device__ __forceinline__ double2 load(int o, int x, int pos) const { return *step(f + (size_t)o * Ny * Nx + x, pos, Nx * 16); }
  __device__ __forceinline__ void tally(int, int, int k, Limbs p, Limbs q, Acc& a) const {
    if (RED) a.add(ikfreq(k, Ny), p, q);
  }
  __device__ __forceinline__ double mline(int, int x) const { return -Om * xc(x); }
  __device__ __forceinline__ Mult mult(double c, int k) const { return mult_of(fma(c, __ldg(nu + k), __ldg(kin + k))); }
  __device__ __forceinline__ void store(int o, int x, int pos, c64 v, const Tile& t, Acc&) const {
    if (t.bad) v.x = kBadElem;
    stc(step(A + (size_t)o * Ny * Nx + x, pos, Nx * 16), v);
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const { put_exp_at(ex, l.o, l.x, l, t.e); }
  __device__ __forceinline__ void sums(const Line& l, const Acc& a, const Tile& t, double* s) const {
    const double2 k = a.get();
    s[0] = l.ok ? ck * k.x : 0.0;
    s[1] = l.ok ? cr * xc(l.x) * k.y : 0.0;
    if (t.bad) s[0] = s[1] = __longlong_as_double(0x7ff8000000000000ll);
  }
};

// z: multiplier nu^2/2 on lines (o = y, x), then Hf = x part + y part + z part
// + (V + beta |phi|^2 + lambda Phi) f, the last term in binary64.
// RED (f = phi) sums: kin_z, V|f|^2, |f|^4, Phi |f|^2, Re(Hf conj f), |f|^2; the
// fifth is the sum of all kinetic and rotation sums, the second, beta times the
// third and lambda times the fourth, which spares two of the 13 binary64 operations
// a point that bound this pass.
template <bool RED> struct IHZ : IOpBase<-1, true, RED ? 6 : 0, false, kSrcF64> {
  const double2* f;
  const double2* phi;
  const double* Phi;
  const c64* AX;
  const c64* AY;
  ExpTab ix, iy;
  double2* Hf;
  const double* kin;
  int Nx, Ny, Nz;
  const double* hx2;  // x_i^2 / 2 of each axis
  const double* hy2;
  const double* hz2;
  double gx2, gy2, gz2, beta, lambda, ck;
  bool same;  // f == phi: phi is not read a second time
  static constexpr bool kMul = true, kLineExp = true;
  static constexpr bool kPdl = false;
  struct Acc : KinAcc {
    double s[4];
  };
  __device__ __forceinline__ bool valid(int, int x) const { return x < Nx; }
  __device__ __forceinline__ double2 load(int o, int x, int pos) const { return *step(f + (size_t)o * Nx + x, pos, Ny * Nx * 16); }
  __device__ __forceinline__ void tally(int, int, int k, Limbs p, Limbs q, Acc& a) const {
    if (RED) a.add(ikfreq(k, Nz), p, q);
  }
  __device__ __forceinline__ Mult mult(double, int k) const { return mult_of(__ldg(kin + k)); }
  __device__ __forceinline__ void store(int o, int x, int pos, c64 v, const Tile& t, Acc& a) const {
    const size_t i0 = (size_t)o * Nx + x;
    const int pl = Ny * Nx;
    const double2 fv = __ldg(step(f + i0, pos, pl * 16));
    const double Pd = __ldg(step(Phi + i0, pos, pl * 8));
    const c64 u = ldc_ro(step(AX + i0, pos, pl * 16)), w = ldc_ro(step(AY + i0, pos, pl * 16));
    const bool bad = t.bad || u.x == kBadElem || w.x == kBadElem;
    const int eu = ix.at_ro(pos * Ny + o, 0), ew = iy.at_ro(pos, x);
    const int e = max(t.e, max(eu, ew)) + 2;  // room for the sum of three
    const int dv = min(e - t.e, 64), du = min(e - eu, 64), dw = min(e - ew, 64);
    const long long sx = shr_clamp(v.x, dv) + shr_clamp(u.x, du) + shr_clamp(w.x, dw);
    const long long sy = shr_clamp(v.y, dv) + shr_clamp(u.y, du) + shr_clamp(w.y, dw);
    double2 kin;
    if (bad) kin.x = kin.y = __longlong_as_double(0x7ff8000000000000ll);
    else if (i2d_ok(e)) kin = make_double2(i2d(sx, e + 1085), i2d(sy, e + 1085));
    else kin = make_double2(i2d_any(sx, e), i2d_any(sy, e));
    const double V = gz2 * hz2[pos] + (gy2 * hy2[o] + gx2 * hx2[x]);
    const double2 pv = RED || same ? fv : __ldg(step(phi + i0, pos, pl * 16));
    const double f2 = pv.x * pv.x + pv.y * pv.y;
    const double wt = V + beta * f2 + lambda * Pd;
    const double ox = kin.x + wt * fv.x, oy = kin.y + wt * fv.y;
    *step(Hf + i0, pos, pl * 16) = make_double2(ox, oy);
    if (RED) {
      a.s[0] += V * f2;
      a.s[1] += f2 * f2;
      a.s[2] += Pd * f2;
      a.s[3] += f2;
    }
  }
  __device__ __forceinline__ void put_exp(const Line&, const Tile&) const {}
  __device__ __forceinline__ void sums(const Line& l, const Acc& a, const Tile& t, double* s) const {
    s[0] = l.ok ? ck * a.get().x : 0.0;
    if (t.bad) s[0] = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
    for (int i = 0; i < 3; ++i) s[1 + i] = a.s[i];
    s[4] = s[0] + fma(lambda, a.s[2], fma(beta, a.s[1], a.s[0]));
    // the sums of the x and y passes lie before this pass's
    if (blockIdx.x + blockIdx.y + threadIdx.x == 0)
      s[4] += (this->sums_out[-4] + this->sums_out[-2]) + (this->sums_out[-3] + this->sums_out[-1]);
    s[5] = a.s[3];
  }
};

// 1 / v and 1 / sqrt(v) as mantissa and exponent: the binary32 estimate y and one
// correction step in integers, off the FP64 pipe (2 operations a clock and SM
// against 64 integer products; the binary64 steps took 4 and 5 operations).  The
// residual e = 1 - v y (|e| < 2^-22), 1 - v y^2 (|e| < 2^-20) is exact to 2^-62,
// so the results are good to 2^-55.  Outside the estimate's range the library's.
__device__ __forceinline__ bool f32_range(double v) {
  return (unsigned)(__double2hiint(v) - 0x39000000) < 0x0e000000u;  // 2^-111 <= v < 2^113
}
// y (1 + f 2^-56), y's mantissa my in [2^23, 2^24), its biased exponent ey
__device__ __forceinline__ Mult mult_corr(unsigned my, int ey, long long f) {
  return Mult{(long long)((unsigned long long)my << 38) + (((long long)my * f) >> 18), ey - 127 + 1023};
}
__device__ __forceinline__ unsigned long long mantissa53(double v) {  // of a normal v
  return (unsigned long long)(((unsigned)__double2hiint(v) & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(v);
}
// To binary64, rounded.
__device__ __forceinline__ double mult_double(Mult w) {
  // the correction may have moved the mantissa a little out of [2^61, 2^62)
  const int h = (int)(w.m >> 32), d = (h >= 0x40000000 ? 1 : 0) - (h < 0x20000000 ? 1 : 0);
  return __longlong_as_double(((w.m + (128ll << (1 + d))) >> (9 + d)) + ((long long)(w.ex - 1 + d) << 52));
}
__device__ __forceinline__ Mult mult_rcp(double v) {
  if (!f32_range(v)) return mult_of(1.0 / v);
  const unsigned yb = __float_as_uint(__frcp_rn(d2f_bits(v))), my = (yb & 0x7fffffu) | 0x800000u;
  const int ey = (int)(yb >> 23);
  const int s = 1150 - ey - (__double2hiint(v) >> 20);  // 0 or 1
  const long long E = (long long)(0ull - (mantissa53(v) << 9) * my) << (1 - s);  // e 2^85; 2^(84 + s) is 0 modulo 2^64
  const int eh = (int)(E >> 32);                                                 // e 2^53
  return mult_corr(my, ey, (E >> 29) + (mulw(eh, eh) >> 50));
}
__device__ __forceinline__ double rsqrt_fast(double v) {
  if (!f32_range(v)) return rsqrt(v);
  const unsigned yb = __float_as_uint(rsqrtf(d2f_bits(v))), my = (yb & 0x7fffffu) | 0x800000u;
  const int ey = (int)(yb >> 23);
  const int s = 1277 - 2 * ey - (__double2hiint(v) >> 20);  // 0 ... 3
  // v y^2 is 2^(60 + s) here; E = e 2^63
  const long long E = (long long)((1ull << (60 + s)) - __umul64hi(mantissa53(v) << 10, ((unsigned long long)my * my) << 16)) << (3 - s);
  const int eh = (int)(E >> 12);  // e 2^51
  // e / 2 + 3/8 e^2 in units 2^-56
  return mult_double(mult_corr(my, ey, (E + 3 * (mulw(eh, eh) >> 41)) >> 8));
}
// max(v, 0), 0 for a NaN, off the FP64 pipe
__device__ __forceinline__ double pos_part(double v) {
  const unsigned h = (unsigned)__double2hiint(v);
  return h < 0x7ff00000u || (h == 0x7ff00000u && __double2loint(v) == 0) ? v : 0.0;
}

// ---- preconditioner (unpadded grid); Wk: [Nz][Ny][Nx] workspace.  The weight
// P_V^{-1/2} of each point is stored in Pw for the x inverse pass, which then
// reads it instead of forming it again.
struct IPXF : IOpBase<-1, false, 0, true, kSrcF64> {
  static constexpr bool kPdl = false;
  const double2* r;
  const double2* phi;
  const double* Phi;
  c64* Wk;
  double* Pw;
  ExpTab ex;
  const double* hx2;
  const double* hy2;
  const double* hz2;
  double gx2, gy2, gz2, beta, alam;
  const double* alpha;
  int Nx, Ny, nl;
  __device__ __forceinline__ bool valid(int o, int) const { return o < nl; }
  __device__ __forceinline__ double2 load(int o, int, int pos) const {
    const size_t i = (size_t)o * Nx + pos;
    const int y = o % Ny, z = o / Ny;
    const double2 pv = __ldg(phi + i);
    // alpha and the terms of y and z are the line's
    const double V = fma(gx2, hx2[pos], *alpha + (gy2 * hy2[y] + gz2 * hz2[z]));
    const double den = fma(alam, pos_part(__ldg(Phi + i)), fma(beta, fma(pv.x, pv.x, pv.y * pv.y), V));
    const double w = rsqrt_fast(den);
    Pw[i] = w;
    const double2 rv = __ldg(r + i);
    return make_double2(rv.x * w, rv.y * w);
  }
  __device__ __forceinline__ void store(int o, int, int pos, c64 v, const Tile&, Acc&) const {
    stc(Wk + (size_t)o * Nx + pos, v);
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const {
    put_exp_at(ex, l.o, 0, l, t.anybad ? kExpNaN : t.e);
  }
};

// y transform of sign S in place: o = z.  LINES: the input's exponents are
// indexed by the row z Ny + y (a line-major pass wrote them), else by y.
template <int S, bool LINES> struct IPY : IOpBase<S, false, 0, false, kSrcInt> {
  c64* Wk;
  ExpTab in, ex;
  int Nx, Ny;
  __device__ __forceinline__ bool valid(int, int x) const { return x < Nx; }
  __device__ __forceinline__ c64 load(int o, int x, int pos) const { return ldc(step(Wk + (size_t)o * Ny * Nx + x, pos, Nx * 16)); }
  __device__ __forceinline__ int lexp(int o, int x, int pos) const { return in.at(LINES ? o * Ny + pos : pos, x); }
  __device__ __forceinline__ void store(int o, int x, int pos, c64 v, const Tile&, typename IPY::Acc&) const {
    stc(step(Wk + (size_t)o * Ny * Nx + x, pos, Nx * 16), v);
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const { put_exp_at(ex, l.o, l.x, l, t.e); }
};

// z forward * 1/((alpha + |nu|^2/2) N) * inverse on lines (o = y, x).
struct IPZ : IOpBase<-1, true, 0, false, kSrcInt> {
  c64* Wk;
  ExpTab in, ex;
  const double* alpha;
  const double* nx2;  // nu^2 / 2 of each axis
  const double* ny2;
  const double* nz2;
  double Nt;  // grid points
  int Nx, Ny;
  static constexpr bool kMul = true;
  __device__ __forceinline__ bool valid(int, int x) const { return x < Nx; }
  __device__ __forceinline__ c64 load(int o, int x, int pos) const { return ldc(step(Wk + (size_t)o * Nx + x, pos, Ny * Nx * 16)); }
  __device__ __forceinline__ int lexp(int, int x, int pos) const { return in.at(pos, x); }
  __device__ __forceinline__ void tally(int, int, int, Limbs, Limbs, Acc&) const {}
  // x may lie beyond the grid for the lines that a tile's last CTA leaves idle
  __device__ __forceinline__ double mline(int o, int x) const { return valid(o, x) ? Nt * (*alpha + (nx2[x] + ny2[o])) : 1.0; }
  __device__ __forceinline__ Mult mult(double c, int k) const { return mult_rcp(fma(Nt, nz2[k], c)); }
  __device__ __forceinline__ void store(int o, int x, int pos, c64 v, const Tile&, Acc&) const {
    stc(step(Wk + (size_t)o * Nx + x, pos, Ny * Nx * 16), v);
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const { put_exp_at(ex, l.o, l.x, l, t.e); }
};

struct IPXI : IOpBase<1, false, 0, true, kSrcInt> {
  static constexpr bool kPdl = false;
  const c64* Wk;
  const double* Pw;
  double2* Pr;
  ExpTab in;
  int Nx, Ny, nl;
  __device__ __forceinline__ bool valid(int o, int) const { return o < nl; }
  __device__ __forceinline__ c64 load(int o, int, int pos) const { return ldc(Wk + (size_t)o * Nx + pos); }
  __device__ __forceinline__ int lexp(int o, int, int pos) const { return in.at(o / Ny, pos); }
  __device__ __forceinline__ void store(int o, int, int pos, c64 v, const Tile& t, Acc&) const {
    const size_t i = (size_t)o * Nx + pos;
    const double w = __ldg(Pw + i);
    double2 d;
    if (i2d_ok(t.e)) d = make_double2(i2d(v.x, t.e + 1085), i2d(v.y, t.e + 1085));
    else d = make_double2(i2d_any(v.x, t.e), i2d_any(v.y, t.e));
    Pr[i] = make_double2(w * d.x, w * d.y);
  }
  __device__ __forceinline__ void put_exp(const Line&, const Tile&) const {}
};

// ---- in-place 3D complex FFT on a plan's (unpadded) grid, sign S: binary64
// in, integers between the passes (the y pass is IPY), binary64 out.
template <int S> struct ICX : IOpBase<S, false, 0, true, kSrcF64> {
  double2* buf;
  ExpTab ex;
  int Nx, nl;
  __device__ __forceinline__ bool valid(int o, int) const { return o < nl; }
  __device__ __forceinline__ double2 load(int o, int, int pos) const { return buf[(size_t)o * Nx + pos]; }
  __device__ __forceinline__ void store(int o, int, int pos, c64 v, const Tile&, typename ICX::Acc&) const {
    stc(reinterpret_cast<c64*>(buf) + (size_t)o * Nx + pos, v);
  }
  __device__ __forceinline__ void put_exp(const Line& l, const Tile& t) const {
    put_exp_at(ex, l.o, 0, l, t.anybad ? kExpNaN : t.e);
  }
};
template <int S> struct ICZ : IOpBase<S, false, 0, false, kSrcInt> {
  double2* buf;
  ExpTab in;
  int Nx, Ny;
  __device__ __forceinline__ bool valid(int, int x) const { return x < Nx; }
  __device__ __forceinline__ c64 load(int o, int x, int pos) const {
    return ldc(reinterpret_cast<const c64*>(buf) + ((size_t)pos * Ny + o) * Nx + x);
  }
  __device__ __forceinline__ int lexp(int, int x, int pos) const { return in.at(pos, x); }
  __device__ __forceinline__ void store(int o, int x, int pos, c64 v, const Tile& t, typename ICZ::Acc&) const {
    double2 d;
    if (i2d_ok(t.e)) d = make_double2(i2d(v.x, t.e + 1085), i2d(v.y, t.e + 1085));
    else d = make_double2(i2d_any(v.x, t.e), i2d_any(v.y, t.e));
    buf[((size_t)pos * Ny + o) * Nx + x] = d;
  }
  __device__ __forceinline__ void put_exp(const Line&, const Tile&) const {}
};

}  // namespace atkm
