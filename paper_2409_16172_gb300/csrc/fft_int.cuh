// FFT passes of the complex128 preconditioner apply, in 64-bit integers.
//
// sm_103a executes 2 FP64 lanes per clock and SM, so an FP64 transform is
// bound by its additions (a radix-4 FP64 engine took 30 clocks per point and
// node in the symbol pass at 480 x 720).  Here a block turns its lines into
// integers of one common unit, runs the mixed-radix Stockham stages on them
// (additions on the 62-lane integer pipe, twiddles as 31-bit limb products),
// and turns the results back: two FP64 conversions per point and pass remain.
//
// Block floating point: the values of a block share one exponent.  Before a
// stage of radix R every component is below 2^(61 - g), g >= log2(R) + 1/2,
// so the stage cannot overflow 2^61; after it the largest component of the
// block is known (one reduction that rides on the stage's barrier) and the
// next stage's reads shift all values to the top of its range again.  A value
// thus keeps at least 55 bits below the largest of its block in every stage.
// Values, products and shifts are rounded to nearest: a truncation's bias adds
// up over a line, above all where a spectrum is a few large entries.  Whole
// apply against extended precision, here (cut instead of rounded; FP64 stages):
// 40 x 48 x 60 noise 3.6e-16 (5.2; 4.7), wide bump 2.6 (5.1; 2.8), plane wave 2.3
// (3.3; 2.4); 240 x 360 noise 3.8 (4.3; 5.7), plane wave 2.8 (5.1; 3.8).
// Rounding costs no time (480 x 720, K = 8: 193 -> 190 us).
// A block's lines belong to one right-hand side, and which lines share a block
// does not depend on the call's other right-hand sides: neither do results.
//
// Stages ping-pong between two shared-memory copies of the lines; a work item
// is one butterfly, so a thread holds one radix of elements, and any thread
// count works for any length.
#pragma once
#include <type_traits>
#include <utility>

#include "fft_engine.cuh"
#include "fixed.cuh"
#include "recip.cuh"

namespace hz {

struct __align__(16) CI {
  long long x, y;
};

template <typename F, int... I>
__device__ __forceinline__ void static_for_seq(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int M, typename F> __device__ __forceinline__ void static_for(F&& f) {
  static_for_seq(f, std::make_integer_sequence<int, M>{});
}

// ---- products with numbers of modulus <= 1, held times 2^61 -----------------
// Limbs v = h 2^31 + l, l symmetric about zero (as those of the twiddle table
// and of the constants): the partial products l l are then left out without
// a bias.
__device__ __forceinline__ int l31l(long long v) { return int(unsigned(v) << 1) >> 1; }
__device__ __forceinline__ int l31h(long long v) { return int(v >> 31) - (l31l(v) >> 31); }
constexpr int q31h(long long c) { return int((c + (1ll << 30)) >> 31); }
constexpr int q31l(long long c) { return int(c - q31h(c) * (1ll << 31)); }
// constants times 2^61, rounded
constexpr long long q61(double c) {
  return c < 0 ? -q61(-c) : (long long)(c * 2305843009213693952.0 + 0.5);
}
// (hh 2^62 + m 2^31) / 2^61 to the nearest integer, where m was begun with
// half; the lowest partial products (below one unit, of mean zero) are left out
constexpr long long HALF61 = 1ll << 29;
__device__ __forceinline__ long long join61(long long hh, long long m) { return (hh << 1) + (m >> 30); }

template <long long C> __device__ __forceinline__ long long mulq(long long v) {
  constexpr int ch = q31h(C), cl = q31l(C);
  const int h = l31h(v), l = l31l(v);
  return join61(mad_w(h, ch, 0), mad_w(h, cl, mad_w(l, ch, HALF61)));
}
// C1 v + C2 w
template <long long C1, long long C2> __device__ __forceinline__ long long mulq2(long long v, long long w) {
  constexpr int ah = q31h(C1), al = q31l(C1), bh = q31h(C2), bl = q31l(C2);
  const int h = l31h(v), l = l31l(v), p = l31h(w), q = l31l(w);
  return join61(mad_w(p, bh, mad_w(h, ah, 0)),
                mad_w(p, bl, mad_w(q, bh, mad_w(h, al, mad_w(l, ah, HALF61)))));
}
template <long long C, long long D> __device__ __forceinline__ CI cmulq(CI a) {  // a (C + i D)
  return CI{mulq2<C, -D>(a.x, a.y), mulq2<D, C>(a.x, a.y)};
}
// a w (S < 0) or a conj(w) (S > 0), w as (re hi, re lo, im hi, im lo)
template <int S> __device__ __forceinline__ CI twiddle_int(CI a, int4 w) {
  const int xh = l31h(a.x), xl = l31l(a.x), yh = l31h(a.y), yl = l31l(a.y);
  const int ih = S > 0 ? -w.z : w.z, il = S > 0 ? -w.w : w.w;  // imaginary part in use
  const int nh = S > 0 ? w.z : -w.z, nl = S > 0 ? w.w : -w.w;  // and its negative
  CI r;
  r.x = join61(mad_w(yh, nh, mad_w(xh, w.x, 0)),
               mad_w(yh, nl, mad_w(yl, nh, mad_w(xh, w.y, mad_w(xl, w.x, HALF61)))));
  r.y = join61(mad_w(yh, w.x, mad_w(xh, ih, 0)),
               mad_w(yh, w.y, mad_w(yl, w.x, mad_w(xh, il, mad_w(xl, ih, HALF61)))));
  return r;
}

// cos and sin of 2 pi m / RR, 0 <= m < RR: series on the first octant
constexpr double oct_cos(double x) {
  double t = 1.0, s = 1.0;
  for (int i = 1; i < 14; ++i) {
    t *= -x * x / double((2 * i - 1) * (2 * i));
    s += t;
  }
  return s;
}
constexpr double oct_sin(double x) {
  double t = x, s = x;
  for (int i = 1; i < 14; ++i) {
    t *= -x * x / double((2 * i) * (2 * i + 1));
    s += t;
  }
  return s;
}
constexpr double wcos(int RR, int m) {
  m = ((m % RR) + RR) % RR;
  if (2 * m > RR) return wcos(RR, RR - m);
  if (4 * m > RR) return -wcos(2 * RR, RR - 2 * m);
  const double a = 6.283185307179586476925287 * m / RR;
  return 8 * m <= RR ? oct_cos(a) : oct_sin(6.283185307179586476925287 * (RR - 4 * m) / (4.0 * RR));
}
constexpr double wsin(int RR, int m) { return wcos(4 * RR, 4 * m - RR); }

// a exp(S 2 pi i M / RR)
template <int RR, int M, int S> __device__ __forceinline__ CI wmul(CI a) {
  constexpr int m = M % RR;
  if constexpr (m == 0) return a;
  else if constexpr (4 * m == RR) return cmul_si<S>(a);
  else if constexpr (2 * m == RR) return CI{-a.x, -a.y};
  else if constexpr (4 * m == 3 * RR) return cmul_si<-S>(a);
  else return cmulq<q61(wcos(RR, m)), q61(S * wsin(RR, m))>(a);
}

template <int RAD, int S> __device__ __forceinline__ void idft(CI* x);

template <int S> __device__ __forceinline__ void idft3(CI* x) {
  constexpr long long h = q61(0.86602540378443864676);  // sin(2 pi / 3)
  const CI s = cadd(x[1], x[2]), d = csub(x[1], x[2]);
  const CI t = CI{x[0].x - (s.x >> 1), x[0].y - (s.y >> 1)};
  const CI e = cmul_si<S>(CI{mulq<h>(d.x), mulq<h>(d.y)});
  x[0] = cadd(x[0], s);
  x[1] = cadd(t, e);
  x[2] = csub(t, e);
}

// the folded 5-point form of fft_engine.cuh's dft5
template <int S> __device__ __forceinline__ void idft5(CI* x) {
  constexpr long long c1 = q61(0.30901699437494742410), c2 = q61(-0.80901699437494742410);
  constexpr long long s1 = q61(0.95105651629515357212), s2 = q61(0.58778525229247312917);
  const CI t1 = cadd(x[1], x[4]), t2 = cadd(x[2], x[3]);
  const CI t3 = csub(x[1], x[4]), t4 = csub(x[2], x[3]);
  const CI a1 = CI{x[0].x + mulq2<c1, c2>(t1.x, t2.x), x[0].y + mulq2<c1, c2>(t1.y, t2.y)};
  const CI a2 = CI{x[0].x + mulq2<c2, c1>(t1.x, t2.x), x[0].y + mulq2<c2, c1>(t1.y, t2.y)};
  const CI b1 = cmul_si<S>(CI{mulq2<s1, s2>(t3.x, t4.x), mulq2<s1, s2>(t3.y, t4.y)});
  const CI b2 = cmul_si<S>(CI{mulq2<s2, -s1>(t3.x, t4.x), mulq2<s2, -s1>(t3.y, t4.y)});
  x[0] = cadd(x[0], cadd(t1, t2));
  x[1] = cadd(a1, b1);
  x[4] = csub(a1, b1);
  x[2] = cadd(a2, b2);
  x[3] = csub(a2, b2);
}

template <int S> __device__ __forceinline__ void idft8(CI* x) {
  constexpr long long r2 = q61(0.70710678118654752440);
  CI e[4] = {x[0], x[2], x[4], x[6]};
  CI o[4] = {x[1], x[3], x[5], x[7]};
  dft4<S>(e);
  dft4<S>(o);
  // w8^1 = r2 (1 + S i), w8^3 = r2 (-1 + S i)
  const CI i1 = cmul_si<S>(o[1]), i3 = cmul_si<S>(o[3]);
  const CI o1 = CI{mulq<r2>(o[1].x + i1.x), mulq<r2>(o[1].y + i1.y)};
  const CI o3 = CI{mulq<r2>(i3.x - o[3].x), mulq<r2>(i3.y - o[3].y)};
  const CI o2 = cmul_si<S>(o[2]);
  x[0] = cadd(e[0], o[0]); x[4] = csub(e[0], o[0]);
  x[1] = cadd(e[1], o1);   x[5] = csub(e[1], o1);
  x[2] = cadd(e[2], o2);   x[6] = csub(e[2], o2);
  x[3] = cadd(e[3], o3);   x[7] = csub(e[3], o3);
}

// radix R1 R2 by one Cooley-Tukey split (as fft_engine.cuh's dft_split)
template <int R1, int R2, int S> __device__ __forceinline__ void isplit(CI* x) {
  constexpr int RR = R1 * R2;
  CI y[RR];
  static_for<R2>([&](auto n2) {
    CI t[R1];
    static_for<R1>([&](auto n1) { t[n1.value] = x[n2.value + R2 * n1.value]; });
    idft<R1, S>(t);
    static_for<R1>([&](auto k1) {
      y[n2.value * R1 + k1.value] = wmul<RR, n2.value * k1.value, S>(t[k1.value]);
    });
  });
  static_for<R1>([&](auto k1) {
    CI t[R2];
    static_for<R2>([&](auto n2) { t[n2.value] = y[n2.value * R1 + k1.value]; });
    idft<R2, S>(t);
    static_for<R2>([&](auto k2) { x[k1.value + R1 * k2.value] = t[k2.value]; });
  });
}

template <int RAD, int S> __device__ __forceinline__ void idft(CI* x) {
  if constexpr (RAD == 2) dft2<S>(x);
  else if constexpr (RAD == 3) idft3<S>(x);
  else if constexpr (RAD == 4) dft4<S>(x);
  else if constexpr (RAD == 5) idft5<S>(x);
  else if constexpr (RAD == 6) isplit<2, 3, S>(x);
  else if constexpr (RAD == 8) idft8<S>(x);
  else if constexpr (RAD == 9) isplit<3, 3, S>(x);
  else if constexpr (RAD == 10) isplit<2, 5, S>(x);
  else if constexpr (RAD == 12) isplit<4, 3, S>(x);
  else static_assert(RAD == 2, "unsupported radix");
}
// bits a stage may add to a component: at least log2(RAD) + 1/2
constexpr int growth(int rad) { return rad <= 2 ? 2 : (rad <= 5 ? 3 : (rad <= 11 ? 4 : 5)); }

// ---- radices -----------------------------------------------------------------
template <int N> struct IPlan;
#define HZ_IPLAN(NN, ...)                                                  \
  template <> struct IPlan<NN> {                                           \
    static constexpr int rads[] = {__VA_ARGS__};                           \
    static constexpr int NST = sizeof(rads) / sizeof(int);                 \
    __host__ __device__ static constexpr int rad(int s) { return rads[s]; } \
  };
HZ_IPLAN(8, 8)
HZ_IPLAN(12, 12)
HZ_IPLAN(16, 4, 4)
HZ_IPLAN(20, 5, 4)
HZ_IPLAN(24, 6, 4)
HZ_IPLAN(32, 8, 4)
HZ_IPLAN(40, 8, 5)
HZ_IPLAN(48, 8, 6)
HZ_IPLAN(60, 10, 6)
HZ_IPLAN(64, 8, 8)
HZ_IPLAN(96, 12, 8)
HZ_IPLAN(120, 12, 10)
HZ_IPLAN(128, 8, 4, 4)
HZ_IPLAN(180, 6, 6, 5)
HZ_IPLAN(192, 8, 6, 4)
HZ_IPLAN(240, 8, 6, 5)
HZ_IPLAN(256, 8, 8, 4)
HZ_IPLAN(360, 9, 8, 5)
HZ_IPLAN(480, 10, 8, 6)
HZ_IPLAN(512, 8, 8, 8)
HZ_IPLAN(720, 10, 9, 8)
HZ_IPLAN(960, 12, 10, 8)
HZ_IPLAN(1024, 8, 8, 4, 4)
HZ_IPLAN(1440, 12, 12, 10)
HZ_IPLAN(1920, 8, 8, 6, 5)
HZ_IPLAN(2048, 8, 8, 8, 4)
HZ_IPLAN(2400, 10, 8, 6, 5)
HZ_IPLAN(2880, 12, 10, 6, 4)
HZ_IPLAN(3600, 10, 10, 6, 6)
HZ_IPLAN(4800, 10, 10, 8, 6)
#undef HZ_IPLAN

// ---- doubles to and from a block's integers -----------------------------------
// x 2^(top + 1023 - E) to the nearest integer; E >= exponent of x, 52 <= top <= 61
__device__ __forceinline__ long long int_of(double x, int E, int top) {
  const int hi = __double2hiint(x);
  const unsigned lo = unsigned(__double2loint(x));
  const int ex = (hi >> 20) & 0x7ff;
  const unsigned mh = ex == 0 ? 0u : unsigned((hi & 0xfffff) | 0x100000);
  unsigned long long t = (static_cast<unsigned long long>(mh) << 32 | (ex == 0 ? 0u : lo)) << (top - 51);
  asm("shr.u64 %0, %0, %1;" : "+l"(t) : "r"(E - ex));
  const long long s = hi >> 31;
  return (static_cast<long long>((t + 1) >> 1) ^ s) - s;
}
// A block of LINES lines of N points.  ROWS: lines one after the other, else
// interleaved (columns).
template <int N_, int LINES_, bool ROWS> struct IBlock {
  static constexpr int N = N_, LINES = LINES_;
  static constexpr bool BY_ROWS = ROWS;
  static constexpr int PADN = N + N / 8 + 1;
  static constexpr int want() {
    // about one butterfly per thread; small blocks more threads, so that the
    // FP64 parts spread over an SM's four units
    const int points = N * LINES;
    int t = (points / (points <= 512 ? 2 : 9) + 31) / 32 * 32;
    if (points <= 512 && t > 128) t = 128;
    return t < 32 ? 32 : (t > 256 ? 256 : t);
  }
  static constexpr int NT = want();
  static constexpr int WARPS = NT / 32;
  static constexpr size_t SMEM = size_t(2) * PADN * LINES * sizeof(CI);
  // one element after every 8 keeps the strided writes of the early stages
  // off each other's banks
  __device__ static __forceinline__ int at(int p, int line) {
    const int q = p + (p >> 3);
    return ROWS ? line * PADN + q : q * LINES + line;
  }
};

// Transforms the lines in shared memory copy A (doubles as bits; E0 = their
// largest biased exponent, known to all threads, copies synchronised) and
// gives every result to store(line, position, re, im).
template <typename B, int S, int STAGE, int NS, typename Store>
__device__ __forceinline__ void int_stage(CI* src, CI* dst, int* red, int E0, int e, int sh,
                                          const int4* __restrict__ tw, Store& store) {
  using P = IPlan<B::N>;
  constexpr int N = B::N, RAD = P::rad(STAGE), M = N / RAD;
  constexpr bool LAST = STAGE == P::NST - 1;
  constexpr int ITEMS = M * B::LINES;
  constexpr int TOP0 = 60 - growth(RAD);  // first stage: values below 2^(61 - growth)
  unsigned bits = 0u;
#pragma unroll 1
  for (int it = threadIdx.x; it < ITEMS; it += B::NT) {
    const int ln = B::BY_ROWS ? it / M : it % B::LINES;
    const int j = B::BY_ROWS ? it - ln * M : it / B::LINES;
    CI x[RAD];
#pragma unroll
    for (int r = 0; r < RAD; ++r) x[r] = src[B::at(j + r * M, ln)];
    if constexpr (STAGE == 0) {
#pragma unroll
      for (int r = 0; r < RAD; ++r)
        x[r] = CI{int_of(__longlong_as_double(x[r].x), E0, TOP0),
                  int_of(__longlong_as_double(x[r].y), E0, TOP0)};
    } else {
      if (sh >= 0) {
#pragma unroll
        for (int r = 0; r < RAD; ++r) x[r] = CI{x[r].x << sh, x[r].y << sh};
      } else {
        const long long half = 1ll << (-sh - 1);
#pragma unroll
        for (int r = 0; r < RAD; ++r) x[r] = CI{(x[r].x + half) >> -sh, (x[r].y + half) >> -sh};
      }
    }
    const int k = NS > 1 ? j % NS : 0;
    if constexpr (NS > 1) {
#pragma unroll
      for (int r = 1; r < RAD; ++r) x[r] = twiddle_int<S>(x[r], __ldg(tw + r * k * (N / (NS * RAD))));
    }
    idft<RAD, S>(x);
    const int d = (j / NS) * NS * RAD + k;
#pragma unroll
    for (int r = 0; r < RAD; ++r) {
      if constexpr (LAST) {
        store(ln, d + r * NS, double_of(x[r].x, e), double_of(x[r].y, e));
      } else {
        dst[B::at(d + r * NS, ln)] = x[r];
        const int hx = int(x[r].x >> 32), hy = int(x[r].y >> 32);
        bits |= unsigned(hx ^ (hx >> 31)) | unsigned(hy ^ (hy >> 31));
      }
    }
  }
  if constexpr (!LAST) {
    // two sets of words in turn: one barrier per stage
    int* rd = red + (STAGE % 2 == 0 ? B::WARPS : 0);
    bits = __reduce_or_sync(0xffffffffu, bits);
    if ((threadIdx.x & 31) == 0) rd[threadIdx.x >> 5] = int(bits);
    __syncthreads();
    unsigned all = unsigned(rd[0]);
#pragma unroll
    for (int i = 1; i < B::WARPS; ++i) all |= unsigned(rd[i]);
    // components are below 2^(64 - clz); the next stage wants 2^(61 - growth)
    const int lead = all ? __clz(int(all)) : 32;
    const int s = 61 - growth(P::rad(STAGE + 1)) - (64 - lead);
    int_stage<B, S, STAGE + 1, NS * RAD>(dst, src, red, E0, e - s, s, tw, store);
  }
}

template <typename B, int S, typename Store>
__device__ __forceinline__ void int_transform(CI* sm, int* red, int E0, const int4* __restrict__ tw,
                                              Store&& store) {
  constexpr int TOP0 = 60 - growth(IPlan<B::N>::rad(0));
  int_stage<B, S, 0, 1>(sm, sm + B::PADN * B::LINES, red, E0, E0 - 1023 - TOP0, 0, tw, store);
}

// largest biased exponent over the block of what the threads have seen (max
// of the high words without sign); one barrier, which also makes copy A visible
template <typename B> __device__ __forceinline__ int block_exp(unsigned hi, int* red) {
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = int(hi);
  __syncthreads();
  unsigned m = unsigned(red[0]);
#pragma unroll
  for (int i = 1; i < B::WARPS; ++i) m = max(m, unsigned(red[i]));
  return int(m >> 20);
}
__device__ __forceinline__ unsigned top_word(double2 v) {
  return max(unsigned(__double2hiint(v.x)) & 0x7fffffffu, unsigned(__double2hiint(v.y)) & 0x7fffffffu);
}
__device__ __forceinline__ CI bits_of(double2 v) {
  return CI{__double_as_longlong(v.x), __double_as_longlong(v.y)};
}

// ---------------------------------------------------------------------------
// The passes (the counterparts in fft_kernels.cuh are complex64).  A block
// that holds an infinity or a NaN gives NaN for all of its lines, as a
// transform of such a line does.
// ---------------------------------------------------------------------------

// Forward along x.  grid (blocks of LINES rows, rhs)
template <int N, int LINES>
__global__ void __launch_bounds__(IBlock<N, LINES, true>::NT)
irow_fwd_kernel(const double2* __restrict__ in, const double* __restrict__ scale, long rows,
                const int4* __restrict__ tw, double2* __restrict__ out,
                const int* __restrict__ active) {
  pdl_wait();
  using B = IBlock<N, LINES, true>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CI* sm = reinterpret_cast<CI*>(smem_raw);
  __shared__ int red[2 * B::WARPS];
  const long rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  const long row0 = long(blockIdx.x) * LINES;
  const int have = int(min(long(LINES), rows - row0));
  const double s = scale ? scale[rhs] : 1.0;
  const double2* src = in + (rhs * rows + row0) * N;
  unsigned hi = 0u;
#pragma unroll 4
  for (int i = threadIdx.x; i < N * LINES; i += B::NT) {
    double2 v = i < N * have ? src[i] : make_double2(0.0, 0.0);
    if (scale) v = make_double2(v.x * s, v.y * s);
    hi = max(hi, top_word(v));
    sm[B::at(i % N, i / N)] = bits_of(v);
  }
  const int E = block_exp<B>(hi, red);
  double2* dst = out + (rhs * rows + row0) * N;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  int_transform<B, -1>(sm, red, E, tw, [&](int line, int p, double re, double im) {
    if (line < have) dst[line * N + p] = E < 0x7ff ? make_double2(re, im) : make_double2(nan, nan);
  });
}

// Inverse along x of the (row, node) lines in use, in place.
// grid (blocks of LINES rows, K, rhs)
template <int N, int LINES>
__global__ void __launch_bounds__(IBlock<N, LINES, true>::NT)
irow_inv_kernel(double2* planes, const unsigned long long* __restrict__ rowmask, int K, long rows,
                long n, const int4* __restrict__ tw, const int* __restrict__ active) {
  pdl_wait();
  using B = IBlock<N, LINES, true>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CI* sm = reinterpret_cast<CI*>(smem_raw);
  __shared__ int red[2 * B::WARPS];
  const long rhs = blockIdx.z;
  const int k = blockIdx.y;
  if (active && !active[rhs]) return;
  const long row0 = long(blockIdx.x) * LINES;
  unsigned long long used = 0ull;  // one bit per line: LINES <= 128
  unsigned long long used2 = 0ull;
  for (int l = 0; l < LINES && row0 + l < rows; ++l) {
    const unsigned long long bit = (rowmask[row0 + l] >> k) & 1ull;
    if (l < 64) used |= bit << l;
    else used2 |= bit << (l - 64);
  }
  if (!(used | used2)) return;
  auto on = [&](int l) { return ((l < 64 ? used >> l : used2 >> (l - 64)) & 1ull) != 0; };
  double2* g = planes + (rhs * K + k) * n + row0 * N;
  unsigned hi = 0u;
#pragma unroll 4
  for (int i = threadIdx.x; i < N * LINES; i += B::NT) {
    const int l = i / N;
    const double2 v = on(l) ? g[i] : make_double2(0.0, 0.0);
    hi = max(hi, top_word(v));
    sm[B::at(i - l * N, l)] = bits_of(v);
  }
  const int E = block_exp<B>(hi, red);
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  int_transform<B, +1>(sm, red, E, tw, [&](int line, int p, double re, double im) {
    if (on(line)) g[line * N + p] = E < 0x7ff ? make_double2(re, im) : make_double2(nan, nan);
  });
}

// Strided axis, in place: TB adjacent columns.  grid (tiles * outer, 1, batch)
template <int N, int SIGN, int TB>
__global__ void __launch_bounds__(IBlock<N, TB, false>::NT)
iline_kernel(double2* data, int nx, int ntile, long S, long ostride, long bstride,
             const unsigned long long* __restrict__ omask, int K, const int4* __restrict__ tw,
             const int* __restrict__ active, int per_rhs) {
  pdl_wait();
  using B = IBlock<N, TB, false>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CI* sm = reinterpret_cast<CI*>(smem_raw);
  __shared__ int red[2 * B::WARPS];
  const int tile = blockIdx.x % ntile;
  const long o = blockIdx.x / ntile;
  if (omask && !((omask[o] >> (blockIdx.z % K)) & 1ull)) return;
  if (active && !active[blockIdx.z / per_rhs]) return;
  const int x0 = tile * TB, have = min(TB, nx - x0);
  double2* base = data + long(blockIdx.z) * bstride + o * ostride + x0;
  const int Si = int(S);
  unsigned hi = 0u;
#pragma unroll 4
  for (int i = threadIdx.x; i < N * TB; i += B::NT) {
    const int col = i % TB, p = i / TB;
    const double2 v = col < have ? base[p * Si + col] : make_double2(0.0, 0.0);
    hi = max(hi, top_word(v));
    sm[B::at(p, col)] = bits_of(v);
  }
  const int E = block_exp<B>(hi, red);
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  int_transform<B, SIGN>(sm, red, E, tw, [&](int col, int p, double re, double im) {
    if (col < have) base[p * Si + col] = E < 0x7ff ? make_double2(re, im) : make_double2(nan, nan);
  });
}

// Last axis: spectrum times q_k (Eqn. 021), inverse, plane k on the rows /
// slabs that use node k.  grid (tiles * outer, K, rhs)
template <int N, int TB, bool HERM>
__global__ void __launch_bounds__(IBlock<N, TB, false>::NT)
isym_kernel(const double2* __restrict__ vhat, double2* __restrict__ planes, int nx, int ntile, long S,
            long ostride, long n, int K, const double* __restrict__ xi2_x,
            const double* __restrict__ xi2_o, const double* __restrict__ xi2_l,
            const double2* __restrict__ symA, const double2* __restrict__ symG,
            const double* __restrict__ symD, const unsigned long long* __restrict__ smask, long smO,
            long smS, const int4* __restrict__ tw, const int* __restrict__ active) {
  pdl_wait();
  using B = IBlock<N, TB, false>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CI* sm = reinterpret_cast<CI*>(smem_raw);
  __shared__ int red[2 * B::WARPS];
  const long rhs = blockIdx.z;
  if (active && !active[rhs]) return;
  const int tile = blockIdx.x % ntile;
  const long o = blockIdx.x / ntile;
  const int k = blockIdx.y;
  const int x0 = tile * TB, have = min(TB, nx - x0);
  const int Si = int(S);
  const double2* src = vhat + rhs * n + o * ostride + x0;
  const double2 A = symA[k], G = symG[k];
  const double D = HERM ? symD[k] : 0.0;
  // a thread keeps its column (the block's columns divide its threads)
  static_assert(B::NT % TB == 0, "one column per thread");
  const int col = threadIdx.x % TB;
  const double sx = (col < have ? xi2_x[x0 + col] : 0.0) + (xi2_o ? xi2_o[o] : 0.0);
  const bool real = G.y == 0.0;  // a real node: the imaginary part of den is constant
  const double ay2 = A.y * A.y;
  unsigned hi = 0u;
#pragma unroll 2
  for (int i = threadIdx.x; i < N * TB; i += B::NT) {
    const int p = i / TB;
    double2 r = make_double2(0.0, 0.0);
    if (col < have) {
      const double2 v = src[p * Si + col];
      // vhat q_k = vhat conj(den) / |den|^2,  den = A - G |xi|^2
      // (|xi|^2 rounded once before the cancellation near the resonance)
      const double s2 = sx + xi2_l[p];
      const double dx = fma(-G.x, s2, A.x);
      double dy = A.y, dy2 = ay2;
      if (!real) {
        dy = fma(-G.y, s2, A.y);
        dy2 = dy * dy;
      }
      const double inv = recip3(fma(dx, dx, dy2));
      const double qx = dx * inv, qy = dy * inv;
      r.x = fma(v.x, qx, v.y * qy);
      r.y = fma(v.y, qx, -(v.x * qy));
      if (HERM && D != 0.0) {
        // derivative plane: vhat dq/dc = vhat q (D |xi|^2 q)
        const double ds = D * s2, ux = qx * ds, uy = qy * ds;
        r = make_double2(fma(r.x, ux, r.y * uy), fma(r.y, ux, -(r.x * uy)));
      }
    }
    hi = max(hi, top_word(r));
    sm[B::at(p, col)] = bits_of(r);
  }
  const int E = block_exp<B>(hi, red);
  double2* dst = planes + (rhs * K + k) * n + o * ostride + x0;
  const unsigned long long* mk = smask + o * smO;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  int_transform<B, +1>(sm, red, E, tw, [&](int col, int p, double re, double im) {
    if (col < have && ((mk[p * int(smS)] >> k) & 1ull))
      dst[p * Si + col] = E < 0x7ff ? make_double2(re, im) : make_double2(nan, nan);
  });
}

// Lines per block.  Rows: about 1024 points.  Columns: 64 bytes or more of
// each row while two copies leave room for several blocks on an SM.
template <int N> struct ICfg {
  static constexpr int ROWS = N >= 768 ? 1 : (1024 / N > 128 ? 128 : 1024 / N);
  static constexpr int TB = N <= 64 ? 16 : (N <= 128 ? 8 : (N <= 512 ? 4 : (N <= 1440 ? 2 : 1)));
  // grids that would leave SMs without a block
  static constexpr int TB_FEW = TB >= 4 ? TB / 4 : 1;
};

}  // namespace hz
