// Finite-difference Helmholtz operator P_N (Eqn. 001 discretised as in
// Section 5: second-order centred differences, periodic boundaries), FP64:
//   (P x)_j = gamma_j^2 sum_axes (x_{j+e} - 2 x_j + x_{j-e}) / h_axis^2
//             + (omega^2 + i omega a_j) x_j,
// with gamma^2 = c^2 (1 - i zeta)^2 (Eqn. Complex_wave_speed).
// Mode RESID computes r = f - P x and per-block partial sums of |r|^2.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "fixed.cuh"
#include "hz_internal.h"
#include "kernels.h"

namespace hz {
namespace {

constexpr int ST_THREADS = 256;

__device__ __forceinline__ double2 ld2(const double2* p, long i) { return p[i]; }
__device__ __forceinline__ double2 ld2(const float2* p, long i) {
  const float2 v = p[i];
  return make_double2(f2d_bits(v.x), f2d_bits(v.y));
}

// The stencil in the form that takes the fewest FP64 instructions per point
// (the FP64 pipe is this kernel's limit): with g = gamma^2 / h_x^2 (stored
// so by the medium), rho_a = h_x^2 / h_a^2 and diag = 2 sum_a rho_a,
//   (P x)_j = g_j [ (x_{j-ex} + x_{j+ex}) + rho_y (x_{j-ey} + x_{j+ey})
//                  (+ rho_z (...)) - diag x_j ] + (omega^2 + i omega a_j) x_j.
template <typename InT, bool RESID>
__global__ void __launch_bounds__(ST_THREADS)
stencil_kernel(const InT* __restrict__ x, double2* __restrict__ y, const double2* __restrict__ f,
               const double2* __restrict__ gs, const double* __restrict__ a, double omega,
               double w2, double rho_y, double rho_z, double diag, int nx, int ny, int nz, long n,
               long in_stride, long out_stride, const int* __restrict__ active,
               double* __restrict__ partial) {
  pdl_wait();
  const int b = blockIdx.y;
  double nrm = 0.0;
  const bool on = !active || active[b];
  if (on) {
    const InT* xb = x + b * in_stride;
    const long i = long(blockIdx.x) * ST_THREADS + threadIdx.x;
    if (i < n) {
      // n < 2^31 per right-hand side: 32-bit division
      const unsigned ui = unsigned(i);
      const unsigned r = ui / unsigned(nx);
      const int ix = int(ui - r * unsigned(nx));
      const unsigned rz = r / unsigned(ny);
      const int iy = int(r - rz * unsigned(ny));
      const int iz = int(rz);
      const long xl = ix == 0 ? i + nx - 1 : i - 1;
      const long xr = ix == nx - 1 ? i - (nx - 1) : i + 1;
      const long sy = nx;
      const long yd = iy == 0 ? i + sy * (ny - 1) : i - sy;
      const long yu = iy == ny - 1 ? i - sy * (ny - 1) : i + sy;
      const double2 c = ld2(xb, i);
      const double2 vxl = ld2(xb, xl), vxr = ld2(xb, xr), vyd = ld2(xb, yd), vyu = ld2(xb, yu);
      double sr = fma(rho_y, vyd.x + vyu.x, vxl.x + vxr.x);
      double si = fma(rho_y, vyd.y + vyu.y, vxl.y + vxr.y);
      if (nz > 1) {
        const long sz = long(nx) * ny;
        const long zd = iz == 0 ? i + sz * (nz - 1) : i - sz;
        const long zu = iz == nz - 1 ? i - sz * (nz - 1) : i + sz;
        const double2 vzd = ld2(xb, zd), vzu = ld2(xb, zu);
        sr = fma(rho_z, vzd.x + vzu.x, sr);
        si = fma(rho_z, vzd.y + vzu.y, si);
      }
      sr = fma(-diag, c.x, sr);
      si = fma(-diag, c.y, si);
      const double2 g = gs[i];
      // g * lap + (w^2 + i w a) x
      double yr = fma(g.x, sr, fma(-g.y, si, w2 * c.x));
      double yi = fma(g.x, si, fma(g.y, sr, w2 * c.y));
      if (a) {
        const double wa = omega * a[i];
        yr = fma(-wa, c.y, yr);
        yi = fma(wa, c.x, yi);
      }
      if (RESID) {
        const double2 fv = f[b * out_stride + i];
        yr = fv.x - yr;
        yi = fv.y - yi;
        nrm = yr * yr + yi * yi;
      }
      y[b * out_stride + i] = make_double2(yr, yi);
    }
  }
  if (RESID) {
    // fixed-shape block reduction of |r|^2
    __shared__ double sh[ST_THREADS];
    sh[threadIdx.x] = nrm;
    __syncthreads();
    for (int s = ST_THREADS / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
      __syncthreads();
    }
    if (threadIdx.x == 0) partial[long(b) * gridDim.x + blockIdx.x] = sh[0];
  }
}


// ---------------------------------------------------------------------------
// The same operator in integers.  The FP64 form above runs at the FP64 pipe
// (2 lanes per clock and SM, 14-18 instructions a point: 1.8 TB/s at 2400^2),
// so larger grids take the products and sums in exact 64-bit integers and use
// the FP64 pipe only to convert the two components of the result.
//
// A block owns 30 x TY (x TZ) points; with the halo these are 32-point rows,
// converted once each into shared memory.  All values of the tile share one
// binary exponent E, the largest of them: v = x 2^(fs_top + 1023 - E) to the
// nearest integer, below 2^(fs_top + 1).  Neighbour sums are exact; g =
// gamma^2 / h_x^2 and omega^2 are integers below 2^60 of a unit for the whole
// medium, and the products of 31-bit limbs are exact up to the last shift.
//
// What the rounding of the values costs a point beside larger ones:
//   complex128, and weighted sums  half a unit 2^-fs_top 2^E in each value,
//     weighted with 2 diag in all, is 2 eps (eps = 2^-53) of the neighbour sum's
//     terms as long as their weighted magnitudes add up to
//     diag 2^(E + 52 - fs_top) at least, separately in the real and the
//     imaginary parts.  A row of 30 points with one below that is done again by
//     the FP64 formula.  Gaussian noise has one such row in thousands.
//   complex64, equal spacings  values have 24 bits: nothing, if none but zeros
//     is below 2^-24 of the tile's largest.  Neighbour sums are then exact, the
//     products exact to 2^-27 of a value's unit, and the result is shifted by
//     its own size before it is cut.  Other tiles are done whole by the FP64
//     formula.
// So every component keeps the FP64 formula's bound, some eps times the
// magnitudes of its own terms, however steep the field is.  A warp whose first
// row is done again leaves all its rows to the FP64 formula.  A tile whose values
// leave the range of normal numbers, or are all zero, is done by it too.
// It is bound by the integer multiply-add pipe, which also takes the 64-bit
// additions (62 lanes per clock and SM, about 130 a point in 2D).  2400^2 damped,
// c128 input: 180 -> 87 us (3.7 TB/s), of which the check takes 3; 192^3, c64
// input: 277 -> 112 us (2.6 TB/s).  Fields that are steep all over (e^-r/8 at
// 2400^2) take 215 us, most of it FP64.
// ---------------------------------------------------------------------------
constexpr int SW = 8;          // warps per block
// bit of the leading one of a value with exponent E: neighbour sums stay below
// 2^61, which in the unweighted form of 3D is 12 values
__host__ __device__ constexpr int fs_top(bool d3, bool unit) { return d3 && unit ? 56 : 57; }
constexpr int FS_KEEP = 3;     // bits of the result kept below 2^62 units

template <bool D3> struct FsTile {
  static constexpr int TY = D3 ? 8 : 32, TZ = D3 ? 8 : 1;
  static constexpr int RY = TY + 2, RZ = D3 ? TZ + 2 : 1;  // rows with the halo
  static constexpr int ROWS = RY * RZ;
  static constexpr int PER = (ROWS + SW - 1) / SW;         // rows per warp
  static constexpr size_t SMEM = size_t(ROWS) * 32 * 16;
};

struct FxStencil {
  int w2h, w2l;                 // omega^2 in units of q_w
  int kh[4], kl[4];             // x, y, z, diagonal weights (general spacing)
  int share[3];                 // x, y, z weights over the diagonal's are 2^-share at least
  int k_out;                    // result = T 2^(E + k_out)
  int uq;                       // unit of g: 2^uq
};

// magnitude of a value, in order of size, from its high word; zero only for
// zeros (and doubles below 2^-1042)
__device__ __forceinline__ int mag_bits(double v) { return __double2hiint(v) & 0x7fffffff; }
__device__ __forceinline__ int mag_bits(float v) { return __float_as_int(v) & 0x7fffffff; }
// biased FP64 exponent of such a magnitude
template <typename T> __device__ __forceinline__ int mag_exp(int m) {
  if constexpr (std::is_same<T, double2>::value) return m >> 20;
  const int e = m >> 23;
  return e == 0 ? 0 : (e == 0xff ? 0x7ff : e + 896);
}
__device__ __forceinline__ long long shr(long long v, int n) {  // n > 63: zero
  asm("shr.u64 %0, %0, %1;" : "+l"(v) : "r"(n));
  return v;
}
// Fixed-point value, rounded to nearest, for the exponent E >= exponent of x.
// Zeros and subnormals need no test: with E at least FS_EMIN their shift is
// past the last bit.
template <typename T> __device__ constexpr int FS_EMIN = 128;
template <> __device__ constexpr int FS_EMIN<float2> = 896 + 60;
template <int TOP> __device__ __forceinline__ long long to_fs(double x, int E) {
  const int hi = __double2hiint(x);
  const unsigned lo = unsigned(__double2loint(x));
  const int ex = (hi >> 20) & 0x7ff;
  const unsigned mh = unsigned((hi & 0xfffff) | 0x100000);
  const unsigned th = __funnelshift_l(lo, mh, TOP - 51), tl = lo << (TOP - 51);
  const long long t =
      (shr(static_cast<long long>(static_cast<unsigned long long>(th) << 32 | tl), E - ex) + 1) >> 1;
  const long long sg = hi >> 31;
  return (t ^ sg) - sg;
}
template <int TOP> __device__ __forceinline__ long long to_fs(float x, int E) {
  const int u = __float_as_int(x);
  const int ex = (u >> 23) & 0xff;
  const int sg = u >> 31;
  const int m = ((u & 0x7fffff) | 0x800000) << (TOP - 54);
  // magnitude first: an arithmetic shift of a negative value would floor
  const long long t =
      (shr(static_cast<long long>(static_cast<unsigned long long>(unsigned(m)) << 32), E - 896 - ex) + 1) >> 1;
  const long long s = sg;
  return (t ^ s) - s;
}
__device__ __forceinline__ long long mul_w(int a, int b) { return static_cast<long long>(a) * b; }
// limbs of 31 bits: v = hi 2^31 + lo, 0 <= lo < 2^31
__device__ __forceinline__ int lim_h(long long v) { return int(v >> 31); }
__device__ __forceinline__ int lim_l(long long v) { return int(unsigned(v) & 0x7fffffffu); }

struct __align__(16) CLong {
  long long x, y;
};
__device__ __forceinline__ int high(long long v) { return int(v >> 32); }
__device__ __forceinline__ int size(long long v, long long w) { return abs(high(v)) + abs(high(w)); }
__device__ __forceinline__ CLong operator+(const CLong& p, const CLong& q) {
  return CLong{p.x + q.x, p.y + q.y};
}

// zero for zeros
__device__ __forceinline__ long long bits(double2 z) {
  return (__double_as_longlong(z.x) | __double_as_longlong(z.y)) << 1;
}

// bits below 2^62 units to keep of hh 2^62 + m 2^31, |m| < 2^63: all that
// leave the sum below 2^63
__device__ __forceinline__ int keep_bits(long long hh) {
  const int h = high(hh);
  return min(__clz(h ^ (h >> 31)) - 2, 28);
}

// Blocks per SM that the registers have to allow: as many as spill next to
// nothing (2400^2 damped: three 98 us, four 92, five 88).
template <typename InT, bool D3, bool UNIT> constexpr int fx_blocks_per_sm() {
  if (D3) return std::is_same<InT, double2>::value || !UNIT ? 3 : 4;
  return UNIT ? 5 : 4;
}

template <typename InT, bool RESID, bool D3, bool UNIT>
__global__ void __launch_bounds__(32 * SW, (fx_blocks_per_sm<InT, D3, UNIT>()))
stencil_fx_kernel(const InT* __restrict__ x, double2* __restrict__ y, const double2* __restrict__ f,
                  const int4* __restrict__ gs, const double* __restrict__ a, double omega, double w2,
                  double rho_y, double rho_z, double diag, FxStencil k, int nx, int ny, int nz,
                  int tiles_x, int tiles_y, long in_stride, long out_stride,
                  const int* __restrict__ active, double* __restrict__ partial) {
  pdl_wait();
  using T = FsTile<D3>;
  constexpr int TOP = fs_top(D3, UNIT);
  // whether points are checked for small terms, and not the tile for small values
  constexpr bool CHECK = std::is_same<InT, double2>::value || !UNIT;
  extern __shared__ CLong tile[];  // [RZ][RY][32]
  __shared__ int red[CHECK ? 2 : 3][SW];
  const int b = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0);
  double nrm = 0.0;
  if (!active || active[b]) {
    const unsigned t = blockIdx.x, r = t / unsigned(tiles_x);
    const int x0 = int(t - r * unsigned(tiles_x)) * 30;
    const int bz = int(r / unsigned(tiles_y));
    const int y0 = int(r - unsigned(bz) * unsigned(tiles_y)) * T::TY, z0 = bz * T::TZ;
    const bool out = lane >= 1 && lane <= 30 && x0 - 1 + lane < nx;
    // periodic indices; those that only unused points need are any valid one
    auto wrap = [](int i, int n) {
      i = i < 0 ? n - 1 : i;
      return i >= n ? (i - n < n ? i - n : 0) : i;
    };
    const int cx = wrap(x0 - 1 + lane, nx);
    const InT* xb = x + b * in_stride;
    // points are counted in 32 bits (a right-hand side has less than 2^31)
    auto point = [&](int q) {  // q-th row of the tile with its halo
      const int rz = D3 ? q / T::RY : 0, ry = D3 ? q - rz * T::RY : q;
      return unsigned(((D3 ? wrap(z0 - 1 + rz, nz) * ny : 0) + wrap(y0 - 1 + ry, ny)) * nx + cx);
    };
    // medium data of the warp's next output row
    unsigned on = 0;
    bool sn = false;
    int4 Gn = make_int4(0, 0, 0, 0);
    double aa = 0.0;
    auto fetch = [&](int q) {
      const int qz = D3 ? q / T::TY : 0, qy = D3 ? q - qz * T::TY : q;
      sn = y0 + qy < ny && (!D3 || z0 + qz < nz);
      on = ((D3 ? unsigned(z0 + qz) * unsigned(ny) : 0u) + unsigned(y0 + qy)) * unsigned(nx) + unsigned(cx);
      if (sn && out) {
        Gn = gs[on];
        if (a) aa = a[on];
      }
    };
    InT v[T::PER];
    int mx = 0, my = 0;  // largest magnitudes of the real and the imaginary parts
    unsigned least = ~0u;  // smallest magnitude but zeros, less one
#pragma unroll
    for (int i = 0; i < T::PER; ++i)
      if (warp + i * SW < T::ROWS) v[i] = xb[point(warp + i * SW)];
#pragma unroll
    for (int i = 0; i < T::PER; ++i)
      if (warp + i * SW < T::ROWS) {
        mx = max(mx, mag_bits(v[i].x));
        my = max(my, mag_bits(v[i].y));
        if (!CHECK) least = min(least, min(unsigned(mag_bits(v[i].x)) - 1u, unsigned(mag_bits(v[i].y)) - 1u));
      }
    fetch(warp);
    mx = __reduce_max_sync(0xffffffffu, mx);
    my = __reduce_max_sync(0xffffffffu, my);
    if (!CHECK) least = __reduce_min_sync(0xffffffffu, least);
    if (lane == 0) {
      red[0][warp] = mx;
      red[1][warp] = my;
      if (!CHECK) red[2][warp] = int(least);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SW; ++i) {
      mx = max(mx, red[0][i]);
      my = max(my, red[1][i]);
      if (!CHECK) least = min(least, unsigned(red[2][i]));
    }
    const int E = mag_exp<InT>(max(mx, my));
    const bool fx = E >= FS_EMIN<InT> && E < 1920 &&
                    (CHECK || int((least + 1u) >> 23) >= (max(mx, my) >> 23) - 24);
    if (fx) {
#pragma unroll
      for (int i = 0; i < T::PER; ++i)
        if (warp + i * SW < T::ROWS)
          tile[(warp + i * SW) * 32 + lane] = CLong{to_fs<TOP>(v[i].x, E), to_fs<TOP>(v[i].y, E)};
    }
    __syncthreads();
    const int ke = E + k.k_out;
    double2* yb = y + b * out_stride;
    const double2* fb = RESID ? f + b * out_stride : nullptr;
    // rows that the FP64 formula does: bit i for the warp's i-th
    unsigned again = fx ? 0u : ~0u;
    // what the magnitudes of a component's terms (high words) have to add up
    // to; a component that is zero in the whole tile is exact
    constexpr int LOW = (UNIT ? (D3 ? 6 : 4) : 1) << (52 - 32);
    const int low_x = mx ? LOW : 0, low_y = my ? LOW : 0;
    if (fx) {
#pragma unroll 4
      for (int q = warp; q < T::TY * T::TZ; q += SW) {
        const unsigned o = on;
        const int4 G = Gn;
        const double an = aa;
        if (!sn) break;  // rows past the grid: so are the warp's later ones
        if (q + SW < T::TY * T::TZ) fetch(q + SW);
        const int qz = D3 ? q / T::TY : 0, qy = D3 ? q - qz * T::TY : q;
        const CLong* c = tile + ((D3 ? qz + 1 : 0) * T::RY + qy + 1) * 32 + lane;
        const CLong v0 = c[0];
        CLong L;
        bool small = false;  // a component of the sum has small terms
        {
          const CLong l = c[-1], r = c[1], d = c[-32], u = c[32];
          const CLong n = D3 ? c[-32 * T::RY] : CLong{0, 0}, f = D3 ? c[32 * T::RY] : CLong{0, 0};
          int sx, sy;
          if (UNIT) {
            L = (l + r) + (d + u);
            if (D3) L = L + (n + f);
            L.x -= (D3 ? 6 : 4) * v0.x;
            L.y -= (D3 ? 6 : 4) * v0.y;
            sx = size(l.x, r.x) + size(d.x, u.x) + (D3 ? 6 : 4) * abs(high(v0.x));
            sy = size(l.y, r.y) + size(d.y, u.y) + (D3 ? 6 : 4) * abs(high(v0.y));
            if (D3) {
              sx += size(n.x, f.x);
              sy += size(n.y, f.y);
            }
          } else {
            // weights in units of 2^ke (host), result in units of 2^(59 + ke)
            // (the lowest products are below 2^62 each: four fit unsigned)
            long long hx = 0, mx = 0, hy = 0, my = 0;
            unsigned long long lx = 0, ly = 0;
            auto term = [&](const CLong& s, int kh, int kl) {
              const int xh = lim_h(s.x), xl = lim_l(s.x), yh = lim_h(s.y), yl = lim_l(s.y);
              hx += mul_w(kh, xh);
              mx += mul_w(kh, xl) + mul_w(kl, xh);
              lx += (unsigned long long)mul_w(kl, xl);
              hy += mul_w(kh, yh);
              my += mul_w(kh, yl) + mul_w(kl, yh);
              ly += (unsigned long long)mul_w(kl, yl);
            };
            sx = abs(high(v0.x));
            sy = abs(high(v0.y));
            auto pair = [&](const CLong& p, const CLong& q, int i) {
              term(p + q, k.kh[i], k.kl[i]);
              sx += size(p.x, q.x) >> k.share[i];
              sy += size(p.y, q.y) >> k.share[i];
            };
            pair(l, r, 0);
            pair(d, u, 1);
            if (D3) pair(n, f, 2);
            term(v0, k.kh[3], k.kl[3]);
            mx += (long long)(lx >> 31) + (1ll << 27);
            my += (long long)(ly >> 31) + (1ll << 27);
            L = CLong{(hx << 3) + (mx >> 28), (hy << 3) + (my >> 28)};
          }
          if (CHECK) small = sx < low_x || sy < low_y;
        }
        // g L + omega^2 v
        const int ah = lim_h(L.x), al = lim_l(L.x), bh = lim_h(L.y), bl = lim_l(L.y);
        const int vxh = lim_h(v0.x), vxl = lim_l(v0.x), vyh = lim_h(v0.y), vyl = lim_l(v0.y);
        const int nz_ = -G.z, nw = -G.w;
        const long long rh = mad_w(k.w2h, vxh, mad_w(nz_, bh, mul_w(G.x, ah)));
        const long long ih = mad_w(k.w2h, vyh, mad_w(G.z, ah, mul_w(G.x, bh)));
        // CHECK: rounded at the last bit kept; |g L + omega^2 v| < 2^121.7, 62.7 bits left
        constexpr long long half = CHECK ? 1ll << (30 - FS_KEEP) : 0;
        long long rm = (mad_w(nw, bl, mul_w(G.y, al)) >> 31) + (mad_w(k.w2l, vxl, half << 31) >> 31);
        long long im = (mad_w(G.w, al, mul_w(G.y, bl)) >> 31) + (mad_w(k.w2l, vyl, half << 31) >> 31);
        rm = mad_w(G.x, al, mad_w(G.y, ah, mad_w(nz_, bl, mad_w(nw, bh, mad_w(k.w2h, vxl, mad_w(k.w2l, vxh, rm))))));
        im = mad_w(G.x, bl, mad_w(G.y, bh, mad_w(G.z, al, mad_w(G.w, ah, mad_w(k.w2h, vyl, mad_w(k.w2l, vyh, im))))));
        double yr, yi;
        if (CHECK) {
          yr = fx_to((rh << FS_KEEP) + (rm >> (31 - FS_KEEP)), ke);
          yi = fx_to((ih << FS_KEEP) + (im >> (31 - FS_KEEP)), ke);
        } else {
          const int kr = keep_bits(rh), ki = keep_bits(ih);
          yr = fx_to((rh << kr) + (rm >> (31 - kr)), ke + FS_KEEP - kr);
          yi = fx_to((ih << ki) + (im >> (31 - ki)), ke + FS_KEEP - ki);
        }
        const bool redo = CHECK && __any_sync(0xffffffffu, out && small);
        again |= unsigned(redo) << (q / SW);
        if (redo && q == warp) {  // a steep field: the other rows would be too
          again = ~0u;
          break;
        }
        if (a) {
          const double2 m = ld2(xb, o);
          const double wa = omega * an;
          yr = fma(-wa, m.y, yr);
          yi = fma(wa, m.x, yi);
        }
        if (RESID) {
          const double2 fv = fb[o];
          yr = fv.x - yr;
          yi = fv.y - yi;
          if (out && !redo) nrm = fma(yr, yr, fma(yi, yi, nrm));
        }
        if (out && !redo) yb[o] = make_double2(yr, yi);
      }
    }
#pragma unroll 1
    for (int q = warp; again && q < T::TY * T::TZ; q += SW, again >>= 1) {
      if (!(again & 1u)) continue;
      const int qz = D3 ? q / T::TY : 0, qy = D3 ? q - qz * T::TY : q;
      if (!(y0 + qy < ny && (!D3 || z0 + qz < nz))) break;
      const int own = ((D3 ? qz + 1 : 0) * T::RY) + qy + 1;  // row of the tile
      const unsigned o = point(own);
      const double2 m = ld2(xb, o), dn = ld2(xb, point(own - 1)), up = ld2(xb, point(own + 1));
      double2 zd = make_double2(0.0, 0.0), zu = zd;
      if (D3) {
        zd = ld2(xb, point(own - T::RY));
        zu = ld2(xb, point(own + T::RY));
      }
      // a row of zeros with neighbours of zeros gives zeros
      const long long any = bits(m) | bits(dn) | bits(up) | bits(zd) | bits(zu);
      const bool zero = !__any_sync(0xffffffffu, any != 0);
      double sr = 0.0, si = 0.0;
      if (!zero) {
        const double2 l = make_double2(__shfl_up_sync(0xffffffffu, m.x, 1), __shfl_up_sync(0xffffffffu, m.y, 1));
        const double2 rr = make_double2(__shfl_down_sync(0xffffffffu, m.x, 1), __shfl_down_sync(0xffffffffu, m.y, 1));
        sr = fma(rho_y, dn.x + up.x, l.x + rr.x);
        si = fma(rho_y, dn.y + up.y, l.y + rr.y);
        if (D3) {
          sr = fma(rho_z, zd.x + zu.x, sr);
          si = fma(rho_z, zd.y + zu.y, si);
        }
        sr = fma(-diag, m.x, sr);
        si = fma(-diag, m.y, si);
      }
      if (!out) continue;
      double yr = 0.0, yi = 0.0;
      if (!zero) {
        const int4 G = gs[o];
        const double gx = fx_to((static_cast<long long>(G.x) << 31) + G.y, k.uq);
        const double gy = fx_to((static_cast<long long>(G.z) << 31) + G.w, k.uq);
        yr = fma(gx, sr, fma(-gy, si, w2 * m.x));
        yi = fma(gx, si, fma(gy, sr, w2 * m.y));
        if (a) {
          const double wa = omega * a[o];
          yr = fma(-wa, m.y, yr);
          yi = fma(wa, m.x, yi);
        }
      }
      if (RESID) {
        const double2 fv = fb[o];
        yr = fv.x - yr;
        yi = fv.y - yi;
        nrm = fma(yr, yr, fma(yi, yi, nrm));
      }
      yb[o] = make_double2(yr, yi);
    }
  }
  if (RESID) {
    __shared__ double sh[SW];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nrm += __shfl_down_sync(0xffffffffu, nrm, o);
    if (lane == 0) sh[warp] = nrm;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = sh[0];
      for (int i = 1; i < SW; ++i) s += sh[i];
      partial[long(b) * gridDim.x + blockIdx.x] = s;
    }
  }
}

}  // namespace

namespace {
struct StencilConsts {
  double w2, rho_y, rho_z, diag;
};
StencilConsts stencil_consts(const hz_medium* m) {
  StencilConsts k;
  k.w2 = m->omega * m->omega;
  k.rho_y = m->inv_h2[1] / m->inv_h2[0];
  k.rho_z = m->dim == 3 ? m->inv_h2[2] / m->inv_h2[0] : 0.0;
  k.diag = 2.0 * (1.0 + k.rho_y + k.rho_z);
  return k;
}

// v = hi 2^31 + lo, 0 <= lo < 2^31
void limbs31(long long v, int* hi, int* lo) {
  *hi = int(v >> 31);
  *lo = int(v & 0x7fffffff);
}

bool unit_spacing(const StencilConsts& c, int dim) {
  return c.rho_y == 1.0 && (dim == 2 || c.rho_z == 1.0);
}

// exponent of the unit of the axis weights: diag < 2^(60 + ke)
int weight_unit(const StencilConsts& c) { return std::ilogb(c.diag) - 59; }

// Integer constants of the medium for the unit q_g = 2^uq of g; false when
// omega^2 would keep fewer than 53 bits.
bool fx_consts(const StencilConsts& c, int dim, int uq, FxStencil* k) {
  const bool unit = unit_spacing(c, dim);
  const int ul = unit ? 0 : 59 + weight_unit(c);  // unit of the neighbour sums, over that of x
  const double w = std::ldexp(c.w2, -(uq + ul));
  if (!(w >= 4503599627370496.0 && w < 1152921504606846976.0)) return false;  // [2^52, 2^60)
  limbs31(std::llrint(w), &k->w2h, &k->w2l);
  if (!unit) {
    const double kap[4] = {1.0, c.rho_y, c.rho_z, -c.diag};
    for (int i = 0; i < 4; ++i)
      limbs31(std::llrint(std::ldexp(kap[i], -weight_unit(c))), &k->kh[i], &k->kl[i]);
    for (int i = 0; i < dim; ++i) k->share[i] = std::min(31, -std::ilogb(kap[i] / c.diag));
  }
  k->uq = uq;
  // a 31 x 31 bit product's high part counts 2^62 units; the sums keep FS_KEEP more bits
  k->k_out = 62 - FS_KEEP + uq + ul - fs_top(dim == 3, unit) - 1023;
  return true;
}

template <bool D3>
long fx_blocks(const hz_medium* m) {
  using T = FsTile<D3>;
  return long((m->nx + 29) / 30) * ((m->ny + T::TY - 1) / T::TY) * ((m->nz + T::TZ - 1) / T::TZ);
}

template <typename InT, bool RESID, bool D3, bool UNIT>
hz_status launch_fx(const hz_medium* m, const StencilConsts& c, const void* x, long in_stride,
                    const double2* f, double2* y, long out_stride, int nrhs, const int* active,
                    double* partial, cudaStream_t st) {
  using T = FsTile<D3>;
  FxStencil k{};
  fx_consts(c, m->dim, m->gunit, &k);
  auto kernel = stencil_fx_kernel<InT, RESID, D3, UNIT>;
  HZ_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(T::SMEM)));
  HZ_CUDA(launch_pdl(kernel, dim3(unsigned(fx_blocks<D3>(m)), unsigned(nrhs)), dim3(32 * SW),
                     T::SMEM, st, static_cast<const InT*>(x), y, f,
                     reinterpret_cast<const int4*>(m->gamma2), m->a, m->omega, c.w2, c.rho_y,
                     c.rho_z, c.diag, k, m->nx, m->ny, m->nz, (m->nx + 29) / 30,
                     (m->ny + T::TY - 1) / T::TY, in_stride, out_stride, active, partial));
  return HZ_OK;
}

template <typename InT, bool RESID>
hz_status launch_any(const hz_medium* m, const void* x, long in_stride, const double2* f,
                     double2* y, long out_stride, int nrhs, const int* active, double* partial,
                     cudaStream_t st) {
  const StencilConsts c = stencil_consts(m);
  if (m->gfix) {
    auto go = m->dim == 2 ? (unit_spacing(c, 2) ? launch_fx<InT, RESID, false, true>
                                                : launch_fx<InT, RESID, false, false>)
                          : (unit_spacing(c, 3) ? launch_fx<InT, RESID, true, true>
                                                : launch_fx<InT, RESID, true, false>);
    return go(m, c, x, in_stride, f, y, out_stride, nrhs, active, partial, st);
  }
  HZ_CUDA(launch_pdl(stencil_kernel<InT, RESID>, dim3(unsigned(stencil_blocks(m)), unsigned(nrhs)),
                     dim3(ST_THREADS), 0, st, static_cast<const InT*>(x), y, f, m->gamma2, m->a,
                     m->omega, c.w2, c.rho_y, c.rho_z, c.diag, m->nx, m->ny, m->nz, m->n, in_stride,
                     out_stride, active, partial));
  return HZ_OK;
}

// g in place as integers of the medium's unit, in limbs of 31 bits
__global__ void gfix_kernel(double2* __restrict__ g, long n, double inv_qg) {
  const long i = blockIdx.x * long(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const double2 v = g[i];
  const long long a = __double2ll_rn(v.x * inv_qg), b = __double2ll_rn(v.y * inv_qg);
  reinterpret_cast<int4*>(g)[i] = make_int4(lim_h(a), lim_l(a), lim_h(b), lim_l(b));
}

}  // namespace

// Chooses the operator's form for a medium whose gamma2 has been written, and
// brings gamma2 into it.  The integer form is for grids that fill the GPU
// (n >= 2^17) and needs |g| within 2^6 of the largest and omega^2 with 53
// bits in the same unit (any medium at 4 to 60 points per wavelength does).
hz_status stencil_prepare(hz_medium* m, double zeta_max, cudaStream_t st) {
  m->gfix = false;
  if (m->n < (1l << 17)) return HZ_OK;
  const StencilConsts c = stencil_consts(m);
  const double ih2 = m->inv_h2[0];
  const double gmax = m->c_max * m->c_max * (1.0 + zeta_max * zeta_max) * ih2;
  const double gmin = m->c_min * m->c_min * ih2;
  if (!(gmax < 1e30 && gmin > 1e-30) || gmax > 64.0 * gmin) return HZ_OK;
  // |g| < 2^eg = 2^60 units; a larger omega^2 coarsens the unit
  const int uq = std::max(std::ilogb(gmax), std::ilogb(c.w2)) + 1 - 60;
  FxStencil k{};
  if (std::ldexp(gmin, -uq) < 4503599627370496.0 || !fx_consts(c, m->dim, uq, &k)) return HZ_OK;
  // omega^2 x is one more term, whose rounding the others have to cover
  if (c.w2 > c.diag * gmin) return HZ_OK;
  gfix_kernel<<<unsigned((m->n + 255) / 256), 256, 0, st>>>(m->gamma2, m->n, std::ldexp(1.0, -uq));
  count_launches(1);
  HZ_CUDA(cudaGetLastError());
  m->gunit = uq;
  m->gfix = true;
  return HZ_OK;
}

int stencil_blocks(const hz_medium* m) {
  if (m->gfix) return int(m->dim == 2 ? fx_blocks<false>(m) : fx_blocks<true>(m));
  return int((m->n + ST_THREADS - 1) / ST_THREADS);
}

hz_status launch_stencil(const hz_medium* m, int in_prec, const void* x, long in_stride,
                         double2* y, long out_stride, int nrhs, const int* active,
                         cudaStream_t st) {
  if (in_prec == 0)
    HZ_TRY((launch_any<double2, false>(m, x, in_stride, nullptr, y, out_stride, nrhs, active,
                                       nullptr, st)));
  else
    HZ_TRY((launch_any<float2, false>(m, x, in_stride, nullptr, y, out_stride, nrhs, active,
                                      nullptr, st)));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_residual(const hz_medium* m, const double2* u, const double2* f, double2* r,
                          long stride, int nrhs, const int* active, double* partial,
                          cudaStream_t st) {
  HZ_TRY((launch_any<double2, true>(m, u, stride, f, r, stride, nrhs, active, partial, st)));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

}  // namespace hz
