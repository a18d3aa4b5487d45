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
// binary exponent E, the largest of them: v = x 2^(FS_TOP + 1023 - E),
// |v| < 2^57, so a value within a factor 2^4 of the largest of its
// neighbourhood keeps all its bits.  Neighbour sums are exact; g =
// gamma^2 / h_x^2 and omega^2 are integers below 2^60 of a unit for the whole
// medium, and the products of 31-bit limbs are exact up to the last shift.  A
// tile whose values leave the range of normal numbers, or are all zero, takes
// the FP64 formula.  It is bound by the integer multiply-add pipe, which also
// takes the 64-bit additions (62 lanes per clock and SM, about 130 a point in
// 2D).  2400^2 damped, c128 input: 180 -> 82 us (3.9 TB/s); 192^3, c64 input:
// 277 -> 115 us (2.5 TB/s).
// ---------------------------------------------------------------------------
constexpr int SW = 8;          // warps per block
constexpr int FS_TOP = 56;
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
  int k_out;                    // result = T 2^(E + k_out)
  double qg;                    // unit of g
};

__device__ __forceinline__ int exp_bits(double2 z) {
  return max((__double2hiint(z.x) >> 20) & 0x7ff, (__double2hiint(z.y) >> 20) & 0x7ff);
}
__device__ __forceinline__ int exp_bits(float2 z) {
  const int e = max((__float_as_int(z.x) >> 23) & 0xff, (__float_as_int(z.y) >> 23) & 0xff);
  return e == 0 ? 0 : (e == 0xff ? 0x7ff : e + 896);
}
__device__ __forceinline__ long long shr(long long v, int n) {  // n > 63: zero
  asm("shr.u64 %0, %0, %1;" : "+l"(v) : "r"(n));
  return v;
}
// Truncated fixed-point value for the exponent E >= exponent of x.  Zeros and
// subnormals need no test: with E at least FS_EMIN their shift is past the
// last bit.
template <typename T> __device__ constexpr int FS_EMIN = 128;
template <> __device__ constexpr int FS_EMIN<float2> = 896 + 60;
__device__ __forceinline__ long long to_fs(double x, int E) {
  const int hi = __double2hiint(x);
  const unsigned lo = unsigned(__double2loint(x));
  const int ex = (hi >> 20) & 0x7ff;
  const unsigned mh = unsigned((hi & 0xfffff) | 0x100000);
  const unsigned th = __funnelshift_l(lo, mh, 4), tl = lo << 4;
  const long long t = shr(static_cast<long long>(static_cast<unsigned long long>(th) << 32 | tl), E - ex);
  const long long sg = hi >> 31;
  return (t ^ sg) - sg;
}
__device__ __forceinline__ long long to_fs(float x, int E) {
  const int u = __float_as_int(x);
  const int ex = (u >> 23) & 0xff;
  const int sg = u >> 31;
  const int m = ((u & 0x7fffff) | 0x800000) << 1;
  // magnitude first: an arithmetic shift of a negative value would floor
  const long long t = shr(static_cast<long long>(static_cast<unsigned long long>(unsigned(m)) << 32), E - 896 - ex);
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
__device__ __forceinline__ CLong operator+(const CLong& p, const CLong& q) {
  return CLong{p.x + q.x, p.y + q.y};
}

template <typename InT, bool RESID, bool D3, bool UNIT>
__global__ void __launch_bounds__(32 * SW)
stencil_fx_kernel(const InT* __restrict__ x, double2* __restrict__ y, const double2* __restrict__ f,
                  const int4* __restrict__ gs, const double* __restrict__ a, double omega, double w2,
                  double rho_y, double rho_z, double diag, FxStencil k, int nx, int ny, int nz,
                  int tiles_x, int tiles_y, long in_stride, long out_stride,
                  const int* __restrict__ active, double* __restrict__ partial) {
  pdl_wait();
  using T = FsTile<D3>;
  extern __shared__ CLong tile[];  // [RZ][RY][32]
  __shared__ int red[SW];
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
    int E = 0;
#pragma unroll
    for (int i = 0; i < T::PER; ++i)
      if (warp + i * SW < T::ROWS) v[i] = xb[point(warp + i * SW)];
#pragma unroll
    for (int i = 0; i < T::PER; ++i)
      if (warp + i * SW < T::ROWS) E = max(E, exp_bits(v[i]));
    fetch(warp);
    E = __reduce_max_sync(0xffffffffu, E);
    if (lane == 0) red[warp] = E;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SW; ++i) E = max(E, red[i]);
    const bool fx = E >= FS_EMIN<InT> && E < 1920;
#pragma unroll
    for (int i = 0; i < T::PER; ++i) {
      if (warp + i * SW < T::ROWS) {
        CLong s;
        if (fx) {
          s = CLong{to_fs(v[i].x, E), to_fs(v[i].y, E)};
        } else {
          const double2 d = ld2(&v[i], 0);
          s = CLong{__double_as_longlong(d.x), __double_as_longlong(d.y)};
        }
        tile[(warp + i * SW) * 32 + lane] = s;
      }
    }
    __syncthreads();
    const int ke = E + k.k_out;
    double2* yb = y + b * out_stride;
    const double2* fb = RESID ? f + b * out_stride : nullptr;
    auto rows = [&](auto fxc) {
    constexpr bool FX = decltype(fxc)::value;
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
      double yr, yi;
      if constexpr (FX) {
        CLong L;
        if (UNIT) {
          L = (c[-1] + c[1]) + (c[-32] + c[32]);
          if (D3) L = L + (c[-32 * T::RY] + c[32 * T::RY]);
          L.x -= (D3 ? 6 : 4) * v0.x;
          L.y -= (D3 ? 6 : 4) * v0.y;
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
          term(c[-1] + c[1], k.kh[0], k.kl[0]);
          term(c[-32] + c[32], k.kh[1], k.kl[1]);
          if (D3) term(c[-32 * T::RY] + c[32 * T::RY], k.kh[2], k.kl[2]);
          term(v0, k.kh[3], k.kl[3]);
          mx += (long long)(lx >> 31);
          my += (long long)(ly >> 31);
          L = CLong{(hx << 3) + (mx >> 28), (hy << 3) + (my >> 28)};
        }
        // g L + omega^2 v
        const int ah = lim_h(L.x), al = lim_l(L.x), bh = lim_h(L.y), bl = lim_l(L.y);
        const int vxh = lim_h(v0.x), vxl = lim_l(v0.x), vyh = lim_h(v0.y), vyl = lim_l(v0.y);
        const int nz_ = -G.z, nw = -G.w;
        const long long rh = mad_w(k.w2h, vxh, mad_w(nz_, bh, mul_w(G.x, ah)));
        const long long ih = mad_w(k.w2h, vyh, mad_w(G.z, ah, mul_w(G.x, bh)));
        // rounded at the last bit kept: |g L + omega^2 v| < 2^121.2, 62.2 bits left
        constexpr long long half = 1ll << (30 - FS_KEEP);
        long long rm = (mad_w(nw, bl, mul_w(G.y, al)) >> 31) + (mad_w(k.w2l, vxl, half << 31) >> 31);
        long long im = (mad_w(G.w, al, mul_w(G.y, bl)) >> 31) + (mad_w(k.w2l, vyl, half << 31) >> 31);
        rm = mad_w(G.x, al, mad_w(G.y, ah, mad_w(nz_, bl, mad_w(nw, bh, mad_w(k.w2h, vxl, mad_w(k.w2l, vxh, rm))))));
        im = mad_w(G.x, bl, mad_w(G.y, bh, mad_w(G.z, al, mad_w(G.w, ah, mad_w(k.w2h, vyl, mad_w(k.w2l, vyh, im))))));
        yr = fx_to((rh << FS_KEEP) + (rm >> (31 - FS_KEEP)), ke);
        yi = fx_to((ih << FS_KEEP) + (im >> (31 - FS_KEEP)), ke);
      } else {
        auto d = [&](int i) {
          return make_double2(__longlong_as_double(c[i].x), __longlong_as_double(c[i].y));
        };
        const double2 l = d(-1), rr = d(1), dn = d(-32), up = d(32), m = d(0);
        double sr = fma(rho_y, dn.x + up.x, l.x + rr.x), si = fma(rho_y, dn.y + up.y, l.y + rr.y);
        if (D3) {
          const double2 zd = d(-32 * T::RY), zu = d(32 * T::RY);
          sr = fma(rho_z, zd.x + zu.x, sr);
          si = fma(rho_z, zd.y + zu.y, si);
        }
        sr = fma(-diag, m.x, sr);
        si = fma(-diag, m.y, si);
        const double gx = fma(double(G.x), 2147483648.0, double(G.y)) * k.qg;
        const double gy = fma(double(G.z), 2147483648.0, double(G.w)) * k.qg;
        yr = fma(gx, sr, fma(-gy, si, w2 * m.x));
        yi = fma(gx, si, fma(gy, sr, w2 * m.y));
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
        if (out) nrm = fma(yr, yr, fma(yi, yi, nrm));
      }
      if (out) yb[o] = make_double2(yr, yi);
    }
    };
    if (fx) rows(std::true_type{});
    else rows(std::false_type{});
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
  }
  k->qg = std::ldexp(1.0, uq);
  // a 31 x 31 bit product's high part counts 2^62 units; the sums keep FS_KEEP more bits
  k->k_out = 62 - FS_KEEP + uq + ul - FS_TOP - 1023;
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
