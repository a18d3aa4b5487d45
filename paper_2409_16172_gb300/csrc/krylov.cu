// FP64 Krylov kernels of restarted (F)GMRES (Section 5, "GMRES
// implementation"): CGS2 Arnoldi (classical Gram-Schmidt applied twice),
// complex Givens rotations on the Hessenberg column, the solution update and
// the deterministic reductions they need.
//
// The basis is stored unnormalised: the true basis vector is
// v_i = sigma_i * V_i, sigma_i = 1 / ||w_i||.  Then
//   h_i   = <v_i, w> = sigma_i * sum conj(V_i) w          (dots)
//   w    -= sum_i h_i v_i = sum_i (sigma_i h_i) V_i         (update)
// so no pass ever rescales a stored vector.
// Layout: V[(i * ldb + b) * n + p] for basis vector i, right-hand side b, 16
// bytes a point; the current vector w is FP64.  Two forms of the basis:
//   block fixed point (fixed.cuh), where the preconditioner's transforms make
//     the vectors: a transform's rounding errors are of one size all over the
//     grid, so that a unit of 2^-54 of the largest of 128 neighbours costs
//     nothing (complex128 solves of 16 steps: solution and Hessenberg entries
//     as close to extended precision as in FP64)
//   FP64, for the unpreconditioned method: its vectors come from the operator
//     alone, which keeps the bits of values however small they are beside
//     their neighbours (a point source's field 1e-8 of its largest value:
//     relative error 2e-15 in FP64, 2e-6 in block fixed point; 128^2, 40 steps)
#include <math.h>

#include <algorithm>

#include "fixed.cuh"
#include "hz_internal.h"
#include "kernels.h"
#include "recip.cuh"

namespace hz {
namespace {

constexpr int KT = 256;   // threads per block

// fixed-order block sum of NV doubles per thread; result in sh[0..NV-1]
template <int NV, int NT = KT>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* sh) {
#pragma unroll
  for (int c = 0; c < NV; ++c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_down_sync(0xffffffffu, v[c], o);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
#pragma unroll
    for (int c = 0; c < NV; ++c) sh[warp * NV + c] = v[c];
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double s = 0.0;
    for (int w = 0; w < NT / 32; ++w) s += sh[w * NV + threadIdx.x];
    sh[NT / 32 * NV + threadIdx.x] = s;
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Gram-Schmidt kernels over the basis in block fixed-point form (fixed.cuh).
//
// What bounds them: past about 16 vectors dots and update run at the basis in
// HBM, 16 bytes a point and vector; before that, and in the kernel that does
// both, at the latency of the tile's phases with 8 to 16 warps per SM.  2^24
// points: dots 6.0 TB/s of basis at j = 20 and 39, update 4.9 and 5.4, update
// and dots in one 1.52 and 3.05 ms; in FP64 the same sums were bound by the
// FP64 pipe at 2.1-2.5 TB/s.  A 256^3 Arnoldi step (j = 17 on average) spends
// 3.2 ms here instead of 9.2.  A block takes one tile of FX_TILE points at a
// time.  Its basis rows (one row: the tile's 128 points of one vector, 2 KB)
// come through shared memory by cp.async, so that the loads in flight do not
// cost registers and run ahead over tile boundaries.
//   update side  a thread owns a point and runs over the vectors
//   dot side     the vectors are dealt to the half warps; a lane takes CG_U
//                points, and the integer sums of CG_NB vectors are folded
//                across the lanes together before they become doubles
// ---------------------------------------------------------------------------
enum CgMode {
  CG_DOTS = 0,     // partial sums of conj(V_i) w, i <= j
  CG_UPDATE_DOTS,  // w -= sum_i sigma_i^2 S[b][i] V_i, then the sums of the new w
  CG_UPDATE,       // w -= ..., |w|^2 sums, the new w as basis vector (unless Vnew is null)
  CG_COMBINE       // w = sum_i sigma_i S[b][i] V_i, i < jn[b]
};

constexpr int CT = FX_TILE;               // threads
constexpr int CG_WARPS = CT / 32;
constexpr int CG_HALVES = 2 * CG_WARPS;   // vectors in work at a time on the dot side
constexpr int CG_U = FX_TILE / 16;        // points per lane on the dot side
constexpr int CG_NB = 4;
constexpr int CG_ROWS = 24;               // ring rows when rows only pass through
constexpr int CG_DEPTH = CG_ROWS / CG_HALVES;  // dot side: rows in flight per half warp
constexpr int CG_NU = 4;                       // update side: rows per copy group
constexpr int CG_GROUPS = CG_ROWS / CG_NU;     // and groups in flight
constexpr int CG_MAXROWS = 52;            // ring rows at most (two blocks per SM)
constexpr int CG_FUSED = 44;              // vectors at most in CG_UPDATE_DOTS
constexpr size_t CG_ROW_BYTES = FX_TILE * sizeof(int4);

__device__ __forceinline__ void copy16(int4* dst, const int4* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   unsigned(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// sum over the 16 lanes of a half warp of 4 values per lane; lane l returns
// the sum of value (l >> 2) & 3 (each step sends the half the partner keeps)
__device__ __forceinline__ long long fold4(const long long (&t)[CG_NB], int lane) {
  const bool u8 = lane & 8, u4 = lane & 4;
  long long a = u8 ? t[2] : t[0], b = u8 ? t[3] : t[1];
  a += __shfl_xor_sync(0xffffffffu, u8 ? t[0] : t[2], 8);
  b += __shfl_xor_sync(0xffffffffu, u8 ? t[1] : t[3], 8);
  long long c = u4 ? b : a;
  c += __shfl_xor_sync(0xffffffffu, u4 ? a : b, 4);
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  return c;
}

// per-warp maxima into red; the block's maximum after a barrier
__device__ __forceinline__ void warp_max(int v, int* red) {
  const int m = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
}
__device__ __forceinline__ int max_of(const int* red) {
  int r = red[0];
#pragma unroll
  for (int i = 1; i < CG_WARPS; ++i) r = max(r, red[i]);
  return r;
}

// a coefficient against the exponent E >= its own; one of a zero (or
// subnormal) part, which fx_from's E may not be too small for, by itself
__device__ __forceinline__ int4 coef_limbs(double2 c, int E) {
  int4 r = fx_pack(c, E);
  if (fx_exp(c.x) == 0) r.x = r.y = 0;
  if (fx_exp(c.y) == 0) r.z = r.w = 0;
  return r;
}

// limb sums of conj(v) y (re, and the two halves of im); no sum takes more
// than two products of a point, so that none is a long chain
struct DotAcc {
  long long rh = 0, rx = 0, ry = 0, ph = 0, px = 0, qh = 0, qx = 0;
  __device__ __forceinline__ void add(const int4& v, const int4& y) {
    rh = mad_w(v.x, y.x, rh);
    ph = mad_w(v.x, y.z, ph);
    qh = mad_w(v.z, y.x, qh);
    rx = mad_w(v.y, y.x, rx);
    ry = mad_w(v.w, y.z, ry);
    px = mad_w(v.y, y.z, px);
    qx = mad_w(v.w, y.x, qx);
    rh = mad_w(v.z, y.z, rh);
    rx = mad_w(v.x, y.y, rx);
    ry = mad_w(v.z, y.w, ry);
    px = mad_w(v.x, y.w, px);
    qx = mad_w(v.z, y.y, qx);
  }
  // |hh| <= 2^58 over a lane's CG_U points: the sum over 16 lanes fits
  __device__ __forceinline__ long long re() const { return fx_sum(rh, rx + ry); }
  __device__ __forceinline__ long long im() const { return fx_sum(ph - qh, px - qx); }
};
// limb sums of c v
struct UpdAcc {
  long long rh = 0, rx = 0, ih = 0, ix = 0;
  __device__ __forceinline__ void add(const int4& c, const int4& v) {
    const int nh = -c.z, nl = -c.w;
    rh = mad_w(nh, v.z, mad_w(c.x, v.x, rh));
    ih = mad_w(c.z, v.x, mad_w(c.x, v.z, ih));
    rx = mad_w(nh, v.w, mad_w(nl, v.z, mad_w(c.x, v.y, mad_w(c.y, v.x, rx))));
    ix = mad_w(c.z, v.y, mad_w(c.w, v.x, mad_w(c.x, v.w, mad_w(c.y, v.z, ix))));
  }
  __device__ __forceinline__ void join(const UpdAcc& o) {
    rh += o.rh;
    rx += o.rx;
    ih += o.ih;
    ix += o.ix;
  }
  // |hh| <= 2 (HZ_MAX_RESTART + 1) 2^54 < 2^63
  __device__ __forceinline__ long long re() const { return fx_sum(rh, rx); }
  __device__ __forceinline__ long long im() const { return fx_sum(ih, ix); }
};

template <int MODE>
__global__ void __launch_bounds__(CT, 4)
cgs_kernel(const int4* __restrict__ V, const int* __restrict__ ev, long ldb, long ntiles,
           double2* __restrict__ w, long wstride, long n, int j, int rows,
           const double2* __restrict__ S, int ldS, const double* __restrict__ sigma, int ldsig,
           const int* __restrict__ active, double2* __restrict__ partial, int4* __restrict__ Vnew,
           int* __restrict__ enew) {
  pdl_wait();
  const int b = blockIdx.y;
  if (MODE == CG_COMBINE) {
    j = active[b] - 1;  // jn
  } else if (!active[b]) {
    return;
  }
  constexpr bool UPD = MODE != CG_DOTS, DOT = MODE <= CG_UPDATE_DOTS;
  extern __shared__ int4 ring[];  // [rows][FX_TILE]
  __shared__ int4 cl[UPD ? HZ_MAX_RESTART : 1];
  __shared__ int4 wl[DOT ? FX_TILE : 1];
  __shared__ double2 sacc[DOT ? HZ_MAX_RESTART : 1];
  __shared__ int redF[CG_WARPS], redw[CG_WARPS];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int hw = tid >> 4, hl = tid & 15;  // half warp, lane of it
  double2* wb = w + b * wstride;
  const int4* Vb = V + long(b) * n;
  const int* eb = ev + long(b) * ntiles;
  const long vs = ldb * n, es = ldb * ntiles;  // strides between basis vectors
  const long dt = gridDim.x;
  long tile = blockIdx.x;

  // ---- update side: coefficients of a tile, as integers of one common unit
  double2 ci = make_double2(0.0, 0.0);  // thread i holds the coefficient of vector i
  if (UPD && tid <= j) {
    const double s = sigma[long(tid) * ldsig + b];
    const double2 h = S[long(b) * ldS + tid];
    const double c = MODE == CG_COMBINE ? s : s * s;
    ci = make_double2(c * h.x, c * h.y);
  }
  const int ec = fx_exp(ci);
  auto tile_exp = [&](long t) { return UPD && tid <= j && t < ntiles ? eb[tid * es + t] : 0; };
  const int e0 = tile_exp(tile);
  int F = 0;
  if (DOT)
    for (int i = tid; i <= j; i += CT) sacc[i] = make_double2(0.0, 0.0);

  // ---- copies into the ring
  long qt = tile;  // next to copy: tile qt, row (group) qr of the thread's
  int qr = 0, qs = 0, rs = 0;
  // CG_DOTS: the half warp's rows i = hw, hw + 8, ...; a lane copies the
  // points that it reads
  const int nr = (j - 2 * warp) / CG_HALVES + 1;  // of the warp's first half (its second: may be one less)
  auto copy_row = [&] {
    if (2 * warp <= j && qt < ntiles) {
      const int i = hw + CG_HALVES * qr;
      if (i <= j) {
        int4* d = ring + (hw * CG_DEPTH + qs) * FX_TILE + hl;
        const int m = int(min(n - qt * FX_TILE, long(FX_TILE))) - hl;
        const int4* s = Vb + i * vs + qt * FX_TILE + hl;
        if (m > 16 * (CG_U - 1)) {
#pragma unroll
          for (int u = 0; u < CG_U; ++u) copy16(d + 16 * u, s + 16 * u);
        } else {
#pragma unroll
          for (int u = 0; u < CG_U; ++u)
            if (16 * u < m) copy16(d + 16 * u, s + 16 * u);
        }
      }
      if (++qr == nr) {
        qr = 0;
        qt += dt;
      }
    }
    copy_commit();
    qs = qs + 1 == CG_DEPTH ? 0 : qs + 1;
  };
  // update-only modes: the thread's own point, rows in groups of CG_NU
  const int ng = (j + CG_NU) / CG_NU;  // groups per tile
  auto copy_group = [&] {
    if (qt < ntiles) {
      const long p = qt * FX_TILE + tid;
      if (p < n) {
        int4* d = ring + qs * CG_NU * FX_TILE + tid;
        const int i0 = qr * CG_NU;
        const int4* s = Vb + i0 * vs + p;
#pragma unroll
        for (int u = 0; u < CG_NU; ++u) {
          if (i0 + u <= j) copy16(d + u * FX_TILE, s);
          s += vs;
        }
      }
      if (++qr == ng) {
        qr = 0;
        qt += dt;
      }
    }
    copy_commit();
    qs = qs + 1 == CG_GROUPS ? 0 : qs + 1;
  };
  // CG_UPDATE_DOTS: all rows of a tile stay until its dots are done.  Row i of
  // the block's even tiles is at ring row i, of its odd ones at rows - 1 - i:
  // the first rows - (j + 1) rows of the next tile never meet this one's.
  auto ring_row = [&](bool odd, int i) { return ring + (odd ? rows - 1 - i : i) * FX_TILE; };
  auto copy_part = [&](long t, bool odd, int lo, int hi) {  // rows lo <= i < hi of tile t
    const long p = t * FX_TILE + tid;
    if (t < ntiles && p < n) {
      int4* d = ring_row(odd, lo) + tid;
      const int step = odd ? -FX_TILE : FX_TILE;
      const int4* s = Vb + lo * vs + p;
#pragma unroll 4
      for (int i = lo; i < hi; ++i) {
        copy16(d, s);
        s += vs;
        d += step;
      }
    }
    copy_commit();
  };
  bool odd = false;
  const int ahead = MODE == CG_UPDATE_DOTS ? min(j + 1, rows - (j + 1)) : 0;
  if (MODE == CG_DOTS) {
    for (int k = 0; k < CG_DEPTH; ++k) copy_row();
  } else if (MODE == CG_UPDATE_DOTS) {
    copy_part(tile, odd, 0, ahead);
  } else {
    for (int k = 0; k < CG_GROUPS; ++k) copy_group();
  }
  auto load_w = [&](long t) {
    const long p = t * FX_TILE + tid;
    return MODE != CG_COMBINE && t < ntiles && p < n ? wb[p] : make_double2(0.0, 0.0);
  };
  double2 xn = load_w(tile);
  if (UPD) {
    warp_max(tid <= j ? fx_exp_sum(ec, e0) : 0, redF);
    __syncthreads();
    F = max_of(redF);
    if (tid <= j) cl[tid] = coef_limbs(ci, F - e0);
    __syncthreads();
  }

  double nrm[1] = {0.0};
  for (; tile < ntiles; tile += dt) {
    const long p = tile * FX_TILE + tid;
    const bool in = p < n;
    double2 x = xn;
    xn = load_w(tile + dt);
    const int e1 = tile_exp(tile + dt);
    if (UPD) {
      UpdAcc a, a2;  // alternate rows: shorter chains
      if (MODE == CG_UPDATE_DOTS) {
        // the rest of this tile's rows, and what fits of the next tile's
        copy_part(tile, odd, ahead, j + 1);
        copy_part(tile + dt, !odd, 0, ahead);
        const int4* s = ring_row(odd, 0) + tid;
        const int step = odd ? -FX_TILE : FX_TILE;
        auto rows_of = [&](int lo, int hi) {
          int i = lo;
#pragma unroll 2
          for (; i + 2 <= hi; i += 2) {
            a.add(cl[i], s[0]);
            a2.add(cl[i + 1], s[step]);
            s += 2 * step;
          }
          if (i < hi) {
            a.add(cl[i], s[0]);
            s += step;
          }
        };
        copy_wait<2>();
        rows_of(0, ahead);
        copy_wait<1>();
        rows_of(ahead, j + 1);
      } else {
        for (int k = 0; k < ng; ++k) {
          copy_wait<CG_GROUPS - 1>();
          const int i0 = k * CG_NU;
          const int4* s = ring + rs * CG_NU * FX_TILE + tid;
          if (i0 + CG_NU <= j + 1) {
#pragma unroll
            for (int u = 0; u < CG_NU; ++u) (u & 1 ? a2 : a).add(cl[i0 + u], s[u * FX_TILE]);
          } else {
#pragma unroll
            for (int u = 0; u < CG_NU; ++u)
              if (i0 + u <= j) (u & 1 ? a2 : a).add(cl[i0 + u], s[u * FX_TILE]);
          }
          copy_group();
          rs = rs + 1 == CG_GROUPS ? 0 : rs + 1;
        }
      }
      a.join(a2);
      const int k = fx_unit(F);
      double dr = double_of(a.re(), k), di = double_of(a.im(), k);
      if (F >= FX_BAD) dr = di = fx_nan();
      x = MODE == CG_COMBINE ? make_double2(dr, di) : make_double2(x.x - dr, x.y - di);
      if (in) wb[p] = x;
      else x = make_double2(0.0, 0.0);
      if (MODE == CG_UPDATE) nrm[0] = fma(x.x, x.x, fma(x.y, x.y, nrm[0]));
      warp_max(tid <= j ? fx_exp_sum(ec, e1) : 0, redF);
    }
    if (MODE != CG_COMBINE) warp_max(fx_exp(x), redw);
    __syncthreads();
    if (UPD) {
      F = max_of(redF);
      if (tid <= j) cl[tid] = coef_limbs(ci, F - e1);
    }
    const int E = MODE != CG_COMBINE ? max(max_of(redw), FX_EMIN) : 0;
    if (MODE == CG_UPDATE && Vnew) {
      if (in) Vnew[long(b) * n + p] = fx_pack(x, E);
      if (tid == 0) enew[long(b) * ntiles + tile] = E;
    }
    if (DOT) wl[tid] = fx_pack_floor(x, E);
    __syncthreads();
    if (DOT) {
      int4 wr[CG_U];
#pragma unroll
      for (int u = 0; u < CG_U; ++u) wr[u] = wl[u * 16 + hl];
      for (int i0 = 2 * warp; i0 <= j; i0 += CG_HALVES * CG_NB) {
        const int is = i0 + (hw & 1) + CG_HALVES * ((lane >> 2) & 3);  // whose sum this lane gets
        const int e = is <= j ? eb[is * es + tile] : 0;
        long long tr[CG_NB], ti[CG_NB];
#pragma unroll
        for (int c = 0; c < CG_NB; ++c) {
          tr[c] = ti[c] = 0;
          if (i0 + CG_HALVES * c <= j) {  // the warp's first half; a second half past j sums what is not used
            int r;
            if (MODE == CG_DOTS) {
              copy_wait<CG_DEPTH - 1>();
              r = hw * CG_DEPTH + rs;
            } else {
              r = min(i0 + (hw & 1) + CG_HALVES * c, j);
              if (odd) r = rows - 1 - r;
            }
            const int4* s = ring + r * FX_TILE + hl;
            DotAcc a;
            // points past the end: wr is zero there, whatever the ring holds
#pragma unroll
            for (int u = 0; u < CG_U; ++u) a.add(s[16 * u], wr[u]);
            tr[c] = a.re();
            ti[c] = a.im();
            if (MODE == CG_DOTS) {
              copy_row();
              rs = rs + 1 == CG_DEPTH ? 0 : rs + 1;
            }
          }
        }
        const long long sr = fold4(tr, lane), si = fold4(ti, lane);
        if ((lane & 3) == 0 && is <= j) {
          const int k = fx_unit(E + e);
          double2 s = sacc[is];
          s.x += max(E, e) < FX_INF ? double_of(sr, k) : fx_nan();
          s.y += max(E, e) < FX_INF ? double_of(si, k) : fx_nan();
          sacc[is] = s;
        }
      }
      if (MODE == CG_UPDATE_DOTS) {
        odd = !odd;
        __syncthreads();  // the tile's rows are free
      }
    }
  }
  copy_wait<0>();
  if (DOT) {
    __syncthreads();
    for (int i = tid; i <= j; i += CT)
      partial[(long(b) * (j + 1) + i) * gridDim.x + blockIdx.x] = sacc[i];
  }
  if (MODE == CG_UPDATE) {
    __shared__ double sh[KT / 32 + 1];
    block_sum<1, CT>(nrm, sh);
    if (tid == 0)
      reinterpret_cast<double*>(partial)[long(b) * gridDim.x + blockIdx.x] = sh[CT / 32];
  }
}

// ---------------------------------------------------------------------------
// The same on an FP64 basis, bound by the FP64 pipe (2^24 points: 2.1-2.5 TB/s
// of basis).
// ---------------------------------------------------------------------------
constexpr int VC = 8;  // basis vectors per dots block at most

// Sums of conj(V_i) w for i in [i0, i0 + nv), i0 = blockIdx.z vpc, nv =
// min(vpc, j + 1 - i0), vpc <= VC.  grid (blocks, rhs, chunks).  The next
// point's operands are loaded before the current point's FMAs, so that the
// FP64 pipe does not wait on memory.
__global__ void __launch_bounds__(KT, 2)
dots_kernel(const double2* __restrict__ V, long ldb, const double2* __restrict__ w, long wstride,
            long n, int j, int vpc, const int* __restrict__ active, double2* __restrict__ partial) {
  pdl_wait();
  const int b = blockIdx.y;
  if (!active[b]) return;
  const int i0 = blockIdx.z * vpc;
  const int nv = min(vpc, j + 1 - i0);
  double sum[2 * VC];
#pragma unroll
  for (int c = 0; c < 2 * VC; ++c) sum[c] = 0.0;
  const double2* wb = w + b * wstride;
  const double2* Vb = V + (long(i0) * ldb + b) * n;
  const long vs = ldb * n;
  const long step = long(gridDim.x) * KT;
  long p = long(blockIdx.x) * KT + threadIdx.x;
  double2 x, v[VC];
  if (p < n) {
    x = wb[p];
#pragma unroll
    for (int c = 0; c < VC; ++c)
      if (c < nv) v[c] = Vb[c * vs + p];
  }
  while (p < n) {
    const long q = p + step;
    double2 xn, vn[VC];
    if (q < n) {
      xn = wb[q];
#pragma unroll
      for (int c = 0; c < VC; ++c)
        if (c < nv) vn[c] = Vb[c * vs + q];
    }
#pragma unroll
    for (int c = 0; c < VC; ++c) {
      if (c < nv) {
        sum[2 * c] = fma(v[c].x, x.x, fma(v[c].y, x.y, sum[2 * c]));
        sum[2 * c + 1] = fma(v[c].x, x.y, fma(-v[c].y, x.x, sum[2 * c + 1]));
      }
    }
    p = q;
    x = xn;
#pragma unroll
    for (int c = 0; c < VC; ++c) v[c] = vn[c];
  }
  __shared__ double sh[(KT / 32 + 1) * 2 * VC];
  block_sum<2 * VC>(sum, sh);
  if (threadIdx.x < nv) {
    const double* s = sh + KT / 32 * 2 * VC + 2 * threadIdx.x;
    partial[(long(b) * (j + 1) + i0 + threadIdx.x) * gridDim.x + blockIdx.x] =
        make_double2(s[0], s[1]);
  }
}

// w -= sum_{i <= j} sigma_i^2 S[b][i] V_i; with partial: |w|^2 sums, and the
// new w as basis vector (unless Vnew is null).
__global__ void __launch_bounds__(KT)
update_kernel(const double2* __restrict__ V, long ldb, double2* __restrict__ w, long wstride,
              long n, int j, const double2* __restrict__ S, int ldS, const double* __restrict__ sigma,
              int ldsig, const int* __restrict__ active, double* __restrict__ partial,
              double2* __restrict__ Vnew) {
  pdl_wait();
  const int b = blockIdx.y;
  if (!active[b]) return;
  __shared__ double2 coef[HZ_MAX_RESTART];
  for (int i = threadIdx.x; i <= j; i += KT) {
    const double s = sigma[long(i) * ldsig + b];
    const double2 h = S[long(b) * ldS + i];
    coef[i] = make_double2(s * s * h.x, s * s * h.y);
  }
  __syncthreads();
  double nrm[1] = {0.0};
  double2* wb = w + b * wstride;
  const double2* Vb = V + long(b) * n;
  const long vs = ldb * n;  // stride between basis vectors
  for (long p = long(blockIdx.x) * KT + threadIdx.x; p < n; p += long(gridDim.x) * KT) {
    // two interleaved partial sums
    double dr0 = 0.0, di0 = 0.0, dr1 = 0.0, di1 = 0.0;
    int i = 0;
    for (; i + 3 <= j; i += 4) {
      const double2 v0 = Vb[(i + 0) * vs + p], v1 = Vb[(i + 1) * vs + p];
      const double2 v2 = Vb[(i + 2) * vs + p], v3 = Vb[(i + 3) * vs + p];
      const double2 c0 = coef[i], c1 = coef[i + 1], c2 = coef[i + 2], c3 = coef[i + 3];
      dr0 = fma(c0.x, v0.x, fma(-c0.y, v0.y, dr0));
      di0 = fma(c0.x, v0.y, fma(c0.y, v0.x, di0));
      dr1 = fma(c1.x, v1.x, fma(-c1.y, v1.y, dr1));
      di1 = fma(c1.x, v1.y, fma(c1.y, v1.x, di1));
      dr0 = fma(c2.x, v2.x, fma(-c2.y, v2.y, dr0));
      di0 = fma(c2.x, v2.y, fma(c2.y, v2.x, di0));
      dr1 = fma(c3.x, v3.x, fma(-c3.y, v3.y, dr1));
      di1 = fma(c3.x, v3.y, fma(c3.y, v3.x, di1));
    }
    for (; i <= j; ++i) {
      const double2 v = Vb[i * vs + p];
      const double2 c = coef[i];
      dr0 = fma(c.x, v.x, fma(-c.y, v.y, dr0));
      di0 = fma(c.x, v.y, fma(c.y, v.x, di0));
    }
    double2 x = wb[p];
    x.x -= dr0 + dr1;
    x.y -= di0 + di1;
    wb[p] = x;
    if (Vnew) Vnew[long(b) * n + p] = x;
    if (partial) nrm[0] = fma(x.x, x.x, fma(x.y, x.y, nrm[0]));
  }
  if (partial) {
    __shared__ double sh[KT / 32 + 1];
    block_sum<1>(nrm, sh);
    if (threadIdx.x == 0) partial[long(b) * gridDim.x + blockIdx.x] = sh[KT / 32];
  }
}

// out[b] = sum_{i < jn[b]} (sigma_i y_i) V_i
__global__ void __launch_bounds__(KT)
combine_kernel(const double2* __restrict__ V, long ldb, double2* __restrict__ out, long ostride,
               long n, const double2* __restrict__ y, int ldy, const double* __restrict__ sigma,
               int ldsig, const int* __restrict__ jn) {
  pdl_wait();
  const int b = blockIdx.y;
  const int J = jn[b];
  __shared__ double2 ys[HZ_MAX_RESTART];
  for (int i = threadIdx.x; i < J; i += KT) {
    const double s = sigma[long(i) * ldsig + b];
    const double2 yy = y[long(b) * ldy + i];
    ys[i] = make_double2(s * yy.x, s * yy.y);
  }
  __syncthreads();
  double2* ob = out + b * ostride;
  for (long p = long(blockIdx.x) * KT + threadIdx.x; p < n; p += long(gridDim.x) * KT) {
    double2 x = make_double2(0.0, 0.0);
    for (int i = 0; i < J; ++i) {
      const double2 v = V[(long(i) * ldb + b) * n + p];
      const double2 c = ys[i];
      x.x = fma(c.x, v.x, fma(-c.y, v.y, x.x));
      x.y = fma(c.x, v.y, fma(c.y, v.x, x.y));
    }
    ob[p] = x;
  }
}

// w as basis vector: the first one of a cycle
__global__ void __launch_bounds__(KT)
copy_kernel(const double2* __restrict__ w, long wstride, long n, const int* __restrict__ active,
            double2* __restrict__ V) {
  pdl_wait();
  const int b = blockIdx.y;
  if (!active[b]) return;
  for (long p = long(blockIdx.x) * KT + threadIdx.x; p < n; p += long(gridDim.x) * KT)
    V[long(b) * n + p] = w[b * wstride + p];
}

// w as basis vector in block fixed point
__global__ void __launch_bounds__(CT)
encode_kernel(const double2* __restrict__ w, long wstride, long n, long ntiles,
              const int* __restrict__ active, int4* __restrict__ V, int* __restrict__ ev) {
  pdl_wait();
  const int b = blockIdx.y;
  if (!active[b]) return;
  __shared__ int red[CG_WARPS];
  const long p = long(blockIdx.x) * FX_TILE + threadIdx.x;
  const double2 x = p < n ? w[b * wstride + p] : make_double2(0.0, 0.0);
  warp_max(fx_exp(x), red);
  __syncthreads();
  const int E = max(max_of(red), FX_EMIN);
  if (p < n) V[long(b) * n + p] = fx_pack(x, E);
  if (threadIdx.x == 0) ev[long(b) * ntiles + blockIdx.x] = E;
}

// Sum partials in a fixed order: q = b * jp1 + i,
// out[b * ldo + i] = sum_blk part[q * nblk + blk].
__global__ void __launch_bounds__(KT)
reduce_c_kernel(const double2* __restrict__ part, int nblk, int jp1, int ldo,
                double2* __restrict__ out) {
  pdl_wait();
  const long q = blockIdx.x;
  double v[2] = {0.0, 0.0};
  for (int i = threadIdx.x; i < nblk; i += KT) {
    const double2 p = part[q * nblk + i];
    v[0] += p.x;
    v[1] += p.y;
  }
  __shared__ double sh[(KT / 32 + 1) * 2];
  block_sum<2>(v, sh);
  if (threadIdx.x == 0)
    out[(q / jp1) * ldo + q % jp1] = make_double2(sh[(KT / 32) * 2], sh[(KT / 32) * 2 + 1]);
}

__global__ void __launch_bounds__(KT)
reduce_r_kernel(const double* __restrict__ part, int nblk, double* __restrict__ out) {
  pdl_wait();
  const long q = blockIdx.x;
  double v[1] = {0.0};
  for (int i = threadIdx.x; i < nblk; i += KT) v[0] += part[q * nblk + i];
  __shared__ double sh[(KT / 32 + 1)];
  block_sum<1>(v, sh);
  if (threadIdx.x == 0) out[q] = sh[KT / 32];
}

__device__ __forceinline__ double2 cmul_d(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ double2 cfma_d(double2 a, double2 b, double2 c) {  // a b + c
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
// max(|a|, |b|) of finite doubles as an integer max of the magnitude bits
// (IEEE order of non-negative doubles is that of their bit patterns), off the
// FP64 pipe
__device__ __forceinline__ long long absbits(double a) {
  return __double_as_longlong(a) & 0x7fffffffffffffffLL;
}

__device__ __forceinline__ double2 shfl_up_d2(double2 v, int o) {
  return make_double2(__shfl_up_sync(0xffffffffu, v.x, o), __shfl_up_sync(0xffffffffu, v.y, o));
}

constexpr int GT = 128;

// One block per right-hand side: form column j of the Hessenberg matrix,
// apply the earlier rotations, build the new one (c real, G [a;b] = [r;0]),
// update g and the residual estimate, and retire converged / broken rows.
// Applying rotations 0..j-1 is a linear recurrence on the running entry,
//   x_0 = h_0,  x_{i+1} = -conj(s_i) x_i + c_i h_{i+1},  r_i = c_i x_i + s_i h_{i+1},
// evaluated by the first warp as a scan of affine maps (each lane composes a contiguous
// chunk, a shuffle scan composes the chunks) instead of j serial steps.
// The other warps meanwhile sum |w|^2 from the update's nblk block sums (fixed
// order) and take its root, and divide the history's entry: one warp doing it
// all in turn held its FP64 unit for 2.3 us a step longer (128^2, 29 steps:
// solve 1759 -> 1690 us).
__global__ void __launch_bounds__(GT)
givens_kernel(KsDev ks, int j, const double* __restrict__ partial, int nblk) {
  pdl_wait();
  const int b = blockIdx.x;
  if (!ks.active[b]) return;
  __shared__ double wsum[GT / 32], shn[3];  // warp sums; |w|^2, 1 / |w|, estimate
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp > 0) {
    double v = 0.0;
    for (int i = threadIdx.x - 32; i < nblk; i += GT - 32) v += partial[long(b) * nblk + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) wsum[warp] = v;
    asm volatile("bar.sync 1, %0;" ::"n"(GT - 32) : "memory");
    if (threadIdx.x == 32) {
      double q = wsum[1];
      for (int i = 2; i < GT / 32; ++i) q += wsum[i];
      shn[0] = q;  // |w|^2 after orthogonalisation
      shn[1] = q > 0.0 ? rsqrt3(q) : 0.0;
    }
    __syncthreads();
    __syncthreads();
    if (threadIdx.x == 32) ks.hist[long(b) * ks.m + j] = shn[2] / ks.bnorm[b];
    return;
  }
  const int m = ks.m;
  __shared__ double2 col[HZ_MAX_RESTART + 2];   // h, the new column before rotation
  __shared__ double2 rcol[HZ_MAX_RESTART + 2];  // rotated column
  double2* colg = ks.H + (long(b) * m + j) * (m + 1);
  const double2* S1 = ks.S1 + long(b) * (m + 1);
  const double2* S2 = ks.S2 + long(b) * (m + 1);
  double* cs = ks.cs + long(b) * m;
  double2* sn = ks.sn + long(b) * m;
  double2* g = ks.g + long(b) * (m + 1);
  long long hbits = 0;  // bits of max |Re h|, |Im h|
  bool bad = false;
  for (int i = lane; i <= j; i += 32) {
    const double s = ks.sigma[long(i) * ks.ldsig + b];
    const double2 h = make_double2(s * (S1[i].x + S2[i].x), s * (S1[i].y + S2[i].y));
    col[i] = h;
    ks.Hraw[(long(b) * m + j) * (m + 1) + i] = h;
    hbits = max(hbits, max(absbits(h.x), absbits(h.y)));
    bad |= !isfinite(h.x) || !isfinite(h.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hbits = max(hbits, __shfl_xor_sync(0xffffffffu, hbits, o));
  const double hmax = __longlong_as_double(hbits);
  __syncwarp();
  // chunk of maps i in [i0, i1) of this lane; composite F(x) = A x + B
  const int per = (j + 31) / 32;
  const int i0 = min(j, lane * per), i1 = min(j, i0 + per);
  double2 A = make_double2(1.0, 0.0), B = make_double2(0.0, 0.0);
  for (int i = i0; i < i1; ++i) {
    const double2 al = make_double2(-sn[i].x, sn[i].y);  // -conj(s_i)
    const double c = cs[i];
    const double2 be = make_double2(c * col[i + 1].x, c * col[i + 1].y);
    if (i == i0) {
      A = al;
      B = be;
    } else {
      A = cmul_d(al, A);
      B = cfma_d(al, B, be);
    }
  }
  // inclusive scan over the lanes that hold a chunk: G_l = F_l o ... o F_0
  const int last = per ? (j - 1) / per : 0;
  for (int o = 1; o <= last; o <<= 1) {
    const double2 Ap = shfl_up_d2(A, o), Bp = shfl_up_d2(B, o);
    if (lane >= o) {
      B = cfma_d(A, Bp, B);
      A = cmul_d(A, Ap);
    }
  }
  const double2 h0 = col[0];
  double2 Ae = shfl_up_d2(A, 1), Be = shfl_up_d2(B, 1);
  if (lane == 0) {
    Ae = make_double2(1.0, 0.0);
    Be = make_double2(0.0, 0.0);
  }
  double2 x = cfma_d(Ae, h0, Be);  // x_{i0}
  for (int i = i0; i < i1; ++i) {
    const double c = cs[i];
    const double2 sv = sn[i], h1 = col[i + 1];
    rcol[i] = cfma_d(sv, h1, make_double2(c * x.x, c * x.y));
    x = cfma_d(make_double2(-sv.x, sv.y), x, make_double2(c * h1.x, c * h1.y));
  }
  const double2 xall = cfma_d(A, h0, B);  // lane last holds the full composition
  const double2 a =
      make_double2(__shfl_sync(0xffffffffu, xall.x, last), __shfl_sync(0xffffffffu, xall.y, last));
  __syncthreads();  // |w|
  const double hn2 = shn[0];
  bad = __any_sync(0xffffffffu, bad) || !isfinite(hn2);
  if (lane == 0) {
    // h_{j+1,j} = hn = |w|; sigma_{j+1} = 1 / hn normalises the next vector
    const double inv_hn = shn[1];
    const double hn = hn2 * inv_hn;
    ks.Hraw[(long(b) * m + j) * (m + 1) + j + 1] = make_double2(hn, 0.0);
    const bool happy = hn <= 1e-14 * hmax;
    ks.sigma[long(j + 1) * ks.ldsig + b] = (hn > 0.0 && !happy) ? inv_hn : 0.0;
    const double aa2 = fma(a.x, a.x, a.y * a.y);
    double c;
    double2 s, r;
    if (hn == 0.0) {
      c = 1.0; s = make_double2(0.0, 0.0); r = a;
    } else if (aa2 == 0.0) {
      c = 0.0; s = make_double2(1.0, 0.0); r = make_double2(hn, 0.0);
    } else {
      // rho = sqrt(|a|^2 + hn^2); c = |a| / rho; s = (a / |a|) hn / rho;
      // r = (a / |a|) rho
      const double rho2 = aa2 + hn2;
      const double inv_aa = rsqrt3(aa2), inv_rho = rsqrt3(rho2);
      const double aa = aa2 * inv_aa, rho = rho2 * inv_rho;
      c = aa * inv_rho;
      const double2 ph = make_double2(a.x * inv_aa, a.y * inv_aa);
      const double hr = hn * inv_rho;
      s = make_double2(ph.x * hr, ph.y * hr);  // ph conj(hn) / rho
      r = make_double2(ph.x * rho, ph.y * rho);
    }
    cs[j] = c;
    sn[j] = s;
    rcol[j] = r;
    rcol[j + 1] = make_double2(0.0, 0.0);
    const double2 gj = g[j];
    const double2 gn = make_double2(-(s.x * gj.x + s.y * gj.y), -(s.x * gj.y - s.y * gj.x));
    g[j + 1] = gn;  // -conj(s) g_j
    g[j] = make_double2(c * gj.x, c * gj.y);
    const double gn2 = fma(gn.x, gn.x, gn.y * gn.y);
    const double est = gn2 > 0.0 ? gn2 * rsqrt3(gn2) : 0.0;
    ks.est[b] = est;
    shn[2] = est;
    ks.jend[b] = j + 1;
    bad |= !isfinite(est) || !isfinite(r.x) || !isfinite(r.y);
    int act = 1;
    if (bad) {
      ks.status[b] = HZ_ERR_BREAKDOWN;
      act = 0;
    } else if (est <= ks.tol * ks.bnorm[b] || happy) {
      act = 0;
    }
    if (!act) {
      ks.active[b] = 0;
      atomicSub(ks.n_active, 1);
    }
  }
  __syncthreads();  // the estimate
  for (int i = lane; i <= j + 1; i += 32) colg[i] = rcol[i];
}

__device__ __forceinline__ double2 widen(double2 v) { return v; }
__device__ __forceinline__ double2 widen(float2 v) { return make_double2(f2d_bits(v.x), f2d_bits(v.y)); }

// u += sum_{i < jn} y[b][i] Z_i  (Z in c64 or c128), one pass.
template <typename ZT>
__global__ void __launch_bounds__(KT)
solution_update_kernel(const ZT* __restrict__ Z, long ldb, double2* __restrict__ u, long ustride,
                       long n, const double2* __restrict__ y, int ldy, const int* __restrict__ jn) {
  pdl_wait();
  const int b = blockIdx.y;
  const int J = jn[b];
  if (J <= 0) return;
  __shared__ double2 ys[HZ_MAX_RESTART];
  for (int i = threadIdx.x; i < J; i += KT) ys[i] = y[long(b) * ldy + i];
  __syncthreads();
  double2* ub = u + b * ustride;
  for (long p = long(blockIdx.x) * KT + threadIdx.x; p < n; p += long(gridDim.x) * KT) {
    // two interleaved partial sums; complex64 Z widened by integer bit moves
    // (off the FP64 pipe, the limit here)
    double2 x = ub[p], x1 = make_double2(0.0, 0.0);
    int i = 0;
    for (; i + 1 < J; i += 2) {
      const double2 z0 = widen(Z[(long(i) * ldb + b) * n + p]);
      const double2 z1 = widen(Z[(long(i + 1) * ldb + b) * n + p]);
      const double2 c0 = ys[i], c1 = ys[i + 1];
      x.x = fma(c0.x, z0.x, fma(-c0.y, z0.y, x.x));
      x.y = fma(c0.x, z0.y, fma(c0.y, z0.x, x.y));
      x1.x = fma(c1.x, z1.x, fma(-c1.y, z1.y, x1.x));
      x1.y = fma(c1.x, z1.y, fma(c1.y, z1.x, x1.y));
    }
    if (i < J) {
      const double2 z0 = widen(Z[(long(i) * ldb + b) * n + p]);
      const double2 c0 = ys[i];
      x.x = fma(c0.x, z0.x, fma(-c0.y, z0.y, x.x));
      x.y = fma(c0.x, z0.y, fma(c0.y, z0.x, x.y));
    }
    ub[p] = make_double2(x.x + x1.x, x.y + x1.y);
  }
}

// u += t (element-wise, FP64), for active right-hand sides with jn > 0
__global__ void axpy_kernel(double2* __restrict__ u, const double2* __restrict__ t, long stride,
                            long n, const int* __restrict__ jn) {
  pdl_wait();
  const int b = blockIdx.y;
  if (jn[b] <= 0) return;
  for (long p = long(blockIdx.x) * KT + threadIdx.x; p < n; p += long(gridDim.x) * KT) {
    const double2 a = u[b * stride + p], c = t[b * stride + p];
    u[b * stride + p] = make_double2(a.x + c.x, a.y + c.y);
  }
}

// out[b] = sigma[b] V[b]: the operator input of an unpreconditioned step
__global__ void scale_copy_kernel(const double2* __restrict__ V, const double* __restrict__ sigma,
                                  double2* __restrict__ out, long n, const int* __restrict__ active) {
  pdl_wait();
  const int b = blockIdx.y;
  if (!active[b]) return;
  const double s = sigma[b];
  for (long p = long(blockIdx.x) * KT + threadIdx.x; p < n; p += long(gridDim.x) * KT) {
    const double2 v = V[b * n + p];
    out[b * n + p] = make_double2(s * v.x, s * v.y);
  }
}

// |x|^2 partials of nrhs vectors
__global__ void __launch_bounds__(KT)
norm2_kernel(const double2* __restrict__ x, long stride, long n, double* __restrict__ partial) {
  pdl_wait();
  const int b = blockIdx.y;
  double v[1] = {0.0};
  for (long p = long(blockIdx.x) * KT + threadIdx.x; p < n; p += long(gridDim.x) * KT) {
    const double2 a = x[b * stride + p];
    v[0] = fma(a.x, a.x, fma(a.y, a.y, v[0]));
  }
  __shared__ double sh[KT / 32 + 1];
  block_sum<1>(v, sh);
  if (threadIdx.x == 0) partial[long(b) * gridDim.x + blockIdx.x] = sh[KT / 32];
}

}  // namespace

// Blocks per right-hand side of the element-wise FP64 kernels: four per SM over
// the whole launch, but at least one point per thread.  Short vectors thus
// still spread over every SM: an FP64 warp instruction holds a sub-partition's
// FP64 unit for ~64 cycles, so a few long-running warps would serialise the
// work.
int krylov_blocks(long n, int nrhs) {
  const long per = (4 * 152 + long(nrhs) - 1) / nrhs;
  return int(std::max(std::min(per, (n + KT - 1) / KT), 1l));
}

namespace {
// Blocks per right-hand side of the Gram-Schmidt kernels: they walk over the
// tiles, so per_sm * 152 blocks are asked for (what fits at a time); with
// several right-hand sides as many whole waves as leave the fewest SMs idle.
int cgs_blocks(long ntiles, int nrhs, int per_sm) {
  const long wave = long(per_sm) * 152;
  long best = 1;
  double fill = 0.0;
  for (int k = 1; k <= 4; ++k) {
    const long per = k * wave / nrhs;
    const double f = double(per) * nrhs / double(k * wave);
    if (per >= 1 && f > fill + 0.03) {
      fill = f;
      best = per;
    }
  }
  return int(std::min(std::min(best, long(HZ_CGS_BLOCKS)), ntiles));
}

template <int MODE>
hz_status launch_cgs(const Basis& Q, int nblk, int rows, double2* w, long wstride, int j, int nrhs,
                     const double2* S, int ldS, const double* sigma, int ldsig, const int* active,
                     double2* partial, int4* Vnew, int* enew, cudaStream_t st) {
  // one limit for every launch: other threads may be launching the same kernel
  // with another number of rows
  constexpr int limit = int((MODE == CG_UPDATE_DOTS ? CG_MAXROWS : CG_ROWS) * CG_ROW_BYTES);
  HZ_CUDA(cudaFuncSetAttribute(cgs_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, limit));
  HZ_CUDA(launch_pdl(cgs_kernel<MODE>, dim3(nblk, nrhs), dim3(CT), rows * CG_ROW_BYTES, st, Q.V,
                     Q.ev, Q.ldb, Q.ntiles, w, wstride, Q.n, j, rows, S, ldS, sigma, ldsig, active, partial,
                     Vnew, enew));
  return HZ_OK;
}

// the FP64 basis
double2* fp64(const Basis& Q, int i = 0) { return reinterpret_cast<double2*>(Q.V) + i * Q.ldb * Q.n; }

hz_status launch_update_f64(const Basis& Q, double2* w, long wstride, int j, int nrhs,
                            const double2* S, int ldS, const double* sigma, int ldsig,
                            const int* active, double* partial, int* nblk, bool keep,
                            cudaStream_t st) {
  *nblk = krylov_blocks(Q.n, nrhs);
  HZ_CUDA(launch_pdl(update_kernel, dim3(*nblk, nrhs), dim3(KT), 0, st, fp64(Q), Q.ldb, w, wstride,
                     Q.n, j, S, ldS, sigma, ldsig, active, partial,
                     keep ? fp64(Q, j + 1) : static_cast<double2*>(nullptr)));
  return HZ_OK;
}
}  // namespace

hz_status launch_dots(const Basis& Q, double2* w, long wstride, int j, int nrhs, const int* active,
                      double2* partial, double2* S, int ldS, cudaStream_t st) {
  int nblk;
  if (Q.fixed) {
    nblk = cgs_blocks(Q.ntiles, nrhs, 4);
    HZ_TRY(launch_cgs<CG_DOTS>(Q, nblk, CG_ROWS, w, wstride, j, nrhs, nullptr, 0, nullptr, 0, active,
                               partial, nullptr, nullptr, st));
  } else {
    // balanced chunks of at most VC vectors, none empty; one wave of two blocks
    // per SM, at least one point per thread
    int nchunk = (j + VC) / VC;
    const int vpc = (j + nchunk) / nchunk;
    nchunk = (j + vpc) / vpc;
    const long per = std::min(2 * 152 / (long(nrhs) * nchunk), (Q.n + KT - 1) / KT);
    nblk = int(std::max(per, 1l));
    HZ_CUDA(launch_pdl(dots_kernel, dim3(nblk, nrhs, nchunk), dim3(KT), 0, st, fp64(Q), Q.ldb, w,
                       wstride, Q.n, j, vpc, active, partial));
  }
  HZ_CUDA(launch_pdl(reduce_c_kernel, dim3(unsigned(nrhs * (j + 1))), dim3(KT), 0, st, partial,
                     nblk, j + 1, ldS, S));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_update_dots(const Basis& Q, double2* w, long wstride, int j, int nrhs,
                             const double2* S1, int ldS, const double* sigma, int ldsig,
                             const int* active, double2* partial, double2* S2,
                             cudaStream_t st) {
  if (!Q.fixed) {
    int unused;
    HZ_TRY(launch_update_f64(Q, w, wstride, j, nrhs, S1, ldS, sigma, ldsig, active, nullptr, &unused,
                             false, st));
    count_launches(1);  // the phase counts two
    return launch_dots(Q, w, wstride, j, nrhs, active, partial, S2, ldS, st);
  }
  // One kernel while a tile's rows fit the shared memory of half an SM, with as
  // many blocks per SM as hold them: what it lacks is warps, not room for the
  // next tile's rows (2^24 points, j = 22: four blocks of 24 rows 1703 us, three
  // of 34 1727, two of 52 2001, two kernels 2270; j = 39: 3050 against 3780).
  if (j + 1 > CG_FUSED) {
    HZ_TRY(launch_cgs<CG_UPDATE>(Q, cgs_blocks(Q.ntiles, nrhs, 4), CG_ROWS, w, wstride, j, nrhs,
                                 S1, ldS, sigma, ldsig, active, partial, nullptr, nullptr, st));
    count_launches(1);  // the phase counts two
    return launch_dots(Q, w, wstride, j, nrhs, active, partial, S2, ldS, st);
  }
  const int per_sm = j + 1 <= CG_ROWS ? 4 : (j + 1 <= 34 ? 3 : 2);
  const int rows = per_sm == 4 ? CG_ROWS : (per_sm == 3 ? 34 : CG_MAXROWS);
  const int nblk = cgs_blocks(Q.ntiles, nrhs, per_sm);
  HZ_TRY(launch_cgs<CG_UPDATE_DOTS>(Q, nblk, rows, w, wstride, j, nrhs, S1, ldS, sigma, ldsig,
                                    active, partial, nullptr, nullptr, st));
  HZ_CUDA(launch_pdl(reduce_c_kernel, dim3(unsigned(nrhs * (j + 1))), dim3(KT), 0, st, partial,
                     nblk, j + 1, ldS, S2));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_update(const Basis& Q, double2* w, long wstride, int j, int nrhs,
                        const double2* S, int ldS, const double* sigma, int ldsig,
                        const int* active, double* partial, int* nblk, bool keep, cudaStream_t st) {
  if (!Q.fixed)
    return launch_update_f64(Q, w, wstride, j, nrhs, S, ldS, sigma, ldsig, active, partial, nblk,
                             keep, st);
  *nblk = cgs_blocks(Q.ntiles, nrhs, 4);
  HZ_TRY(launch_cgs<CG_UPDATE>(Q, *nblk, CG_ROWS, w, wstride, j, nrhs, S, ldS, sigma, ldsig, active,
                               reinterpret_cast<double2*>(partial),
                               keep ? Q.V + (j + 1) * Q.ldb * Q.n : nullptr,
                               keep ? Q.ev + (j + 1) * Q.ldb * Q.ntiles : nullptr, st));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_encode(const Basis& Q, const double2* w, long wstride, int i, int nrhs,
                        const int* active, cudaStream_t st) {
  if (!Q.fixed)
    HZ_CUDA(launch_pdl(copy_kernel, dim3(krylov_blocks(Q.n, nrhs), nrhs), dim3(KT), 0, st, w,
                       wstride, Q.n, active, fp64(Q, i)));
  else
    HZ_CUDA(launch_pdl(encode_kernel, dim3(unsigned(Q.ntiles), nrhs), dim3(CT), 0, st, w, wstride,
                       Q.n, Q.ntiles, active, Q.V + i * Q.ldb * Q.n, Q.ev + i * Q.ldb * Q.ntiles));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_givens(const KsDev& ks, int j, int nrhs, const double* partial, int nblk,
                        cudaStream_t st) {
  HZ_CUDA(launch_pdl(givens_kernel, dim3(nrhs), dim3(GT), 0, st, ks, j, partial, nblk));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_solution_update(int zprec, const void* Z, long ldb, double2* u, long ustride,
                                 long n, int nrhs, const double2* y, int ldy, const int* jn,
                                 cudaStream_t st) {
  const int nblk = krylov_blocks(n, nrhs);
  if (zprec == 0)
    HZ_CUDA(launch_pdl(solution_update_kernel<double2>, dim3(nblk, nrhs), dim3(KT), 0, st,
                       static_cast<const double2*>(Z), ldb, u, ustride, n, y, ldy, jn));
  else
    HZ_CUDA(launch_pdl(solution_update_kernel<float2>, dim3(nblk, nrhs), dim3(KT), 0, st,
                       static_cast<const float2*>(Z), ldb, u, ustride, n, y, ldy, jn));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_combine(const Basis& Q, double2* out, long ostride, int nrhs, const double2* y,
                         int ldy, const double* sigma, int ldsig, const int* jn, cudaStream_t st) {
  if (Q.fixed)
    HZ_TRY(launch_cgs<CG_COMBINE>(Q, cgs_blocks(Q.ntiles, nrhs, 4), CG_ROWS, out, ostride, 0, nrhs, y,
                                  ldy, sigma, ldsig, jn, nullptr, nullptr, nullptr, st));
  else
    HZ_CUDA(launch_pdl(combine_kernel, dim3(krylov_blocks(Q.n, nrhs), nrhs), dim3(KT), 0, st,
                       fp64(Q), Q.ldb, out, ostride, Q.n, y, ldy, sigma, ldsig, jn));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_scale_copy(const double2* V, const double* sigma, double2* out, long n, int nrhs,
                           const int* active, cudaStream_t st) {
  const int nblk = krylov_blocks(n, nrhs);
  HZ_CUDA(launch_pdl(scale_copy_kernel, dim3(nblk, nrhs), dim3(KT), 0, st, V, sigma, out, n,
                     active));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_axpy(double2* u, const double2* t, long stride, long n, int nrhs, const int* jn,
                      cudaStream_t st) {
  const int nblk = krylov_blocks(n, nrhs);
  HZ_CUDA(launch_pdl(axpy_kernel, dim3(nblk, nrhs), dim3(KT), 0, st, u, t, stride, n, jn));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_norm2(const double2* x, long stride, long n, int nrhs, double* partial, int nblk,
                       double* out, cudaStream_t st) {
  HZ_CUDA(launch_pdl(norm2_kernel, dim3(nblk, nrhs), dim3(KT), 0, st, x, stride, n, partial));
  HZ_CUDA(launch_pdl(reduce_r_kernel, dim3(unsigned(nrhs)), dim3(KT), 0, st, partial, nblk, out));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status launch_reduce_r(const double* partial, int nblk, int nq, double* out, cudaStream_t st) {
  HZ_CUDA(launch_pdl(reduce_r_kernel, dim3(unsigned(nq)), dim3(KT), 0, st, partial, nblk, out));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

}  // namespace hz
