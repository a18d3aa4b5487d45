// Instantiates the FFT pass kernels for one axis length, HZ_FFT_N, and
// exposes them as an FftOps table.  The build compiles this file once per
// supported length, in parallel.
#include <algorithm>

#include "fft_int.cuh"
#include "fft_kernels.cuh"

#ifndef HZ_FFT_N
#error "HZ_FFT_N must be defined"
#endif

namespace hz {
namespace {

constexpr int N = HZ_FFT_N;

template <typename K>
hz_status smem_attr(K kernel, size_t bytes) {
  if (bytes > 48 * 1024) {
    HZ_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes)));
  }
  return HZ_OK;
}

hz_status row_fwd_c64(const double2* in, const double* scale, long rows_per_rhs, long nrows,
                      const void* tw, void* out, cudaStream_t st, const int* active, void* zero,
                      long zero_row_bytes) {
  if (zero && zero_row_bytes % 16 != 0) return HZ_ERR_INVALID_ARG;
  uint4* z = static_cast<uint4*>(zero);
  const int zc = int(zero_row_bytes / 16);
  using C = LineCfg<float, N>;
  using V = float2;
  // blocks of ROW_LINES lines, or one line per block when that leaves the
  // GPU under-filled (few rows)
  const bool small = (nrows + C::ROW_LINES - 1) / C::ROW_LINES < 2L * 152;
  if (small) {
    auto k = row_fwd_kernel<float, N, 1>;
    HZ_TRY(smem_attr(k, C::row_smem(1)));
    HZ_CUDA(launch_pdl(k, dim3(unsigned(nrows)), dim3(C::TPL_ROW), C::row_smem(1), st, in, scale,
                       rows_per_rhs, nrows, static_cast<const V*>(tw), static_cast<V*>(out),
                       active, z, zc));
    HZ_CUDA(cudaGetLastError());
    return HZ_OK;
  }
  constexpr int lines = C::ROW_LINES;
  auto k = row_fwd_kernel<float, N, C::ROW_LINES>;
  HZ_TRY(smem_attr(k, C::row_smem(lines)));
  const long blocks = (nrows + lines - 1) / lines;
  HZ_CUDA(launch_pdl(k, dim3(unsigned(blocks)), dim3(lines * C::TPL_ROW), C::row_smem(lines), st,
                     in, scale, rows_per_rhs, nrows, static_cast<const V*>(tw),
                     static_cast<V*>(out), active, z, zc));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

// complex128 passes (fft_int.cuh): blocks of full size, or of one line (a
// quarter of the columns) where those of one right-hand side would leave SMs
// without a block.  The lines of a block share an exponent, so the choice may
// not depend on how many right-hand sides a call has: each gives bit for bit
// the result that it gives alone.  (By the whole call's blocks eight of 128^2
// took 79 us instead of 81, eight of 48 x 40 x 24 238 instead of 253.)
constexpr long kFew = 2 * 152;

template <int LINES>
hz_status irow_fwd_t(const double2* in, const double* scale, long rows, long nrhs, const int4* tw,
                     double2* out, cudaStream_t st, const int* active) {
  using B = IBlock<N, LINES, true>;
  auto k = irow_fwd_kernel<N, LINES>;
  HZ_TRY(smem_attr(k, B::SMEM));
  HZ_CUDA(launch_pdl(k, dim3(unsigned((rows + LINES - 1) / LINES), unsigned(nrhs)), dim3(B::NT),
                     B::SMEM, st, in, scale, rows, tw, out, active));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status row_fwd(int prec, const double2* in, const double* scale, long rows_per_rhs, long nrows,
                  const void* tw, void* out, cudaStream_t st, const int* active, void* zero,
                  long zero_row_bytes) {
  if (prec == 0) {
    // the complex128 x-inverse ends in a gather: nothing to clear
    constexpr int L = ICfg<N>::ROWS;
    const long nrhs = nrows / rows_per_rhs;
    const bool few = (rows_per_rhs + L - 1) / L < kFew;
    return (few ? irow_fwd_t<1> : irow_fwd_t<L>)(in, scale, rows_per_rhs, nrhs,
                                                 static_cast<const int4*>(tw),
                                                 static_cast<double2*>(out), st, active);
  }
  return row_fwd_c64(in, scale, rows_per_rhs, nrows, tw, out, st, active, zero, zero_row_bytes);
}

template <int LINES>
hz_status irow_inv_t(double2* planes, const unsigned long long* rowmask, int K, long rows,
                     long nrhs, long n, const int4* tw, cudaStream_t st, const int* active) {
  using B = IBlock<N, LINES, true>;
  auto k = irow_inv_kernel<N, LINES>;
  HZ_TRY(smem_attr(k, B::SMEM));
  HZ_CUDA(launch_pdl(k, dim3(unsigned((rows + LINES - 1) / LINES), unsigned(K), unsigned(nrhs)),
                     dim3(B::NT), B::SMEM, st, planes, rowmask, K, rows, n, tw, active));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

// complex128: every (row, node) line in place, then the weighted gather
hz_status row_inv_c128(const void* planes, const void* rec, const uchar2* segtab,
                       const unsigned long long* rowmask, int K, long rows_per_rhs, long nrows,
                       long n, double inv_n, const void* tw, void* out, cudaStream_t st,
                       const int* active, const uchar4* gnode, const void* gw) {
  constexpr int L = ICfg<N>::ROWS;
  const long nrhs = nrows / rows_per_rhs;
  const bool few = (rows_per_rhs + L - 1) / L * K < kFew;
  double2* pl = static_cast<double2*>(const_cast<void*>(planes));
  HZ_TRY((few ? irow_inv_t<1> : irow_inv_t<L>)(pl, rowmask, K, rows_per_rhs, nrhs, n,
                                               static_cast<const int4*>(tw), st, active));
  const long total = nrows * N;
  const long gblocks = std::min<long>((total + 255) / 256, 152L * 16);
  if (gnode)
    HZ_CUDA(launch_pdl(weighted_gather4_kernel<double, double2>, dim3(unsigned(gblocks)), dim3(256),
                       0, st, pl, gnode, static_cast<const double2*>(gw), K, n, total, inv_n,
                       static_cast<double2*>(out), active));
  else
    HZ_CUDA(launch_pdl(weighted_gather_kernel<double, double2>, dim3(unsigned(gblocks)), dim3(256),
                       0, st, pl, static_cast<const double*>(rec), segtab, K, n, total, inv_n,
                       static_cast<double2*>(out), active));
  HZ_CUDA(cudaGetLastError());
  count_launches(1);  // the phase counts one
  return HZ_OK;
}

template <typename OutT>
hz_status row_inv_acc_c64(const void* planes, const void* rec, const uchar2* segtab, int nseg,
                          const unsigned long long* rowmask, int K, long rows_per_rhs, long nrows,
                          long n, double inv_n, const void* tw, void* out, cudaStream_t st,
                          const int* active, int mode, const unsigned long long* items,
                          long nitems, const uchar4* gnode, const void* gw) {
  using C = LineCfg<float, N>;
  using V = float2;
  using GW = GwT<float>::T;
  if (gnode && mode != 3) {
    // per-point (node, weight) records: lines in place, then the gather
    auto ki = row_inv_inplace_kernel<float, N, C::ROW_LINES>;
    HZ_TRY(smem_attr(ki, C::row_smem()));
    dim3 grid(unsigned((nrows + C::ROW_LINES - 1) / C::ROW_LINES), unsigned(K));
    HZ_CUDA(launch_pdl(ki, dim3(grid), dim3(C::ROW_THREADS), C::row_smem(), st,
                       static_cast<V*>(const_cast<void*>(planes)), rowmask, K, rows_per_rhs, nrows,
                       n, static_cast<const V*>(tw), active));
    HZ_CUDA(cudaGetLastError());
    const long total = nrows * N;
    const long gblocks = std::min<long>((total + 255) / 256, 152L * 16);
    HZ_CUDA(launch_pdl(weighted_gather4_kernel<float, OutT>, dim3(unsigned(gblocks)), dim3(256), 0, st,
                       static_cast<const V*>(planes), gnode, static_cast<const GW*>(gw), K, n,
                       total, float(inv_n), static_cast<OutT*>(out), active));
    HZ_CUDA(cudaGetLastError());
    count_launches(1);  // the phase counts one
    return HZ_OK;
  }
  if (mode == 3) {
    // one line per (row, node) item, added into the cleared output
    if (!items || nitems <= 0) return nitems == 0 ? HZ_OK : HZ_ERR_INVALID_ARG;
    const long rhs = nrows / rows_per_rhs;
    if (rhs > 65535) return HZ_ERR_INVALID_ARG;
    auto ks = gnode ? row_inv_scatter_kernel<float, N, OutT, C::ROW_LINES, true>
                    : row_inv_scatter_kernel<float, N, OutT, C::ROW_LINES, false>;
    // line buffers, then (two-node records) one weight table per line
    const size_t smem = C::row_smem() + (gnode ? 0 : size_t(C::ROW_LINES) * HZ_MAX_SEG * sizeof(V));
    HZ_TRY(smem_attr(ks, smem));
    dim3 grid(unsigned((nitems + C::ROW_LINES - 1) / C::ROW_LINES), unsigned(rhs));
    HZ_CUDA(launch_pdl(ks, dim3(grid), dim3(C::ROW_THREADS), smem, st,
                       static_cast<const V*>(planes), static_cast<const RecT<float>::T*>(rec),
                       segtab, nseg, items, nitems, K, n, float(inv_n), static_cast<const V*>(tw),
                       static_cast<OutT*>(out), active, gnode, static_cast<const GW*>(gw)));
    HZ_CUDA(cudaGetLastError());
    return HZ_OK;
  }
  // fewer blocks of ROW_LINES rows than SMs: few rows
  const bool small = (nrows + C::ROW_LINES - 1) / C::ROW_LINES < 152L;
  if (mode == 1 || (mode == 0 && small)) {
    // few rows: (row, node) lines in parallel, in place, then the gather
    auto ki = row_inv_inplace_kernel<float, N, C::ROW_LINES>;
    HZ_TRY(smem_attr(ki, C::row_smem()));
    dim3 grid(unsigned((nrows + C::ROW_LINES - 1) / C::ROW_LINES), unsigned(K));
    HZ_CUDA(launch_pdl(ki, dim3(grid), dim3(C::ROW_THREADS), C::row_smem(), st,
                       static_cast<V*>(const_cast<void*>(planes)), rowmask, K, rows_per_rhs, nrows,
                       n, static_cast<const V*>(tw), active));
    HZ_CUDA(cudaGetLastError());
    const long total = nrows * N;
    const long gblocks = std::min<long>((total + 255) / 256, 152L * 16);
    HZ_CUDA(launch_pdl(weighted_gather_kernel<float, OutT>, dim3(unsigned(gblocks)), dim3(256), 0, st,
                       static_cast<const V*>(planes), static_cast<const RecT<float>::T*>(rec),
                       segtab, K, n, total, float(inv_n), static_cast<OutT*>(out), active));
    HZ_CUDA(cudaGetLastError());
    count_launches(1);  // the phase counts one
    return HZ_OK;
  }
  constexpr int lines = C::ROW_LINES;
  auto k = row_inv_acc_kernel<float, N, OutT, C::ROW_LINES>;
  HZ_TRY(smem_attr(k, C::row_acc_smem(lines)));
  const long blocks = (nrows + lines - 1) / lines;
  HZ_CUDA(launch_pdl(k, dim3(unsigned(blocks)), dim3(lines * C::TPL_ROW), C::row_acc_smem(lines),
                     st, static_cast<const V*>(planes),
                     static_cast<const RecT<float>::T*>(rec), segtab, nseg, rowmask, K,
                     rows_per_rhs, nrows, n, float(inv_n), static_cast<const V*>(tw),
                     static_cast<OutT*>(out), active));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status row_inv_acc(int prec, int out_kind, const void* planes, const void* rec,
                      const uchar2* segtab, int nseg, const unsigned long long* rowmask, int K,
                      long rows_per_rhs, long nrows, long n, double inv_n, const void* tw,
                      void* out, cudaStream_t st, const int* active, int mode,
                      const unsigned long long* items, long nitems, const uchar4* gnode,
                      const void* gw) {
  if (prec == 0)
    return row_inv_c128(planes, rec, segtab, rowmask, K, rows_per_rhs, nrows, n, inv_n, tw, out, st,
                        active, gnode, gw);
  if (out_kind == 0)
    return row_inv_acc_c64<float2>(planes, rec, segtab, nseg, rowmask, K, rows_per_rhs,
                                        nrows, n, inv_n, tw, out, st, active, mode, items, nitems, gnode, gw);
  return row_inv_acc_c64<double2>(planes, rec, segtab, nseg, rowmask, K, rows_per_rhs,
                                       nrows, n, inv_n, tw, out, st, active, mode, items, nitems, gnode, gw);
}

template <int SIGN>
hz_status line_pass_c64(void* data, int nx, long outer, long S, long ostride, long bstride,
                        int batch, const unsigned long long* omask, int K, const void* tw,
                        cudaStream_t st, const int* active, int per_rhs) {
  using C = LineCfg<float, N>;
  using V = float2;
  auto k = line_pass_kernel<float, N, SIGN>;
  HZ_TRY(smem_attr(k, C::col_smem()));
  const int ntile = (nx + C::TB - 1) / C::TB;
  dim3 grid(unsigned(ntile * outer), 1, unsigned(batch));
  HZ_CUDA(launch_pdl(k, dim3(grid), dim3(C::COL_THREADS), C::col_smem(), st, static_cast<V*>(data),
                     nx, ntile, S, ostride, bstride, omask, K, static_cast<const V*>(tw), active,
                     per_rhs));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

template <int SIGN, int TB>
hz_status iline_t(double2* data, int nx, long outer, long S, long ostride, long bstride, int batch,
                  const unsigned long long* omask, int K, const int4* tw, cudaStream_t st,
                  const int* active, int per_rhs) {
  using B = IBlock<N, TB, false>;
  auto k = iline_kernel<N, SIGN, TB>;
  HZ_TRY(smem_attr(k, B::SMEM));
  const int ntile = (nx + TB - 1) / TB;
  HZ_CUDA(launch_pdl(k, dim3(unsigned(ntile * outer), 1, unsigned(batch)), dim3(B::NT), B::SMEM, st,
                     data, nx, ntile, S, ostride, bstride, omask, K, tw, active, per_rhs));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status line_pass(int prec, int sign, void* data, int nx, long outer, long S, long ostride,
                    long bstride, int batch, const unsigned long long* omask, int K,
                    const void* tw, cudaStream_t st, const int* active, int per_rhs) {
  if (prec == 0) {
    constexpr int TB = ICfg<N>::TB, TF = ICfg<N>::TB_FEW;
    const bool few = (nx + TB - 1) / TB * outer * per_rhs < kFew;
    auto go = sign < 0 ? (few ? iline_t<-1, TF> : iline_t<-1, TB>)
                       : (few ? iline_t<+1, TF> : iline_t<+1, TB>);
    return go(static_cast<double2*>(data), nx, outer, S, ostride, bstride, batch, omask, K,
              static_cast<const int4*>(tw), st, active, per_rhs);
  }
  return sign < 0 ? line_pass_c64<-1>(data, nx, outer, S, ostride, bstride, batch, omask, K, tw, st, active, per_rhs)
                  : line_pass_c64<+1>(data, nx, outer, S, ostride, bstride, batch, omask, K, tw, st, active, per_rhs);
}

// L: the length, so that the node loop is compiled for its lengths only
template <int L>
hz_status line_sym_inv_c64(const void* vhat, void* planes, int nx, long outer, long S, long ostride,
                           long n, int K, int batch, const void* xi2_x, const void* xi2_o,
                           const void* xi2_l, const void* symA, const void* symG,
                           const void* symD, const unsigned long long* smask, long smO, long smS,
                           const void* tw, const void* tw2, cudaStream_t st, const int* active,
                           int kpb, int pair) {
  using C = LineCfg<float, N>;
  using V = float2;
  if constexpr (L == 128 || L == 256) {
    // more nodes than that: the loop over nodes with the spectrum in shared memory
    if (kpb > SYM_KPB_MAX && tw2 && nx % 2 == 0) {
      constexpr int TB = C::template tb_p<1>();
      constexpr int NT = TB * C::template tpl_p<1>();
      auto k = symD ? line_sym_inv_loop_kernel<L, TB, true> : line_sym_inv_loop_kernel<L, TB, false>;
      constexpr size_t smem = C::col_pair_smem(TB) + size_t(N) * TB * 16 + size_t(N) * 12;
      HZ_TRY(smem_attr(k, smem));
      const int ntile = (nx / 2 + TB - 1) / TB;
      HZ_CUDA(launch_pdl(k, dim3(unsigned(ntile * outer), unsigned((K + kpb - 1) / kpb), unsigned(batch)),
                         dim3(NT), smem, st, static_cast<const float2*>(vhat),
                         static_cast<float2*>(planes), nx, ntile, S, ostride, n, K, kpb,
                         static_cast<const float*>(xi2_x), static_cast<const float*>(xi2_o),
                         static_cast<const float*>(xi2_l), static_cast<const float2*>(symA),
                         static_cast<const float2*>(symG), static_cast<const float*>(symD), smask,
                         smO, smS, static_cast<const float4*>(tw2), active));
      HZ_CUDA(cudaGetLastError());
      return HZ_OK;
    }
  }
  // nodes per block: 1, 2 or 4
  kpb = kpb >= 4 ? 4 : (kpb >= 2 ? 2 : 1);
  if (tw2 && nx % 2 == 0) {
    // pair > 1: half-size blocks
    const bool half = pair > 1;
    constexpr int T1 = C::template tb_p<1>(), T1H = C::template tb_p_half<1>();
    constexpr int Tn = C::template tb_p<2>(), TnH = C::template tb_p_half<2>();
    // the Hermite derivative planes (symD) are a compiled variant, so
    // that other media run without their test
    // a square 2D grid (line stride N): the one-node form with compile-time offsets
    const bool sq = kpb == 1 && !half && outer == 1 && S == N;
    auto k = sq ? (symD ? line_sym_inv_pair_kernel<N, 1, T1, true, N>
                        : line_sym_inv_pair_kernel<N, 1, T1, false, N>)
           : symD ? (kpb == 1 ? (half ? line_sym_inv_pair_kernel<N, 1, T1H, true>
                                      : line_sym_inv_pair_kernel<N, 1, T1, true>)
                     : kpb == 2 ? (half ? line_sym_inv_pair_kernel<N, 2, TnH, true>
                                        : line_sym_inv_pair_kernel<N, 2, Tn, true>)
                                : (half ? line_sym_inv_pair_kernel<N, 4, TnH, true>
                                        : line_sym_inv_pair_kernel<N, 4, Tn, true>))
                  : (kpb == 1 ? (half ? line_sym_inv_pair_kernel<N, 1, T1H, false>
                                      : line_sym_inv_pair_kernel<N, 1, T1, false>)
                     : kpb == 2 ? (half ? line_sym_inv_pair_kernel<N, 2, TnH, false>
                                        : line_sym_inv_pair_kernel<N, 2, Tn, false>)
                                : (half ? line_sym_inv_pair_kernel<N, 4, TnH, false>
                                        : line_sym_inv_pair_kernel<N, 4, Tn, false>));
    const int tb = kpb == 1 ? (half ? T1H : T1) : (half ? TnH : Tn);
    const int tpl = kpb == 1 ? C::template tpl_p<1>() : C::template tpl_p<2>();
    HZ_TRY(smem_attr(k, C::col_pair_smem(tb)));
    const int ntile = (nx / 2 + tb - 1) / tb;
    dim3 grid(unsigned(ntile * outer), unsigned((K + kpb - 1) / kpb), unsigned(batch));
    HZ_CUDA(launch_pdl(k, dim3(grid), dim3(tb * tpl), C::col_pair_smem(tb), st,
                       static_cast<const float2*>(vhat), static_cast<float2*>(planes), nx, ntile,
                       S, ostride, n, K, static_cast<const float*>(xi2_x),
                       static_cast<const float*>(xi2_o), static_cast<const float*>(xi2_l),
                       static_cast<const float2*>(symA), static_cast<const float2*>(symG),
                       static_cast<const float*>(symD), smask, smO, smS,
                       static_cast<const float4*>(tw2), active));
    HZ_CUDA(cudaGetLastError());
    return HZ_OK;
  }
  auto k = symD ? (kpb == 4 ? line_sym_inv_kernel<float, N, 4, true>
                            : (kpb == 2 ? line_sym_inv_kernel<float, N, 2, true>
                                        : line_sym_inv_kernel<float, N, 1, true>))
                : (kpb == 4 ? line_sym_inv_kernel<float, N, 4, false>
                            : (kpb == 2 ? line_sym_inv_kernel<float, N, 2, false>
                                        : line_sym_inv_kernel<float, N, 1, false>));
  HZ_TRY(smem_attr(k, C::col_smem()));
  const int ntile = (nx + C::TB - 1) / C::TB;
  dim3 grid(unsigned(ntile * outer), unsigned((K + kpb - 1) / kpb), unsigned(batch));
  HZ_CUDA(launch_pdl(k, dim3(grid), dim3(C::COL_THREADS), C::col_smem(), st,
                     static_cast<const V*>(vhat), static_cast<V*>(planes), nx, ntile, S, ostride, n,
                     K, static_cast<const float*>(xi2_x), static_cast<const float*>(xi2_o),
                     static_cast<const float*>(xi2_l), static_cast<const V*>(symA),
                     static_cast<const V*>(symG), static_cast<const float*>(symD), smask, smO, smS,
                     static_cast<const V*>(tw), active));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

template <int TB>
hz_status isym_t(const void* vhat, void* planes, int nx, long outer, long S, long ostride, long n,
                 int K, int batch, const void* xi2_x, const void* xi2_o, const void* xi2_l,
                 const void* symA, const void* symG, const void* symD,
                 const unsigned long long* smask, long smO, long smS, const void* tw,
                 cudaStream_t st, const int* active) {
  using B = IBlock<N, TB, false>;
  auto k = symD ? isym_kernel<N, TB, true> : isym_kernel<N, TB, false>;
  HZ_TRY(smem_attr(k, B::SMEM));
  const int ntile = (nx + TB - 1) / TB;
  HZ_CUDA(launch_pdl(k, dim3(unsigned(ntile * outer), unsigned(K), unsigned(batch)), dim3(B::NT),
                     B::SMEM, st, static_cast<const double2*>(vhat), static_cast<double2*>(planes),
                     nx, ntile, S, ostride, n, K, static_cast<const double*>(xi2_x),
                     static_cast<const double*>(xi2_o), static_cast<const double*>(xi2_l),
                     static_cast<const double2*>(symA), static_cast<const double2*>(symG),
                     static_cast<const double*>(symD), smask, smO, smS,
                     static_cast<const int4*>(tw), active));
  HZ_CUDA(cudaGetLastError());
  return HZ_OK;
}

hz_status line_sym_inv(int prec, const void* vhat, void* planes, int nx, long outer, long S,
                       long ostride, long n, int K, int batch, const void* xi2_x,
                       const void* xi2_o, const void* xi2_l, const void* symA, const void* symG,
                       const void* symD, const unsigned long long* smask, long smO, long smS,
                       const void* tw, const void* tw2, cudaStream_t st, const int* active,
                       int kpb, int pair) {
  if (prec == 0) {
    constexpr int TB = ICfg<N>::TB, TF = ICfg<N>::TB_FEW;
    const bool few = (nx + TB - 1) / TB * outer * K < kFew;
    return (few ? isym_t<TF> : isym_t<TB>)(vhat, planes, nx, outer, S, ostride, n, K, batch, xi2_x,
                                           xi2_o, xi2_l, symA, symG, symD, smask, smO, smS, tw, st,
                                           active);
  }
  return line_sym_inv_c64<N>(vhat, planes, nx, outer, S, ostride, n, K, batch, xi2_x, xi2_o, xi2_l,
                               symA, symG, symD, smask, smO, smS, tw, tw2, st, active, kpb, pair);
}

const FftOps ops = {N, row_fwd, row_inv_acc, line_pass, line_sym_inv};

}  // namespace

#define HZ_CAT2(a, b) a##b
#define HZ_CAT(a, b) HZ_CAT2(a, b)
const FftOps* HZ_CAT(fft_ops_, HZ_FFT_N)() { return &ops; }

}  // namespace hz
