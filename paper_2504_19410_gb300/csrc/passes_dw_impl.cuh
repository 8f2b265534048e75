// Launchers of the paired double-word passes (passes_dw.cuh), included by the
// instance units inst_dw_*.cu.
#pragma once
#include "passes_dw.cuh"
#include "passes_impl.cuh"

namespace fsa {
namespace detail {

template <int M> struct InstDw {
  using G = GeoDw<M>;
  static constexpr bool kUnpadded = true;
  static constexpr int W = G::W, NT = G::NT, WX = G::WX, NTX = G::T * WX;
  template <bool PAD> static constexpr int SM_R2C = SmR2cDw<M, WX, PAD>::BYTES;
  template <bool FWD, bool PAD> static constexpr int SM_ROW = SmRowDw<M, W, FWD, PAD>::BYTES;
  template <bool PAD> static constexpr int SM_MID = SmMidDw<M, W, PAD>::BYTES;
  static constexpr int SM_C2R = SmC2rDw<M, WX>::BYTES;
  // A plane has only n0 + 1 rows and n1 real columns: narrow tiles (two lines,
  // or two warps' worth of short ones)
  static constexpr int WM = G::T >= 32 ? 2 : 64 / G::T;
  static constexpr int NTM = G::T * WM;
  static constexpr int SM_R2CP = SmR2cDw<M, WM>::BYTES, SM_ROWM = SmRowMidDw<M, WM>::BYTES, SM_C2RP = SmC2rDw<M, WM>::BYTES;

  static cudaError_t prepare() {
    cudaError_t e = cudaSuccess;
    auto set = [&](const void* f, int bytes) {
      if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    set((const void*)kd_r2c_ax0<M, WX>, SM_R2C<true>);
    set((const void*)kd_row<M, W, true>, SM_ROW<true, true>);
    set((const void*)kd_col_mid<M, W>, SM_MID<true>);
    set((const void*)kd_row<M, W, false>, SM_ROW<false, true>);
    set((const void*)kd_c2r_ax0<M, WX>, SM_C2R);
    set((const void*)kd_r2c_ax0<M, WM>, SM_R2CP);
    set((const void*)kd_row_mid<M, WM>, SM_ROWM);
    set((const void*)kd_c2r_ax0<M, WM>, SM_C2RP);
    set((const void*)kd_col_mid<M, W, kMulDdiKernel>, SM_MID<true>);
    set((const void*)kd_c2r_ax0<M, WX, true, true>, SM_C2R);
    set((const void*)kd_r2c_ax0<M, WX, false>, SM_R2C<false>);
    set((const void*)kd_row<M, W, true, false>, SM_ROW<true, false>);
    set((const void*)kd_col_mid<M, W, kMulDdiGrid>, SM_MID<false>);
    set((const void*)kd_row<M, W, false, false>, SM_ROW<false, false>);
    set((const void*)kd_c2r_ax0<M, WX, false>, SM_C2R);
    return e;
  }
  static Geometry geometry(PassKind) {
    Geometry g;
    g.W = W;
    g.threads = NT;
    g.smem = SM_MID<true>;
    return g;
  }
  // lines / columns: the launch's extent; per: how many one CTA takes
  // One CTA per tile: the kernels hand their tiles out themselves (TileQueue).
  template <class F, class... A>
  static cudaError_t go(F f, int per, int nt, int smem, long long extent, const Jobs& jobs, cudaStream_t s, A... a) {
    const long long tiles = (extent + per - 1) / per * jobs.count;
    if (tiles > 0x7fffffff) return cudaErrorInvalidValue;
    Jobs jj = jobs;
    jj.fault = device_fault_word();
    f<<<(unsigned)tiles, nt, smem, s>>>(jj, a...);
    return cudaGetLastError();
  }
  template <class F> static cudaError_t mid(F f, int smem, const Jobs& jobs, int M2, int planes, cudaStream_t s) {
    const long long tiles = (long long)((M2 + W - 1) / W) * planes * jobs.count;
    if (tiles > 0x7fffffff) return cudaErrorInvalidValue;
    Jobs jj = jobs;
    jj.fault = device_fault_word();
    f<<<(unsigned)tiles, NT, smem, s>>>(jj, M2, planes);
    return cudaGetLastError();
  }
  static cudaError_t r2c(const Jobs& j, long long C, cudaStream_t s) {
    return go(kd_r2c_ax0<M, WX>, 2 * WX, NTX, SM_R2C<true>, C, j, s, C);
  }
  static cudaError_t rowf(const Jobs& j, long long rows, cudaStream_t s) {
    return go(kd_row<M, W, true>, W, NT, (SM_ROW<true, true>), rows, j, s, rows);
  }
  static cudaError_t colm(const Jobs& j, int M2, int planes, cudaStream_t s) {
    return mid(kd_col_mid<M, W>, SM_MID<true>, j, M2, planes, s);
  }
  static cudaError_t rowi(const Jobs& j, long long rows, cudaStream_t s) {
    return go(kd_row<M, W, false>, W, NT, (SM_ROW<false, true>), rows, j, s, rows);
  }
  static cudaError_t c2r(const Jobs& j, long long C, cudaStream_t s) {
    return go(kd_c2r_ax0<M, WX>, 2 * WX, NTX, SM_C2R, C, j, s, C);
  }
  // d = 2
  static cudaError_t rowm(const Jobs& j, long long rows, cudaStream_t s) {
    return go(kd_row_mid<M, WM>, WM, NTM, SM_ROWM, rows, j, s, rows);
  }
  static cudaError_t r2c_plane(const Jobs& j, long long C, cudaStream_t s) {
    return go(kd_r2c_ax0<M, WM>, 2 * WM, NTM, SM_R2CP, C, j, s, C);
  }
  static cudaError_t c2r_plane(const Jobs& j, long long C, cudaStream_t s) {
    return go(kd_c2r_ax0<M, WM>, 2 * WM, NTM, SM_C2RP, C, j, s, C);
  }
  // 3-D DDI: the kernel reading's middle pass, the grid reading's C2R with the
  // local term and its unpadded passes of length M
  static cudaError_t colm_ddi(const Jobs& j, int M2, int planes, cudaStream_t s) {
    return mid(kd_col_mid<M, W, kMulDdiKernel>, SM_MID<true>, j, M2, planes, s);
  }
  static cudaError_t c2r_epi(const Jobs& j, long long C, cudaStream_t s) {
    return go(kd_c2r_ax0<M, WX, true, true>, 2 * WX, NTX, SM_C2R, C, j, s, C);
  }
  static cudaError_t r2c_per(const Jobs& j, long long C, cudaStream_t s) {
    return go(kd_r2c_ax0<M, WX, false>, 2 * WX, NTX, SM_R2C<false>, C, j, s, C);
  }
  static cudaError_t rowf_per(const Jobs& j, long long rows, cudaStream_t s) {
    return go(kd_row<M, W, true, false>, W, NT, (SM_ROW<true, false>), rows, j, s, rows);
  }
  static cudaError_t colm_per(const Jobs& j, int M2, int planes, cudaStream_t s) {
    return mid(kd_col_mid<M, W, kMulDdiGrid>, SM_MID<false>, j, M2, planes, s);
  }
  static cudaError_t rowi_per(const Jobs& j, long long rows, cudaStream_t s) {
    return go(kd_row<M, W, false, false>, W, NT, (SM_ROW<false, false>), rows, j, s, rows);
  }
  static cudaError_t c2r_per(const Jobs& j, long long C, cudaStream_t s) {
    return go(kd_c2r_ax0<M, WX, false>, 2 * WX, NTX, SM_C2R, C, j, s, C);
  }
};

}  // namespace detail
}  // namespace fsa

#define FSA_REG_DW(M) fsa::register_pass_fns(fsa::kArithDW, M, fsa::fns_of<fsa::detail::InstDw<M>>());
