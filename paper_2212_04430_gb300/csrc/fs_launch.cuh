// Kernel launchers, instantiated once per storage precision (fs_kern_*.cu).
#pragma once

#include <algorithm>

#include "fs_engine.h"

namespace fs {

template <typename Ts>
using MathOf = typename std::conditional<std::is_same<Ts, double>::value, double, float>::type;

// Directions kept in flight by the prefetching hop kernel (shared-memory ring slots).
template <typename Ts> constexpr int hop_pf() { return sizeof(Ts) == 2 ? 4 : 3; }

// Ring depth of the persistent paired kernel: four operands in flight for 16-bit storage
// (measured on the 16^3x32 hop: 2 or 3 slots leave the 10-operand launches waiting on L2), which
// keeps three 128-thread blocks resident per SM; FP32 storage has twice the bytes per operand.
// The autotuner may pick the other depth of hop_pk_depths for a tile.
template <typename Ts>
constexpr int hop_pk_depth() {
  return sizeof(Ts) <= 2 ? 4 : 2;
}
template <typename Ts>
constexpr int hop_pk_alt_depth() {
  return 3;
}

// The persistent paired hop for 32-system chunks (hop_kernel_pk) at ring depth PF: 128-thread
// blocks of 8 sites, as many as are resident (capped at l.pk_blocks per SM when set), never more
// blocks than site chunks.
template <typename Ts, typename Tg, int R, int C, int D, int PF, bool CLV = false, int LPS = 16>
cudaError_t launch_hop_pk_at(const HopArgs& a, const Launch& l) {
  auto kern = hop_kernel_pk<Ts, Tg, R, C, D, PF, CLV, LPS>;
  const size_t smem = hop_pk_smem<Ts, PF, DotK<D>::K>();
  const LaunchSetup pg = launch_setup((const void*)kern, smem, 128);
  if (pg.err) return pg.err;
  const int per_sm = l.pk_blocks > 0 ? std::min(l.pk_blocks, pg.blocks_per_sm) : pg.blocks_per_sm;
  const int gy = l.grid_y;
  const int gx = std::max(1, std::min(a.sh.nchunk, per_sm * pg.nsm / std::max(gy, 1)));
  kern<<<dim3(gx, gy), 128, smem, l.stream>>>(a);
  note_launch();
  return cudaGetLastError();
}

template <typename Ts, typename Tg, typename Tm, int R, int C, int D, bool CLV = false>
cudaError_t launch_hop_pk(const HopArgs& a, const Launch& l) {
  if (l.pk_depth == hop_pk_alt_depth<Ts>())
    return launch_hop_pk_at<Ts, Tg, R, C, D, hop_pk_alt_depth<Ts>(), CLV>(a, l);
  return launch_hop_pk_at<Ts, Tg, R, C, D, hop_pk_depth<Ts>(), CLV>(a, l);
}

// the shapes the persistent paired kernel serves: 32-system chunks of 8 sites
inline bool pk_shape(const HopArgs& a, const Launch& l) { return a.sh.NB == 32 && a.sh.SB == 8 && l.block == 256; }
// Systems of a chunk (32, 16 or 8) with which it takes a tile of N systems in a solve, by the padded count at each
// chunk's cost per system; 0: the other kernels do. Shifted solves on 12^3 x 16 / 16^3 x 32 in FP16, ms, hop_kernel_pf
// and chunks of 8 / 16 / 32: N = 3 5.6 | 6.1 / 6.6 / 10.2 and 15.1 | 16.1 / 24.5 / 38.0; N = 4 5.8 | 5.7 / 6.7 / 9.4 and
// 19.7 | 16.9 / 23.1 / 37.1; N = 8 8.8 | 7.1 / 8.0 / 10.8 and 32.1 | 23.4 / 28.5 / 43.4; N = 12 11.4 | 10.1 / 10.0 / 12.1
// and 51.1 | 38.3 / 33.9 / 47.7; N = 24 21.8 | 15.1 / 16.1 / 15.9 and 100.7 | 61.2 / 62.8 / 62.0; N = 48 39.3 | 27.0 /
// 25.3 / 27.1 and 207 | 122 / 110 / 120; N = 60 47.1 | 34.4 / 31.3 / 31.1 and 243 | 161 / 146 / 145. FP32, 16^3 x 32:
// N = 2 12.3 | 17.3, N = 4 22.3 | 20.4, N = 24 110 | 82 / 76 / 73, N = 48 219 | 172 / 137 / 143.
template <typename Ts>
int pk_chunk(int N) {
  if (N < 4) return 0;
  const int c8 = (N + 7) / 8 * 8 * (sizeof(Ts) == 2 ? 130 : 150), c16 = (N + 15) / 16 * 16 * 105;
  const int c32 = (N + 31) / 32 * 32 * 100;
  return c32 <= c16 && c32 <= c8 ? 32 : (c16 <= c8 ? 16 : 8);
}

template <typename Ts, typename Tg, typename Tm, int R, int C, int D, bool CLV>
cudaError_t launch_hop_chunks(const HopArgs& a, const Launch& l, int nb) {
  HopArgs b = a;
  Launch m = l;
  b.sh.NB = nb;
  b.sh.SB = 256 / nb;
  b.sh.nchunk = (a.g.Vh + b.sh.SB - 1) / b.sh.SB;
  m.grid_y = (a.sh.N + nb - 1) / nb;
  if (nb == 8) return launch_hop_pk_at<Ts, Tg, R, C, D, hop_pk_depth<Ts>(), CLV, 4>(b, m);
  if (nb == 16) return launch_hop_pk_at<Ts, Tg, R, C, D, hop_pk_depth<Ts>(), CLV, 8>(b, m);
  return launch_hop_pk<Ts, Tg, Tm, R, C, D, CLV>(b, m);
}

template <typename Ts, typename Tg, typename Tm, int R, int C, int D>
cudaError_t launch_hop_pf(const HopArgs& a, const Launch& l) {
  if (a.sysmajor) return cudaErrorInvalidValue;  // inner-precision fields are tile-layout only
  // 32-system chunks, 8 sites per block: the persistent paired kernel
  if (pk_shape(a, l)) return launch_hop_pk<Ts, Tg, Tm, R, C, D>(a, l);
  if constexpr (C != COEF_DSLASH)
    if (const int nb = pk_chunk<Ts>(a.sh.N)) return launch_hop_chunks<Ts, Tg, Tm, R, C, D, false>(a, l, nb);
  constexpr int PF = hop_pf<Ts>();
  const size_t smem = hop_pf_smem<Ts, PF>(l.block);
  auto kern = hop_kernel_pf<Ts, Tg, Tm, R, C, D, PF>;
  if (cudaError_t e = launch_setup((const void*)kern, hop_pf_smem<Ts, PF>(256), 256).err) return e;
  kern<<<dim3(l.grid_x, l.grid_y), l.block, smem, l.stream>>>(a);
  note_launch();
  return cudaGetLastError();
}

// FP64 fields: the hop in integer arithmetic (fs_hopfx.cuh), over the tile or the system-major work list
inline cudaError_t launch_hop_fx(int coef, int dot, const HopArgs& a, const Launch& l) {
  const bool wl = a.sysmajor != 0, fi = a.in_ex != nullptr, fo = a.out_ex != nullptr;
  // Wilson-clover M-hat and D_sw: C X comes in through Y
  const bool clv = a.clover && (coef == COEF_MHAT || coef == COEF_DSLASH);
#define FS_FX(C, D, WL, CLV, FI, FO)                                                                  \
  if (coef == C && dot == D && wl == WL && clv == CLV && fi == FI && fo == FO) {                      \
    note_launch();                                                                                    \
    if constexpr (!WL)                                                                                \
      if (fx_few(a.sh.N, a.g.Vh)) return launch_hop_fx_at(hop_kernel_fx<C, D, WL, CLV, FI, FO, true>, a, l.stream); \
    return launch_hop_fx_at(hop_kernel_fx<C, D, WL, CLV, FI, FO>, a, l.stream);                       \
  }
  FS_FX(COEF_PLAIN, DOT_NONE, false, false, false, false)    // FP64 storage: the iteration's hops
  FS_FX(COEF_MHAT, DOT_R, false, false, false, false)
  FS_FX(COEF_MHAT, DOT_TS, false, false, false, false)
  FS_FX(COEF_MHAT, DOT_R, false, true, false, false)
  FS_FX(COEF_MHAT, DOT_TS, false, true, false, false)
  FS_FX(COEF_DSLASH, DOT_NONE, false, false, false, false)
  FS_FX(COEF_DSLASH, DOT_NONE, false, true, false, false)
  FS_FX(COEF_PLAIN, DOT_NONE, true, false, true, true)       // reliable updates
  FS_FX(COEF_PLAIN, DOT_NONE, true, false, true, false)      // (Wilson-clover: a pass follows)
  FS_FX(COEF_TRUERES, DOT_NORM, true, false, true, false)
  FS_FX(COEF_TRUERES, DOT_NORM, true, false, false, false)   // (Wilson-clover, CGNR fallback)
  FS_FX(COEF_PREP, DOT_NORM, true, false, false, false)
  FS_FX(COEF_RECON, DOT_NONE, true, false, false, false)
  FS_FX(COEF_FULLRES, DOT_NORM, true, false, false, false)
  FS_FX(COEF_KAPPA, DOT_NONE, true, false, false, false)     // hopping parameter expansion
  FS_FX(COEF_PLAIN, DOT_NONE, true, false, false, false)     // CGNR fallback
  FS_FX(COEF_MHAT, DOT_NORM, true, false, false, false)      // q = M p, ||q||^2
  FS_FX(COEF_MHAT, DOT_NONE, true, false, false, false)      // M gamma5 s
  FS_FX(COEF_MHAT, DOT_NORM, true, true, false, false)
  FS_FX(COEF_MHAT, DOT_NONE, true, true, false, false)
#undef FS_FX
  return cudaErrorInvalidValue;
}

template <typename Ts>
cudaError_t launch_hop(int coef, int dot, int nr, const HopArgs& a, const Launch& l) {
  if constexpr (std::is_same<Ts, double>::value) {
    return nr == 18 ? launch_hop_fx(coef, dot, a, l) : cudaErrorInvalidValue;
  } else {
    using Tg = typename GaugeOf<Ts>::T;
    using Tm = MathOf<Ts>;
    const dim3 grid(l.grid_x, l.grid_y), block(l.block);
    if (a.sysmajor) return cudaErrorInvalidValue;  // inner-precision fields are tile-layout only
    // Wilson-clover M-hat and D_sw on the tile layout, with the Y operand (C X): the persistent
    // paired kernel for the M-hat of four systems or more, else the generic one
#define FS_HOP_CLV(C, D, R)                                                                  \
  if (coef == C && dot == D && nr == R) {                                                    \
    if constexpr (C == COEF_MHAT)                                                            \
      if (const int nb = pk_chunk<Ts>(a.sh.N))                                               \
        return launch_hop_chunks<Ts, Tg, Tm, R, C, D, true>(a, l, nb);                       \
    hop_kernel<Ts, Tg, Tm, R, C, D><<<grid, block, 0, l.stream>>>(a);                        \
    note_launch();                                                                           \
    return cudaGetLastError();                                                               \
  }
    if (a.clover && (coef == COEF_MHAT || coef == COEF_DSLASH)) {
      FS_HOP_CLV(COEF_MHAT, DOT_R, 18)
      FS_HOP_CLV(COEF_MHAT, DOT_TS, 18)
      FS_HOP_CLV(COEF_DSLASH, DOT_NONE, 18)
      FS_HOP_CLV(COEF_MHAT, DOT_R, 12)
      FS_HOP_CLV(COEF_MHAT, DOT_TS, 12)
      FS_HOP_CLV(COEF_DSLASH, DOT_NONE, 12)
      return cudaErrorInvalidValue;
    }
#undef FS_HOP_CLV
#define FS_HOP_PF(C, D, R) \
  if (coef == C && dot == D && nr == R) return launch_hop_pf<Ts, Tg, Tm, R, C, D>(a, l);
    FS_HOP_PF(COEF_PLAIN, DOT_NONE, 18)
    FS_HOP_PF(COEF_DSLASH, DOT_NONE, 18)
    FS_HOP_PF(COEF_MHAT, DOT_R, 18)
    FS_HOP_PF(COEF_MHAT, DOT_TS, 18)
    FS_HOP_PF(COEF_PLAIN, DOT_NONE, 12)
    FS_HOP_PF(COEF_DSLASH, DOT_NONE, 12)
    FS_HOP_PF(COEF_MHAT, DOT_R, 12)
    FS_HOP_PF(COEF_MHAT, DOT_TS, 12)
#undef FS_HOP_PF
    return cudaErrorInvalidValue;
  }
}

template <typename Ts>
cudaError_t launch_blas(int op, const BlasArgs& a, const Launch& l) {
  using Tx = typename XOf<Ts>::T;
  using Tm = MathOf<Ts>;
  const dim3 grid(l.grid_x, l.grid_y), block(l.block);
  // the per-iteration solver updates run on the tile shape; the FP64-field operations
  // (x_hi updates, residual restarts, norms) on the system-major work list
  if ((op == OP_S || op == OP_XRP) == (a.sysmajor != 0)) return cudaErrorInvalidValue;
  switch (op) {
    case OP_S: blas_kernel<Ts, Tx, Tm, OP_S, false><<<grid, block, 0, l.stream>>>(a); break;
    case OP_XRP: blas_kernel<Ts, Tx, Tm, OP_XRP, false><<<grid, block, 0, l.stream>>>(a); break;
    case OP_ACCX: blas_kernel<Ts, Tx, Tm, OP_ACCX, true><<<grid, block, 0, l.stream>>>(a); break;
    case OP_ZEROX: blas_kernel<Ts, Tx, Tm, OP_ZEROX, true><<<grid, block, 0, l.stream>>>(a); break;
    case OP_SETR: blas_kernel<Ts, Tx, Tm, OP_SETR, true><<<grid, block, 0, l.stream>>>(a); break;
    case OP_NORM64: blas_kernel<Ts, Tx, Tm, OP_NORM64, true><<<grid, block, 0, l.stream>>>(a); break;
    case OP_RECON: blas_kernel<Ts, Tx, Tm, OP_RECON, true><<<grid, block, 0, l.stream>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  note_launch();
  return cudaGetLastError();
}

template <typename Ts, typename Tg, int NR>
cudaError_t launch_small_at(const SmallArgs& a, cudaStream_t s) {
  auto kern = small_iter_kernel<Ts, Tg, NR>;
  const SmallShape sh = small_shape(a.g.Vh);
  const size_t smem = (size_t)(sh.threads / 32) * FX_WARP_WORDS * 16;
  // (256 threads at most, 128 with FP64 storage)
  const int most = std::is_same<Ts, double>::value ? 128 : 256;
  if (cudaError_t e = launch_setup((const void*)kern, (size_t)(most / 32) * FX_WARP_WORDS * 16, most).err) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(a.N * sh.cluster);
  cfg.blockDim = dim3(sh.threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = sh.cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  note_launch();
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <typename Ts>
cudaError_t launch_small(int nr, const SmallArgs& a, cudaStream_t s) {
  using Tg = typename GaugeOf<Ts>::T;
  if (nr == 18) return launch_small_at<Ts, Tg, 18>(a, s);
  if constexpr (!std::is_same<Ts, double>::value)
    if (nr == 12) return launch_small_at<Ts, Tg, 12>(a, s);
  return cudaErrorInvalidValue;
}

template <typename Ts>
cudaError_t launch_clover(int mode, const ClovArgs& a, const Launch& l) {
  using Tm = MathOf<Ts>;
  using Tc = typename std::conditional<std::is_same<Ts, double>::value, double, float>::type;
  const dim3 grid(l.grid_x, l.grid_y), block(l.block);
  if (a.sysmajor && !std::is_same<Ts, double>::value) return cudaErrorInvalidValue;  // FP64 fields only
  // the paired pass where the block rows hold an even number of systems that divides 512
  const bool paired = !std::is_same<Ts, double>::value && !a.sysmajor && a.sh.NB % 2 == 0 && 256 % (a.sh.NB / 2) == 0;
#define FS_CLV(M)                                                                                         \
  if (mode == M) {                                                                                        \
    if constexpr (!std::is_same<Ts, double>::value)                                                       \
      if (paired) {                                                                                       \
        clover_kernel_pk<Ts, M><<<grid, 256, 0, l.stream>>>(a);                                           \
        note_launch();                                                                                    \
        return cudaGetLastError();                                                                        \
      }                                                                                                   \
    if (a.sysmajor) clover_kernel<Ts, Tc, Tm, M, true><<<grid, block, 0, l.stream>>>(a);                 \
    else clover_kernel<Ts, Tc, Tm, M, false><<<grid, block, 0, l.stream>>>(a);                           \
    note_launch();                                                                                        \
    return cudaGetLastError();                                                                            \
  }
  FS_CLV(CLV_MUL)
  FS_CLV(CLV_SUB)
  FS_CLV(CLV_INV)
  if (mode == CLV_INV_MUL) {  // tile layout only
    if (a.sysmajor) return cudaErrorInvalidValue;
    if constexpr (!std::is_same<Ts, double>::value)
      if (paired) {
        clover_kernel_pk<Ts, CLV_INV_MUL><<<grid, 256, 0, l.stream>>>(a);
        note_launch();
        return cudaGetLastError();
      }
    clover_kernel<Ts, Tc, Tm, CLV_INV_MUL, false><<<grid, block, 0, l.stream>>>(a);
    note_launch();
    return cudaGetLastError();
  }
#undef FS_CLV
  return cudaErrorInvalidValue;
}

template <typename Ts>
cudaError_t launch_pack(void* fe, void* fo, const double* canon, const int* vec, const Geom& g, const Shape& sh,
                        const Launch& l, bool sysmajor) {
  pack_kernel<Ts><<<dim3(l.grid_x, l.grid_y), l.block, 0, l.stream>>>(fe, fo, canon, vec, g, sh, sysmajor);
  note_launch();
  return cudaGetLastError();
}

template <typename Ts>
cudaError_t launch_unpack(double* canon, const void* fe, const void* fo, const int* vec, const Geom& g,
                          const Shape& sh, const Launch& l, bool sysmajor) {
  unpack_kernel<Ts><<<dim3(l.grid_x, l.grid_y), l.block, 0, l.stream>>>(canon, fe, fo, vec, g, sh, sysmajor);
  note_launch();
  return cudaGetLastError();
}

template <typename Tg>
cudaError_t launch_gauge_pack(void* out, const double* canon, const Geom& g, int nr, cudaStream_t s) {
  const int n = 8 * g.Vh;
  const int blocks = (n + 255) / 256;
  if (nr == 18) gauge_pack_kernel<Tg, 18><<<blocks, 256, 0, s>>>(out, canon, g);
  else if (nr == 12) gauge_pack_kernel<Tg, 12><<<blocks, 256, 0, s>>>(out, canon, g);
  else return cudaErrorInvalidValue;
  note_launch();
  return cudaGetLastError();
}

#define FS_INSTANTIATE(TS)                                                                                   \
  template cudaError_t launch_hop<TS>(int, int, int, const HopArgs&, const Launch&);                        \
  template cudaError_t launch_small<TS>(int, const SmallArgs&, cudaStream_t);                               \
  template cudaError_t launch_blas<TS>(int, const BlasArgs&, const Launch&);                                \
  template cudaError_t launch_clover<TS>(int, const ClovArgs&, const Launch&);                              \
  template cudaError_t launch_pack<TS>(void*, void*, const double*, const int*, const Geom&, const Shape&,   \
                                       const Launch&, bool);                                                \
  template cudaError_t launch_unpack<TS>(double*, const void*, const void*, const int*, const Geom&,         \
                                         const Shape&, const Launch&, bool);

}  // namespace fs
