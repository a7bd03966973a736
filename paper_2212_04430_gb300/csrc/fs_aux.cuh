// Z4 noise on the device, canonical <-> even-odd layout conversion, gauge packing.
#pragma once

#include "fs_hop.cuh"

namespace fs {

// ---- Philox4x32-10 (Salmon et al., SC'11), written from its definition ----
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; r++) {
    if (r > 0) { k.x += 0x9E3779B9u; k.y += 0xBB67AE85u; }
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

// Noise source of one tile slot: z(x, s, c) = i^k, k = (Philox(x, sample, level, job; seed).x >> 2(3s+c)) & 3.
// Probing and dilution (Sec. 2.1, Eq. (probing_vectors); Sec. 3.1) restrict it to the sites whose
// probing colour is `color` (NOISE_COLOR) and to the one spin-colour index comp = 3 s + c
// (NOISE_COMP): the pieces of one sample share its Z4 vector.
struct NoiseSpec {
  uint32_t key0, key1, job, level, sample;
  uint32_t flags;  // NOISE_* bits
  int32_t color;   // probing colour of the piece (NOISE_COLOR)
  int32_t comp;    // spin-colour index of the piece, 0..11 (NOISE_COMP)
};
// gamma_5 z ; has a noise identity ; z is the rhs ; colour-restricted ; one spin-colour index
enum { NOISE_G5 = 1, NOISE_VALID = 2, NOISE_RHS = 4, NOISE_COLOR = 8, NOISE_COMP = 16 };

// Spin-colour indices (bit j = 3 s + c) that noise n keeps at canonical site lex; colors is the
// probing colour of every site, read only for a colour-restricted source.
__device__ __forceinline__ unsigned noise_keep(const NoiseSpec& n, const int* colors, int lex) {
  unsigned keep = 0xFFFu;
  if ((n.flags & NOISE_COLOR) && colors[lex] != n.color) keep = 0u;
  if (n.flags & NOISE_COMP) keep &= 1u << n.comp;
  return keep;
}

__device__ __forceinline__ void z4_site(const NoiseSpec& n, int lex, double (&z)[24], unsigned keep = 0xFFFu) {
  const uint4 o = philox4x32_10(make_uint4((uint32_t)lex, n.sample, n.level, n.job), make_uint2(n.key0, n.key1));
#pragma unroll
  for (int j = 0; j < 12; j++) {
    const uint32_t k = (o.x >> (2 * j)) & 3u;
    const bool on = (keep >> j) & 1u;
    // i^k: 0 -> 1, 1 -> i, 2 -> -1, 3 -> -i
    double re = !on ? 0.0 : ((k == 0) ? 1.0 : ((k == 2) ? -1.0 : 0.0));
    double im = !on ? 0.0 : ((k == 1) ? 1.0 : ((k == 3) ? -1.0 : 0.0));
    if ((n.flags & NOISE_G5) && j >= 6) { re = -re; im = -im; }
    z[2 * j] = re;
    z[2 * j + 1] = im;
  }
}

// Finished slots to staged columns, all of them and their four parities in one launch (they were four copies
// and an upload each: 5 us of an 8^3 x 16 system, and as much of the host's time).
struct StageMoves {
  int n;
  short slot[64], col[64];
  char with_y[64];
};
#ifdef FS_ENGINE_KERNELS
// z for slots flagged INIT with a noise source, both parities (FP64 e/o tile fields).
__global__ void __launch_bounds__(256) noise_kernel(double* z_e, double* z_o, const NoiseSpec* spec,
                                                    const SysState* st, const int* colors, Geom g, Shape sh) {
  const int lsys = threadIdx.x % sh.NB, lsite = threadIdx.x / sh.NB;
  const int sys = blockIdx.y * sh.NB + lsys;
  if (sys >= sh.N || !(st[sys].flags & FLAG_INIT) || !(spec[sys].flags & NOISE_RHS)) return;
  const NoiseSpec n = spec[sys];
  for (int chunk = blockIdx.x; chunk < 2 * sh.nchunk; chunk += gridDim.x) {
    const int par = chunk >= sh.nchunk ? 1 : 0;
    const int site = (chunk - par * sh.nchunk) * sh.SB + lsite;
    if (site >= g.Vh) continue;
    int x[4];
    cb_coords(g, par, site, x);
    double z[24];
    const int lex = lex_index(g, x);
    z4_site(n, lex, z, noise_keep(n, colors, lex));
    make_field<double>(par ? z_o : z_e, g.Vh, sh.N, true).store(site, sys, z);
  }
}

struct StageArgs {
  StageMoves mv;
  const double* from[4];  // x even, x odd, y even, y odd
  double* to[4];
  const NoiseSpec* spec;
  NoiseSpec* stage_spec;
  size_t colsz;           // doubles of a column
};
__global__ void __launch_bounds__(256) stage_kernel(StageArgs a) {
  const int k = blockIdx.y >> 2, f = blockIdx.y & 3;
  if (f >= 2 && !a.mv.with_y[k]) return;
  const int slot = a.mv.slot[k], col = a.mv.col[k];
  const double2* src = reinterpret_cast<const double2*>(a.from[f] + (size_t)slot * a.colsz);
  double2* dst = reinterpret_cast<double2*>(a.to[f] + (size_t)col * a.colsz);
  const size_t n = a.colsz / 2, step = (size_t)gridDim.x * 256;  // colsz = 24 Vh
  size_t i = blockIdx.x * (size_t)256 + threadIdx.x;
  for (; i + 3 * step < n; i += 4 * step) {
    const double2 v0 = src[i], v1 = src[i + step], v2 = src[i + 2 * step], v3 = src[i + 3 * step];
    dst[i] = v0;
    dst[i + step] = v1;
    dst[i + 2 * step] = v2;
    dst[i + 3 * step] = v3;
  }
  for (; i < n; i += step) dst[i] = src[i];
  if (f == 0 && blockIdx.x == 0 && threadIdx.x == 0) a.stage_spec[col] = a.spec[slot];
}

// Integer Z4 codes of one noise vector in canonical order (bit-exact RNG check).
__global__ void noise_codes_kernel(uint8_t* codes, NoiseSpec n, int V) {
  const int lex = blockIdx.x * blockDim.x + threadIdx.x;
  if (lex >= V) return;
  const uint4 o = philox4x32_10(make_uint4((uint32_t)lex, n.sample, n.level, n.job), make_uint2(n.key0, n.key1));
#pragma unroll
  for (int j = 0; j < 12; j++) codes[(size_t)lex * 12 + j] = (uint8_t)((o.x >> (2 * j)) & 3u);
}
#endif  // FS_ENGINE_KERNELS

// canonical FP64 [nvec][V][24]  ->  e/o tile fields of type Ts (slot j <- vector vec[j], -1 skips)
template <typename Ts>
__global__ void __launch_bounds__(256) pack_kernel(void* f_e, void* f_o, const double* canon, const int* vec,
                                                  Geom g, Shape sh, bool sysmajor) {
  const int lsys = threadIdx.x % sh.NB, lsite = threadIdx.x / sh.NB;
  const int sys = blockIdx.y * sh.NB + lsys;
  if (sys >= sh.N) return;
  const int vi = vec[sys];
  if (vi < 0) return;
  for (int chunk = blockIdx.x; chunk < 2 * sh.nchunk; chunk += gridDim.x) {
    const int par = chunk >= sh.nchunk ? 1 : 0;
    const int site = (chunk - par * sh.nchunk) * sh.SB + lsite;
    if (site >= g.Vh) continue;
    int x[4];
    cb_coords(g, par, site, x);
    const double* src = canon + ((size_t)vi * g.V + lex_index(g, x)) * 24;
    double v[24];
#pragma unroll
    for (int k = 0; k < 24; k += 2) {
      const double2 w = *reinterpret_cast<const double2*>(src + k);
      v[k] = w.x; v[k + 1] = w.y;
    }
    make_field<Ts>(par ? f_o : f_e, g.Vh, sh.N, sysmajor).store(site, sys, v);
  }
}

template <typename Ts>
__global__ void __launch_bounds__(256) unpack_kernel(double* canon, const void* f_e, const void* f_o,
                                                    const int* vec, Geom g, Shape sh, bool sysmajor) {
  const int lsys = threadIdx.x % sh.NB, lsite = threadIdx.x / sh.NB;
  const int sys = blockIdx.y * sh.NB + lsys;
  if (sys >= sh.N) return;
  const int vi = vec[sys];
  if (vi < 0) return;
  for (int chunk = blockIdx.x; chunk < 2 * sh.nchunk; chunk += gridDim.x) {
    const int par = chunk >= sh.nchunk ? 1 : 0;
    const int site = (chunk - par * sh.nchunk) * sh.SB + lsite;
    if (site >= g.Vh) continue;
    int x[4];
    cb_coords(g, par, site, x);
    double v[24];
    make_field<Ts>(const_cast<void*>(par ? f_o : f_e), g.Vh, sh.N, sysmajor).load(site, sys, v);
    double* dst = canon + ((size_t)vi * g.V + lex_index(g, x)) * 24;
#pragma unroll
    for (int k = 0; k < 24; k += 2) *reinterpret_cast<double2*>(dst + k) = make_double2(v[k], v[k + 1]);
  }
}

// canonical FP64 links [4][V][18] -> [parity][mu][Vh][RP] of type Tg, NR = 18 or 12 stored reals
template <typename Tg, int NR>
__global__ void gauge_pack_kernel(void* out, const double* canon, Geom g) {
  constexpr int RP = link_pad<Tg>(NR);
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 8 * g.Vh) return;
  const int site = idx % g.Vh;
  const int pm = idx / g.Vh;  // parity * 4 + mu
  const int par = pm / 4, mu = pm % 4;
  int x[4];
  cb_coords(g, par, site, x);
  const double* src = canon + ((size_t)mu * g.V + lex_index(g, x)) * 18;
  Tg* dst = reinterpret_cast<Tg*>(out) + ((size_t)pm * g.Vh + site) * RP;
  constexpr int VW = Store<Tg>::VW;
  double tmp[RP];
#pragma unroll
  for (int k = 0; k < RP; k++) tmp[k] = k < NR ? src[k] : 0.0;
#pragma unroll
  for (int c = 0; c < RP / VW; c++) store_vec<Tg, double>(dst + c * VW, tmp + c * VW);
}

}  // namespace fs
