// The FP64 hopping kernel in integer arithmetic.
//
// GB300 issues FP64 multiply-adds at 0.62 T/s (2 a clock per SM) and 32x32+64-bit integer
// multiply-adds (mad.wide) at 18.9 T/s. An FP64 hop in FP64 instructions is bound by that pipe (1.5 ns per
// (site, system), 0.74 of its rate), so its products are formed on the integer units instead:
//  - a neighbour spinor is brought to 60-bit integers under its own exponent (the largest of its
//    24 entries), a link to 59-bit integers under its own, when the links are packed
//    (gauge_fx_kernel);
//  - an integer is two limbs, v = v1 2^32 + v0 with v0 signed, and a product is the three 64-bit products
//    hh += a1 b1, xx += a1 b0 + a0 b1, rounded in units of 2^64 as hh + ((xx + 2^31) >> 32): a dropped
//    a0 b0 is at most a quarter of a unit, and |xx| < 7.5 x 2^60 over the six terms;
//  - the eight directions are summed as integers under a running exponent, and only the sums
//    go back to FP64, where the epilogue and the dot products stay.
// The unit of the sum is 2^-55 of the largest neighbouring entry, its range 2^61.6 of 2^63. Error of H psi
// against 80-bit arithmetic (Gaussian spinors, Haar links): 0.4 x 2^-53 of its rms, the FP64 chains' 1.4 x 2^-53.
// The exponents are per spinor and per link, so any finite field is taken: spinors of tiny entries are rescaled
// (fx_spinor), zero ones add nothing, non-finite ones give NaN in all 24 entries of the sites that read them. The precision
// is that of a spinor's (a link's) largest entry: an entry more than 2^7 below it has fewer than 53 bits and one 2^60
// below counts as zero. Sums over colours and spins round small results to that anyway; where links do not mix the colours
// (diagonal ones), FP64 chains would keep each colour's own 53 bits and this hop does not.
// Measured at 16^3x32, 8 systems: a reliable update's two hops 1.50 + 1.61 -> 0.40 + 0.49 ns per (site,
// system), the preparation's 1.52 -> 0.62 ns (its input is converted in the hop). What bounds it now: the FMA-heavy pipe
// that mad.wide runs on (54% busy in an update's first hop) and the latency of 11 warps an SM (issue 48%, the
// largest stall fixed-latency dependencies); the preparation adds the conversions on the ALU pipe (52%).
#pragma once

#include <algorithm>
#include <climits>

#include "fs_device.h"
#include "fs_hop.cuh"

namespace fs {

// ---- links ------------------------------------------------------------------------------------
// [parity][mu][entry 9][Vh] of {re1, re0, im1, im0}: consecutive sites are consecutive 16-byte words
// (the work lists run one system over consecutive sites), and a site's word is one broadcast where a
// warp holds its systems. |b| < 2^59, b1 in 28 bits and a sign; the link's exponent (biased by 1023 + 64: links
// below the smallest normal double have one too) is in the top three bits of the four b1 of entries 0 and 4. The t
// boundary phase is folded into the links.
constexpr int FX_BITS = 60;       // spinors
constexpr int FX_LINK_BITS = 59;  // links
constexpr int FX_LINK_BIAS = 64;
constexpr int FX_LINK_BAD = 0xfff;  // exponent of a link with an entry that is not finite
__host__ __device__ constexpr size_t fx_gauge_bytes(int Vh) { return (size_t)8 * 9 * Vh * sizeof(int4); }

// The products negate low limbs in 32 bits, which -2^31 does not survive: an integer of which a low limb is
// negated (links; the left vectors of a contraction) is moved away from zero by one unit where its low word is
// 0x80000000: odd multiples of 2^-28 of the link's power of two. Random doubles meet that once in 10^8; of links
// that were once stored in single precision a quarter have such an entry.
__device__ __forceinline__ long long fx_negatable(long long v) {
  return (int)v == INT_MIN ? v + (v < 0 ? -1 : 1) : v;
}
// v = hi 2^32 + lo, lo signed (the low word as it is)
__device__ __forceinline__ void fx_limbs(long long v, int& hi, int& lo) {
  lo = (int)v;
  hi = (int)(v >> 32) - (lo >> 31);
}

// A matrix of doubles as a link's nine words
__device__ __forceinline__ void fx_link(const double (&u)[18], int4 (&o)[9]) {
  unsigned m = 0;
#pragma unroll
  for (int k = 0; k < 18; k++) m = max(m, (unsigned)__double2hiint(u[k]) & 0x7fffffffu);
  int e = (int)(m >> 20);
  const bool bad = e == 0x7ff;
  if (e == 0) {  // all below the smallest normal double
    m = 0;
#pragma unroll
    for (int k = 0; k < 18; k++) m = max(m, (unsigned)__double2hiint(u[k] * 0x1p512) & 0x7fffffffu);
    e = m == 0 ? -FX_LINK_BIAS : (int)(m >> 20) - 512;
  }
  const int ex = bad ? FX_LINK_BAD : e + FX_LINK_BIAS;
#pragma unroll
  for (int k = 0; k < 9; k++) {
    long long v[2];
#pragma unroll
    for (int q = 0; q < 2; q++)
      v[q] = bad ? 0 : fx_negatable(__double2ll_rn(scalbn(u[2 * k + q], FX_LINK_BITS + 1022 - e)));
    int4 w;
    fx_limbs(v[0], w.x, w.y);
    fx_limbs(v[1], w.z, w.w);
    if (k == 0 || k == 4) {
      const int sh = k == 0 ? 0 : 6;
      w.x = (w.x & 0x1fffffff) | (((ex >> sh) & 7) << 29);
      w.z = (w.z & 0x1fffffff) | (((ex >> (sh + 3)) & 7) << 29);
    }
    o[k] = w;
  }
}
// a link's exponent, from words 0 and 4, and these two without it
__device__ __forceinline__ int fx_link_exponent(const int4& w0, const int4& w4) {
  return (int)(((unsigned)w0.x >> 29) | (((unsigned)w0.z >> 29) << 3) | (((unsigned)w4.x >> 29) << 6) |
               (((unsigned)w4.z >> 29) << 9));
}

#ifdef FS_ENGINE_KERNELS
// canonical FP64 links [4][V][18] -> the integer links
__global__ void __launch_bounds__(256) gauge_fx_kernel(int4* out, const double* canon, Geom g) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 8 * g.Vh) return;
  const int site = idx % g.Vh;
  const int pm = idx / g.Vh;  // parity * 4 + mu
  const int mu = pm % 4;
  int x[4];
  cb_coords(g, pm / 4, site, x);
  const double* src = canon + ((size_t)mu * g.V + lex_index(g, x)) * 18;
  const double sgn = (mu == 3 && x[3] == g.L[3] - 1) ? (double)g.bc_t : 1.0;
  double u[18];
#pragma unroll
  for (int k = 0; k < 18; k++) u[k] = sgn * src[k];
  int4 w[9];
  fx_link(u, w);
#pragma unroll
  for (int k = 0; k < 9; k++) out[((size_t)pm * 9 + k) * g.Vh + site] = w[k];
}
#endif  // FS_ENGINE_KERNELS

// ---- spinors -----------------------------------------------------------------------------------
constexpr int FX_ZERO = -100000;  // exponent of a spinor of zeros: below every sum's
constexpr int FX_BAD = 1 << 20;   // exponent of a spinor with an entry that is not finite

// 24 doubles -> integers below 2^60 (truncated) under the returned biased exponent. On the integer
// pipes: cvt.rni.s64.f64 issues at the FP64 rate here (0.62 T/s measured), and a hop converts every spinor in
// each of its eight neighbours: with it the hop took 0.85 ns per (site, system), half of it conversions.
__device__ __forceinline__ int fx_spinor(double (&v)[24], long long (&p)[24]) {
  unsigned m = 0;
#pragma unroll
  for (int k = 0; k < 24; k++) m = max(m, (unsigned)__double2hiint(v[k]) << 1);
  int e = (int)(m >> 21), es = e;
  if ((unsigned)(e - 70) > 1900u) {
    if (e == 0x7ff) {
      e = FX_BAD;
    } else if (e < 70) {
      // entries all below 1e-286: scaled up, so that zeros shift out below (e, which stands for the
      // spinor in the sum, may leave a double's range)
      const double f = __hiloint2double((512 + 1023) << 20, 0);
      m = 0;
#pragma unroll
      for (int k = 0; k < 24; k++) {
        v[k] *= f;
        m = max(m, (unsigned)__double2hiint(v[k]) << 1);
      }
      es = (int)(m >> 21);
      e = es - 512;
      if (m == 0) { es = 1023; e = FX_ZERO; }
    }
  }
  const int c = es + 64 - FX_BITS;
#pragma unroll
  for (int k = 0; k < 24; k++) {
    const unsigned hi = (unsigned)__double2hiint(v[k]), lo = (unsigned)__double2loint(v[k]);
    // the mantissa with its leading one at bit 63, shifted down; a zero (exponent 0) shifts out
    unsigned long long w = ((unsigned long long)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | (lo << 11);
    const int sh = c - (int)((hi << 1) >> 21);
    asm("shr.u64 %0, %0, %1;" : "+l"(w) : "r"(sh));
    const long long sg = (long long)((int)hi >> 31);
    p[k] = ((long long)w ^ sg) - sg;
  }
  return e;
}

// a 2^(es - 1023) on the integer pipes, rounded to nearest (ties up in magnitude), 70 <= es <= 1870
__device__ __forceinline__ double fx_double(long long a, int es) {
  const int sg = (int)(a >> 63);
  unsigned long long w = (unsigned long long)((a ^ (long long)sg) - (long long)sg);
  const int z = __clzll((long long)w);
  asm("shl.b64 %0, %0, %1;" : "+l"(w) : "r"(z));  // leading one at bit 63
  const unsigned long long r = (w >> 11) + ((w >> 10) & 1);  // the leading one adds 1 to the exponent below
  const unsigned hi = ((unsigned)(r >> 32) + ((unsigned)(es + 62 - z) << 20)) | ((unsigned)sg & 0x80000000u);
  return w == 0 ? 0.0 : __hiloint2double((int)hi, (int)r);
}

// ---- the hop ---------------------------------------------------------------------------------------
// Upper spins of (1 + S gamma_MU) psi (project(), on integers)
template <int MU, int S>
__device__ __forceinline__ void fx_project(const long long (&p)[24], long long (&w)[12]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const long long p2r = p[12 + 2 * c], p2i = p[13 + 2 * c], p3r = p[18 + 2 * c], p3i = p[19 + 2 * c];
    long long g0r, g0i, g1r, g1i;  // G psi_dn
    if (MU == 0) {
      g0r = -p3i; g0i = p3r; g1r = -p2i; g1i = p2r;
    } else if (MU == 1) {
      g0r = -p3r; g0i = -p3i; g1r = p2r; g1i = p2i;
    } else if (MU == 2) {
      g0r = -p2i; g0i = p2r; g1r = p3i; g1i = -p3r;
    } else {
      g0r = p2r; g0i = p2i; g1r = p3r; g1i = p3i;
    }
    w[2 * c] = p[2 * c] + S * g0r;
    w[2 * c + 1] = p[2 * c + 1] + S * g0i;
    w[6 + 2 * c] = p[6 + 2 * c] + S * g1r;
    w[7 + 2 * c] = p[7 + 2 * c] + S * g1i;
  }
}

// lower spins of acc += S G^dag z
template <int MU, int S>
__device__ __forceinline__ void fx_lower(long long (&acc)[24], const long long (&z)[12]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const long long z0r = z[2 * c], z0i = z[2 * c + 1], z1r = z[6 + 2 * c], z1i = z[7 + 2 * c];
    long long d0r, d0i, d1r, d1i;  // G^dag z
    if (MU == 0) {
      d0r = z1i; d0i = -z1r; d1r = z0i; d1i = -z0r;
    } else if (MU == 1) {
      d0r = z1r; d0i = z1i; d1r = -z0r; d1i = -z0i;
    } else if (MU == 2) {
      d0r = z0i; d0i = -z0r; d1r = -z1i; d1i = z1r;
    } else {
      d0r = z0r; d0i = z0i; d1r = z1r; d1i = z1i;
    }
    acc[12 + 2 * c] += S * d0r; acc[13 + 2 * c] += S * d0i;
    acc[18 + 2 * c] += S * d1r; acc[19 + 2 * c] += S * d1i;
  }
}

// a b + c as the one instruction it is (written in C++, products of a negated operand become a wide
// multiply and a 64-bit subtraction: 1068 instructions a direction instead of 662)
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
// The eight directions are a rolled loop, only the spin projections and additions unrolled: all of it unrolled is
// 80 to 150 KB of instructions, more than the instruction caches hold (no_instruction was then the largest stall).
// A warp works alone on `nst` consecutive sites of 32 / nst systems. The next direction's spinors (12 words of
// 16 bytes a lane) and links (9 words a site, once for the systems that share it) come through shared
// memory by cp.async while the current one is computed: about 700 instructions (1100 with FP64 input) on 3
// warps a scheduler, which with plain loads waited on memory for more than half of their time.
constexpr int FX_WARP_WORDS = 12 * 32 + 9 * 32;  // 16-byte words per warp
constexpr int FX_BLOCK = 128;  // three blocks per SM (168 registers; four, at 128, measured 6% slower)
constexpr size_t FX_SMEM = (size_t)(FX_BLOCK / 32) * FX_WARP_WORDS * 16;

template <bool FXIN>
struct FxHop {
  const double* in;    // the system's field, entry word 0 of site 0
  size_t cstride, sitestride;
  const int* in_ex;    // the system's exponents
  const int4* gauge;
  int L0, L1, L2, L3, Lh0, Vh;
  int p_out;
  int x0, x1, x2, x3, site;
  int4* sp;            // this lane's spinor words, 32 apart
  int4* lw;            // the warp's link words, [entry][slot]
  int lane, nst, lst;  // slots (sites) of the warp, log2; a power of two
  int slot, rep;       // this lane's slot; lanes between the representatives of slots 0, 1, ...
  int E;
  bool bad;

  __device__ __forceinline__ int neighbour(int d) const {
    const int s = (d & 1) ? -1 : 1;
    int y0 = x0, y1 = x1, y2 = x2, y3 = x3;
    const int mu = d >> 1;
    if (mu == 0) { y0 += s; y0 = y0 == L0 ? 0 : (y0 < 0 ? L0 - 1 : y0); }
    if (mu == 1) { y1 += s; y1 = y1 == L1 ? 0 : (y1 < 0 ? L1 - 1 : y1); }
    if (mu == 2) { y2 += s; y2 = y2 == L2 ? 0 : (y2 < 0 ? L2 - 1 : y2); }
    if (mu == 3) { y3 += s; y3 = y3 == L3 ? 0 : (y3 < 0 ? L3 - 1 : y3); }
    return (y0 >> 1) + Lh0 * (y1 + L1 * (y2 + L2 * y3));
  }
  __device__ __forceinline__ int issue_spinor(int nb) const {
    const double* b = in + (size_t)nb * sitestride;
#pragma unroll
    for (int c = 0; c < 12; c++) {
      cp_async16(sp + c * 32, b);
      b += cstride;
    }
    cp_async_commit();
    return FXIN ? __ldcg(in_ex + nb) : 0;  // (the L2: another block of a cluster may have written it)
  }
  __device__ __forceinline__ void issue_link(int d, int nb) const {
    const bool dag = d & 1;
    const int ls = dag ? nb : site;
    const int4* lk = gauge + (size_t)((dag ? 1 - p_out : p_out) * 4 + (d >> 1)) * 9 * Vh;
    const int n = 9 * nst;
    for (int w0 = 0; w0 < n; w0 += 32) {
      const int w = w0 + lane;
      const int s = __shfl_sync(0xffffffffu, ls, (w & (nst - 1)) * rep);
      if (w < n) cp_async16(lw + w, lk + (size_t)(w >> lst) * Vh + s);
    }
    cp_async_commit();
  }

  // Directions first .. last - 1 of H in: 24 integers and their common exponent E, value = acc 2^(E - FX_UNIT) (the
  // bits of spinor and link, the exponents' biases, units of 2^64). The whole warp takes part.
  __device__ __forceinline__ void run(long long (&acc)[24], int first = 0, int last = 8) {
#pragma unroll
    for (int k = 0; k < 24; k++) acc[k] = 0;
    E = -50000;  // below every exponent but a zero spinor's
    bad = false;
    const int nb = neighbour(first);
    int e = issue_spinor(nb);
    issue_link(first, nb);
#pragma unroll 1
    for (int d = first; d < last; d++) {
      const bool dag = d & 1;
      cp_async_wait<1>();  // the spinor is here (each lane reads its own)
      long long p[24];
      if constexpr (FXIN) {
#pragma unroll
        for (int c = 0; c < 12; c++) {
          const longlong2 w = *reinterpret_cast<const longlong2*>(sp + c * 32);
          p[2 * c] = w.x;
          p[2 * c + 1] = w.y;
        }
      } else {
        double v[24];
#pragma unroll
        for (int c = 0; c < 12; c++) {
          const double2 w = *reinterpret_cast<const double2*>(sp + c * 32);
          v[2 * c] = w.x;
          v[2 * c + 1] = w.y;
        }
        e = fx_spinor(v, p);
      }
      int nb_next = 0, e_next = 0;
      if (d + 1 < last) {
        nb_next = neighbour(d + 1);
        e_next = issue_spinor(nb_next);
      } else {
        cp_async_commit();  // keeps the count of groups in flight
      }
      // the upper spins of (1 -+ gamma_mu) psi (the branches are the same for every lane)
      long long w[12];
      switch (d) {
        case 0: fx_project<0, -1>(p, w); break;
        case 1: fx_project<0, +1>(p, w); break;
        case 2: fx_project<1, -1>(p, w); break;
        case 3: fx_project<1, +1>(p, w); break;
        case 4: fx_project<2, -1>(p, w); break;
        case 5: fx_project<2, +1>(p, w); break;
        case 6: fx_project<3, -1>(p, w); break;
        default: fx_project<3, +1>(p, w); break;
      }
      int h1[12], h0[12];
#pragma unroll
      for (int k = 0; k < 12; k++) fx_limbs(w[k], h1[k], h0[k]);
      cp_async_wait<1>();  // the links are here, every lane's part of them
      __syncwarp();
      const int4* lk = lw + slot;
      const int4 w0 = lk[0], w4 = lk[4 << lst];
      const int eu = fx_link_exponent(w0, w4);
      bad = bad || e == FX_BAD || eu == FX_LINK_BAD;
      const int et = e + eu;
      if (__any_sync(0xffffffffu, et > E)) {
        // the sum goes under a larger exponent, with a bit to spare: spinors of like size then raise it once
        const int en = et > E ? et + 1 : E, s = min(en - E, 62);
        const long long half = (1ll << s) >> 1;
#pragma unroll
        for (int k = 0; k < 24; k++) acc[k] = (acc[k] + half) >> s;
        E = en;
      }
      const int s = min(E - et, 62);
      const long long half = (1ll << s) >> 1;
      // z = U h (U^dag h for the backward hop), row by row
      const int sa = (dag ? 1 : 3) << lst, sb = (dag ? 3 : 1) << lst;
      const int sg = dag ? -1 : 1;
      long long z[12];
#pragma unroll
      for (int a = 0; a < 3; a++) {
        long long hh[4], xx[4];
#pragma unroll
        for (int q = 0; q < 4; q++) { hh[q] = half; xx[q] = 1ll << 31; }
#pragma unroll
        for (int b = 0; b < 3; b++) {
          int4 u = lk[a * sa + b * sb];
          if (a == b && a < 2) {  // entries 0 and 4 carry the exponent in their top bits
            u.x = (u.x << 3) >> 3;
            u.z = (u.z << 3) >> 3;
          }
          const int r1 = u.x, r0 = u.y, i1 = sg * u.z, i0 = sg * u.w, ni1 = -i1, ni0 = -i0;
#pragma unroll
          for (int t = 0; t < 2; t++) {
            const int kr = 6 * t + 2 * b, ki = kr + 1;
            hh[2 * t] = fx_mad(h1[kr], r1, hh[2 * t]);
            hh[2 * t + 1] = fx_mad(h1[ki], r1, hh[2 * t + 1]);
            hh[2 * t] = fx_mad(h1[ki], ni1, hh[2 * t]);
            hh[2 * t + 1] = fx_mad(h1[kr], i1, hh[2 * t + 1]);
            xx[2 * t] = fx_mad(h1[kr], r0, xx[2 * t]);
            xx[2 * t + 1] = fx_mad(h1[ki], r0, xx[2 * t + 1]);
            xx[2 * t] = fx_mad(h0[kr], r1, xx[2 * t]);
            xx[2 * t + 1] = fx_mad(h0[ki], r1, xx[2 * t + 1]);
            xx[2 * t] = fx_mad(h1[ki], ni0, xx[2 * t]);
            xx[2 * t + 1] = fx_mad(h1[kr], i0, xx[2 * t + 1]);
            xx[2 * t] = fx_mad(h0[ki], ni1, xx[2 * t]);
            xx[2 * t + 1] = fx_mad(h0[kr], i1, xx[2 * t + 1]);
          }
        }
#pragma unroll
        for (int t = 0; t < 2; t++) {
          z[6 * t + 2 * a] = (hh[2 * t] + (int)(xx[2 * t] >> 32)) >> s;
          z[6 * t + 2 * a + 1] = (hh[2 * t + 1] + (int)(xx[2 * t + 1] >> 32)) >> s;
        }
      }
      __syncwarp();  // every lane is done with the links
      if (d + 1 < last) issue_link(d + 1, nb_next);
#pragma unroll
      for (int k = 0; k < 12; k++) acc[k] += z[k];
      switch (d) {
        case 0: fx_lower<0, -1>(acc, z); break;
        case 1: fx_lower<0, +1>(acc, z); break;
        case 2: fx_lower<1, -1>(acc, z); break;
        case 3: fx_lower<1, +1>(acc, z); break;
        case 4: fx_lower<2, -1>(acc, z); break;
        case 5: fx_lower<2, +1>(acc, z); break;
        case 6: fx_lower<3, -1>(acc, z); break;
        default: fx_lower<3, +1>(acc, z); break;
      }
      if (FXIN) e = e_next;
    }
    cp_async_wait<0>();
  }
};
constexpr int FX_UNIT = FX_BITS + FX_LINK_BITS + 2 * 1022 + FX_LINK_BIAS - 64;

// The sums as doubles, h = acc 2^(E - FX_UNIT)
__device__ __forceinline__ void fx_values(double (&h)[24], const long long (&acc)[24], int E, bool bad) {
  const int es = E - FX_UNIT + 1023;
  if ((unsigned)(es - 70) > 1800u || bad) {  // beyond a double's range (all sums zero among them)
#pragma unroll
    for (int k = 0; k < 24; k++)
      h[k] = bad ? __longlong_as_double(0x7ff8000000000000ll) : (E < -4000 ? 0.0 : scalbn(__ll2double_rn(acc[k]), E - FX_UNIT));
  } else {
#pragma unroll
    for (int k = 0; k < 24; k++) h[k] = fx_double(acc[k], es);
  }
}

// The sums brought below 2^FX_BITS and stored as an integer spinor with its exponent
__device__ __forceinline__ void fx_store(const Field<double>& out, int* out_ex, int Vh, long long (&acc)[24], int E, bool bad,
                                         int site, int sys) {
  long long m = 0;
#pragma unroll
  for (int k = 0; k < 24; k++) m |= acc[k] ^ (acc[k] >> 63);
  const int sh = max(0, 64 - __clzll(m) - FX_BITS);
  double* b = out.ptr + out.off(site, sys);
#pragma unroll
  for (int c = 0; c < 12; c++)
    *reinterpret_cast<longlong2*>(b + c * out.cstride) = make_longlong2(acc[2 * c] >> sh, acc[2 * c + 1] >> sh);
  out_ex[(size_t)sys * Vh + site] = bad ? FX_BAD : (m == 0 ? FX_ZERO : E + sh + FX_BITS + 1022 - FX_UNIT);
}

// out = a X + b (H in) + c Y over FP64 fields, with the dot products of DOT (fs_hop.cuh). Warps take items, no
// block barriers:
//  WL: the system-major work list, items (32 / w sites, w selected systems), w = 4, 2 or 1 by how many are
//      selected: systems that share a warp share its links (1152 bytes a site, three quarters of the
//      spinors' traffic).
//  else the tile layout, items (8 sites, 4 systems).
//  FEW: a tile of one or two systems (fx_few), items of 32 or 16 sites. A variant of its own, since a run-time split
//      costs three systems and more 2 to 3%.
// The sites of an 8-site group are in one warp: its dot products are summed there, in one order.
//  FXIN / FXOUT: `in` / `out` hold integer spinors with the exponents in_ex / out_ex [system][Vh].
template <int COEF, int DOT, bool WL = false, bool CLV = false, bool FXIN = false, bool FXOUT = false, bool FEW = false>
__global__ void __launch_bounds__(FX_BLOCK, 3) hop_kernel_fx(HopArgs a) {
  if (a.gate != nullptr && *a.gate == 0) return;
  constexpr int K = DotK<DOT>::K;
  static_assert(!(WL && FEW), "the work list has its own split");
  static_assert(!FXOUT || (COEF == COEF_PLAIN && DOT == DOT_NONE), "integer output is H in itself");
  extern __shared__ int4 fx_words[];  // FX_WARP_WORDS per warp
  const int N = a.sh.N, Vh = a.g.Vh;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int nw = FX_BLOCK / 32;
  __shared__ int slist[64];
  int nsel = N, lsy = FEW ? N - 1 : 2;  // systems to go through; log2 of the systems of a warp
  if constexpr (WL) {
    nsel = selected_list(a.st, N, a.mask, slist);
    lsy = (nsel >= 7 || nsel == 4) ? 2 : (nsel >= 3 || nsel == 2) ? 1 : 0;
  }
  FxHop<FXIN> f;
  f.gauge = (const int4*)a.gauge;
  f.L0 = a.g.L[0]; f.L1 = a.g.L[1]; f.L2 = a.g.L[2]; f.L3 = a.g.L[3]; f.Lh0 = a.g.Lh0; f.Vh = Vh;
  f.p_out = a.p_out;
  f.sp = fx_words + (size_t)warp * FX_WARP_WORDS + lane;
  f.lw = fx_words + (size_t)warp * FX_WARP_WORDS + 12 * 32;
  f.lane = lane;
  f.lst = 5 - lsy;
  f.nst = 1 << f.lst;
  // lanes: system-major fields take sites fastest, the tile layout systems
  f.slot = WL ? (lane & (f.nst - 1)) : (lane >> lsy);
  f.rep = WL ? 1 : 1 << lsy;
  const int lsys = WL ? (lane >> f.lst) : (lane & ((1 << lsy) - 1));
  const Field<double> fin = make_field<double>(const_cast<void*>(a.in), Vh, N, WL);
  f.cstride = fin.cstride;
  f.sitestride = fin.sitestride;
  const int nsg = (nsel + (1 << lsy) - 1) >> lsy, nchunk = (Vh + f.nst - 1) >> f.lst;
  for (int item = blockIdx.x * nw + warp; item < nsg * nchunk; item += gridDim.x * nw) {
    const int chunk = item / nsg;
    const int k = ((item - chunk * nsg) << lsy) + lsys;
    const int site0 = (chunk << f.lst) + f.slot;
    bool act = k < nsel && site0 < Vh;
    // a lane without work of its own goes along on a neighbour's operands and stores nothing
    const int sys = WL ? slist[min(k, nsel - 1)] : min(k, N - 1), site = min(site0, Vh - 1);
    if constexpr (!WL) {
      act = act && selected(a.st, sys, a.mask);
      if (!__any_sync(0xffffffffu, act)) continue;
    }
    if (a.work != nullptr) {  // profiling: (site, system) pairs computed, one atomic per warp
      const unsigned m = __ballot_sync(0xffffffffu, act);
      if (lane == 0 && m) atomicAdd(a.work, (unsigned long long)__popc(m));
    }
    f.site = site;
    f.in = fin.ptr + (size_t)sys * fin.sysstride;
    f.in_ex = a.in_ex + (size_t)sys * Vh;
    {
      int x[4];
      cb_coords(a.g, a.p_out, site, x);
      f.x0 = x[0]; f.x1 = x[1]; f.x2 = x[2]; f.x3 = x[3];
    }
    double o[24], dv[K > 0 ? K : 1];
    {
      long long acc[24];
      f.run(acc);
      if constexpr (FXOUT) {
        if (act) fx_store(make_field<double>(a.out, Vh, N, WL), a.out_ex, Vh, acc, f.E, f.bad, site, sys);
        continue;
      }
      fx_values(o, acc, f.E, f.bad);
    }
    // with the clover term the site factors A^-1 come from clover passes on the operands (in = A_oo^-1 H x,
    // z_o pre-inverted, x_o inverted afterwards) and C x enters through Y
    double ca = 0, cb = 1;
    const SysState& s = a.st[sys];
    const bool cl = a.clover != 0;
    if (COEF == COEF_MHAT) { ca = s.cd[C_A]; cb = cl ? -0.25 : s.cd[C_MINV4A]; }
    else if (COEF == COEF_DSLASH) { ca = s.cd[C_A]; cb = -0.5; }
    else if (COEF == COEF_PREP) { cb = cl ? 0.5 : s.cd[C_INV2A]; }
    else if (COEF == COEF_RECON) { ca = cl ? 1 : s.cd[C_INVA]; cb = cl ? 0.5 : s.cd[C_INV2A]; }
    else if (COEF == COEF_TRUERES) { ca = s.cd[C_MINVA]; cb = cl ? 0.25 : s.cd[C_INV4A]; }
    else if (COEF == COEF_FULLRES) { ca = s.cd[C_MINVA]; cb = 0.5; }
    else if (COEF == COEF_KAPPA) { cb = cl ? 0.5 : s.cd[C_INV2A]; }
    if constexpr (COEF == COEF_KAPPA) {
#pragma unroll
      for (int q = 0; q < 24; q++) o[q] = cb * o[q];
    } else if constexpr (COEF != COEF_PLAIN) {
      double xv[24];
      make_field<double>(const_cast<void*>(a.X), Vh, N, WL).load(site, sys, xv);
      if constexpr (CLV) {
        double yv[24];
        make_field<double>(const_cast<void*>(a.Y), Vh, N, WL).load(site, sys, yv);
#pragma unroll
        for (int q = 0; q < 24; q++) o[q] = fmadd(ca, xv[q], fmadd(cb, o[q], yv[q]));
      } else if constexpr (COEF == COEF_TRUERES || COEF == COEF_FULLRES) {
        double yv[24];
        make_field<double>(const_cast<void*>(a.Y), Vh, N, WL).load(site, sys, yv);
#pragma unroll
        for (int q = 0; q < 24; q++) o[q] = fmadd(cb, o[q], fmadd(ca, xv[q], yv[q]));
      } else if constexpr (COEF == COEF_PREP) {
#pragma unroll
        for (int q = 0; q < 24; q++) o[q] = fmadd(cb, o[q], xv[q]);
      } else {
#pragma unroll
        for (int q = 0; q < 24; q++) o[q] = axpby(ca, xv[q], cb, o[q]);
      }
      if constexpr (DOT == DOT_TS) {
        double rv[24];
        make_field<double>(const_cast<void*>(a.R), Vh, N, WL).load(site, sys, rv);
        ts_dots(dv, o, xv, rv);
      }
    }
    if constexpr (DOT == DOT_R) {
      double rv[24];
      make_field<double>(const_cast<void*>(a.R), Vh, N, WL).load(site, sys, rv);
      double sr = 0, si = 0;
#pragma unroll
      for (int q = 0; q < 24; q += 2) dot_acc(sr, si, rv[q], rv[q + 1], o[q], o[q + 1]);
      dv[0] = sr; dv[1] = si;
    }
    if constexpr (DOT == DOT_NORM) {
      double nn = 0;
#pragma unroll
      for (int q = 0; q < 24; q += 2) norm_acc(nn, o[q], o[q + 1]);
      dv[0] = nn;
    }
    if (act) make_field<double>(a.out, Vh, N, WL).store(site, sys, o);
    if constexpr (K > 0) {
      // the 8-site groups: lane sums of value v, system y over the group's sites in site order, from the
      // warp's spinor words (free now); a lane that stands in for another adds nothing of its own
      double* buf = reinterpret_cast<double*>(fx_words + (size_t)warp * FX_WARP_WORDS);
      __syncwarp();
#pragma unroll
      for (int v = 0; v < K; v++) buf[(v * 33 + (WL ? lane : (lsys << f.lst) + f.slot))] = dv[v];
      __syncwarp();
      // sums: 4 groups of 8 (by lane order: site fastest) per value
      for (int q = lane; q < 4 * K; q += 32) {
        const int v = q >> 2, gl = (q & 3) * 8;
        double t = 0.0;
#pragma unroll
        for (int j = 0; j < 8; j++) t += buf[v * 33 + gl + j];
        const int gsy = gl >> f.lst, gs = (chunk << f.lst) + (gl & (f.nst - 1));
        const int gk = ((item - chunk * nsg) << lsy) + gsy;
        if (gk < nsel && gs < Vh) {
          const int gsys = WL ? slist[gk] : gk;
          a.partial[((size_t)gsys * K + v) * (Vh / 8) + gs / 8] = t;
        }
      }
      __syncwarp();
    }
  }
}

// Tiles that take the FEW variants: with items of 8 sites and 4 systems three quarters or half of the lanes go along idle.
// FP64 solves of 1 / 2 systems, ms: 16^4 13.8 / 14.0, now 6.1 / 9.9; 12^3x16 6.8 / 6.9, now 4.4 / 5.6. Up to 4096 sites
// the warps are too few to fill the SMs and more of them serve as well or better: 8^3x16 4.62 / 4.58 both ways, the
// operator on 4^4 66.5 / 69.0 us against 69.1 / 70.8 with larger items.
inline bool fx_few(int N, int Vh) { return N <= 2 && Vh > 4096; }
// Three resident blocks per SM at most; items go to the warps in turn, so a block beyond the resident
// ones would run its share last.
template <typename Kern>
cudaError_t launch_hop_fx_at(Kern kern, const HopArgs& a, cudaStream_t s) {
  const LaunchSetup pg = launch_setup((const void*)kern, FX_SMEM, FX_BLOCK);
  if (pg.err) return pg.err;
  // a warp for every item (8 sites, 4 systems; FEW: 32 or 16 sites)
  const int lsy = !a.sysmajor && fx_few(a.sh.N, a.g.Vh) ? a.sh.N - 1 : 2, nst = 32 >> lsy;
  const long long items = (long long)((a.g.Vh + nst - 1) / nst) * ((a.sh.N + (1 << lsy) - 1) >> lsy);
  const int grid = (int)std::max(1ll, std::min(3ll * pg.nsm, (items + FX_BLOCK / 32 - 1) / (FX_BLOCK / 32)));
  kern<<<grid, FX_BLOCK, FX_SMEM, s>>>(a);
  return cudaGetLastError();
}

}  // namespace fs
