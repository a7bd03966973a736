// The Gamma Omega_p contractions of the level traces and the variance sampling:
// c_p = sum_x L(x)^dag Gamma W(x, x + p z) R(x + p z).
//
// The straight path products W(x, x + q z) = U_z(x) U_z(x + z) ... U_z(x + (q-1) z) depend on
// the gauge field alone, so they are built once (transport_kernel), as the integer links of fs_hopfx.cuh.
//
// FP64 multiply-adds issue at 0.62 T/s here, 64 clocks a warp: 190 of them a site for every pair of
// vectors and displacement bound the contraction (24^3 x 64, 40 pairs, 9 displacements: 115 ms; here 21). So:
//  - the products are formed in integers (mad.wide, 18.9 T/s), R, W and xi = Gamma^dag L under exponents of their
//    own; the 24-term sums of a site are kept in units of 2^-60 of the largest product, those of a warp are
//    added exactly (redux of 22-bit limbs) and go to FP64 as one value;
//  - W R, two thirds of the products, is formed once for up to four left vectors, whose xi wait in
//    shared memory through all displacements.
// Pairs with the same right vector make such a group (up to 2 / 3 / 4 left vectors: 25.6 / 21.9 / 20.7 ms); the groups
// of one run of sites are neighbouring blocks, so that W and the left vectors come from the L2. What bounds it now is
// latency in 8 warps an SM, about 1300 integer instructions a site and displacement. Error against 80-bit sums
// over the same vectors (8^2 x 16^2, p = 0, 1, 2, 4, 8), in 1e-18 |L| |R|: 0.4 / 16 / 6.2 / 0.9 / 0.6, the FP64 chains'
// 0.6 / 16 / 5.5 / 1.0 / 0.7 (p = 1 and 2: the last rounding of a large sum).
#pragma once

#include "fs_aux.cuh"
#include "fs_hopfx.cuh"

namespace fs {

struct ContractPair {
  int right;      // slot holding the right vector (solution)
  int left;       // slot of the left vector
  int left_kind;  // 0: noise of slot `left` ; 1: gamma_5 * solution of slot `left`
  int out;        // output row
  int right_kind = 0;  // 0: the solution of slot `right` ; 1: slot `right` of the pair y_e / y_o
};
constexpr int CONTRACT_MAXP = 16;
constexpr int CONTRACT_LEFTS = 4;      // left vectors of a group, at most: 98 KB of xi in a block, two blocks an SM
constexpr int CONTRACT_BLOCK = 128;    // threads, a site each
constexpr int CONTRACT_RUN = 256;      // sites of a block

struct ContractGroup {  // pairs with the same right vector
  int n;
  int pair[CONTRACT_LEFTS];
};

struct ContractArgs {
  const double* x_e;
  const double* x_o;
  const double* y_e;      // right vectors of the right_kind 1 pairs (hopping parameter expansion)
  const double* y_o;
  const int4* wline;      // W(x, x + q z) for the requested q > 0: [k][9][2 Vh], k counts them
  const NoiseSpec* spec;
  const int* colors;      // probing colour per canonical site (colour-restricted noise only)
  const ContractPair* pairs;
  const ContractGroup* groups;
  double* partial;        // [npairs][np][2][nblk]
  double gamma[32];       // Gamma, 4x4 complex, row major
  int gmono;              // 1: Gamma is a monomial matrix with entries in {+-1, +-i}
  int gperm[4];           // (Gamma psi)_s = i^gphase[s] psi_{gperm[s]} when gmono
  int gphase[4];
  Geom g;
  int N;
  int ngroups;
  int pmask;              // bit q set: displacement q requested
  int pmax;
  int np;
  int nblk;
};

#ifdef FS_ENGINE_KERNELS
// W(x, x + q z) for every site x (thread fs = parity * Vh + checkerboard index) and every q with
// bit q of qmask set (q >= 1), stored as the words w[k][entry][fs], k counting the set bits in increasing q.
__global__ void __launch_bounds__(256) transport_kernel(int4* w, const double* gauge64, Geom g, int qmask,
                                                        int qmax) {
  const int fs = blockIdx.x * blockDim.x + threadIdx.x;
  if (fs >= 2 * g.Vh) return;
  const int par = fs >= g.Vh ? 1 : 0;
  const int site = fs - par * g.Vh;
  int x[4];
  cb_coords(g, par, site, x);
  const size_t stride = (size_t)2 * g.Vh;
  double W[18];
#pragma unroll
  for (int r = 0; r < 18; r++) W[r] = (r == 0 || r == 8 || r == 16) ? 1.0 : 0.0;
  int k = 0;
  for (int q = 1; q <= qmax; q++) {
    int v[4] = {x[0], x[1], x[2], x[3]};
    v[2] = (x[2] + q - 1) % g.L[2];
    const int vpar = (v[0] + v[1] + v[2] + v[3]) & 1;
    const double* lk = gauge64 + ((size_t)(vpar * 4 + 2) * g.Vh + cb_index(g, v)) * 18;
    double nw[18];
#pragma unroll
    for (int j = 0; j < 3; j++) {
      // column j of W U = W times column j of U
      double col[6], out[6];
#pragma unroll
      for (int i = 0; i < 3; i++) {
        col[2 * i] = lk[(i * 3 + j) * 2];
        col[2 * i + 1] = lk[(i * 3 + j) * 2 + 1];
      }
      su3_mul<false, double>(W, col, out);
#pragma unroll
      for (int i = 0; i < 3; i++) {
        nw[(i * 3 + j) * 2] = out[2 * i];
        nw[(i * 3 + j) * 2 + 1] = out[2 * i + 1];
      }
    }
#pragma unroll
    for (int r = 0; r < 18; r++) W[r] = nw[r];
    if ((qmask >> q) & 1) {
      int4 o[9];
      fx_link(W, o);
#pragma unroll
      for (int r = 0; r < 9; r++) w[((size_t)k * 9 + r) * stride + fs] = o[r];
      k++;
    }
  }
}

// xi = Gamma^dag L
__device__ __forceinline__ void contract_left(const ContractArgs& a, const double (&l)[24], double (&xi)[24]) {
#pragma unroll
  for (int k = 0; k < 24; k++) xi[k] = 0.0;
  if (a.gmono) {
    // every Clifford product is a signed / phased permutation in this basis
#pragma unroll
    for (int s = 0; s < 4; s++) {
      const int ph = a.gphase[s];
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const double re = l[s * 6 + c * 2], im = l[s * 6 + c * 2 + 1];
        const double gr = ph == 0 ? re : (ph == 1 ? im : (ph == 2 ? -re : -im));
        const double gi = ph == 0 ? im : (ph == 1 ? -re : (ph == 2 ? -im : re));
#pragma unroll
        for (int t = 0; t < 4; t++)
          if (a.gperm[s] == t) { xi[t * 6 + c * 2] = gr; xi[t * 6 + c * 2 + 1] = gi; }
      }
    }
    return;
  }
#pragma unroll
  for (int s = 0; s < 4; s++)
#pragma unroll
    for (int t = 0; t < 4; t++) {
      const double Gr = a.gamma[(s * 4 + t) * 2], Gi = a.gamma[(s * 4 + t) * 2 + 1];
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const double re = l[s * 6 + c * 2], im = l[s * 6 + c * 2 + 1];
        xi[t * 6 + c * 2] += Gr * re + Gi * im;
        xi[t * 6 + c * 2 + 1] += Gr * im - Gi * re;
      }
    }
}

// v / 2^s, ties to even: rounded up, the ties of every site would add up (2^-58 of |L| |R| at any volume, measured)
__device__ __forceinline__ long long contract_shift(long long v, int s) {
  const long long q = v >> s;
  return (v + ((1ll << s) >> 1) - (s > 0 ? 1 - (q & 1) : 0)) >> s;
}
// The warp's sum of v >> s over its lanes, |v| < 2^60.7, in units of 8: exact but for the shifts' roundings
__device__ __forceinline__ long long contract_warp_sum(long long v, int s) {
  const long long d = contract_shift(v, s);
  const int lo = (int)(d & 0x3fffff), mi = (int)((d >> 22) & 0x3fffff), hi = (int)(d >> 44);
  const long long s0 = __reduce_add_sync(0xffffffffu, lo), s1 = __reduce_add_sync(0xffffffffu, mi);
  const long long s2 = __reduce_add_sync(0xffffffffu, hi);
  return s2 * (1ll << 41) + s1 * (1ll << 19) + contract_shift(s0, 3);
}

__global__ void __launch_bounds__(CONTRACT_BLOCK, 2) contract_kernel(ContractArgs a) {
  constexpr int NW = CONTRACT_RUN / 32, VALUES = CONTRACT_MAXP * CONTRACT_LEFTS;
  extern __shared__ longlong2 xi_words[];            // [left][12][thread]
  __shared__ int xi_ex[CONTRACT_LEFTS][CONTRACT_BLOCK];
  __shared__ long long wsum[2][VALUES][NW];          // the warps' sums and exponents
  __shared__ int wex[VALUES][NW];
  const ContractGroup grp = a.groups[blockIdx.x % a.ngroups];
  const int blk = blockIdx.x / a.ngroups;
  const ContractPair pr0 = a.pairs[grp.pair[0]];     // (every pair has the same right vector)
  const Geom g = a.g;
  const int tid = threadIdx.x, lane = tid & 31;
  const size_t stride = (size_t)2 * g.Vh;
#pragma unroll 1
  for (int half = 0; half < CONTRACT_RUN / CONTRACT_BLOCK; half++) {
    const int slot = half * (CONTRACT_BLOCK / 32) + (tid >> 5);
    const int at = blk * CONTRACT_RUN + half * CONTRACT_BLOCK + tid;
    const bool in = at < 2 * g.Vh;
    const int fs = in ? at : 2 * g.Vh - 1;
    const int par = fs >= g.Vh ? 1 : 0;
    const int site = fs - par * g.Vh;
    int x[4];
    cb_coords(g, par, site, x);
    const int lex = lex_index(g, x);
    bool act = false;  // a site where every left vector vanishes contributes nothing
#pragma unroll 1
    for (int l = 0; l < grp.n; l++) {
      const ContractPair pr = a.pairs[grp.pair[l]];
      double lv[24], xi[24];
      if (pr.left_kind == 0) {
        z4_site(a.spec[pr.left], lex, lv, in ? noise_keep(a.spec[pr.left], a.colors, lex) : 0u);
      } else {
        make_field<double>(const_cast<double*>(par ? a.x_o : a.x_e), g.Vh, a.N, true).load(site, pr.left, lv);
#pragma unroll
        for (int k = 0; k < 24; k++) lv[k] = !in ? 0.0 : (k < 12 ? lv[k] : -lv[k]);
      }
      contract_left(a, lv, xi);
      long long p[24];
      const int e = fx_spinor(xi, p);
      xi_ex[l][tid] = e;
      act = act || e != FX_ZERO;
#pragma unroll
      for (int c = 0; c < 12; c++)
        xi_words[(l * 12 + c) * CONTRACT_BLOCK + tid] = make_longlong2(p[2 * c], fx_negatable(p[2 * c + 1]));
    }
    const bool any = __any_sync(0xffffffffu, act);
    // the right vector and the path of a displacement, read while the one before is worked on
    double psi[24];
    int4 wn[9];
    auto fetch = [&](int q, int k) {
      if (act) {
        int y[4] = {x[0], x[1], x[2], x[3]};
        y[2] = (x[2] + q) % g.L[2];
        const int ypar = (y[0] + y[1] + y[2] + y[3]) & 1;
        const double* rf = pr0.right_kind ? (ypar ? a.y_o : a.y_e) : (ypar ? a.x_o : a.x_e);
        make_field<double>(const_cast<double*>(rf), g.Vh, a.N, true).load(cb_index(g, y), pr0.right, psi);
      } else {
#pragma unroll
        for (int i = 0; i < 24; i++) psi[i] = 0.0;
      }
      if (q > 0 && any) {
#pragma unroll
        for (int r = 0; r < 9; r++) wn[r] = __ldg(a.wline + ((size_t)k * 9 + r) * stride + fs);
      }
    };
    int qi = 0, k = 0;
    int q = __ffs(a.pmask) - 1;
    fetch(q, 0);
#pragma unroll 1
    while (q <= a.pmax) {
      long long z[24];  // W R, below 2^60
      int X = 0;        // value = z 2^X
      bool bad = false;
      if (any) {
        X = fx_spinor(psi, z);
        bad = X == FX_BAD;
        X -= 1022 + FX_BITS;
        if (q > 0) {
          int4 w[9];
#pragma unroll
          for (int r = 0; r < 9; r++) w[r] = wn[r];
          const int eu = fx_link_exponent(w[0], w[4]);
          bad = bad || (act && eu == FX_LINK_BAD);
          w[0].x = (w[0].x << 3) >> 3;
          w[0].z = (w[0].z << 3) >> 3;
          w[4].x = (w[4].x << 3) >> 3;
          w[4].z = (w[4].z << 3) >> 3;
          X += eu - FX_LINK_BIAS - 1022 - FX_LINK_BITS + 64 - 4;
          long long m = 0;
#pragma unroll
          for (int t = 0; t < 4; t++) {
            int h1[6], h0[6];
#pragma unroll
            for (int i = 0; i < 6; i++) fx_limbs(z[6 * t + i], h1[i], h0[i]);
#pragma unroll
            for (int i = 0; i < 3; i++) {
              // six products of 60 and 59 bits: |hh| < 2^57.6, |xx| < 2^62.2; four bits below 2^64 are kept
              long long hr = 0, hi = 0, xr = 1 << 27, xi = 1 << 27;
#pragma unroll
              for (int b = 0; b < 3; b++) {
                const int4 u = w[3 * i + b];
                const int r1 = h1[2 * b], r0 = h0[2 * b], i1 = h1[2 * b + 1], i0 = h0[2 * b + 1];
                hr = fx_mad(r1, u.x, hr);
                hi = fx_mad(i1, u.x, hi);
                hr = fx_mad(i1, -u.z, hr);
                hi = fx_mad(r1, u.z, hi);
                xr = fx_mad(r1, u.y, xr);
                xi = fx_mad(i1, u.y, xi);
                xr = fx_mad(r0, u.x, xr);
                xi = fx_mad(i0, u.x, xi);
                xr = fx_mad(i1, -u.w, xr);
                xi = fx_mad(r1, u.w, xi);
                xr = fx_mad(i0, -u.z, xr);
                xi = fx_mad(r0, u.z, xi);
              }
              const long long vr = (hr << 4) + (xr >> 28), vi = (hi << 4) + (xi >> 28);
              z[6 * t + 2 * i] = vr;
              z[6 * t + 2 * i + 1] = vi;
              m |= (vr ^ (vr >> 63)) | (vi ^ (vi >> 63));
            }
          }
          const int sh = max(0, 64 - __clzll(m) - FX_BITS);  // |z| < 2^61.6
          if (__any_sync(0xffffffffu, sh > 0)) {
            const long long h = (1ll << sh) >> 1;
#pragma unroll
            for (int i = 0; i < 24; i++) z[i] = (z[i] + h) >> sh;
          }
          X += sh;
        }
      }
      k += q > 0;
      do { q++; } while (q <= a.pmax && !((a.pmask >> q) & 1));
      if (q <= a.pmax) fetch(q, k);
      int z1[24], z0[24];
#pragma unroll
      for (int i = 0; i < 24; i++) fx_limbs(any ? z[i] : 0, z1[i], z0[i]);
#pragma unroll 1
      for (int l = 0; l < grp.n; l++) {
        const int v = qi * CONTRACT_LEFTS + l;
        if (!any) {
          if (lane == 0) {
            wsum[0][v][slot] = wsum[1][v][slot] = 0;
            wex[v][slot] = 0;
          }
          continue;
        }
        // conj(xi) . z: 24 products of 60 bits, |hh| < 2^60.7; |xx| < 2^62.7 over the six of a spin
        long long dr = 0, di = 0, fr = 0, fi = 0;  // fr, fi: what is below 2^64
#pragma unroll
        for (int t = 0; t < 4; t++) {
          long long xr = 0, xi = 0;
#pragma unroll
          for (int c = 0; c < 3; c++) {
            const longlong2 w = xi_words[(l * 12 + 3 * t + c) * CONTRACT_BLOCK + tid];
            int a1, a0, b1, b0;
            fx_limbs(w.x, a1, a0);
            fx_limbs(w.y, b1, b0);
            const int r1 = z1[6 * t + 2 * c], r0 = z0[6 * t + 2 * c], i1 = z1[6 * t + 2 * c + 1], i0 = z0[6 * t + 2 * c + 1];
            dr = fx_mad(a1, r1, dr);
            di = fx_mad(a1, i1, di);
            dr = fx_mad(b1, i1, dr);
            di = fx_mad(-b1, r1, di);
            xr = fx_mad(a1, r0, xr);
            xi = fx_mad(a1, i0, xi);
            xr = fx_mad(a0, r1, xr);
            xi = fx_mad(a0, i1, xi);
            xr = fx_mad(b1, i0, xr);
            xi = fx_mad(-b1, r0, xi);
            xr = fx_mad(b0, i1, xr);
            xi = fx_mad(-b0, r1, xi);
          }
          dr += xr >> 32;
          di += xi >> 32;
          fr += (unsigned)xr;
          fi += (unsigned)xi;
        }
        dr += contract_shift(fr, 32);
        di += contract_shift(fi, 32);
        const int eL = xi_ex[l][tid];
        const bool nan = __any_sync(0xffffffffu, eL == FX_BAD || (bad && eL != FX_ZERO));
        const int XD = eL == FX_BAD ? FX_ZERO : X + eL - 1022 - FX_BITS + 64;
        const int E = __reduce_max_sync(0xffffffffu, bad ? FX_ZERO : XD);
        const int s = min(max(E - XD, 0), 62);
        const long long tr = contract_warp_sum(dr, s), ti = contract_warp_sum(di, s);
        if (lane == 0) {
          wsum[0][v][slot] = tr;
          wsum[1][v][slot] = ti;
          wex[v][slot] = nan ? INT_MAX : E + 3;
        }
      }
      qi++;
    }
  }
  __syncthreads();
  // the warps' sums in one order, a thread per value
  for (int i = tid; i < a.np * grp.n * 2; i += CONTRACT_BLOCK) {
    const int c = i & 1, l = (i >> 1) % grp.n, qi = (i >> 1) / grp.n, v = qi * CONTRACT_LEFTS + l;
    double sum = 0.0;
#pragma unroll
    for (int w = 0; w < NW; w++) {
      const int e = wex[v][w];
      sum += e == INT_MAX ? __longlong_as_double(0x7ff8000000000000ll) : scalbn((double)wsum[c][v][w], e);
    }
    a.partial[(((size_t)grp.pair[l] * a.np + qi) * 2 + c) * a.nblk + blk] = sum;
  }
}

// result[pair.out][qi] = sum over blocks, fixed order
__global__ void __launch_bounds__(256) contract_finalize(const double* partial, const ContractPair* pairs,
                                                         double* result, int np, int nblk) {
  __shared__ double sm[256 * 2];
  const int pi = blockIdx.x / np, qi = blockIdx.x % np;
  const size_t base = (((size_t)pi * np + qi) * 2) * nblk;
  double r = 0, im = 0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) { r += partial[base + b]; im += partial[base + nblk + b]; }
  sm[threadIdx.x * 2] = r;
  sm[threadIdx.x * 2 + 1] = im;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sm[threadIdx.x * 2] += sm[(threadIdx.x + w) * 2];
      sm[threadIdx.x * 2 + 1] += sm[(threadIdx.x + w) * 2 + 1];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int row = pairs[pi].out;
    result[((size_t)row * np + qi) * 2] = sm[0];
    result[((size_t)row * np + qi) * 2 + 1] = sm[1];
  }
}
#endif  // FS_ENGINE_KERNELS

}  // namespace fs
