// BiCGStab iterations of a small lattice in one launch: a cluster of blocks per system.
//
// On a small lattice an iteration of 14 launches waits for launches and for latencies inside nearly
// empty grids (8^4, 15 systems in FP32: 74 us an iteration, no kernel above 11; here 35). The systems of a tile are
// independent, so here each has a cluster of up to 8 blocks that goes through whole iterations, reliable
// updates among them, with a cluster barrier (0.22 us) where the launches were. The vectors stay in global
// memory (L2-resident at these sizes), system-major, so that a warp's sites are contiguous; a thread keeps its sites,
// so only what a hop reads from neighbours crosses a barrier, through the L2 (ld.cg).
//  - Hops of the inner precisions: a thread per site, the roundings of the other hop kernels.
//  - FP64 hops (the updates', all of them with FP64 storage): integer arithmetic (fs_hopfx.cuh), the four
//    directions mu of 32 sites in four warps, whose integer sums are added through shared memory and whose lanes
//    then finish one spin each: a quarter of the latency that a warp with all eight directions has.
//  - Dot products: per thread over its sites, over the block in FP64, then the blocks' sums in rank order, read by
//    every block of the cluster (distributed shared memory): each runs the scalar step on its own copy of
//    the state, with the same bits, so all take the same branches. Barriers are the hardware's; nothing spins.
// The shape depends on the lattice alone, so a system's result does not depend on its tile.
#pragma once

#include <cooperative_groups.h>

#include "fs_blas.cuh"
#include "fs_hopfx.cuh"

namespace fs {

// Sites per parity up to which the cluster kernel serves, by storage precision. Above, 8 SMs a system are too few and
// the tile kernels, which share links between systems, are ahead. Shifted solves of 8 / 32 systems, cluster against
// tile kernels, ms: 4^4 FP64 1.7 / 2.0 against 4.1 / 4.5, FP16 1.0 / 1.5 against 2.5 / 2.6; 4x4x8x16 FP64 9.1 / 11.4
// against 9.2 / 12.5, FP32 2.6 / 3.3 against 5.2 / 5.6; 8^4 FP64 9.2 / 13.6 against 6.6 / 14.0, FP16 2.2 / 3.3 against
// 3.6 / 5.2, FP32 2.3 / 3.4 against 3.7 / 4.4; 6x10x14x12 (5040) FP32 6.2 / 11.1 against 5.3 / 9.3. Near the limits, two
// shifts, tiles of 1 / 8 / 32 / 64 systems: 8^3x16 FP16 3.7 / 4.0 / 6.1 / 11.5 against 3.7 / 4.9 / 8.2 / 12.8, BF16
// 4.2 / 4.6 / 7.0 / 13.3 against 3.9 / 5.4 / 9.4 / 14.5, FP32 3.8 / 4.2 / 7.0 / 13.1 against 3.3 / 4.2 / 7.5 / 13.1;
// 8x8x10x16 (5120) FP16 4.2 / 4.8 / 7.4 / 14.1 against 3.7 / 5.3 / 9.7 / 14.5; 6x10x14x12 FP16 4.8 / 5.4 / 8.8 / 15.9
// against 4.0 / 5.5 / 9.9 / 14.9, BF16 5.6 / 6.2 / 10.1 / 18.6 against 4.2 / 5.9 / 10.8 / 16.8. So there the tile kernels
// would serve one to four systems better (by up to a third in BF16, whose FP64 updates run on 8 SMs here) and about
// 8 to 48 worse. The line is drawn by the lattice alone, so that a system's bits do not depend on its tile.
constexpr int SMALL_MAX_VH_16 = 5120;
constexpr int SMALL_MAX_VH_F32 = 4096;
constexpr int SMALL_MAX_VH_F64 = 1024;
template <typename Ts>
constexpr int small_max_vh() {
  return sizeof(Ts) == 8 ? SMALL_MAX_VH_F64 : sizeof(Ts) == 4 ? SMALL_MAX_VH_F32 : SMALL_MAX_VH_16;
}
constexpr int SMALL_CLUSTER = 8;

struct SmallShape {
  int threads, cluster;
};
inline SmallShape small_shape(int Vh) {
  SmallShape s;
  // 128 threads finish 32 sites of an FP64 hop at a time: no more blocks than that keeps busy
  s.threads = Vh <= SMALL_MAX_VH_F64 ? 128 : 256;
  s.cluster = 1;
  while (s.cluster < SMALL_CLUSTER && s.cluster * s.threads < 4 * Vh) s.cluster *= 2;
  return s;
}

struct SmallArgs {
  void *x_lo, *r, *rhat, *p, *v, *s, *t, *tmp;  // system-major
  double *x_hi, *bhat, *r_hi, *tmp64;
  int *ex_r, *ex_t;
  SysState* st;
  const void* gauge;  // inner precision
  const int4* gauge_fx;
  Geom g;
  int N;
  int iters;
  FinArgs fin;
};

template <typename Ts>
struct SysField {  // one system's parity, system-major, through the L2
  Ts* ptr;
  int Vh;
  template <typename Tm>
  __device__ __forceinline__ void load(int site, Tm (&v)[24]) const {
    constexpr int VW = Store<Ts>::VW;
#pragma unroll
    for (int c = 0; c < 24 / VW; c++) {
      const uint4 w = __ldcg(reinterpret_cast<const uint4*>(ptr + ((size_t)c * Vh + site) * VW));
      load_vec<Ts, Tm>(reinterpret_cast<const Ts*>(&w), v + c * VW);
    }
  }
  template <typename Tm>
  __device__ __forceinline__ void store(int site, const Tm (&v)[24]) const {
    constexpr int VW = Store<Ts>::VW;
#pragma unroll
    for (int c = 0; c < 24 / VW; c++) store_vec<Ts, Tm>(ptr + ((size_t)c * Vh + site) * VW, v + c * VW);
  }
  // stores v and leaves in it what was stored (rounded)
  template <typename Tm>
  __device__ __forceinline__ void store_round(int site, Tm (&v)[24]) const {
    constexpr int VW = Store<Ts>::VW;
#pragma unroll
    for (int c = 0; c < 24 / VW; c++) {
      uint4 w;
      store_vec<Ts, Tm>(reinterpret_cast<Ts*>(&w), v + c * VW);
      *reinterpret_cast<uint4*>(ptr + ((size_t)c * Vh + site) * VW) = w;
      load_vec<Ts, Tm>(reinterpret_cast<const Ts*>(&w), v + c * VW);
    }
  }
  // one spin's six reals (FP64 storage: a thread's share of a site)
  __device__ __forceinline__ void load(int site, int spin, double (&v)[6]) const {
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const double2 d = __ldcg(reinterpret_cast<const double2*>(ptr + ((size_t)(3 * spin + c) * Vh + site) * 2));
      v[2 * c] = d.x;
      v[2 * c + 1] = d.y;
    }
  }
  __device__ __forceinline__ void store(int site, int spin, const double (&v)[6]) const {
#pragma unroll
    for (int c = 0; c < 3; c++)
      *reinterpret_cast<double2*>(ptr + ((size_t)(3 * spin + c) * Vh + site) * 2) = make_double2(v[2 * c], v[2 * c + 1]);
  }
  // the share of a thread: a site, or a spin of it
  template <typename Tm> __device__ __forceinline__ void load(int site, int, Tm (&v)[24]) const { load(site, v); }
  template <typename Tm> __device__ __forceinline__ void store(int site, int, const Tm (&v)[24]) const { store(site, v); }
  template <typename Tm> __device__ __forceinline__ void store_round(int site, int, Tm (&v)[24]) const { store_round(site, v); }
  __device__ __forceinline__ void store_round(int site, int spin, double (&v)[6]) const { store(site, spin, v); }
};

// o += (cr + i ci) a over a thread's share
template <typename Tm, int NE>
__device__ __forceinline__ void share_acc(Tm (&o)[NE], const Tm (&a)[NE], Tm cr, Tm ci) {
#pragma unroll
  for (int k = 0; k < NE; k += 2) {
    o[k] += cr * a[k] - ci * a[k + 1];
    o[k + 1] += cr * a[k + 1] + ci * a[k];
  }
}

// A stored link, and its matrix with the third row and the boundary phase
template <typename Tg, int NR>
struct RawLink {
  static constexpr int C = link_pad<Tg>(NR) * (int)sizeof(Tg) / 16;
  uint4 w[C];
  __device__ __forceinline__ void load(const Tg* gauge, int Vh, int parity, int mu, int site) {
    const uint4* p = reinterpret_cast<const uint4*>(gauge + ((size_t)(parity * 4 + mu) * Vh + site) * link_pad<Tg>(NR));
#pragma unroll
    for (int c = 0; c < C; c++) w[c] = __ldg(p + c);
  }
  __device__ __forceinline__ void expand(float (&u)[18]) const {
    constexpr int VW = Store<Tg>::VW;
    float t[link_pad<Tg>(NR)];
#pragma unroll
    for (int c = 0; c < C; c++) load_vec<Tg, float>(reinterpret_cast<const Tg*>(&w[c]), t + c * VW);
#pragma unroll
    for (int k = 0; k < NR; k++) u[k] = t[k];
    if constexpr (NR == 12) link_row3(u);
  }
};

template <typename Ts, typename Tg, int NR>
__global__ void __launch_bounds__(std::is_same<Ts, double>::value ? 128 : 256, 2) small_iter_kernel(SmallArgs a) {
  namespace cg = cooperative_groups;
  using Tm = typename std::conditional<std::is_same<Ts, double>::value, double, float>::type;
  using Tx = Tm;
  constexpr bool F64 = std::is_same<Ts, double>::value;
  constexpr int NE = F64 ? 6 : 24;  // reals of a thread's share in the vector updates
  extern __shared__ int4 fx_words[];  // FX_WARP_WORDS per warp
  __shared__ double red[8][256];      // dot values of the block's threads
  __shared__ double tot[2][FIN_MAXV];  // the block's sums, by parity of the reduction
  __shared__ SysState state;
  __shared__ int fxE[8][32];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), C = (int)cl.num_blocks();
  const int sys = blockIdx.x / C;
  const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const Geom g = a.g;
  const int Vh = g.Vh;
  {
    const SysState& s0 = a.st[sys];
    if (s0.status != SYS_ACTIVE || (s0.flags & FLAG_CG)) return;  // the whole cluster
  }
  constexpr int words = (int)(sizeof(SysState) / 4);
  int* const sw = reinterpret_cast<int*>(&state);
  for (int w = tid; w < words; w += T) sw[w] = reinterpret_cast<const int*>(a.st + sys)[w];
  cl.sync();  // every block has its copy of the state (block 0 writes it at the end)

  const size_t so = (size_t)sys * 24 * Vh;
  auto f = [&](void* q) { return SysField<Ts>{(Ts*)q + so, Vh}; };
  auto fd = [&](double* q) { return SysField<double>{q + so, Vh}; };
  const SysField<Ts> r = f(a.r), rh = f(a.rhat), p = f(a.p), v = f(a.v), s = f(a.s), t = f(a.t), tmp = f(a.tmp);
  const SysField<Tx> xl{(Tx*)a.x_lo + so, Vh};
  const SysField<double> xh = fd(a.x_hi), bh = fd(a.bhat), rhi = fd(a.r_hi), t64 = fd(a.tmp64);
  int* const exr = a.ex_r + (size_t)sys * Vh;
  int* const ext = a.ex_t + (size_t)sys * Vh;
  // The vector updates: a thread per site (32-site runs dealt to the warps of the blocks in turn), or with FP64
  // storage per spin of a site, as the FP64 hop leaves them: an FP64 instruction costs a warp 64 clocks.
  const int grp = warp >> 2, spin = warp & 3, ngrp = T / 128;
  const int first = F64 ? (rank * ngrp + grp) * 32 + lane : (warp * C + rank) * 32 + lane;
  const int step = F64 ? C * ngrp * 32 : C * T;

  // a block's K values (per thread in w) and the scalar step op on the cluster's sums
  int par = 0;
  auto reduce = [&](auto Kc, const auto* w, int op) {
    constexpr int K = decltype(Kc)::value;
#pragma unroll
    for (int k = 0; k < K; k++) red[k][tid] = (double)w[k];
    __syncthreads();
    for (int k = warp; k < K; k += T / 32) {
      double q = red[k][lane] + red[k][lane + 32], q1 = red[k][lane + 64] + red[k][lane + 96];
      if (T > 128) {
        q += red[k][lane + 128] + red[k][lane + 160];
        q1 += red[k][lane + 192] + red[k][lane + 224];
      }
      q += q1;
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) q += __shfl_down_sync(0xffffffffu, q, d);
      if (lane == 0) tot[par][k] = q;
    }
    cl.sync();
    if (warp == 0) {
      // lane (rank group, value): the loads of the blocks' sums side by side, added up in one fixed order
      const int k = lane & 7;
      double q = 0.0;
#pragma unroll
      for (int h = 0; h < SMALL_CLUSTER / 4; h++) {
        const int c = (lane >> 3) + 4 * h;
        if (k < K && c < C) q += *cl.map_shared_rank(&tot[par][k], c);
      }
      q += __shfl_xor_sync(0xffffffffu, q, 8);
      q += __shfl_xor_sync(0xffffffffu, q, 16);
      double sum[FIN_MAXV];
#pragma unroll
      for (int i = 0; i < FIN_MAXV; i++) sum[i] = i < K ? lane_of(q, i) : 0.0;
      fin_logic(a.fin, op, state, sum);
    }
    par ^= 1;  // a buffer is written again two reductions, so at least one cluster barrier, later
    __syncthreads();
  };

  // ---- FP64 hop of 32 sites by four warps: the direction mu = warp & 3 of each, added up, then spin warp & 3 of
  // each site: o[6] is finished by `epi(site, spin, h)`, h = (H in) of that spin. Every thread takes part.
  auto fx_hop = [&](auto FXINc, const double* in, const int* in_ex, int p_out, auto&& store_fx, auto&& epi) {
    constexpr bool FXIN = decltype(FXINc)::value;
    FxHop<FXIN> h;
    h.gauge = a.gauge_fx;
    h.L0 = g.L[0]; h.L1 = g.L[1]; h.L2 = g.L[2]; h.L3 = g.L[3]; h.Lh0 = g.Lh0; h.Vh = Vh;
    h.p_out = p_out;
    h.sp = fx_words + (size_t)warp * FX_WARP_WORDS + lane;
    h.lw = fx_words + (size_t)warp * FX_WARP_WORDS + 12 * 32;
    h.lane = lane;
    h.lst = 5;
    h.nst = 32;
    h.slot = lane;
    h.rep = 1;
    h.cstride = (size_t)Vh * 2;
    h.sitestride = 2;
    h.in = in + so;
    h.in_ex = in_ex;
    const int q = spin;
    for (int base = (rank * ngrp + grp) * 32; base - grp * 32 < Vh; base += C * ngrp * 32) {
      const int site = min(base + lane, Vh - 1);
      const bool act = base + lane < Vh;
      h.site = site;
      int x[4];
      cb_coords(g, p_out, site, x);
      h.x0 = x[0]; h.x1 = x[1]; h.x2 = x[2]; h.x3 = x[3];
      long long acc[24];
      h.run(acc, 2 * q, 2 * q + 2);
      // this warp's sums over its spinor words (done with), [entry][lane]
      long long* const mine = reinterpret_cast<long long*>(fx_words + (size_t)warp * FX_WARP_WORDS);
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 24; k++) mine[k * 32 + lane] = acc[k];
      fxE[warp][lane] = h.bad ? FX_BAD : h.E;
      __syncthreads();
      int E = -50000;
      bool bad = false;
#pragma unroll
      for (int w = 0; w < 4; w++) {
        const int e = fxE[grp * 4 + w][lane];
        bad = bad || e == FX_BAD;
        E = max(E, e == FX_BAD ? -50000 : e);
      }
      long long z[6];
#pragma unroll
      for (int k = 0; k < 6; k++) z[k] = 0;
#pragma unroll
      for (int w = 0; w < 4; w++) {
        const long long* o = reinterpret_cast<const long long*>(fx_words + (size_t)(grp * 4 + w) * FX_WARP_WORDS);
        const int e = fxE[grp * 4 + w][lane], sh = min(E - (e == FX_BAD ? E : e), 62);
        const long long half = (1ll << sh) >> 1;
#pragma unroll
        for (int k = 0; k < 6; k++) z[k] += (o[(6 * q + k) * 32 + lane] + half) >> sh;
      }
      store_fx(site, q, act, z, E, bad);
      epi(site, q, act, z, E, bad);
      __syncthreads();  // the words are free again
    }
  };
  auto value6 = [&](double (&h)[6], const long long (&z)[6], int E, bool bad) {
    const int es = E - FX_UNIT + 1023;
    if ((unsigned)(es - 70) > 1800u || bad) {
#pragma unroll
      for (int k = 0; k < 6; k++)
        h[k] = bad ? __longlong_as_double(0x7ff8000000000000ll)
                   : (E < -4000 ? 0.0 : scalbn(__ll2double_rn(z[k]), E - FX_UNIT));
    } else {
#pragma unroll
      for (int k = 0; k < 6; k++) h[k] = fx_double(z[k], es);
    }
  };
  auto no_store = [](int, int, bool, const long long (&)[6], int, bool) {};

  // tmp = H_oe in, then out = M-hat in and the dot products of DOT with rhat; Tm sums in w
  auto mhat = [&](auto DOTc, const SysField<Ts>& in, const SysField<Ts>& out, Tm* w) {
    constexpr int DOT = decltype(DOTc)::value;
    constexpr int K = DOT == DOT_R ? 2 : 8;
#pragma unroll
    for (int k = 0; k < K; k++) w[k] = 0;
    if constexpr (F64) {
      fx_hop(BoolC<false>{}, (const double*)in.ptr - so, nullptr, 1, no_store,
             [&](int site, int q, bool act, const long long (&z)[6], int E, bool bad) {
               double h[6];
               value6(h, z, E, bad);
               if (act) tmp.store(site, q, h);
             });
      cl.sync();
      const double ca = state.cd[C_A], cb = state.cd[C_MINV4A];
      fx_hop(BoolC<false>{}, (const double*)tmp.ptr - so, nullptr, 0, no_store,
             [&](int site, int q, bool act, const long long (&z)[6], int E, bool bad) {
               if (!act) return;
               double o[6], x[6], rv[6];
               value6(o, z, E, bad);
               in.load(site, q, x);
               rh.load(site, q, rv);
#pragma unroll
               for (int k = 0; k < 6; k++) o[k] = axpby(ca, x[k], cb, o[k]);
               out.store(site, q, o);
#pragma unroll
               for (int k = 0; k < 6; k += 2) {
                 if constexpr (DOT == DOT_R) {
                   dot_acc(w[0], w[1], rv[k], rv[k + 1], o[k], o[k + 1]);
                 } else {
                   dot_acc(w[0], w[1], o[k], o[k + 1], x[k], x[k + 1]);
                   norm_acc(w[2], o[k], o[k + 1]);
                   norm_acc(w[3], x[k], x[k + 1]);
                   dot_acc(w[4], w[5], rv[k], rv[k + 1], x[k], x[k + 1]);
                   dot_acc(w[6], w[7], rv[k], rv[k + 1], o[k], o[k + 1]);
                 }
               }
             });
    } else {
      // A thread's operands (8 neighbour spinors, then X and rhat) come through a ring of its own in the
      // shared memory of the FP64 hop, PF ahead of the arithmetic, its links one direction ahead in registers: with
      // plain loads a hop is a chain of eight L2 latencies. M-hat takes 7 us at 4^3x8, 11 us on 8^4, of iterations
      // of 27 and 35 us; each of the two sums with its scalar step 3.5 to 6.
      constexpr int CV = chunks16<Ts>(), VW = Store<Ts>::VW, PF = sizeof(Ts) == 2 ? 6 : 3;
      static_assert(PF * CV * 16 * 32 <= FX_WARP_WORDS * 16, "the ring fits");
      static_assert(PF >= 2, "the eight directions issue all ten operands");
      uint4* const ring = reinterpret_cast<uint4*>(fx_words) + tid;
      const float ca = state.cf[C_A], cb = state.cf[C_MINV4A];
#pragma unroll 1
      for (int half = 0; half < 2; half++) {  // one copy of the hop's code
        if (half) cl.sync();
        const SysField<Ts>& src = half ? tmp : in;
        const int p_out = half ? 0 : 1;
        for (int site = first; site < Vh; site += step) {
          int x[4], nb[8];
          float ph[2] = {1.f, 1.f};  // t forward / backward boundary phase
          cb_coords(g, p_out, site, x);
#pragma unroll
          for (int m = 0; m < 4; m++) {
            int y[4] = {x[0], x[1], x[2], x[3]};
            y[m] = x[m] + 1;
            if (y[m] == g.L[m]) { y[m] = 0; if (m == 3) ph[0] = (float)g.bc_t; }
            nb[2 * m] = cb_index(g, y);
            y[m] = x[m] - 1;
            if (y[m] < 0) { y[m] = g.L[m] - 1; if (m == 3) ph[1] = (float)g.bc_t; }
            nb[2 * m + 1] = cb_index(g, y);
          }
          auto issue = [&](int item) {
            if (item < 8 || (half && item < 10)) {
              const Ts* q = item < 8 ? src.ptr + (size_t)nb[item & 7] * VW : (item == 8 ? in.ptr : rh.ptr) + (size_t)site * VW;
#pragma unroll
              for (int c = 0; c < CV; c++) cp_async16(ring + (item % PF * CV + c) * T, q + (size_t)c * Vh * VW);
            }
            cp_async_commit();  // one group per item (empty when idle) keeps the wait counts uniform
          };
          auto fetch = [&](int item, float (&o)[24]) {
#pragma unroll
            for (int c = 0; c < CV; c++) {
              const uint4 z = ring[(item % PF * CV + c) * T];
              load_vec<Ts, float>(reinterpret_cast<const Ts*>(&z), o + c * VW);
            }
          };
          RawLink<Tg, NR> lk;
          auto link = [&](int d) {
            lk.load((const Tg*)a.gauge, Vh, (d & 1) ? 1 - p_out : p_out, d >> 1, (d & 1) ? nb[d] : site);
          };
#pragma unroll
          for (int i = 0; i < PF; i++) issue(i);
          link(0);
          float acc[24], xf[12];
#pragma unroll
          for (int k = 0; k < 24; k++) acc[k] = 0.f;
#pragma unroll
          for (int d = 0; d < 8; d++) {
            float u[18], psi[24];
            lk.expand(u);
            if (d < 7) link(d + 1);
            cp_async_wait<PF - 1>();
            fetch(d, psi);
            issue(d + PF);
            switch (d) {
              case 0: hop_fwd<0>(xf, psi, u, 1.f); break;
              case 1: hop_bwd<0>(acc, xf, psi, u, 1.f); break;
              case 2: hop_fwd<1>(xf, psi, u, 1.f); break;
              case 3: hop_bwd<1>(acc, xf, psi, u, 1.f); break;
              case 4: hop_fwd<2>(xf, psi, u, 1.f); break;
              case 5: hop_bwd<2>(acc, xf, psi, u, 1.f); break;
              case 6: hop_fwd<3>(xf, psi, u, ph[0]); break;
              default: hop_bwd<3>(acc, xf, psi, u, ph[1]); break;
            }
          }
          cp_async_wait<0>();
          if (!half) {
            tmp.store(site, acc);
            continue;
          }
          float xv[24];
          fetch(8, xv);
#pragma unroll
          for (int k = 0; k < 24; k++) acc[k] = axpby(ca, xv[k], cb, acc[k]);
          out.store(site, acc);
          float rv[24];
          fetch(9, rv);
#pragma unroll
          for (int k = 0; k < 24; k += 2) {
            if constexpr (DOT == DOT_R) {
              dot_acc(w[0], w[1], rv[k], rv[k + 1], acc[k], acc[k + 1]);
            } else {
              dot_acc(w[0], w[1], acc[k], acc[k + 1], xv[k], xv[k + 1]);
              norm_acc(w[2], acc[k], acc[k + 1]);
              norm_acc(w[3], xv[k], xv[k + 1]);
              dot_acc(w[4], w[5], rv[k], rv[k + 1], xv[k], xv[k + 1]);
              dot_acc(w[6], w[7], rv[k], rv[k + 1], acc[k], acc[k + 1]);
            }
          }
        }
      }
    }
  };

#pragma unroll 1
  for (int it = 0; it < a.iters; it++) {
    Tm w[8];
    // (the p that its neighbours read was written before a cluster barrier: the previous launch, or the
    // barrier at the end of this loop)
    mhat(IntC<DOT_R>{}, p, v, w);
    reduce(IntC<2>{}, w, FIN_ALPHA);
    if (!(state.flags & FLAG_RESTART)) {
      {
        const Tm c0r = coef<Tm>(state, C_ALPHA), c0i = coef<Tm>(state, C_ALPHA + 1);
        for (int site = first; site < Vh; site += step) {
          Tm rv[NE], vv[NE];
          r.load(site, spin, rv);
          v.load(site, spin, vv);
          share_acc(rv, vv, -c0r, -c0i);
          s.store(site, spin, rv);
        }
      }
      cl.sync();
      mhat(IntC<DOT_TS>{}, s, t, w);
      reduce(IntC<8>{}, w, FIN_OMEGA);
      if (!(state.flags & FLAG_RESTART)) {
        const Tm c0r = coef<Tm>(state, C_ALPHA), c0i = coef<Tm>(state, C_ALPHA + 1);
        const Tm c1r = coef<Tm>(state, C_OMEGA), c1i = coef<Tm>(state, C_OMEGA + 1);
        const Tm c2r = coef<Tm>(state, C_BETA), c2i = coef<Tm>(state, C_BETA + 1);
        for (int site = first; site < Vh; site += step) {
          Tm xv[NE], pv[NE], sv[NE], tv[NE];
          p.load(site, spin, pv);
          s.load(site, spin, sv);
          xl.load(site, spin, xv);
          share_acc(xv, pv, c0r, c0i);
          share_acc(xv, sv, c1r, c1i);
          xl.store(site, spin, xv);
          t.load(site, spin, tv);
          share_acc(sv, tv, -c1r, -c1i);  // r = s - omega t
          r.store_round(site, spin, sv);  // the rounded r, as the next iteration sees it
          v.load(site, spin, tv);
          share_acc(pv, tv, -c1r, -c1i);  // p - omega v
          share_acc(sv, pv, c2r, c2i);    // r + beta (p - omega v)
          p.store(site, spin, sv);
        }
      }
    }
    if (state.flags & FLAG_UPDATE) {
      // ---- reliable update: x_hi += x_lo / scale, r = bhat - M x_hi in FP64, restart of the sloppy residual
      const bool keep = !(state.flags & FLAG_RESTART);
      const double isc = state.cd[C_INVSCALE];
      for (int site = first; site < Vh; site += step) {
        double hv[NE];
        xh.load(site, spin, hv);
        {
          Tx lv[NE];
          xl.load(site, spin, lv);
#pragma unroll
          for (int k = 0; k < NE; k++) {
            if (keep) hv[k] += isc * (double)lv[k];
            lv[k] = 0;
          }
          xl.store(site, spin, lv);
        }
        xh.store(site, spin, hv);
        if constexpr (!F64) {
          // x_hi as integers in r_hi, which the hop reads eight times
          long long z[24];
          exr[site] = fx_spinor(hv, z);
#pragma unroll
          for (int c = 0; c < 12; c++)
            *reinterpret_cast<longlong2*>(rhi.ptr + ((size_t)c * Vh + site) * 2) = make_longlong2(z[2 * c], z[2 * c + 1]);
        }
      }
      cl.sync();
      // tmp64 <- H_oe x_hi, as integers below 2^FX_BITS (the four warps of a group bring a site under one exponent)
      fx_hop(BoolC<!F64>{}, F64 ? a.x_hi : a.r_hi, exr, 1,
             [&](int site, int q, bool act, const long long (&z)[6], int E, bool bad) {
               // |sum| < 2^62: two bits down, under one exponent for the site's four threads
               if (!act) return;
#pragma unroll
               for (int c = 0; c < 3; c++)
                 *reinterpret_cast<longlong2*>(t64.ptr + ((size_t)(3 * q + c) * Vh + site) * 2) =
                     make_longlong2(z[2 * c] >> 2, z[2 * c + 1] >> 2);
               if (q == 0) ext[site] = bad ? FX_BAD : (E < -4000 ? FX_ZERO : E + 2 + FX_BITS + 1022 - FX_UNIT);
             },
             [](int, int, bool, const long long (&)[6], int, bool) {});
      cl.sync();
      double nd = 0.0;
      {
        const double ca = state.cd[C_MINVA], cb = state.cd[C_INV4A];
        fx_hop(BoolC<true>{}, a.tmp64, ext, 0, no_store,
               [&](int site, int q, bool act, const long long (&z)[6], int E, bool bad) {
                 if (!act) return;
                 double h[6], x[6], y[6];
                 value6(h, z, E, bad);
                 xh.load(site, q, x);
                 bh.load(site, q, y);
#pragma unroll
                 for (int k = 0; k < 6; k++) h[k] = fmadd(cb, h[k], fmadd(ca, x[k], y[k]));
                 rhi.store(site, q, h);
#pragma unroll
                 for (int k = 0; k < 6; k += 2) norm_acc(nd, h[k], h[k + 1]);
               });
      }
      reduce(IntC<1>{}, &nd, FIN_TRUE);  // (FP64 sums whatever the storage)
      if (state.status != SYS_ACTIVE) break;
      const bool reset = (state.flags & FLAG_RESTART) != 0;
      const double sc = state.cd[C_SCALE];
      const Tm ratio = coef<Tm>(state, C_RATIO);
      Tm dr = 0, di = 0, n2 = 0;
      for (int site = first; site < Vh; site += step) {
        double sv[NE];
        rhi.load(site, spin, sv);
        Tm iv[NE], o[NE], hv[NE];
        if (!reset) r.load(site, spin, iv);  // the iterated residual, replaced below
#pragma unroll
        for (int k = 0; k < NE; k++) o[k] = (Tm)(sc * sv[k]);
        r.store_round(site, spin, o);
        if (reset) {
          p.store(site, spin, o);
          Tm z[NE];
#pragma unroll
          for (int k = 0; k < NE; k++) { hv[k] = o[k]; z[k] = 0; }
          if (state.flags & FLAG_RESTART) {  // after a breakdown another rhat
            const int n = state.restarts;
#pragma unroll
            for (int k = 0; k < NE; k++) hv[k] *= restart_weight<Tm>(site, (F64 ? 3 * spin : 0) + (k >> 1), n);
          }
          rh.store_round(site, spin, hv);
          v.store(site, spin, z);
        } else {
          rh.load(site, spin, hv);
          Tm pv[NE];
          p.load(site, spin, pv);
#pragma unroll
          for (int k = 0; k < NE; k++) pv[k] = fmadd(ratio, pv[k] - iv[k], o[k]);
          p.store(site, spin, pv);
        }
#pragma unroll
        for (int k = 0; k < NE; k += 2) {
          dr += hv[k] * o[k] + hv[k + 1] * o[k + 1];
          di += hv[k] * o[k + 1] - hv[k + 1] * o[k];
          n2 += o[k] * o[k] + o[k + 1] * o[k + 1];
        }
      }
      Tm w3[3] = {dr, di, n2};
      reduce(IntC<3>{}, w3, FIN_UPDATE);
    }
    cl.sync();  // p and r are written
  }
  cl.sync();  // no block leaves while another may still read its sums
  if (rank == 0)
    for (int w = tid; w < words; w += T) reinterpret_cast<int*>(a.st + sys)[w] = sw[w];
}

}  // namespace fs
