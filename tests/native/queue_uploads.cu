// Host model of a tile for run_queue (csrc/fs_driver.cu), linked without the CUDA runtime: every stream operation waits
// in a queue until the host synchronises, the latest that stream order allows, and a copy from a pinned mirror reads it
// only then. A host write that does not wait for a pending copy shows as a wrong result.
// usage: queue_uploads staged|single|chain ; exit status 0 and "ok" if every row is right
#include <cstdio>
#include <cstring>
#include <deque>
#include <functional>
#include <limits>
#include <vector>

#include "fs_engine.h"
#include "fsmlmc.h"

#ifndef __CUDA_ARCH__  // (host code only)
namespace {
std::deque<std::function<void()>> pending;
void later(std::function<void()> f) { pending.push_back(std::move(f)); }
void run_all() {
  while (!pending.empty()) {
    auto f = std::move(pending.front());
    pending.pop_front();
    f();
  }
}
struct Event { int queued = 0; };
}  // namespace

extern "C" {
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  later([=] { memcpy(d, s, n); });
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { run_all(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t) new Event; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { run_all(); delete (Event*)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
  Event* v = (Event*)e;
  v->queued++;
  later([=] { v->queued--; });
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  while (((Event*)e)->queued > 0) {
    auto f = std::move(pending.front());
    pending.pop_front();
    f();
  }
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
int fs_probing_colors(const int*, int, int, int32_t*, int*) { return FS_ERR_ARG; }
}

namespace fs {

// One number stands for a vector: a solution is its right-hand side + 1, a kappa H application adds 100.
class ModelTile : public TileBase {
 public:
  std::vector<SysState> sth, std_;
  std::vector<NoiseSpec> sph, spd, stage_spec;
  std::vector<int> vh, vd, left;
  std::vector<double> z, x, pair[3], stage_x, stage_y;
  int alloc(Ctx*, int n, int) override {
    N = n;
    sth.assign(n, SysState{}); std_ = sth;
    sph.assign(n, NoiseSpec{}); spd = sph;
    vh.assign(n, -1); vd = vh;
    left.assign(n, 0);
    z.assign(n, 0.0); x = z;
    for (auto& p : pair) p = z;
    st_h = sth.data(); st_d = std_.data(); spec_h = sph.data(); spec_d = spd.data();
    vec_h = vh.data(); vec_d = vd.data();
    return 0;
  }
  void set_shape(const PkShape&) override {}
  int clover_alloc() override { return 0; }
  int iters_per_check(int every) const override { return every; }
  cudaError_t enqueue_rhs_from_canon(const double* canon) override {
    later([=] {
      for (int j = 0; j < N; j++)
        if ((std_[j].flags & FLAG_INIT) && vd[j] >= 0) z[j] = canon[vd[j]];
    });
    return cudaSuccess;
  }
  cudaError_t enqueue_noise() override {
    later([=] {
      for (int j = 0; j < N; j++)
        if ((std_[j].flags & FLAG_INIT) && (spd[j].flags & NOISE_RHS)) z[j] = spd[j].sample;
    });
    return cudaSuccess;
  }
  cudaError_t enqueue_init() override {
    later([=] {
      for (int j = 0; j < N; j++) {
        if (!(std_[j].flags & FLAG_INIT)) continue;
        std_[j].flags = 0;
        std_[j].status = SYS_ACTIVE;
        left[j] = 1 + (int)spd[j].sample % 4;  // looks until it has converged
      }
    });
    return cudaSuccess;
  }
  cudaError_t enqueue_iter() override { return cudaErrorInvalidValue; }
  cudaError_t enqueue_iters(int) override {
    later([=] {
      for (int j = 0; j < N; j++)
        if (std_[j].status == SYS_ACTIVE && --left[j] <= 0) std_[j].status = SYS_CONVERGED;
    });
    return cudaSuccess;
  }
  cudaError_t enqueue_recon() override {
    later([=] {
      for (int j = 0; j < N; j++)
        if (std_[j].flags & FLAG_HARVEST) x[j] = z[j] + 1;
    });
    return cudaSuccess;
  }
  cudaError_t enqueue_verify() override { return cudaSuccess; }
  cudaError_t enqueue_solution_to_canon(double* canon) override {
    later([=] {
      for (int j = 0; j < N; j++)
        if (vd[j] >= 0) canon[vd[j]] = x[j];
    });
    return cudaSuccess;
  }
  cudaError_t enqueue_dslash(double*) override { return cudaErrorInvalidValue; }
  double* field_pair(int, int) override { return nullptr; }
  cudaError_t enqueue_kappa_hop(int from, int to) override {
    later([=] {
      for (int j = 0; j < N; j++)
        if (std_[j].flags & FLAG_HPE) pair[to][j] = (from == PAIR_X ? x[j] : pair[from][j]) + 100;
    });
    return cudaSuccess;
  }
  cudaError_t enqueue_site_inverse(int, int) override { return cudaErrorInvalidValue; }
  int stage_alloc(int S, bool) override {
    stage_cols = S;
    stage_x.assign(S, 0.0); stage_y = stage_x;
    stage_spec.assign(S, NoiseSpec{});
    return 0;
  }
  cudaError_t enqueue_stage(const StageMoves& mv, int right_pair) override {
    later([=] {
      for (int k = 0; k < mv.n; k++) {
        stage_x[mv.col[k]] = x[mv.slot[k]];
        if (mv.with_y[k]) stage_y[mv.col[k]] = pair[right_pair][mv.slot[k]];
        stage_spec[mv.col[k]] = spd[mv.slot[k]];
      }
    });
    return cudaSuccess;
  }
  int cg_alloc() override { return 3; }
  cudaError_t enqueue_cg_init() override { return cudaErrorInvalidValue; }
  cudaError_t enqueue_cg_iter() override { return cudaErrorInvalidValue; }
};

int Ctx::cuda_fail(cudaError_t, const char* where) { return fail(FS_ERR_CUDA, where); }
TileBase* Ctx::tile(int, int, int) { return nullptr; }
int upload_colors(Ctx*, const int*) { return FS_ERR_ARG; }
// row <- 1e6 x left noise + right vector
int contract_tile(Ctx*, TileBase* T, const std::vector<ContractPair>& pairs, const double*, const std::vector<int>&,
                  std::vector<double>& result, int rows, int right_pair, const StageView* sv) {
  run_all();
  ModelTile& t = *(ModelTile*)T;
  result.assign((size_t)rows * 2, 0.0);
  for (const ContractPair& p : pairs) {
    const NoiseSpec& l = sv ? t.stage_spec[p.left] : t.spd[p.left];
    const double r = p.right_kind ? (sv ? t.stage_y[p.right] : t.pair[right_pair][p.right])
                                  : (sv ? t.stage_x[p.right] : t.x[p.right]);
    result[(size_t)p.out * 2] = 1e6 * l.sample + r;
  }
  return 0;
}

}  // namespace fs

int main(int argc, char** argv) {
  using namespace fs;
  if (argc != 2) return 2;
  const bool staged = !strcmp(argv[1], "staged"), chain = !strcmp(argv[1], "chain");
  const double none = std::numeric_limits<double>::quiet_NaN();
  Ctx c;
  ModelTile T;
  T.alloc(&c, 7, 18);
  std::vector<double> canon(64, 0.0);
  c.canon_d = canon.data();
  SolveOpts o{};
  o.m = 0.1; o.tol = 1e-8; o.max_iter = 100; o.check_every = 1;
  std::vector<QJob> jobs;
  std::vector<double> want;
  const int K = chain ? 0 : 3;
  for (int n = 0; n < 40; n++) {
    // groups of two systems (staged), of one, and of one with a follow-up solve; every third takes the expansion
    QJob q;
    const int members = staged && n % 3 ? 2 : 1;
    for (int m = 0; m < members; m++) {
      SysSpec s{};
      s.sigma = 0.1 * m;
      s.noise.sample = 1 + 2 * n + m;
      s.noise.flags = NOISE_VALID;
      s.hpe = !chain && n % 3 == 0;
      q.sys.push_back(s);
      q.chain.push_back(chain && n % 2 ? 0.7 : none);
    }
    ContractPair p{members - 1, 0, 0, n};
    p.right_kind = q.sys[0].hpe;
    q.pairs.push_back(p);
    want.push_back(1e6 * (1 + 2 * n) + (1 + 2 * n + members - 1) + 1 + (p.right_kind ? 100 * K : 0) +
                   (chain && n % 2 ? 1 : 0));
    jobs.push_back(q);
  }
  std::vector<double> got(2 * want.size(), 0.0);
  const std::vector<int> plist = {0};
  QOut out;
  out.plist = &plist;
  out.rows = (int)want.size();
  out.result = &got;
  out.hpe_order = K;
  int rc = run_queue(&c, &T, jobs, o, out);
  run_all();
  int bad = 0;
  for (size_t n = 0; n < want.size(); n++)
    if (got[2 * n] != want[n]) {
      bad++;
      printf("row %zu: %.0f, not %.0f\n", n, got[2 * n], want[n]);
    }
  printf("%s\n", rc == 0 && bad == 0 ? "ok" : "failed");
  return rc == 0 && bad == 0 ? 0 : 1;
}
#endif
