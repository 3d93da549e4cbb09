// Grouped Chebyshev filter over many independent problems (Alg. 4 applied to
// a batch of Hermitian matrices of different sizes).
//
// The paper filters one matrix at a time; a batch of small problems (N of a
// few hundred to a few thousand) leaves most of GB300's 152 SMs idle when
// each product is its own launch.  Here every degree step of the filter is
// one launch over the output tiles of all problems that still have active
// columns: CTA t finds its problem by binary search over the step's tile
// prefix, so the hardware block scheduler hands the next tile of any problem
// to whichever SM frees up (problems are ordered by decreasing N, longest
// tiles first).  Per problem the columns are sorted by degree (Alg. 4 lines
// 12-14 keep an active suffix), the recurrence coefficients of Eq. 7 are
// computed on the host once per call, and the whole sequence of step
// launches is captured into a CUDA graph and launched once.
//
// Products run as residue GEMMs (rns.cu): per step one launch slices the
// active columns of every problem, one multiplies, one puts the products
// together.  FP64 batches that are too small for that, and those for which the
// caller names a tile shape, run on the DMMA kernel; its shape is chosen by
// timing the first step (which only writes the second buffer, so it can be
// repeated), and the choice is cached per batch shape.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <limits>
#include <map>
#include <mutex>
#include <numeric>
#include <tuple>
#include <vector>

#include "chase.h"
#include "common.cuh"
#include "context.hpp"

namespace chase {
namespace {

constexpr int kMaxDegree = 1024;

// Per-problem constants of Alg. 4 lines 2-3 and the problem's place in the
// grouped order.
struct Coef {
  int q;  // index into the caller's input list
  double c, e, sigma1;
};

// Step list of degree step i (1-based): FP64 tiles of bm x bn complex columns,
// or (nmod > 0) residue products with tiles bn columns wide.  sigma_prev[k] is
// sigma after step i - 1 of problem k (Alg. 4 line 11).
struct StepTotals {
  int tiles = 0, cols = 0, blocks = 0;
};
void build_step(const std::vector<GroupedFilterInput>& in, const std::vector<Coef>& co, int i,
                int bm, int bn, int nmod, const std::vector<double>& sigma_prev,
                std::vector<GroupedStep>& out, StepTotals* totals) {
  out.clear();
  StepTotals t;
  for (size_t k = 0; k < co.size(); ++k) {
    const GroupedFilterInput& pi = in[co[k].q];
    if (i > pi.maxdeg) continue;
    const int s = pi.start[i];
    if (s >= pi.b) continue;
    GroupedStep g{};
    g.prob = static_cast<int>(k);
    g.s = s;
    g.tile0 = t.tiles;
    g.col0 = t.cols;
    g.blk0 = t.blocks;
    if (i == 1) {  // Alg. 4 line 4
      g.alpha = co[k].sigma1 / co[k].e;
      g.beta = 0.0;
    } else {  // lines 8-9
      const double sigma = sigma_prev[k];
      const double tau = 1.0 / (2.0 / co[k].sigma1 - sigma);
      g.alpha = 2.0 * tau / co[k].e;
      g.beta = -tau * sigma;
    }
    g.shift = co[k].c;
    const int cols = pi.b - s;
    if (nmod > 0) {
      g.sc = rns_scale(nmod, g.alpha, g.beta, g.shift);
      t.tiles += rns_grouped_tiles(nmod, bn, pi.n, cols);
      t.blocks += rns_grouped_crt_blocks(pi.n, cols);
    } else {
      t.tiles += (pi.n + bm - 1) / bm * ((cols + bn - 1) / bn);
    }
    t.cols += cols;
    out.push_back(g);
  }
  GroupedStep sentinel{};
  sentinel.prob = -1;
  sentinel.tile0 = t.tiles;
  sentinel.col0 = t.cols;
  sentinel.blk0 = t.blocks;
  out.push_back(sentinel);
  *totals = t;
}

// Width of the residue tiles of degree step i: the one with the least work,
// counting a tile's padding columns.
int residue_tile_width(const std::vector<GroupedFilterInput>& in, const std::vector<Coef>& co,
                       int i, int nmod) {
  int best = 32;
  double best_cost = 0.0;
  for (int bn = 32; bn <= 256; bn += 32) {
    double cost = 0.0;
    for (const Coef& c : co) {
      const GroupedFilterInput& pi = in[c.q];
      if (i > pi.maxdeg || pi.start[i] >= pi.b) continue;
      // two stages' time for the start and the end of a tile
      cost += rns_grouped_tiles(nmod, bn, pi.n, pi.b - pi.start[i]) * ((pi.n + 63) / 64 + 2.0) *
              rns_stage_cost(bn);
    }
    if (best_cost == 0.0 || cost < 0.995 * best_cost) {
      best_cost = cost;
      best = bn;
    }
  }
  return best;
}

std::mutex g_tune_mu;
std::map<std::tuple<int, long long, long long, int, int>, int> g_tune_cache;

double now_s() {
  return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

struct GraphGuard {
  cudaGraph_t g = nullptr;
  cudaGraphExec_t x = nullptr;
  cudaStream_t cs = nullptr;
  ~GraphGuard() {
    if (x) cudaGraphExecDestroy(x);
    if (g) cudaGraphDestroy(g);
    if (cs) cudaStreamDestroy(cs);
  }
};

struct EventPool {
  std::vector<cudaEvent_t> ev;
  cudaEvent_t get() {
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    ev.push_back(e);
    return e;
  }
  ~EventPool() {
    for (auto e : ev) cudaEventDestroy(e);
  }
};

float elapsed_ms(cudaEvent_t a, cudaEvent_t b) {
  float ms = 0.f;
  if (cudaEventElapsedTime(&ms, a, b) != cudaSuccess) return 0.f;
  return ms;
}

}  // namespace

namespace {
// Estimates of one degree step in microseconds, where all columns are active.
// FP64 tiles of 64 x 8: the longest tile, or what the SMs get through (32
// problems of N = 256, 19 columns: 368 us; 300 of N = 64, 8: 73; 2000 of N = 16,
// 8: 134).  Residue products of small problems: three launches and 1.27 us a
// tile and pair (8 of N = 256: 31; 300 of N = 64: 160 with 14 moduli, 134 with
// 11; 2000 of N = 16: 947 and 777); larger tiles take longer, but there the FP64
// tiles are far behind.
double fp64_step_us(const std::vector<GroupedFilterInput>& in) {
  double longest = 0.0, sum = 0.0;
  for (const GroupedFilterInput& g : in) {
    if (g.n == 0 || g.b == 0) continue;
    longest = std::max(longest, 8.0 + 0.5 * g.n);
    sum += ((g.n + 63) / 64) * ((g.b + 7) / 8) * static_cast<double>(g.n) / 260.0;
  }
  return std::max(longest, sum);
}
double residue_step_us(const std::vector<GroupedFilterInput>& in, int nmod) {
  double tiles = 0.0;
  for (const GroupedFilterInput& g : in)
    if (g.n > 0 && g.b > 0)
      tiles += rns_grouped_tiles(nmod, std::min(256, (g.b + 31) / 32 * 32), g.n, g.b);
  return 25.0 + 1.27 * tiles / 76.0;
}
}  // namespace

// Residue products, for an FP64 batch from 2e7 FLOPs a degree step on (a cautious
// line: 8 problems of N = 128, 10 columns, 1e7, take 70 us a step on the tiles,
// 28 as 11-moduli residues), unless the FP64 tiles are done sooner: many problems of few rows each fill the device
// with FP64 tiles, where each of their residue planes pads a tile of 256 rows.
// 2000 problems of N = 16, ten steps in all: 11.2 ms on the FP64 tiles, 20.4 and
// 18.8 ms as residues (14 and 11 moduli); 200 of N = 100: 3.0, 2.8 and 2.5 ms.
int grouped_moduli(const std::vector<GroupedFilterInput>& in, bool split, int tile, bool rr) {
  int64_t most = 0;
  double step = 0.0;
  for (const GroupedFilterInput& g : in) {
    most = std::max<int64_t>(most, g.n);
    step += 8.0 * g.n * static_cast<double>(g.n) * g.b;
  }
  const int nmod = !split ? kRnsFp64 : rr ? kRnsSplitRR : rns_split_moduli(most, true);
  if (!split && (tile != CHASE_TILE_AUTO || step < 2e7)) return 0;
  return residue_step_us(in, nmod) < fp64_step_us(in) ? nmod : 0;
}

void grouped_rns_release(Dev& d, std::vector<GroupedFilterInput>& in, GroupedWork& w) {
  for (void* p : {w.block, w.planes})
    if (p) d.release(p);
  w = GroupedWork{};
  for (GroupedFilterInput& g : in) {
    g.A = g.Bsl = g.G = nullptr;
    g.E = g.F = nullptr;
    g.Dg = nullptr;
    g.bcap = g.sym = 0;
  }
}

namespace {
// Parts of one allocation, each on a 256-byte boundary: an allocation (and its
// release) per part cost about 5 us a problem on the host.
struct Parts {
  unsigned char* base = nullptr;
  size_t at = 0;
  void* take(size_t bytes) {
    void* p = base ? base + at : nullptr;
    at += (bytes + 255) / 256 * 256;
    return p;
  }
};

// Exponents, diagonals and the planes of the blocks of every problem; without a
// base only their sum is formed.
void block_parts(std::vector<GroupedFilterInput>& in, const std::vector<int>& bcap, int nmod,
                 Parts& parts) {
  for (size_t q = 0; q < in.size(); ++q) {
    GroupedFilterInput& g = in[q];
    if (g.n == 0) continue;
    g.bcap = std::max(bcap[q], 1);
    const size_t block = static_cast<size_t>(2 * nmod) * g.bcap * rns_k_padded(g.n) * 2;
    g.E = static_cast<int*>(parts.take(sizeof(int) * g.n));
    g.Dg = static_cast<double*>(parts.take(sizeof(double) * g.n));
    g.Bsl = parts.take(block);
    g.G = parts.take(block);
    g.F = static_cast<int*>(parts.take(sizeof(int) * g.bcap));
  }
}
void plane_parts(std::vector<GroupedFilterInput>& in, int nmod, Parts& parts) {
  for (GroupedFilterInput& g : in)
    if (g.n > 0)
      g.A = parts.take(static_cast<size_t>(g.sym ? nmod : 2 * nmod) * g.n * rns_k_padded(g.n) * 2);
}

int prepare_planes(Dev& d, std::vector<GroupedFilterInput>& in, const std::vector<int>& bcap,
                   int nmod, size_t reserve, GroupedWork& w) {
  std::vector<GroupedSliceH> all;
  std::vector<size_t> owner;
  int rows = 0;
  double entries = 0.0;
  Parts parts;
  block_parts(in, bcap, nmod, parts);
  const size_t block_bytes = parts.at;
  for (size_t q = 0; q < in.size(); ++q) {
    GroupedFilterInput& g = in[q];
    if (g.n == 0) continue;
    entries += static_cast<double>(g.n) * rns_k_padded(g.n);
    GroupedSliceH sh{};
    sh.H = reinterpret_cast<const double2*>(g.H);
    sh.ldh = g.ldh;
    sh.Kp = rns_k_padded(g.n);
    sh.n = g.n;
    sh.row0 = rows;
    all.push_back(sh);
    owner.push_back(q);
    rows += g.n;
  }
  if (all.empty()) return CHASE_OK;
  const int P = static_cast<int>(all.size());
  CHASE_TRY(d.alloc_bytes(&w.block, block_bytes));
  parts = Parts{static_cast<unsigned char*>(w.block)};
  block_parts(in, bcap, nmod, parts);
  for (int p = 0; p < P; ++p) {
    all[p].E = in[owner[p]].E;
    all[p].Dg = in[owner[p]].Dg;
  }
  // one list on the device per launch: all problems, then those with one
  // scale, then the others
  struct Lists {
    Dev& d;
    GroupedSliceH* problems = nullptr;
    int* minmax = nullptr;
    ~Lists() {
      if (problems) d.release(problems);
      if (minmax) d.release(minmax);
    }
  } lists{d};
  CHASE_TRY(d.alloc(&lists.problems, 3 * all.size()));
  CHASE_TRY(d.alloc(&lists.minmax, 2 * all.size()));
  GroupedSliceH* const dl = lists.problems;
  int* const mm = lists.minmax;
  std::vector<int> hmm(2 * all.size());
  for (int p = 0; p < P; ++p) {
    hmm[2 * p] = std::numeric_limits<int>::max();
    hmm[2 * p + 1] = -std::numeric_limits<int>::max();
  }
  auto upload = [&](GroupedSliceH* to, const std::vector<GroupedSliceH>& v) -> int {
    CHASE_CUDA(cudaMemcpyAsync(to, v.data(), sizeof(GroupedSliceH) * v.size(),
                               cudaMemcpyHostToDevice, d.st));
    return CHASE_OK;
  };
  if (rns_sym_pays(2 * nmod, entries)) {
    CHASE_TRY(upload(dl, all));
    CHASE_CUDA(cudaMemcpyAsync(mm, hmm.data(), sizeof(int) * hmm.size(), cudaMemcpyHostToDevice,
                               d.st));
    CHASE_TRY(rns_grouped_row_exponents(d, nmod, dl, P, rows, mm));
    CHASE_CUDA(cudaMemcpyAsync(hmm.data(), mm, sizeof(int) * hmm.size(), cudaMemcpyDeviceToHost,
                               d.st));
    CHASE_TRY(d.sync_check("grouped row scales of H"));
  }
  for (int p = 0; p < P; ++p)
    in[owner[p]].sym = rns_same_scale(hmm[2 * p], hmm[2 * p + 1]) ? 1 : 0;
  parts = Parts{};
  plane_parts(in, nmod, parts);
  size_t free_b = 0;
  CHASE_TRY(d.free_bytes(&free_b));
  if (parts.at + reserve > free_b) {
    set_error("residue planes of a batch: %zu bytes do not fit the memory", parts.at);
    return CHASE_OUT_OF_MEMORY;
  }
  CHASE_TRY(d.alloc_bytes(&w.planes, parts.at));
  parts = Parts{static_cast<unsigned char*>(w.planes)};
  plane_parts(in, nmod, parts);
  std::vector<GroupedSliceH> one, each;
  int tiles = 0, erows = 0;
  for (int p = 0; p < P; ++p) {
    const GroupedFilterInput& g = in[owner[p]];
    GroupedSliceH sh = all[p];
    sh.A = g.A;
    sh.s = hmm[2 * p];
    if (g.sym) {
      sh.tile0 = tiles;
      tiles += rns_sym_tiles(g.n);
      one.push_back(sh);
    } else {
      sh.row0 = erows;
      erows += g.n;
      each.push_back(sh);
    }
  }
  if (!one.empty()) {
    CHASE_TRY(upload(dl + P, one));
    CHASE_TRY(rns_grouped_prepare_sym(d, nmod, dl + P, static_cast<int>(one.size()), tiles));
  }
  if (!each.empty()) {
    CHASE_TRY(upload(dl + 2 * P, each));
    CHASE_TRY(rns_grouped_prepare_h(d, nmod, dl + 2 * P, static_cast<int>(each.size()), erows));
  }
  // the host arrays must outlive the copies
  return d.sync_check("grouped residues of H");
}
}  // namespace

int grouped_rns_prepare(Dev& d, std::vector<GroupedFilterInput>& in, const std::vector<int>& bcap,
                        int nmod, size_t reserve, GroupedWork& w) {
  const int st = prepare_planes(d, in, bcap, nmod, reserve, w);
  if (st != CHASE_OK) grouped_rns_release(d, in, w);
  return st;
}

namespace {
// The whole of `in` at once; prepared for residue products where nmod > 0.
int filter_part(Dev& d, const std::vector<GroupedFilterInput>& in, int nmod, int tile,
                GroupedFilterTimes* times) {
  const bool rns = nmod > 0;
  const long long launches0 = chase_kernel_launches();
  GroupedFilterTimes tt;
  // active problems, longest tiles first: the block scheduler then balances the tail
  std::vector<Coef> co;
  int maxdeg = 0;
  for (size_t q = 0; q < in.size(); ++q) {
    const GroupedFilterInput& g = in[q];
    if (g.n == 0 || g.b == 0) continue;
    Coef c;
    c.q = static_cast<int>(q);
    c.c = 0.5 * (g.b_sup + g.mu_nn);  // Alg. 4 line 2
    c.e = 0.5 * (g.b_sup - g.mu_nn);
    c.sigma1 = c.e / (g.mu1 - c.c);   // line 3
    co.push_back(c);
    maxdeg = std::max(maxdeg, g.maxdeg);
  }
  std::stable_sort(co.begin(), co.end(),
                   [&](const Coef& x, const Coef& y) { return in[x.q].n > in[y.q].n; });
  const int Q = static_cast<int>(co.size());
  if (Q == 0) {
    if (times) *times = tt;
    return CHASE_OK;
  }
  EventPool evp;
  const int nmaps = rns ? 1 + 8 : 3;  // residues: H and a block map per tile width
  CUtensorMap* dmaps = nullptr;
  CHASE_TRY(d.alloc_bytes(reinterpret_cast<void**>(&dmaps), sizeof(CUtensorMap) * nmaps * Q));
  GroupedProblem* dprobs = nullptr;
  CHASE_TRY(d.alloc(&dprobs, Q));
  std::vector<GroupedProblem> probs(Q);
  std::vector<CUtensorMap> maps(static_cast<size_t>(nmaps) * Q);
  for (int k = 0; k < Q; ++k) {
    const GroupedFilterInput& pi = in[co[k].q];
    GroupedProblem& g = probs[k];
    g = GroupedProblem{};
    g.n = pi.n;
    g.b = pi.b;
    g.buf0 = reinterpret_cast<double2*>(pi.X);
    g.ld0 = pi.ldx;
    g.buf1 = reinterpret_cast<double2*>(pi.W);
    g.ld1 = pi.ldw;
    g.mapA = dmaps + nmaps * k;
    g.mapB0 = dmaps + nmaps * k + 1;
    g.mapB1 = rns ? nullptr : dmaps + nmaps * k + 2;
    if (rns) {
      if (!pi.A || !pi.Bsl || pi.bcap < pi.b) {
        set_error("grouped filter: residue workspace missing or too small");
        return CHASE_INVALID_ARG;
      }
      g.Kp = rns_k_padded(pi.n);
      g.E = pi.E;
      g.F = pi.F;
      g.Dg = pi.Dg;
      g.Bsl = pi.Bsl;
      g.G = pi.G;
      g.bcap = pi.bcap;
      g.sym = pi.sym;
    }
  }
  CHASE_CUDA(cudaMemcpyAsync(dprobs, probs.data(), sizeof(GroupedProblem) * Q, cudaMemcpyHostToDevice,
                             d.st));
  // FP64 maps depend on the tile shape: encoded after the tile choice.
  auto encode_fp64_maps = [&](int cfg) -> int {
    int bm = 0, bn = 0;
    grouped_fp64_tile(cfg, &bm, &bn);
    for (int k = 0; k < Q; ++k) {
      const GroupedFilterInput& pi = in[co[k].q];
      CHASE_TRY(make_tmap_c64(&maps[nmaps * k], pi.H, pi.n, pi.n, pi.ldh, bm, 16));
      CHASE_TRY(make_tmap_c64(&maps[nmaps * k + 1], pi.X, pi.n, pi.b, pi.ldx, 16, bn));
      CHASE_TRY(make_tmap_c64(&maps[nmaps * k + 2], pi.W, pi.n, pi.b, pi.ldw, 16, bn));
    }
    CHASE_CUDA(cudaMemcpyAsync(dmaps, maps.data(), sizeof(CUtensorMap) * maps.size(),
                               cudaMemcpyHostToDevice, d.st));
    // the host array is rewritten by the next encoding: finish this copy first
    CHASE_CUDA(cudaStreamSynchronize(d.st));
    return CHASE_OK;
  };

  int cfg = -1;
  std::vector<int> width(maxdeg + 1, 0);  // residues: tile width of each step
  if (rns) {
    bool used[8] = {};
    for (int i = 1; i <= maxdeg; ++i) {
      width[i] = residue_tile_width(in, co, i, nmod);
      used[width[i] / 32 - 1] = true;
    }
    for (int k = 0; k < Q; ++k) {
      const GroupedFilterInput& pi = in[co[k].q];
      for (int w = 0; w < 8; ++w)
        if (used[w])
          CHASE_TRY(rns_grouped_maps(&maps[nmaps * k], &maps[nmaps * k + 1 + w], nmod, 32 * (w + 1),
                                     pi.sym != 0, pi.A, pi.Bsl, pi.n, pi.b, pi.bcap));
    }
    CHASE_CUDA(cudaMemcpyAsync(dmaps, maps.data(), sizeof(CUtensorMap) * maps.size(),
                               cudaMemcpyHostToDevice, d.st));
  } else if (tile != CHASE_TILE_AUTO) {
    cfg = tile;
  } else {
    long long sum_n = 0, sum_nb = 0;
    int max_n = 0;
    for (const Coef& c : co) {
      sum_n += in[c.q].n;
      sum_nb += static_cast<long long>(in[c.q].n) * in[c.q].b;
      max_n = std::max(max_n, in[c.q].n);
    }
    const auto key = std::make_tuple(Q, sum_n, sum_nb, max_n, maxdeg);
    {
      std::lock_guard<std::mutex> lk(g_tune_mu);
      auto it = g_tune_cache.find(key);
      if (it != g_tune_cache.end()) cfg = it->second;
    }
    if (cfg < 0) {
      // time step 1 (reads X, writes W only) with every tile shape
      const double ta = now_s();
      float best = 0.f;
      std::vector<double> sigma0(Q, 0.0);
      for (int c = 0; c < kGroupedFp64Cfgs; ++c) {
        int bm = 0, bn = 0;
        grouped_fp64_tile(c, &bm, &bn);
        std::vector<GroupedStep> one;
        StepTotals tot;
        build_step(in, co, 1, bm, bn, 0, sigma0, one, &tot);
        GroupedStep* dst1 = nullptr;
        CHASE_TRY(d.alloc(&dst1, one.size()));
        CHASE_CUDA(cudaMemcpyAsync(dst1, one.data(), sizeof(GroupedStep) * one.size(),
                                   cudaMemcpyHostToDevice, d.st));
        CHASE_TRY(encode_fp64_maps(c));
        cudaEvent_t ea = evp.get(), eb = evp.get();
        if (!ea || !eb) {
          set_error("grouped filter: event creation failed");
          return CHASE_CUDA_ERROR;
        }
        const int na = static_cast<int>(one.size()) - 1;
        // one untimed launch, then the timed one
        CHASE_TRY(zgemm_grouped_fp64(d, c, dprobs, dst1, na, tot.tiles, 0));
        CHASE_CUDA(cudaEventRecord(ea, d.st));
        CHASE_TRY(zgemm_grouped_fp64(d, c, dprobs, dst1, na, tot.tiles, 0));
        CHASE_CUDA(cudaEventRecord(eb, d.st));
        CHASE_TRY(d.sync_check("grouped filter autotune"));
        const float ms = elapsed_ms(ea, eb);
        if (cfg < 0 || ms < best) {
          best = ms;
          cfg = c;
        }
      }
      tt.t_autotune = now_s() - ta;
      std::lock_guard<std::mutex> lk(g_tune_mu);
      g_tune_cache[key] = cfg;
    }
  }
  int bm = 0, bn = 0;
  if (!rns) {
    grouped_fp64_tile(cfg, &bm, &bn);
    CHASE_TRY(encode_fp64_maps(cfg));
  }
  // ---- every step's list, uploaded once ----
  std::vector<GroupedStep> all, one;
  std::vector<int> first(maxdeg + 1, 0), nact(maxdeg + 1, 0);
  std::vector<StepTotals> tot(maxdeg + 1);
  {
    std::vector<double> sigma(Q, 0.0);
    for (int i = 1; i <= maxdeg; ++i) {
      build_step(in, co, i, bm, rns ? width[i] : bn, nmod, sigma, one, &tot[i]);
      first[i] = static_cast<int>(all.size());
      nact[i] = static_cast<int>(one.size()) - 1;
      all.insert(all.end(), one.begin(), one.end());
      for (int k = 0; k < Q; ++k) {  // Alg. 4 line 11
        if (i == 1)
          sigma[k] = co[k].sigma1;
        else if (i <= in[co[k].q].maxdeg)
          sigma[k] = 1.0 / (2.0 / co[k].sigma1 - sigma[k]);
      }
    }
  }
  GroupedStep* dsteps = nullptr;
  CHASE_TRY(d.alloc(&dsteps, all.size()));
  CHASE_CUDA(cudaMemcpyAsync(dsteps, all.data(), sizeof(GroupedStep) * all.size(),
                             cudaMemcpyHostToDevice, d.st));

  // Small problems: a pair takes tiles that follow one another, mostly planes of
  // one problem, whose description it then finds in L1 and whose tensor maps it
  // acquires once (200 problems of N = 100: 134 -> 99 us a step).  Larger ones
  // differ in length and share H's rows, so the pairs take turns.
  const bool in_row = in[co[0].q].n <= 256;

  // ---- the degree steps, captured into one graph ----
  CHASE_TRY(rns ? rns_grouped_ready() : zgemm_grouped_fp64_prepare(cfg));
  const double tg = now_s();
  GraphGuard gg;
  CHASE_CUDA(cudaStreamCreateWithFlags(&gg.cs, cudaStreamNonBlocking));
  std::vector<cudaEvent_t> pev;  // product start / end per step, inside the graph
  for (int i = 1; i <= maxdeg; ++i) {
    if (tot[i].tiles == 0) continue;
    cudaEvent_t a = evp.get(), z = evp.get();
    if (!a || !z) {
      set_error("grouped filter: event creation failed");
      return CHASE_CUDA_ERROR;
    }
    pev.push_back(a);
    pev.push_back(z);
  }
  cudaEvent_t g_begin = evp.get(), g_end = evp.get();
  if (!g_begin || !g_end) {
    set_error("grouped filter: event creation failed");
    return CHASE_CUDA_ERROR;
  }
  {
    cudaStream_t user = d.st;
    d.st = gg.cs;
    int st = CHASE_OK;
    if (cudaStreamBeginCapture(gg.cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      d.st = user;
      set_error("grouped filter: stream capture failed to start");
      return CHASE_CUDA_ERROR;
    }
    size_t k = 0;
    for (int i = 1; i <= maxdeg && st == CHASE_OK; ++i) {
      if (tot[i].tiles == 0) continue;
      const int parity = (i - 1) & 1;
      const GroupedStep* sp = dsteps + first[i];
      if (rns) st = rns_grouped_slice_x(d, nmod, dprobs, sp, nact[i], tot[i].cols, parity);
      if (st != CHASE_OK) break;
      // external records: real event nodes of the graph, so the product
      // launches can be timed apart from the slicing
      if (cudaEventRecordWithFlags(pev[k], gg.cs, cudaEventRecordExternal) != cudaSuccess)
        st = CHASE_CUDA_ERROR;
      if (st == CHASE_OK)
        st = rns ? rns_grouped_gemm(d, nmod, width[i], dprobs, sp, nact[i], tot[i].tiles, in_row)
                 : zgemm_grouped_fp64(d, cfg, dprobs, sp, nact[i], tot[i].tiles, parity);
      if (st == CHASE_OK &&
          cudaEventRecordWithFlags(pev[k + 1], gg.cs, cudaEventRecordExternal) != cudaSuccess)
        st = CHASE_CUDA_ERROR;
      if (st == CHASE_OK && rns)
        st = rns_grouped_crt(d, nmod, dprobs, sp, nact[i], tot[i].blocks, parity);
      k += 2;
    }
    const cudaError_t ec = cudaStreamEndCapture(gg.cs, &gg.g);
    d.st = user;
    if (st != CHASE_OK) return st;
    if (ec != cudaSuccess || !gg.g) {
      set_error("grouped filter: stream capture failed: %s", cudaGetErrorString(ec));
      return CHASE_CUDA_ERROR;
    }
  }
  CHASE_CUDA(cudaGraphInstantiate(&gg.x, gg.g, 0));
  tt.t_graph_build = now_s() - tg;
  CHASE_CUDA(cudaEventRecord(g_begin, d.st));
  CHASE_CUDA(cudaGraphLaunch(gg.x, d.st));
  CHASE_CUDA(cudaEventRecord(g_end, d.st));
  CHASE_TRY(d.sync_check("grouped filter"));
  // With even degrees the last product of every column lands in X.
  for (const Coef& c : co) {
    const GroupedFilterInput& pi = in[c.q];
    for (int i = 1; i <= pi.maxdeg; ++i) {
      const int a = pi.b - pi.start[i];
      tt.matvecs += a;
      tt.flops += 8.0 * pi.n * static_cast<double>(pi.n) * a;
    }
  }
  for (size_t k = 0; k < pev.size(); k += 2) tt.t_product += 1e-3 * elapsed_ms(pev[k], pev[k + 1]);
  tt.t_steps = 1e-3 * elapsed_ms(g_begin, g_end);
  cudaGetLastError();  // a timing query that failed leaves no error behind
  tt.tile_config = cfg;
  tt.steps = maxdeg;
  tt.launches = static_cast<int>(chase_kernel_launches() - launches0);
  if (times) *times = tt;
  return CHASE_OK;
}

void add_times(GroupedFilterTimes& to, const GroupedFilterTimes& t) {
  to.tile_config = t.tile_config;
  to.steps = std::max(to.steps, t.steps);
  to.launches += t.launches;
  to.matvecs += t.matvecs;
  to.flops += t.flops;
  to.t_autotune += t.t_autotune;
  to.t_graph_build += t.t_graph_build;
  to.t_steps += t.t_steps;
  to.t_product += t.t_product;
}

// What filter_part allocates for `in` (maps, problems, step lists).
size_t list_bytes(const std::vector<GroupedFilterInput>& in) {
  size_t bytes = size_t(1) << 20;
  for (const GroupedFilterInput& g : in)
    bytes += 9 * sizeof(CUtensorMap) + sizeof(GroupedProblem) + (g.maxdeg + 1) * 2 * sizeof(GroupedStep);
  return bytes;
}

// Residue planes for `in`, made and given back here; halves of the batch in
// turn where they do not all fit (filter_part runs out of memory only before it
// touches a block), and FP64 tiles for a problem whose own do not.
int filter_parts(Dev& d, std::vector<GroupedFilterInput> in, int nmod, int tile,
                 GroupedFilterTimes& times) {
  std::vector<int> bcap;
  for (const GroupedFilterInput& g : in) bcap.push_back(g.b);
  GroupedFilterTimes t;
  GroupedWork w;
  int st = grouped_rns_prepare(d, in, bcap, nmod, list_bytes(in), w);
  if (st == CHASE_OK) {
    st = filter_part(d, in, nmod, tile, &t);
    grouped_rns_release(d, in, w);
  }
  if (st == CHASE_OUT_OF_MEMORY) {
    if (in.size() > 1) {
      const auto mid = in.begin() + static_cast<std::ptrdiff_t>(in.size() / 2);
      CHASE_TRY(filter_parts(d, std::vector<GroupedFilterInput>(in.begin(), mid), nmod, tile, times));
      return filter_parts(d, std::vector<GroupedFilterInput>(mid, in.end()), nmod, tile, times);
    }
    t = GroupedFilterTimes{};
    st = filter_part(d, in, 0, CHASE_TILE_AUTO, &t);
  }
  if (st == CHASE_OK) add_times(times, t);
  return st;
}
}  // namespace

int grouped_filter_sorted(Dev& d, const std::vector<GroupedFilterInput>& in, int nmod, int tile,
                          GroupedFilterTimes* times) {
  bool ready = true;
  for (const GroupedFilterInput& g : in) ready = ready && (g.n == 0 || g.b == 0 || g.A);
  if (nmod == 0 || ready) return filter_part(d, in, nmod, tile, times);
  GroupedFilterTimes t;
  CHASE_TRY(filter_parts(d, in, nmod, tile, t));
  if (times) *times = t;
  return CHASE_OK;
}

}  // namespace chase

using namespace chase;

extern "C" int chase_filter_batched(int P, const chase_c64* const* H, const int64_t* N,
                                    const int64_t* ldh, chase_c64* const* V, const int64_t* ldv,
                                    const int* b, const int* const* degrees, const double* b_sup,
                                    const double* mu1, const double* mu_nevnex, int precision,
                                    int tile, chase_batch_stats* stats, void* stream) {
  const double t0 = now_s();
  const long long launches0 = chase_kernel_launches();
  if (stats) *stats = chase_batch_stats{};
  if (precision != CHASE_FP64 && precision != CHASE_SPLIT_BF16) {
    set_error("chase_filter_batched: unknown precision %d", precision);
    return CHASE_INVALID_ARG;
  }
  if (tile < CHASE_TILE_AUTO || tile >= kGroupedFp64Cfgs) {
    set_error("chase_filter_batched: tile must be CHASE_TILE_AUTO or 0..%d", kGroupedFp64Cfgs - 1);
    return CHASE_INVALID_ARG;
  }
  if (P < 0 || (P > 0 && (!H || !N || !ldh || !V || !ldv || !b || !degrees || !b_sup || !mu1 ||
                          !mu_nevnex))) {
    set_error("chase_filter_batched: invalid problem count or NULL array");
    return CHASE_INVALID_ARG;
  }
  // ---- validation and the column order of every problem ----
  std::vector<int> idx;                    // caller's index of each problem with work
  std::vector<std::vector<int>> perm, start;
  for (int p = 0; p < P; ++p) {
    const int64_t n = N[p];
    if (n < 0 || b[p] < 0 || n > (1 << 20) || ldh[p] < std::max<int64_t>(1, n) ||
        ldv[p] < std::max<int64_t>(1, n)) {
      set_error("chase_filter_batched: problem %d: invalid size or leading dimension", p);
      return CHASE_INVALID_ARG;
    }
    if (n == 0 || b[p] == 0) continue;
    if (!H[p] || !V[p] || !degrees[p]) {
      set_error("chase_filter_batched: problem %d: NULL array", p);
      return CHASE_INVALID_ARG;
    }
    if (!is_device_ptr(H[p]) || !is_device_ptr(V[p])) {
      set_error("chase_filter_batched: problem %d: H and V must be device arrays", p);
      return CHASE_INVALID_ARG;
    }
    if (!(mu1[p] < mu_nevnex[p] && mu_nevnex[p] < b_sup[p]) || !std::isfinite(b_sup[p]) ||
        !std::isfinite(mu1[p])) {
      set_error("chase_filter_batched: problem %d: need mu1 < mu_nevnex < b_sup", p);
      return CHASE_INVALID_ARG;
    }
    const int* deg = degrees[p];
    int mx = 0;
    for (int j = 0; j < b[p]; ++j) {
      const int m = deg[j];
      if (m < 2 || m > kMaxDegree || (m & 1)) {
        set_error("chase_filter_batched: problem %d column %d: degree %d not even in [2, %d]", p, j,
                  m, kMaxDegree);
        return CHASE_INVALID_ARG;
      }
      mx = std::max(mx, m);
    }
    std::vector<int> pm(b[p]);
    std::iota(pm.begin(), pm.end(), 0);
    std::stable_sort(pm.begin(), pm.end(), [&](int x, int y) { return deg[x] < deg[y]; });
    std::vector<int> st(mx + 2, 0);  // Alg. 4 lines 12-14: columns of degree < i
    int s = 0;
    for (int i = 0; i <= mx + 1; ++i) {
      while (s < b[p] && deg[pm[s]] < i) ++s;
      st[i] = s;
    }
    idx.push_back(p);
    perm.push_back(std::move(pm));
    start.push_back(std::move(st));
  }
  const int Q = static_cast<int>(idx.size());
  if (Q == 0) return CHASE_OK;
  const bool split = precision == CHASE_SPLIT_BF16;

  Dev d(stream);
  CHASE_TRY(d.init());
  // sorted copies of the blocks (the filter's X), V is the second buffer
  std::vector<size_t> off0(Q);
  size_t tot0 = 0, totperm = 0;
  for (int q = 0; q < Q; ++q) {
    off0[q] = tot0;
    tot0 += (static_cast<size_t>(N[idx[q]]) * b[idx[q]] + 15) / 16 * 16;  // 256-byte aligned
    totperm += b[idx[q]];
  }
  chase_c64* buf0 = nullptr;
  int* dperm = nullptr;
  GroupedPermute* dgather = nullptr;
  GroupedPermute* dscatter = nullptr;
  CHASE_TRY(d.alloc(&buf0, tot0));
  CHASE_TRY(d.alloc(&dperm, totperm));
  CHASE_TRY(d.alloc(&dgather, Q));
  CHASE_TRY(d.alloc(&dscatter, Q));
  std::vector<int> hperm;
  hperm.reserve(totperm);
  std::vector<GroupedPermute> gat(Q), sca(Q);
  std::vector<GroupedFilterInput> in(Q);
  int total_cols = 0;
  for (int q = 0; q < Q; ++q) {
    const int p = idx[q];
    GroupedPermute& g = gat[q];
    g.src = reinterpret_cast<const double2*>(V[p]);
    g.lds = ldv[p];
    g.dst = reinterpret_cast<double2*>(buf0 + off0[q]);
    g.ldd = N[p];
    g.perm = dperm + hperm.size();
    g.n = static_cast<int>(N[p]);
    g.col0 = total_cols;
    GroupedPermute& h = sca[q];
    h = g;
    h.src = g.dst;
    h.lds = g.ldd;
    h.dst = reinterpret_cast<double2*>(V[p]);
    h.ldd = ldv[p];
    total_cols += b[p];
    hperm.insert(hperm.end(), perm[q].begin(), perm[q].end());
    GroupedFilterInput& f = in[q];
    f.H = H[p];
    f.ldh = ldh[p];
    f.n = static_cast<int>(N[p]);
    f.X = buf0 + off0[q];
    f.ldx = N[p];
    f.W = V[p];
    f.ldw = ldv[p];
    f.b = b[p];
    f.start = start[q].data();
    f.maxdeg = static_cast<int>(start[q].size()) - 2;
    f.b_sup = b_sup[p];
    f.mu1 = mu1[p];
    f.mu_nn = mu_nevnex[p];
  }
  CHASE_CUDA(cudaMemcpyAsync(dperm, hperm.data(), sizeof(int) * hperm.size(), cudaMemcpyHostToDevice,
                             d.st));
  CHASE_CUDA(cudaMemcpyAsync(dgather, gat.data(), sizeof(GroupedPermute) * Q, cudaMemcpyHostToDevice,
                             d.st));
  CHASE_CUDA(cudaMemcpyAsync(dscatter, sca.data(), sizeof(GroupedPermute) * Q,
                             cudaMemcpyHostToDevice, d.st));
  CHASE_TRY(launch_grouped_permute(d, dgather, Q, total_cols, false));
  GroupedFilterTimes tt;
  CHASE_TRY(grouped_filter_sorted(d, in, grouped_moduli(in, split, tile), split ? CHASE_TILE_AUTO : tile, &tt));
  // every result is in the sorted copy (even degrees): back to the caller's order
  CHASE_TRY(launch_grouped_permute(d, dscatter, Q, total_cols, true));
  CHASE_TRY(d.sync_check("chase_filter_batched"));
  if (stats) {
    stats->problems = Q;
    stats->steps = tt.steps;
    stats->tile_config = tt.tile_config;
    stats->launches = static_cast<int>(chase_kernel_launches() - launches0);
    stats->matvecs = tt.matvecs;
    stats->flops = tt.flops;
    stats->t_autotune = tt.t_autotune;
    stats->t_graph_build = tt.t_graph_build;
    stats->t_steps = tt.t_steps;
    stats->t_product = tt.t_product;
    stats->t_total = now_s() - t0;
  }
  return CHASE_OK;
}
