// C ABI, argument checking, plans and orchestration of the GB300 SARABANDE path.
//
// Per measured field (Sec. 3, Fig. workflow):
//   delta (FP64 mean, FP32 data) -> delta-hat = FFT(delta)
//   for each (l, m >= 0) [3D] or m >= 0 [2D]: kernel spectra G^b (Algorithms 1-2,
//     cached in the plan like the paper's saved kernels) -> a^b = IFFT(delta-hat G^b)
//     (Algorithms 3-4), product fused into the first inverse pass
//   3PCF: delta-weighted Gram of each group (Algorithms 5, 7)
//   4PCF: pair x single contraction over x (Algorithms 6, 8) + FP64 couplings.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <queue>
#include <set>
#include <string>
#include <system_error>
#include <thread>
#include <tuple>
#include <unordered_map>
#include <vector>

#include "sarabande_gb300.h"
#include "sbg_host.h"
#include "sbg_kernels.cuh"

using namespace sbg;

namespace {

constexpr int kMaxBins = 20;
constexpr int kMaxL3 = 10;
constexpr int kMaxL4 = 5;
constexpr int kMaxM = 10;
constexpr int kStages = 7;

struct DevBuf {
  void* p = nullptr;
  size_t bytes = 0;
};

// ---------------------------------------------------------------- 3j (host) --
// Racah's closed form for the Wigner 3j symbol in long double (l <= 10 here).
long double lfact(int n) {
  long double f = 1.0L;
  for (int i = 2; i <= n; ++i) f *= i;
  return f;
}

double three_j(int j1, int j2, int j3, int m1, int m2, int m3) {
  if (m1 + m2 + m3 != 0) return 0.0;
  if (j3 < std::abs(j1 - j2) || j3 > j1 + j2) return 0.0;
  if (std::abs(m1) > j1 || std::abs(m2) > j2 || std::abs(m3) > j3) return 0.0;
  const long double delta = lfact(j1 + j2 - j3) * lfact(j1 - j2 + j3) * lfact(-j1 + j2 + j3) / lfact(j1 + j2 + j3 + 1);
  const long double pref = std::sqrt(delta * lfact(j1 + m1) * lfact(j1 - m1) * lfact(j2 + m2) * lfact(j2 - m2) *
                                     lfact(j3 + m3) * lfact(j3 - m3));
  const int kmin = std::max(0, std::max(j2 - j3 - m1, j1 - j3 + m2));
  const int kmax = std::min(j1 + j2 - j3, std::min(j1 - m1, j2 + m2));
  long double s = 0.0L;
  for (int k = kmin; k <= kmax; ++k) {
    const long double den = lfact(k) * lfact(j1 + j2 - j3 - k) * lfact(j1 - m1 - k) * lfact(j2 + m2 - k) *
                            lfact(j3 - j2 + m1 + k) * lfact(j3 - j1 - m2 + k);
    s += ((k & 1) ? -1.0L : 1.0L) / den;
  }
  const int ph = j1 - j2 - m3;
  return (double)(((ph % 2) ? -1.0L : 1.0L) * pref * s);
}

// ------------------------------------------------------------ geometry ----
bool pow2_in(int64_t n, int64_t lo, int64_t hi) { return n >= lo && n <= hi && (n & (n - 1)) == 0; }

std::vector<double> snap_e2(const double* edges, int nb) {
  std::vector<double> e2(nb + 1);
  for (int i = 0; i <= nb; ++i) {
    double v = edges[i] * edges[i];
    double r = std::nearbyint(v);
    if (std::fabs(v - r) <= 1e-9 * std::max(v, 1.0)) v = r;
    e2[i] = v;
  }
  return e2;
}

std::vector<double> cell_counts(int n, int dim, const std::vector<double>& e2, int nb) {
  std::vector<double> c(nb, 0.0);
  // edges[nbins] < N/2, so every binned offset has |component| < N/2 and is a
  // distinct cell of the periodic grid
  const int R = (int)std::ceil(std::sqrt(e2[nb])) + 1;
  const int rz = dim == 3 ? R : 0;
  for (int z = -rz; z <= rz; ++z)
    for (int y = -R; y <= R; ++y)
      for (int x = -R; x <= R; ++x) {
        const double r2 = (double)x * x + (double)y * y + (double)z * z;
        if (!(r2 > e2[0]) || r2 > e2[nb]) continue;
        int b = 0;
        while (b < nb - 1 && r2 > e2[b + 1]) ++b;
        c[b] += 1.0;
      }
  return c;
}

double ylm_norm(int l, int m) {
  long double r = (2.0L * l + 1.0L) / (4.0L * 3.14159265358979323846264338327950288L);
  for (int k = l - m + 1; k <= l + m; ++k) r /= k;
  return (double)std::sqrt(r);
}

std::vector<float2> twiddles(int n) {
  std::vector<float2> t(n);
  for (int j = 0; j < n; ++j) {
    const double a = 2.0 * 3.14159265358979323846 * j / n;
    t[j] = make_float2((float)std::cos(a), (float)std::sin(a));
  }
  return t;
}

// ---------------------------------------------------------- 4PCF tables ----
struct Single { int l, m, b; };

struct Tables4 {
  // host
  std::vector<Tile4> tiles;     // FP32: in the order of the plan's two launches
  SimtPlan simt{};              // FP32 tiles
  std::vector<Row4> rows;
  std::vector<int> cols, uniq;
  std::vector<BGroup> bgroups;  // tensor-core tiles: column groups and their B images
  long long img_stride = 0;     // bytes of B images per K-block
  int chunks_per_kb = 0;
  std::vector<int> ptr, idx;
  std::vector<double> coef;
  long long tcount = 0;  // outputs of T (complex counted once)
  bool tc = false;       // tiles built for the tensor-core kernel
  int covering = 0;      // 0: bin-half (tensor) or b3 >= b2 (SIMT) rows; 1: greedy cover
  int nout = 0;
  // device
  DevBuf d_tiles, d_rows, d_cols, d_uniq, d_bgroups, d_ptr, d_idx, d_coef;
};

}  // namespace

struct sbg_context {
  int device = 0;
  int nsm = 148;
  cudaStream_t own = nullptr;
  cudaStream_t stream = nullptr;
  size_t budget = 0, used = 0;
  std::string err;
  // bound of every wait inside the tensor-core kernel, and the test switch that
  // withholds its MMA issuer (sbg_set_wait_limit)
  unsigned long long wait_ns = 1000000000ull;
  int stall = 0;
  double timings[kStages] = {0};
  long long nlaunch = 0;   // kernels launched by the current/last measurement call
  long long last_launches = 0;
  // two sets of timing events: a batch keeps one field in flight while the
  // previous one is completed; ev / kev point at the set of the current call
  cudaEvent_t evs[2][kStages + 1] = {};
  cudaEvent_t kevs[2][2] = {};
  cudaEvent_t* ev = evs[0];
  cudaEvent_t* kev = kevs[0];   // around the 4PCF contraction kernel(s)
  bool kev_used = false;
  double contraction_ms = 0.0;
  std::map<std::string, DevBuf> bufs;
  // full-plan cache
  std::string gkey;
  DevBuf gcache;
  bool gcached = false;
  // projected kernel spectra of the last few slab geometries, most recently
  // used first (a batch of uneven sizes alternates between them)
  static constexpr int kG2Cache = 4;
  std::vector<std::pair<std::string, DevBuf>> g2cache;
  // 4PCF tables of the last few geometries (dim, bins, order, kernel, parity),
  // so that calls alternating between them (e.g. sbg_full and sbg_full_odd on
  // each field) do not rebuild a plan per call; t4 is the current one
  static constexpr int kT4Cache = 4;
  std::vector<std::pair<std::string, Tables4*>> t4cache;  // most recently used first
  Tables4* t4 = nullptr;
  // pinned host staging for results and status words, so downloads are plain
  // DMA on the stream and the host copies out after the stream is idle
  void* hpin = nullptr;
  size_t hpin_bytes = 0;
  // batch pipelining: with `defer` set, a measurement call stages its results
  // in pinned slot `cur` and returns without waiting; the batch loop completes
  // it after the next field has been queued
  struct Pending {
    bool live = false;
    double* zeta3 = nullptr;
    double* zeta4 = nullptr;
    size_t off3 = 0, off4 = 0, b3 = 0, b4 = 0;
    long long launches = 0;
    bool kev_used = false;
  };
  bool defer = false;
  int cur = 0;
  // host tables that the device already holds (see Tables): what the transform
  // table in buffer "xf" was made for, the sides whose twiddles are uploaded, the
  // squared edges, and the support lines of (side, outermost squared edge)
  std::string xf_key;
  std::set<int> tw_sides;
  std::vector<double> e2_up;
  std::pair<int, double> lines_key{0, 0.0};
  int nlines = 0, rsup = 0;
  // autotuner: launch choices measured on their first use, by key
  std::map<std::string, int> tune;
  cudaEvent_t tev[2] = {};
  bool autotune_on = true;
  size_t slot_bytes = 0;
  Pending pend[2];
};

namespace {

sbg_status fail(sbg_context* c, sbg_status s, const std::string& msg) {
  if (c) c->err = msg;
  return s;
}

#define CU(call)                                                                                 \
  do {                                                                                           \
    cudaError_t e_ = (call);                                                                     \
    if (e_ != cudaSuccess)                                                                       \
      return fail(ctx, SBG_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));        \
  } while (0)

#define KL(call)        \
  do {                  \
    ++ctx->nlaunch;     \
    CU(call);           \
  } while (0)

#define ST(call)                       \
  do {                                 \
    sbg_status s_ = (call);            \
    if (s_ != SBG_OK) return s_;       \
  } while (0)

sbg_status dev_alloc(sbg_context* ctx, DevBuf& b, size_t bytes) {
  if (b.p && b.bytes >= bytes) return SBG_OK;
  if (b.p) {
    cudaFree(b.p);
    ctx->used -= b.bytes;
    b.p = nullptr;
    b.bytes = 0;
  }
  if (bytes == 0) return SBG_OK;
  if (ctx->budget && ctx->used + bytes > ctx->budget)
    return fail(ctx, SBG_ERR_OUT_OF_MEMORY, "allocation of " + std::to_string(bytes) + " bytes exceeds the budget");
  cudaError_t e = cudaMalloc(&b.p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    b.p = nullptr;
    return fail(ctx, SBG_ERR_OUT_OF_MEMORY, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  }
  b.bytes = bytes;
  ctx->used += bytes;
  return SBG_OK;
}

void dev_free(sbg_context* ctx, DevBuf& b) {
  if (b.p) {
    cudaFree(b.p);
    ctx->used -= b.bytes;
  }
  b.p = nullptr;
  b.bytes = 0;
}

sbg_status buf(sbg_context* ctx, const char* name, size_t bytes, void** out) {
  DevBuf& b = ctx->bufs[name];
  ST(dev_alloc(ctx, b, bytes));
  *out = b.p;
  return SBG_OK;
}

template <class T>
sbg_status upload(sbg_context* ctx, DevBuf& b, const std::vector<T>& v) {
  ST(dev_alloc(ctx, b, std::max<size_t>(v.size() * sizeof(T), 16)));
  if (!v.empty()) CU(cudaMemcpyAsync(b.p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, ctx->stream));
  return SBG_OK;
}

// Angular part of a single: 3D (l, m), 2D (m) with l = -1.
int store_index(int dim, int nb, int l, int m_abs, int b) {
  return dim == 3 ? ((l * (l + 1) / 2 + m_abs) * nb + b) : (m_abs * nb + b);
}

// Shared-memory slots of the staged row singles of one tensor-core tile.  A
// quarter-warp of producer threads (8 consecutive rows) reads the same 16-byte
// chunk of the first single of each of its rows, then of the second; the raw
// stage pads each slot's 256-byte row to 272 bytes, so chunk k of slot s lies in
// bank quad (s + k) mod 8 and two distinct singles read together collide in a
// bank only when their slots agree mod 8 (their colour).  Colours are chosen greedily, singles shared by
// the most quarter-warp groups first, best of a few tie-breaking orders; colour
// c owns slots c, c + 8, ...  Unused slots hold -1 (not loaded).
sbg_status colour_slots(sbg_context* ctx, Tables4& t, Tile4& tl, const std::map<int, int>& local) {
  const int nl = (int)local.size();
  const int cap = kTcMaxRowSlots / 8;
  std::vector<int> store(nl);
  for (const auto& kv : local) store[kv.second] = kv.first;
  std::vector<std::vector<int>> groups;       // distinct local singles per (quarter-warp, operand)
  std::vector<std::vector<int>> member(nl);   // groups containing each single
  for (int q = 0; q < tl.nrows; q += 8)
    for (int k = 0; k < 2; ++k) {
      std::vector<int> g;
      for (int r = q; r < std::min(q + 8, tl.nrows); ++r) {
        const Row4& rw = t.rows[tl.row0 + r];
        const int u = k ? rw.u2 : rw.u1;
        if (std::find(g.begin(), g.end(), u) == g.end()) g.push_back(u);
      }
      for (int u : g) member[u].push_back((int)groups.size());
      groups.push_back(std::move(g));
    }
  std::vector<int> base(nl);
  for (int i = 0; i < nl; ++i) base[i] = i;
  std::stable_sort(base.begin(), base.end(), [&](int a, int b) { return member[a].size() > member[b].size(); });
  std::vector<int> best_col;
  long long best_cost = LLONG_MAX;
  uint32_t rng = 12345u;
  for (int trial = 0; trial < 16; ++trial) {
    std::vector<int> col(nl, -1), left(8, cap), tie(nl);
    for (int i = 0; i < nl; ++i) {
      rng = rng * 1664525u + 1013904223u;
      tie[i] = (int)(rng >> 8);
    }
    for (int u : base) {
      int score[8] = {0};
      for (int gi : member[u])
        for (int o : groups[gi])
          if (col[o] >= 0) ++score[col[o]];
      int pick = -1;
      for (int c = 0; c < 8; ++c) {
        const int cc = (c + tie[u]) & 7;  // rotate the tie-break per single and trial
        if (!left[cc]) continue;
        if (pick < 0 || score[cc] < score[pick]) pick = cc;
      }
      if (pick < 0)
        for (int c = 0; c < 8; ++c)
          if (left[c]) { pick = c; break; }
      col[u] = pick;
      --left[pick];
    }
    long long cost = 0;
    for (const auto& g : groups) {
      int cnt[8] = {0}, mx = 0;
      for (int u : g) mx = std::max(mx, ++cnt[col[u]]);
      cost += mx;
    }
    if (cost < best_cost) {
      best_cost = cost;
      best_col = col;
    }
  }
  std::vector<int> slot(nl), used(8, 0);
  int nslot = 0;
  for (int u = 0; u < nl; ++u) {
    slot[u] = best_col[u] + 8 * used[best_col[u]]++;
    nslot = std::max(nslot, slot[u] + 1);
  }
  if (nslot > kTcMaxRowSlots) return fail(ctx, SBG_ERR_INTERNAL, "4PCF tiling: slot colouring overflow");
  for (int r = tl.row0; r < tl.row0 + tl.nrows; ++r) {
    t.rows[r].u1 = slot[t.rows[r].u1];
    t.rows[r].u2 = slot[t.rows[r].u2];
  }
  std::vector<int> slots(nslot, -1);
  for (int u = 0; u < nl; ++u) slots[slot[u]] = store[u];
  tl.nuniq = nslot;
  for (int v : slots) t.uniq.push_back(v);
  return SBG_OK;
}

// Build the pair x single contraction tables of the 4PCF and the coupling CSR.
// T[s1, s2, s3] = sum_x delta a_s1 a_s2 a_s3 is symmetric under permutations of
// its singles s = (l, m, b) and T[-M] = conj T[M] (real delta), so a computed
// entry (pair row, column single) serves every ordering of its triple and the
// triple with all m negated (Re T unchanged; conj for the complex 2D T).  The
// coupling CSR finds each needed triple by trying its orderings and signs.
//   tc = false: FP32 SIMT tiles; for each m3 >= 0 and bin b2, rows (alpha1,
//               b1 <= b2, alpha2) with m1 + m2 = -m3 and cols (b3 >= b2,
//               l3 >= m3), or the greedy cover below when it computes fewer
//               entries; of each row the l3 that the couplings take; tiles as
//               simt_geometry() has them, <= 128 staged singles each.
//   tc = true : tensor-core tiles of 128 rows (M of the MMA), <= kTcMaxRowSlots
//               staged singles, <= 64 B-operand rows (2D: 2 per column single);
//               one block per m3 >= 0 with columns (b3, l3 >= m3).
sbg_status build_tables4(sbg_context* ctx, Tables4& t, int dim, int nb, int L, bool tc, bool odd = false,
                         bool to_device = true) {
  // complex T for the projected 4PCF; the odd-parity 3D 4PCF (whose M-sum is
  // imaginary, Eq. mu with E(Lambda) = -1) keeps one real entry per (row,
  // column), the imaginary part, and single-column B operands of the form
  // (Im v, Re v)
  const bool cplx = dim == 2;
  struct Ang { int l, m; };
  std::vector<Ang> angs;
  if (dim == 3) {
    for (int l = 0; l <= L; ++l)
      for (int m = -l; m <= l; ++m) angs.push_back({l, m});
  } else {
    for (int m = -L; m <= L; ++m) angs.push_back({-1, m});
  }
  const int na = (int)angs.size();
  // position in angs: 3D l^2 + l + m, 2D m + L; -1 if there is none
  auto ang_index = [&](int l, int m) -> int {
    if (dim == 3) return (l < 0 || l > L || std::abs(m) > l) ? -1 : l * l + l + m;
    return (l != -1 || std::abs(m) > L) ? -1 : m + L;
  };
  // Two ways of choosing the formed pairs (rows) so that every canonical triple
  // has one of its pairs among the rows and its third single among the columns:
  //  tc = false (SIMT): bins sorted b1 <= b2 <= b3; rows (alpha1, b1 <= b2, alpha2),
  //                     columns (b3 >= b2, l3) -> one block per (m3, b2);
  //  tc = true (tensor): bins split in two halves; rows are pairs within one half
  //                     (any triple has two bins in the same half), columns are
  //                     every (b3, l3) -> one block per m3 with uniform columns;
  //                     the greedy cover below replaces these rows when it packs
  //                     into fewer tiles.
  auto half = [&](int b) { return b < (nb + 1) / 2 ? 0 : 1; };
  struct RowKey { int a1, b1, a2, b2; };
  struct Block {
    int m3 = 0, b2 = 0;
    std::vector<RowKey> rows;
    std::unordered_map<long long, int> row_of;
    std::vector<int> l3s;
    int ncols = 0, bcol0 = 0;  // columns: b3 in [bcol0, nb) x l3s, b3-major
    long long first = 0;                    // entry (row, column) is number first + row ncols + column of the plan's
    std::vector<float> sign;                // [row]
    std::vector<unsigned> used;             // [row] bit i: the output takes entries of column l3s[i]
  };
  auto rkey = [](int a1, int b1, int a2, int b2) -> long long {
    return (((long long)a1 * 64 + b1) * 4096 + a2) * 64 + b2;
  };
  std::vector<Block> blocks;
  bool uniform = tc;  // one block per m3 >= 0 whose columns are every (b3, l3)
  auto block_of = [&](int m3, int b2) -> int { return uniform ? m3 : m3 * nb + b2; };
  for (int m3 = 0; m3 <= L; ++m3)
    for (int b2 = 0; b2 < (tc ? 1 : nb); ++b2) {
      Block bk;
      bk.m3 = m3;
      bk.b2 = b2;
      if (dim == 3) {
        for (int l3 = m3; l3 <= L; ++l3) bk.l3s.push_back(l3);
      } else {
        bk.l3s.push_back(-1);
      }
      if (!tc) {
        bk.bcol0 = b2;
        // rows ordered (alpha1, b1, alpha2): rows sharing alpha1 share their staged singles
        for (int a1 = 0; a1 < na; ++a1)
          for (int b1 = 0; b1 <= b2; ++b1)
            for (int a2 = 0; a2 < na; ++a2)
              if (angs[a1].m + angs[a2].m == -m3) bk.rows.push_back({a1, b1, a2, b2});
      } else {
        bk.bcol0 = 0;
        for (int b1 = 0; b1 < nb; ++b1)
          for (int bb = b1; bb < nb; ++bb) {
            if (half(b1) != half(bb)) continue;
            for (int a1 = 0; a1 < na; ++a1)
              for (int a2 = (bb == b1 ? a1 : 0); a2 < na; ++a2) {
                if (angs[a1].m + angs[a2].m != -m3) continue;
                if (m3 == 0) {
                  // the row with every m negated gives conj of this row's entries:
                  // keep one of the two (the lookup finds it through M -> -M)
                  int f1 = ang_index(angs[a1].l, -angs[a1].m), f2 = ang_index(angs[a2].l, -angs[a2].m);
                  if (bb == b1 && f2 < f1) std::swap(f1, f2);
                  if (f1 < a1 || (f1 == a1 && f2 < a2)) continue;
                }
                bk.rows.push_back({a1, b1, a2, bb});
              }
          }
      }
      bk.ncols = (nb - bk.bcol0) * (int)bk.l3s.size();
      blocks.push_back(std::move(bk));
    }
  const int col_chunk = tc ? (cplx ? 32 : 64) : 64;
  const int max_u = tc ? kTcMaxRowSlots : kSimtSpanUniq;
  auto sidx = [&](int a, int b) { return store_index(dim, nb, angs[a].l, std::abs(angs[a].m), b); };
  // tiles of at most `most` rows and max_u singles that a packing in order makes of a block's rows
  auto count_tiles = [&](const std::vector<RowKey>& rows, int most = 128) -> long long {
    long long n = 0;
    int nr = 0;
    std::vector<int> local;
    auto has = [&](int v) { return std::find(local.begin(), local.end(), v) != local.end(); };
    for (const RowKey& rk : rows) {
      const int s1 = sidx(rk.a1, rk.b1), s2 = sidx(rk.a2, rk.b2);
      const int need = (has(s1) ? 0 : 1) + ((has(s2) || s2 == s1) ? 0 : 1);
      if (nr == most || (int)local.size() + need > max_u) {  // the row opens the next tile
        ++n;
        nr = 0;
        local.clear();
      }
      if (!has(s1)) local.push_back(s1);
      if (!has(s2)) local.push_back(s2);
      ++nr;
    }
    return n + (nr ? 1 : 0);
  };
  {
    // Second covering: a greedy set cover of the triples the output needs, in
    // blocks of one m3 >= 0 with every (b3, l3) column.  A candidate row is a
    // pair (s1, s2) with m1 + m2 = -m3; it covers the triples (s1, s2, s3) for
    // every column s3 = (l3, m3, b3) of its block that the output needs (3D:
    // l1 + l2 + l3 even and |l1 - l2| <= l3 <= l1 + l2, the terms of the even-
    // parity 4PCF; 2D: every b3).  Triples are counted once up to the order of
    // their singles and M -> -M.  Any element of a triple may be its column and
    // rows that meet no needed column are left out.  The tensor-core kernel
    // pays per tile, so its greedy counts rows and the plan keeps the covering
    // with fewer tiles (at lmax 4, 10 bins: 30 instead of 65); the SIMT kernel
    // pays per (row, column) entry, so its greedy weighs a row by its block's
    // columns and the plan keeps the covering with fewer entries (134,320
    // instead of 239,360).
    std::vector<int> l3_of[kMaxL4 > kMaxM ? kMaxL4 + 1 : kMaxM + 1];
    for (int m3 = 0; m3 <= L; ++m3) {
      if (dim == 3) {
        for (int l3 = m3; l3 <= L; ++l3) l3_of[m3].push_back(l3);
      } else {
        l3_of[m3].push_back(-1);
      }
    }
    auto ucols = [&](int m3) { return nb * (int)l3_of[m3].size(); };
    std::vector<int> nega(na);
    for (int a = 0; a < na; ++a) nega[a] = ang_index(angs[a].l, -angs[a].m);
    const long long S = (long long)na * nb;
    auto key3 = [&](int x, int y, int z) -> long long {  // single s = a * nb + b
      int u[3] = {x, y, z}, v[3] = {nega[x / nb] * nb + x % nb, nega[y / nb] * nb + y % nb, nega[z / nb] * nb + z % nb};
      std::sort(u, u + 3);
      std::sort(v, v + 3);
      if (std::lexicographical_compare(v, v + 3, u, u + 3)) std::copy(v, v + 3, u);
      return ((long long)u[0] * S + u[1]) * S + u[2];
    };
    auto needed = [&](int l1, int l2, int l3) {
      return dim == 2 || (((l1 + l2 + l3) & 1) == (odd ? 1 : 0) && std::abs(l1 - l2) <= l3 && l3 <= l1 + l2);
    };
    auto canon = [](int a1, int b1, int a2, int b2) -> RowKey {  // b1 <= b2; a1 <= a2 when b1 == b2
      if (b1 > b2 || (b1 == b2 && a1 > a2)) return {a2, b2, a1, b1};
      return {a1, b1, a2, b2};
    };
    auto less = [](const RowKey& p, const RowKey& q) {
      return std::make_tuple(p.a1, p.b1, p.a2, p.b2) < std::make_tuple(q.a1, q.b1, q.a2, q.b2);
    };
    struct Cand { int m3; RowKey rk; int off, n; };
    std::vector<Cand> cands;
    std::vector<int> cov;
    std::unordered_map<long long, int> tid;
    for (int m3 = 0; m3 <= L; ++m3)
      for (int a1 = 0; a1 < na; ++a1)
        for (int b1 = 0; b1 < nb; ++b1)
          for (int a2 = 0; a2 < na; ++a2)
            for (int b2 = 0; b2 < nb; ++b2) {
              if (angs[a1].m + angs[a2].m != -m3) continue;
              const RowKey rk{a1, b1, a2, b2};
              const RowKey ck = canon(a1, b1, a2, b2);
              if (ck.a1 != a1 || ck.b1 != b1 || ck.a2 != a2 || ck.b2 != b2) continue;  // the other order
              // m3 = 0: the pair with every m negated covers the same triples
              if (m3 == 0 && less(canon(nega[a1], b1, nega[a2], b2), rk)) continue;
              const int off = (int)cov.size();
              for (int l3 : l3_of[m3]) {
                if (!needed(angs[a1].l, angs[a2].l, l3)) continue;
                const int z = ang_index(l3, m3) * nb;
                for (int b3 = 0; b3 < nb; ++b3) {
                  auto ins = tid.emplace(key3(a1 * nb + b1, a2 * nb + b2, z + b3), (int)tid.size());
                  cov.push_back(ins.first->second);
                }
              }
              std::sort(cov.begin() + off, cov.end());
              cov.erase(std::unique(cov.begin() + off, cov.end()), cov.end());
              if ((int)cov.size() > off) cands.push_back({m3, rk, off, (int)cov.size() - off});
            }
    // lazy greedy: take the candidate with the most uncovered triples (SIMT:
    // per column of its block, as if the tiles took all of them; they take the
    // l3 that are used, and forming a row costs about 10 columns more: see
    // simt_cost; ties: the first enumerated); a popped value that went stale
    // is pushed back
    auto value = [&](const Cand& c, int fresh) { return tc ? (double)fresh : (double)fresh / ucols(c.m3); };
    std::vector<char> done(tid.size(), 0);
    long long left = (long long)tid.size();
    std::priority_queue<std::pair<double, int>> heap;
    for (int i = 0; i < (int)cands.size(); ++i) heap.push({value(cands[i], cands[i].n), -i});
    std::vector<std::vector<RowKey>> grows(L + 1);
    std::vector<char> chosen(cands.size(), 0);
    while (left > 0 && !heap.empty()) {
      const auto top = heap.top();
      heap.pop();
      const Cand& c = cands[-top.second];
      int fresh = 0;
      for (int k = c.off; k < c.off + c.n; ++k) fresh += done[cov[k]] ? 0 : 1;
      if (fresh == 0) continue;
      if (value(c, fresh) < top.first) {
        heap.push({value(c, fresh), top.second});
        continue;
      }
      for (int k = c.off; k < c.off + c.n; ++k) done[cov[k]] = 1;
      left -= fresh;
      chosen[-top.second] = 1;
    }
    if (left > 0) return fail(ctx, SBG_ERR_INTERNAL, "4PCF greedy covering left triples uncovered");
    auto sort_rows = [&](std::vector<RowKey>& g) {
      // rows sharing singles sit together: sorted by the stored index of each single
      std::sort(g.begin(), g.end(), [&](const RowKey& p, const RowKey& q) {
        return std::make_pair(sidx(p.a1, p.b1), sidx(p.a2, p.b2)) < std::make_pair(sidx(q.a1, q.b1), sidx(q.a2, q.b2));
      });
    };
    auto block_rows = [&](int m3) {
      std::vector<RowKey> g;
      for (size_t i = 0; i < cands.size(); ++i)
        if (chosen[i] && cands[i].m3 == m3) g.push_back(cands[i].rk);
      sort_rows(g);
      return g;
    };
    if (tc) {
      // Tile trimming: the tensor-core kernel pays per 128-row tile, so a block
      // whose last tile holds few rows is worth emptying.  Rows of that block
      // are dropped while every triple that only they cover can be re-covered
      // by unchosen candidates of other blocks that stay within their tile
      // counts (the last triple of a row may go to any single as the column,
      // so coverage moves between blocks); the moves of one attempt are kept
      // only if the plan's tile count (with the staged-singles limit) drops.
      std::vector<int> tstart(tid.size() + 1, 0), tcand;
      for (const Cand& c : cands)
        for (int k = c.off; k < c.off + c.n; ++k) ++tstart[cov[k] + 1];
      for (size_t t = 0; t < tid.size(); ++t) tstart[t + 1] += tstart[t];
      tcand.resize(tstart.back());
      {
        std::vector<int> fill(tstart.begin(), tstart.end() - 1);
        for (int i = 0; i < (int)cands.size(); ++i)
          for (int k = cands[i].off; k < cands[i].off + cands[i].n; ++k) tcand[fill[cov[k]]++] = i;
      }
      std::vector<int> cnt(tid.size(), 0);  // chosen rows covering each triple
      std::vector<long long> nrow(L + 1, 0), tb(L + 1, 0);
      for (size_t i = 0; i < cands.size(); ++i)
        if (chosen[i]) {
          ++nrow[cands[i].m3];
          for (int k = cands[i].off; k < cands[i].off + cands[i].n; ++k) ++cnt[cov[k]];
        }
      for (int m3 = 0; m3 <= L; ++m3) tb[m3] = count_tiles(block_rows(m3));
      auto total = [&](const std::vector<long long>& v) {
        long long x = 0;
        for (long long y : v) x += y;
        return x;
      };
      for (int round = 0; round < 8; ++round) {
        bool improved = false;
        std::vector<int> order;
        for (int m3 = 0; m3 <= L; ++m3)
          if (tb[m3] > 0) order.push_back(m3);
        std::sort(order.begin(), order.end(), [&](int x, int y) {
          return nrow[x] - 128 * (tb[x] - 1) < nrow[y] - 128 * (tb[y] - 1);
        });
        for (int B : order) {
          const std::vector<char> chosen0 = chosen;
          const std::vector<int> cnt0 = cnt;
          const std::vector<long long> nrow0 = nrow;
          // rows of B, those covering the fewest triples alone first
          std::vector<std::pair<int, int>> inB;
          for (int i = 0; i < (int)cands.size(); ++i)
            if (chosen[i] && cands[i].m3 == B) {
              int alone = 0;
              for (int k = cands[i].off; k < cands[i].off + cands[i].n; ++k) alone += cnt[cov[k]] == 1;
              inB.push_back({alone, i});
            }
          std::sort(inB.begin(), inB.end());
          for (const auto& e : inB) {
            if (nrow[B] <= 128 * (tb[B] - 1)) break;
            const int c = e.second;
            const Cand& cc = cands[c];
            chosen[c] = 0;
            --nrow[B];
            for (int k = cc.off; k < cc.off + cc.n; ++k) --cnt[cov[k]];
            std::vector<int> added;
            bool ok = true;
            for (int k = cc.off; k < cc.off + cc.n && ok; ++k) {
              const int t0 = cov[k];
              if (cnt[t0] > 0) continue;
              // the unchosen candidate outside B (with room) covering the most
              // of c's still uncovered triples
              int best = -1, bestv = 0;
              for (int q = tstart[t0]; q < tstart[t0 + 1]; ++q) {
                const int c2 = tcand[q];
                const Cand& d = cands[c2];
                if (chosen[c2] || d.m3 == B || nrow[d.m3] >= 128 * std::max(tb[d.m3], 1LL)) continue;
                int v = 0;
                for (int k2 = d.off; k2 < d.off + d.n; ++k2) v += cnt[cov[k2]] == 0;
                if (v > bestv) {
                  bestv = v;
                  best = c2;
                }
              }
              if (best < 0) {
                ok = false;
                break;
              }
              chosen[best] = 1;
              ++nrow[cands[best].m3];
              for (int k2 = cands[best].off; k2 < cands[best].off + cands[best].n; ++k2) ++cnt[cov[k2]];
              added.push_back(best);
            }
            if (!ok) {  // undo this row's move
              for (int c2 : added) {
                chosen[c2] = 0;
                --nrow[cands[c2].m3];
                for (int k2 = cands[c2].off; k2 < cands[c2].off + cands[c2].n; ++k2) --cnt[cov[k2]];
              }
              chosen[c] = 1;
              ++nrow[B];
              for (int k = cc.off; k < cc.off + cc.n; ++k) ++cnt[cov[k]];
            }
          }
          std::vector<long long> tb2(L + 1, 0);
          for (int m3 = 0; m3 <= L; ++m3) tb2[m3] = count_tiles(block_rows(m3));
          if (total(tb2) < total(tb)) {
            tb = tb2;
            improved = true;
          } else {
            chosen = chosen0;
            cnt = cnt0;
            nrow = nrow0;
          }
        }
        if (!improved) break;
      }
    }
    for (int m3 = 0; m3 <= L; ++m3) grows[m3] = block_rows(m3);
    if (tc) {
      long long t_half = 0, t_greedy = 0;
      for (int m3 = 0; m3 <= L; ++m3) {
        t_half += count_tiles(blocks[m3].rows);
        t_greedy += count_tiles(grows[m3]);
      }
      if (t_greedy < t_half) {
        for (int m3 = 0; m3 <= L; ++m3) blocks[m3].rows = std::move(grows[m3]);
        t.covering = 1;
      }
    } else {
      long long e_cur = 0, e_greedy = 0;
      for (const Block& bk : blocks) e_cur += (long long)bk.rows.size() * bk.ncols;
      for (int m3 = 0; m3 <= L; ++m3) e_greedy += (long long)grows[m3].size() * ucols(m3);
      if (e_greedy < e_cur) {
        std::vector<Block> ub(L + 1);
        for (int m3 = 0; m3 <= L; ++m3) {
          ub[m3].m3 = m3;
          ub[m3].l3s = l3_of[m3];
          ub[m3].ncols = ucols(m3);
          ub[m3].rows = std::move(grows[m3]);
        }
        blocks = std::move(ub);
        uniform = true;
        t.covering = 1;
      }
    }
  }
  // The sign of a row's pair, a_{l,-m} = (-1)^m conj(a_lm) (3D): the kernels
  // leave it to the couplings
  auto row_sign = [&](const RowKey& k) {
    auto odd_negative = [&](int a) { return angs[a].m < 0 && (angs[a].m & 1); };
    return dim == 3 && odd_negative(k.a1) != odd_negative(k.a2) ? -1.0f : 1.0f;
  };
  long long nentries = 0;
  for (Block& bk : blocks) {
    bk.row_of.reserve(bk.rows.size() * 2);
    for (int r = 0; r < (int)bk.rows.size(); ++r) {
      const RowKey& k = bk.rows[r];
      bk.row_of[rkey(k.a1, k.b1, k.a2, k.b2)] = r;
    }
    bk.first = nentries;
    nentries += (long long)bk.rows.size() * bk.ncols;
    bk.used.assign(bk.rows.size(), 0u);
    bk.sign.reserve(bk.rows.size());
    for (const RowKey& k : bk.rows) bk.sign.push_back(row_sign(k));
  }
  // Entry of a triple of singles (any order, any sign of M): twice its number, plus
  // one if it is the conjugate's (all m negated); -1: none.  rowsign receives its
  // row's sign.
  auto find_entry = [&](const Single& x, const Single& y, const Single& z, bool neg, float* rowsign) -> long long {
    const int m3 = z.m;
    if (m3 < 0 || m3 > L) return -1;
    if (x.m + y.m != -m3) return -1;
    const int bi = block_of(m3, tc ? 0 : y.b);
    if (bi < 0 || bi >= (int)blocks.size()) return -1;
    Block& bk = blocks[bi];
    int i1 = ang_index(x.l, x.m), i2 = ang_index(y.l, y.m);
    int b1 = x.b, b2 = y.b;
    if (uniform && b1 == b2 && i2 < i1) std::swap(i1, i2);
    auto it = bk.row_of.find(rkey(i1, b1, i2, b2));
    if (it == bk.row_of.end()) return -1;
    const int row = it->second;
    if (z.b < bk.bcol0) return -1;
    const int l3pos = dim == 3 ? z.l - m3 : 0;
    const int col = (z.b - bk.bcol0) * (int)bk.l3s.size() + l3pos;
    if (col >= bk.ncols) return -1;
    bk.used[row] |= 1u << l3pos;
    if (rowsign) *rowsign = bk.sign[row];
    return 2 * (bk.first + (long long)row * bk.ncols + col) + neg;
  };
  auto lookup = [&](Single s[3], float* rowsign) -> long long {
    static const int perms[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
    for (int neg = 0; neg < 2; ++neg)
      for (const auto& p : perms) {
        Single x = s[p[0]], y = s[p[1]], z = s[p[2]];
        if (neg) { x.m = -x.m; y.m = -y.m; z.m = -z.m; }
        if (x.b > y.b) continue;
        if (!uniform && z.b < y.b) continue;
        const long long e = find_entry(x, y, z, neg != 0, rowsign);
        if (e >= 0) return e;
      }
    return -1;
  };

  // coupling CSR: one output per (Lambda, b1, b2, b3) [3D] or (m1, m2, b1, b2, b3) [2D]
  // (entries become T indices once the tiles are cut)
  std::vector<long long> entries;
  t.ptr.clear();
  t.idx.clear();
  t.coef.clear();
  t.ptr.push_back(0);
  if (dim == 3) {
    for (int l1 = 0; l1 <= L; ++l1)
      for (int l2 = 0; l2 <= L; ++l2)
        for (int l3 = std::abs(l1 - l2); l3 <= std::min(l1 + l2, L); ++l3) {
          if (((l1 + l2 + l3) & 1) != (odd ? 1 : 0)) continue;
          struct Term { int m1, m2; double c; };
          std::vector<Term> terms;  // the nonzero E(Lambda) C^Lambda_M of this Lambda
          for (int m1 = -l1; m1 <= l1; ++m1)
            for (int m2 = -l2; m2 <= l2; ++m2) {
              const int m3 = -(m1 + m2);
              if (std::abs(m3) > l3) continue;
              // E(Lambda) C^Lambda_M = (-1)^(l1+l2+l3) (3j), times E = -1 for odd Lambda
              const double c = (((l1 + l2 + l3) & 1) ? -1.0 : 1.0) * (odd ? -1.0 : 1.0) *
                               three_j(l1, l2, l3, m1, m2, m3);
              if (c != 0.0) terms.push_back({m1, m2, c});
            }
          for (int b1 = 0; b1 < nb; ++b1)
            for (int b2 = 0; b2 < nb; ++b2)
              for (int b3 = 0; b3 < nb; ++b3) {
                for (const Term& tm : terms) {
                  Single sg[3] = {{l1, tm.m1, b1}, {l2, tm.m2, b2}, {l3, -(tm.m1 + tm.m2), b3}};
                  float rs = 1.0f;
                  const long long e = lookup(sg, &rs);
                  if (e < 0) return fail(ctx, SBG_ERR_INTERNAL, "4PCF table lookup failed");
                  // the entry with every m negated holds the conjugate: Re T is
                  // the same, Im T (odd Lambda) changes sign
                  const double sgn = (e & 1) && odd ? -1.0 : 1.0;
                  entries.push_back(e);
                  t.coef.push_back(sgn * tm.c * rs);
                }
                t.ptr.push_back((int)entries.size());
              }
        }
  } else {
    for (int m1 = -L; m1 <= L; ++m1)
      for (int m2 = -L; m2 <= L; ++m2)
        for (int b1 = 0; b1 < nb; ++b1)
          for (int b2 = 0; b2 < nb; ++b2)
            for (int b3 = 0; b3 < nb; ++b3) {
              const int m3 = -(m1 + m2);
              if (std::abs(m3) <= L) {
                Single sg[3] = {{-1, m1, b1}, {-1, m2, b2}, {-1, m3, b3}};
                const long long e = lookup(sg, nullptr);
                if (e < 0) return fail(ctx, SBG_ERR_INTERNAL, "2D 4PCF table lookup failed");
                entries.push_back(e);
              }
              t.ptr.push_back((int)entries.size());
            }
  }
  long long so = 0;
  t.tc = tc;
  // Appends the block's rows rows[r], rows[r + 1], ... to a tile, at most TR rows
  // and tile_u singles.  Returns how many it took.
  auto cut_tile = [&](Block& bk, const std::vector<int>& rows, size_t r, int TR, int tile_u, Tile4& tl,
                      std::map<int, int>& local) -> int {
    tl.row0 = (int)t.rows.size();
    tl.uniq0 = (int)t.uniq.size();
    int nr = 0;
    for (; r < rows.size() && nr < TR; ++r, ++nr) {
      const RowKey rk = bk.rows[rows[r]];
      const Ang a1 = angs[rk.a1], a2 = angs[rk.a2];
      const int s1 = store_index(dim, nb, a1.l, std::abs(a1.m), rk.b1);
      const int s2 = store_index(dim, nb, a2.l, std::abs(a2.m), rk.b2);
      const int need = (local.count(s1) ? 0 : 1) + ((local.count(s2) || s2 == s1) ? 0 : 1);
      if ((int)local.size() + need > tile_u) break;
      if (!local.count(s1)) { const int k = (int)local.size(); local[s1] = k; if (!tc) t.uniq.push_back(s1); }
      if (!local.count(s2)) { const int k = (int)local.size(); local[s2] = k; if (!tc) t.uniq.push_back(s2); }
      Row4 rw;
      rw.u1 = local[s1];
      rw.u2 = local[s2];
      rw.flags = (a1.m < 0 ? 1 : 0) | (a2.m < 0 ? 2 : 0);
      t.rows.push_back(rw);
    }
    tl.nrows = nr;
    tl.nuniq = (int)local.size();
    return nr;
  };
  // FP32 tiles of n rows and nc columns, in entries of the accumulation: the
  // lanes of their warps, forming the rows (about as long as 10 columns' FMAs)
  // and about 2000 per tile for staging and barriers
  auto simt_cost = [&](long long n, int nc) -> double {
    if (n == 0 || nc == 0) return 0.0;
    const SimtGeometry g = simt_geometry(cplx ? 1 : 0, nc);
    auto tile = [&](long long rows) {
      const long long thr = (rows + g.rt - 1) / g.rt * g.ncg;
      return (double)((thr + 31) / 32 * 32 * g.rt * g.ct) + 10.0 * rows + 2000.0;
    };
    const long long full = n / g.max_rows, rest = n % g.max_rows;
    return full * tile(g.max_rows) + (rest ? tile(rest) : 0.0);
  };
  struct Group { unsigned mask; std::vector<int> rows; };
  std::vector<int> index(nentries, -1);  // [entry] its place in T
  for (Block& bk : blocks) {
    const int nrows_blk = (int)bk.rows.size();
    if (nrows_blk == 0) continue;
    const int nl3 = (int)bk.l3s.size();
    for (int c0 = 0; c0 < bk.ncols; c0 += col_chunk) {
      const int nc = std::min(col_chunk, bk.ncols - c0);
      const int cls = tc ? 0 : (nc <= 16 ? 0 : (nc <= 32 ? 1 : 2));
      std::vector<Group> groups;
      auto columns = [&](unsigned mask) {
        int n = 0;
        for (int c = c0; c < c0 + nc; ++c) n += mask >> (c % nl3) & 1;
        return n;
      };
      if (tc) {
        groups.push_back({~0u, {}});
        for (int r = 0; r < nrows_blk; ++r) groups[0].rows.push_back(r);
      } else {
        // the units of the span grid: rows x columns of 4096 entries, cut in order
        const int span_rows = cls == 0 ? 256 : (cls == 1 ? 128 : 64);
        t.simt.span_tiles[cls] += (int)count_tiles(bk.rows, span_rows);
        // The output takes a row's entries of a few l3 only (3D: l1 + l2 + l3 of
        // one parity within the triangle, and not those another row covers):
        // the rows of one set of l3 share tiles of its columns, about half of
        // the block's (lmax 4, 10 bins: 75,500 of 134,320 entries).  Sets too
        // small to fill their tiles join another one while that costs less.
        std::map<unsigned, std::vector<int>> sets;
        for (int r = 0; r < nrows_blk; ++r)
          if (bk.used[r]) sets[bk.used[r]].push_back(r);
        for (auto& kv : sets) groups.push_back({kv.first, std::move(kv.second)});
        for (;;) {
          double gain = 0.0;
          size_t ga = 0, gb = 0;
          for (size_t i = 0; i < groups.size(); ++i)
            for (size_t j = i + 1; j < groups.size(); ++j) {
              const Group &p = groups[i], &q = groups[j];
              const double d = simt_cost(p.rows.size(), columns(p.mask)) + simt_cost(q.rows.size(), columns(q.mask)) -
                               simt_cost(p.rows.size() + q.rows.size(), columns(p.mask | q.mask));
              if (d > gain) {
                gain = d;
                ga = i;
                gb = j;
              }
            }
          if (gain <= 0.0) break;
          groups[ga].mask |= groups[gb].mask;
          groups[ga].rows.insert(groups[ga].rows.end(), groups[gb].rows.begin(), groups[gb].rows.end());
          std::sort(groups[ga].rows.begin(), groups[ga].rows.end());
          groups.erase(groups.begin() + gb);
        }
      }
      for (const Group& gr : groups) {
        std::vector<int> gcols;  // the block's columns of the group
        const int col0 = (int)t.cols.size();
        for (int c = c0; c < c0 + nc; ++c) {
          if (!(gr.mask >> (c % nl3) & 1)) continue;
          gcols.push_back(c);
          t.cols.push_back(store_index(dim, nb, bk.l3s[c % nl3], bk.m3, bk.bcol0 + c / nl3));
        }
        const int gc = (int)t.cols.size() - col0;
        if (gc == 0) continue;
        int TR = 128, tile_u = max_u;
        SimtGeometry geo{};
        if (!tc) {
          geo = simt_geometry(cplx ? 1 : 0, gc);
          tile_u = geo.max_uniq;
          TR = geo.max_rows;
        }
        int bgroup = -1;
        if (tc) {
          BGroup g{};
          g.col0 = col0;
          g.ncols = gc;
          g.n = ((cplx ? 2 * gc : gc) + 7) & ~7;  // the MMAs take 2n and n rounded up to 16
          // the kernel's B stage holds 2n rows of 128 bytes and its inner
          // accumulator 3n TMEM columns: n <= 64
          if (g.n > 64) return fail(ctx, SBG_ERR_INTERNAL, "tensor-core column group wider than 64");
          g.off = t.img_stride;
          t.img_stride += (long long)g.n * 256;
          t.chunks_per_kb += g.n * 8;
          bgroup = (int)t.bgroups.size();
          t.bgroups.push_back(g);
        }
        for (size_t r = 0; r < gr.rows.size();) {
          Tile4 tl{};
          tl.col0 = col0;
          tl.ncols = gc;
          tl.bgroup = bgroup;
          std::map<int, int> local;
          const int nr = cut_tile(bk, gr.rows, r, TR, tile_u, tl, local);
          if (nr == 0) return fail(ctx, SBG_ERR_INTERNAL, "4PCF tiling: a row needs more staged singles than allowed");
          if (tc) ST(colour_slots(ctx, t, tl, local));
          tl.tout = so;
          if (tc) {
            so += (long long)nr * gc;
          } else {
            tl.cls = cls;
            tl.nrg = (nr + geo.rt - 1) / geo.rt;
            tl.ncg = geo.ncg;
            so += (long long)geo.rt * geo.ct * tl.nrg * tl.ncg;
            const int k = geo.launch;
            t.simt.threads[k] = std::max(t.simt.threads[k], tl.nrg * tl.ncg);
            t.simt.smem[k] = std::max(t.simt.smem[k], simt_tile_smem(tl, geo));
            t.simt.uses[k][cls] = true;
            ++t.simt.ntiles[k];
          }
          for (int q = 0; q < nr; ++q)
            for (int c = 0; c < gc; ++c)
              index[bk.first + (long long)gr.rows[r + q] * bk.ncols + gcols[c]] =
                  (int)(tc ? tl.tout + (long long)q * gc + c : simt_entry(tl, geo, q, c));
          t.tiles.push_back(tl);
          r += nr;
        }
      }
    }
  }
  t.tcount = so;

  // T indices of the couplings; 2D, negative: the entry's conjugate
  t.idx.resize(entries.size());
  for (size_t i = 0; i < entries.size(); ++i) {
    const int ti = index[entries[i] >> 1];
    if (ti < 0) return fail(ctx, SBG_ERR_INTERNAL, "4PCF entry without a tile");
    t.idx[i] = dim == 2 && (entries[i] & 1) ? -ti - 1 : ti;
  }
  t.nout = (int)t.ptr.size() - 1;
  if (!tc) {
    // the tiles of each launch together, in the order they were cut
    std::stable_partition(t.tiles.begin(), t.tiles.end(),
                          [&](const Tile4& x) { return simt_geometry(cplx ? 1 : 0, x.ncols).launch == 0; });
    t.simt.first[1] = t.simt.ntiles[0];
  }
  if (!to_device) return SBG_OK;
  ST(upload(ctx, t.d_tiles, t.tiles));
  ST(upload(ctx, t.d_rows, t.rows));
  ST(upload(ctx, t.d_cols, t.cols));
  ST(upload(ctx, t.d_uniq, t.uniq));
  ST(upload(ctx, t.d_bgroups, t.bgroups));
  ST(upload(ctx, t.d_ptr, t.ptr));
  ST(upload(ctx, t.d_idx, t.idx));
  if (dim == 3) ST(upload(ctx, t.d_coef, t.coef));  // 2D: every coefficient is 1
  return SBG_OK;
}

void free_tables4(sbg_context* ctx, Tables4* t) {
  if (!t) return;
  dev_free(ctx, t->d_tiles);
  dev_free(ctx, t->d_rows);
  dev_free(ctx, t->d_cols);
  dev_free(ctx, t->d_uniq);
  dev_free(ctx, t->d_bgroups);
  dev_free(ctx, t->d_ptr);
  dev_free(ctx, t->d_idx);
  dev_free(ctx, t->d_coef);
  delete t;
}

sbg_status ensure_tables4(sbg_context* ctx, int dim, int nb, int L, bool tc, bool odd = false) {
  const std::string key = std::to_string(dim) + "/" + std::to_string(nb) + "/" + std::to_string(L) + (tc ? "/tc" : "/simt") +
                          (odd ? "/odd" : "");
  auto& cache = ctx->t4cache;
  for (size_t i = 0; i < cache.size(); ++i)
    if (cache[i].first == key) {
      std::rotate(cache.begin(), cache.begin() + i, cache.begin() + i + 1);
      ctx->t4 = cache.front().second;
      return SBG_OK;
    }
  Tables4* t = new Tables4();
  sbg_status s = build_tables4(ctx, *t, dim, nb, L, tc, odd);
  if (s == SBG_ERR_OUT_OF_MEMORY && !cache.empty()) {
    // make room: the cached tables of other geometries are only a speed-up
    free_tables4(ctx, t);
    cudaStreamSynchronize(ctx->stream);  // queued work may still read them
    for (auto& kv : cache) free_tables4(ctx, kv.second);
    cache.clear();
    ctx->t4 = nullptr;
    ctx->err.clear();
    t = new Tables4();
    s = build_tables4(ctx, *t, dim, nb, L, tc, odd);
  }
  if (s != SBG_OK) {
    free_tables4(ctx, t);
    return s;
  }
  cache.insert(cache.begin(), {key, t});
  if ((int)cache.size() > sbg_context::kT4Cache) {
    // the evicted tables may still be read by queued work of this stream
    cudaStreamSynchronize(ctx->stream);
    free_tables4(ctx, cache.back().second);
    cache.pop_back();
  }
  ctx->t4 = t;
  return SBG_OK;
}

void rec(sbg_context* ctx, int i) { cudaEventRecord(ctx->ev[i], ctx->stream); }

// ---------------------------------------------------------------- autotuner --
// The choice under `key` among `cands`: measured on its first use by running
// run(c) for every candidate (one warm-up run each, then three rounds in which
// every candidate runs once, each run timed with CUDA events on the context's
// stream, so that drifts of clock or memory state fall on all of them), kept
// for the life of the context.  The first candidate is the default: another
// must be more than 3% faster in total to be taken.  run(c) must leave the
// caller's data as it found it (it writes scratch).
template <class F>
sbg_status autotune(sbg_context* ctx, const std::string& key, const std::vector<int>& cands, F run, int* choice) {
  auto it = ctx->tune.find(key);
  if (it != ctx->tune.end()) {
    *choice = it->second;
    return SBG_OK;
  }
  if (cands.size() == 1 || !ctx->autotune_on) {
    *choice = cands[0];  // the default (not recorded: a later enabled call measures)
    return SBG_OK;
  }
  if (!ctx->tev[0]) {
    CU(cudaEventCreate(&ctx->tev[0]));
    CU(cudaEventCreate(&ctx->tev[1]));
  }
  std::vector<float> total(cands.size(), 0.f);
  for (size_t i = 0; i < cands.size(); ++i) CU(run(cands[i]));
  for (int r = 0; r < 3; ++r)
    for (size_t i = 0; i < cands.size(); ++i) {
      CU(cudaEventRecord(ctx->tev[0], ctx->stream));
      CU(run(cands[i]));
      CU(cudaEventRecord(ctx->tev[1], ctx->stream));
      CU(cudaEventSynchronize(ctx->tev[1]));
      float ms = 0.f;
      CU(cudaEventElapsedTime(&ms, ctx->tev[0], ctx->tev[1]));
      total[i] += ms;
    }
  size_t best = 0;
  for (size_t i = 1; i < cands.size(); ++i)
    if (total[i] < 0.97f * total[0] && total[i] < total[best]) best = i;
  ctx->tune[key] = *choice = cands[best];
  return SBG_OK;
}

// Lines per CTA of a strided FFT pass (N >= 128): the default, half or twice
// it, timed on the pass's own input (its whole batch, up to 4 GB of output),
// writing a scratch buffer; one choice per (N, direction, load, axis).
sbg_status tune_fft(sbg_context* ctx, int n, FftPass& p) {
  if (p.inner == 1 || n < 128) return SBG_OK;
  char key[96];
  snprintf(key, sizeof key, "fft/%d/%d/%d/%s", n, p.sign, p.load, p.inner == (long long)n * n ? "z" : "y");
  if (ctx->tune.count(key)) {
    p.tl = ctx->tune[key];
    return SBG_OK;
  }
  if (!ctx->autotune_on) return SBG_OK;
  FftPass q = p;
  q.batch = (int)std::max<long long>(
      1, std::min<long long>(p.nb_per_field ? p.nb_per_field : p.batch, (4ll << 30) / (q.bstride * 8)));
  q.nb_per_field = 0;
  q.shared_stride = 0;
  q.field_points = 0;
  void* scratch;
  ST(buf(ctx, "tune", (size_t)q.batch * (size_t)q.bstride * 8, &scratch));
  q.out = (float2*)scratch;
  std::vector<int> cands = {0, 1};
  // twice the lines: up to N = 512, and N = 256 for the product passes (which
  // also stage delta-hat in shared memory)
  const bool product = p.load == LOAD_MUL || p.load == LOAD_MUL2 || p.load == LOAD_MULT;
  if (n <= (product ? 256 : 512)) cands.push_back(2);
  int tl = 0;
  ST(autotune(ctx, key, cands, [&](int c) { q.tl = c; return fft_axis_pass(n, q, ctx->stream); }, &tl));
  p.tl = tl;
  return SBG_OK;
}

// -------------------------------------------------------- FFT helpers ----
// Transform of `batch` arrays in three (dim 3) or two axis passes, in place in
// `out` after the first.  prune_r >= 0 (dim 3): the input is zero beyond
// minimum-image distance prune_r on every axis, so z-lines outside the (y, x)
// support and, after that pass, y-lines outside the x support stay zero and are
// skipped.
sbg_status fft_all(sbg_context* ctx, int dim, int n, int sign, int load, const void* in, float2* out, int batch,
                   const float2* tw, int prune_r = -1) {
  FftPass p{};
  p.twiddle = tw;
  p.batch = batch;
  p.bstride = dim == 3 ? (long long)n * n * n : (long long)n * n;
  p.sign = sign;
  p.in = in; p.out = out; p.load = load;
  if (dim == 3) {  // z axis
    p.outer = 1; p.inner = (long long)n * n;
    if (prune_r >= 0) { p.prune_mode = 1; p.prune_r = prune_r; }
    ST(tune_fft(ctx, n, p));
    KL(fft_axis_pass(n, p, ctx->stream));
    p.tl = 0;
    p.in = out; p.load = LOAD_COMPLEX;
  }
  p.outer = dim == 3 ? n : 1; p.inner = n;  // y axis
  if (prune_r >= 0) p.prune_mode = 2;
  ST(tune_fft(ctx, n, p));
  KL(fft_axis_pass(n, p, ctx->stream));
  p.tl = 0;
  p.prune_mode = 0;
  p.in = out; p.load = LOAD_COMPLEX;
  p.outer = dim == 3 ? (long long)n * n : n; p.inner = 1;  // x axis
  KL(fft_axis_pass(n, p, ctx->stream));
  return SBG_OK;
}

// The inverse transforms of the convolutions: those of the stored groups
// (g < ngroups4) go to the blocked coefficient store, where an m = 0 group (real
// kernels, so real coefficients) takes two bins per transform; the other groups
// take one transform per bin.  By group, or (pairs_first) the stored groups'
// packed transforms before their others, so that one launch of each kind serves
// every group.
struct ConvTable {
  std::vector<FftXf> xf;
  std::vector<int> first;  // by group: first transform of each group, and the count
  std::vector<char> real;  // by group: its transforms are packed real ones
  int stored = 0;          // transforms of stored groups
  int packed = 0;          // packed ones
};
ConvTable conv_table(int dim, int nb, int ngroups, int ngroups4, bool pairs_first) {
  ConvTable t;
  std::vector<FftXf> single;
  for (int g = 0, l = 0; g < ngroups; ++g) {
    if (g == ngroups4) t.xf.insert(t.xf.end(), single.begin(), single.end());
    t.first.push_back((int)t.xf.size());
    while (dim == 3 && (l + 1) * (l + 2) / 2 <= g) ++l;
    const bool m0 = dim == 3 ? g == l * (l + 1) / 2 : g == 0;
    t.real.push_back(m0 && g < ngroups4);
    if (t.real[g]) {
      for (int b = 0; b < nb; b += 2) t.xf.push_back({g * nb + b, b + 1 < nb ? g * nb + b + 1 : -1, g * nb + b, 0});
      t.packed += (nb + 1) / 2;
    } else {
      auto& to = pairs_first && g < ngroups4 ? single : t.xf;
      for (int b = 0; b < nb; ++b) to.push_back({g * nb + b, -1, g * nb + b, 0});
    }
    if (g < ngroups4) t.stored += m0 ? (nb + 1) / 2 : nb;
  }
  if (ngroups <= ngroups4) t.xf.insert(t.xf.end(), single.begin(), single.end());
  t.first.push_back((int)t.xf.size());
  return t;
}

// Groups whose convolutions one launch of each pass takes: as many as keep the
// arrays between the passes (`bytes` each, for all fields of a slab) within
// kConvBytes, so that small grids take few launches, and at least one.  Measured
// (convolutions and Gram): 64^2, 20 transforms, 85 -> 18 us and 256^2, 55
// transforms, 216 -> 60 us against one group per launch; beyond that size more
// transforms per launch gain nothing (256^3, 10 of two arrays instead of 5: 80
// instead of 73 us each), and fewer than a group's, to keep the arrays in L2,
// lose (1024^2, 20 bins: 1.54 ms by groups, 1.88 ms by 32 MB).
constexpr long long kConvBytes = 48 << 20;
int conv_groups(int nb, long long bytes) { return (int)std::max<long long>(1, kConvBytes / (bytes * nb)); }

// Convolutions a = IFFT(delta-hat G) of the transforms [t0, t1) of the table d_xf
// (device) in one launch per pass: product and z (dim 3) or y pass, y pass (dim
// 3), x pass.  `load` says how the product takes its factors; G holds the factor
// arrays from array a0 on (LOAD_MUL: those of t0 ...).  astore != null: the x pass
// writes the blocked store of nsingle singles, through `work`; else the
// transforms go to work, [field][transform].
sbg_status conv_run(sbg_context* ctx, int dim, int n, const FftXf* d_xf, int t0, int t1, int load, const float2* G,
                    int a0, const float2* dhat, const float2* tw, float2* work, float2* astore, int nsingle,
                    int nfld = 1) {
  if (t0 >= t1) return SBG_OK;
  const long long ng = dim == 3 ? (long long)n * n * n : (long long)n * n;
  FftPass p{};
  p.twiddle = tw;
  p.batch = nfld * (t1 - t0);
  p.bstride = ng;
  p.sign = +1;
  p.xf = astore ? d_xf + t0 : nullptr;
  p.a0 = a0;
  if (nfld > 1) {
    p.nb_per_field = t1 - t0;
    p.shared_stride = ng;
    p.field_points = ng;
  }
  p.out = work; p.mul = G; p.shared = dhat; p.load = load;
  p.outer = 1; p.inner = ng / n;
  ST(tune_fft(ctx, n, p));
  KL(fft_axis_pass(n, p, ctx->stream));
  p.tl = 0;
  p.in = work; p.load = LOAD_COMPLEX; p.mul = nullptr; p.shared = nullptr;
  if (dim == 3) {
    p.outer = n; p.inner = n;
    ST(tune_fft(ctx, n, p));
    KL(fft_axis_pass(n, p, ctx->stream));
    p.tl = 0;
  }
  p.outer = ng / n; p.inner = 1;
  if (astore) { p.out = astore; p.out_blocked = load == LOAD_MUL2 ? 2 : 1; p.nsingle = nsingle; }
  KL(fft_axis_pass(n, p, ctx->stream));
  return SBG_OK;
}

// Every stored group's convolutions, at most `most` transforms of one kind per
// launch (table in pairs_first order).
sbg_status conv_stored(sbg_context* ctx, int dim, int n, const FftXf* d_xf, const ConvTable& t, int most, const float2* G,
                       const float2* dhat, const float2* tw, float2* work, float2* astore, int nsingle, int nfld = 1) {
  for (int i = 0, c; i < t.stored; i += c) {
    const bool packed = i < t.packed;
    c = std::min(most, (packed ? t.packed : t.stored) - i);
    ST(conv_run(ctx, dim, n, d_xf, i, i + c, packed ? LOAD_MUL2 : LOAD_MULT, G, 0, dhat, tw, work, astore, nsingle, nfld));
  }
  return SBG_OK;
}

// The table of the stored groups' transforms, the first ones of t.xf, on the device
// (kept while it stays the same).  The others need none: they take factor arrays and
// outputs in order.
sbg_status conv_upload(sbg_context* ctx, const ConvTable& t, int dim, int nb, int ngroups, int ngroups4, bool pairs_first,
                       FftXf** out) {
  *out = nullptr;
  if (!t.stored) return SBG_OK;
  const size_t bytes = t.stored * sizeof(FftXf);
  ST(buf(ctx, "xf", bytes, (void**)out));
  const std::string key = std::to_string(dim) + "/" + std::to_string(nb) + "/" + std::to_string(ngroups) + "/" +
                          std::to_string(ngroups4) + (pairs_first ? "/p" : "");
  if (ctx->xf_key != key) {
    ctx->xf_key.clear();
    CU(cudaMemcpyAsync(*out, t.xf.data(), bytes, cudaMemcpyHostToDevice, ctx->stream));
    ctx->xf_key = key;
  }
  return SBG_OK;
}

// Groups per launch of a call's convolutions (see conv_groups) and the buffer
// "group" that holds their arrays.  A context with a budget takes one (its other
// buffers have to fit as well).
sbg_status conv_buffer(sbg_context* ctx, int nb, int ngroups, long long bytes, int* per, float2** out) {
  *per = ctx->budget ? 1 : std::min(ngroups, conv_groups(nb, bytes));
  return buf(ctx, "group", (size_t)*per * nb * bytes, (void**)out);
}

sbg_status check_edges(sbg_context* ctx, const double* edges, int nb, int n) {
  for (int i = 0; i <= nb; ++i)
    if (!std::isfinite(edges[i])) return fail(ctx, SBG_ERR_BIN_RANGE, "non-finite bin edge");
  if (edges[0] < 0) return fail(ctx, SBG_ERR_BIN_RANGE, "edges[0] < 0");
  for (int i = 0; i < nb; ++i)
    if (!(edges[i + 1] > edges[i])) return fail(ctx, SBG_ERR_BIN_RANGE, "bin edges are not strictly increasing");
  if (!(edges[nb] < 0.5 * n)) return fail(ctx, SBG_ERR_BIN_RANGE, "edges[nbins] must be < N/2");
  return SBG_OK;
}

// Pinned host staging of at least `bytes` bytes (grown, never shrunk).
sbg_status host_staging(sbg_context* ctx, size_t bytes, void** out) {
  if (bytes > ctx->hpin_bytes) {
    CU(cudaStreamSynchronize(ctx->stream));
    if (ctx->hpin) cudaFreeHost(ctx->hpin);
    ctx->hpin = nullptr;
    ctx->hpin_bytes = 0;
    CU(cudaMallocHost(&ctx->hpin, bytes));
    ctx->hpin_bytes = bytes;
  }
  *out = ctx->hpin;
  return SBG_OK;
}

sbg_status finish_timings(sbg_context* ctx) {
  CU(cudaStreamSynchronize(ctx->stream));
  ctx->last_launches = ctx->nlaunch;
  for (int i = 0; i < kStages; ++i) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, ctx->ev[i], ctx->ev[i + 1]) != cudaSuccess) {
      cudaGetLastError();
      ms = 0.f;
    }
    ctx->timings[i] = ms;
  }
  ctx->contraction_ms = 0.0;
  if (ctx->kev_used) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, ctx->kev[0], ctx->kev[1]) != cudaSuccess) {
      cudaGetLastError();
      ms = 0.f;
    }
    ctx->contraction_ms = ms;
  }
  return SBG_OK;
}

// Key of the kernel spectra kept between calls: side, order and the squared edges
// themselves, all their bits (edges that differ by less than any printed digits can
// lie on either side of an integer, and then hold other cells).
std::string spectra_key(int dim, int n, int L, const std::vector<double>& e2) {
  std::string key = std::to_string(dim) + "/" + std::to_string(n) + "/" + std::to_string(L) + "/";
  key.append((const char*)e2.data(), e2.size() * sizeof(double));
  return key;
}

// Uploads of small host tables are skipped while the device holds the same ones
// (each costs several microseconds of host time before the first kernel).  A call
// that fails forgets them: its queued uploads may not have run.
struct TableGuard {
  sbg_context* ctx;
  bool ok = false;
  ~TableGuard() {
    if (ok) return;
    ctx->xf_key.clear();
    ctx->tw_sides.clear();
    ctx->e2_up.clear();
    ctx->lines_key = {0, 0.0};
  }
};

// Twiddles of side n, squared edges and (normalised calls only) bin volumes.
sbg_status geometry_tables(sbg_context* ctx, int n, const std::vector<double>& e2, const std::vector<double>& vb, float2** tw,
                           double** d_e2, double** d_vb) {
  const std::string name = "tw" + std::to_string(n);
  ST(buf(ctx, name.c_str(), n * 8, (void**)tw));
  ST(buf(ctx, "e2", (kMaxBins + 1) * 8, (void**)d_e2));
  *d_vb = nullptr;
  if (!vb.empty()) ST(buf(ctx, "vb", kMaxBins * 8, (void**)d_vb));
  if (!ctx->tw_sides.count(n)) {
    const std::vector<float2> t = twiddles(n);
    CU(cudaMemcpyAsync(*tw, t.data(), n * 8, cudaMemcpyHostToDevice, ctx->stream));
    ctx->tw_sides.insert(n);
  }
  if (ctx->e2_up != e2) {
    ctx->e2_up.clear();
    CU(cudaMemcpyAsync(*d_e2, e2.data(), e2.size() * 8, cudaMemcpyHostToDevice, ctx->stream));
    ctx->e2_up = e2;
  }
  if (!vb.empty()) CU(cudaMemcpyAsync(*d_vb, vb.data(), vb.size() * 8, cudaMemcpyHostToDevice, ctx->stream));
  return SBG_OK;
}

// Copies of results from pinned staging to the caller's arrays, by as many host
// threads as copy_threads() gives.
struct HostCopy {
  void* dst;
  const void* src;
  size_t bytes;
};
void copy_out(const std::vector<HostCopy>& c) {
  size_t total = 0;
  for (const HostCopy& x : c) total += x.bytes;
  auto part = [&](size_t b0, size_t b1) {  // bytes [b0, b1) of the copies in a row
    size_t at = 0;
    for (const HostCopy& x : c) {
      const size_t lo = std::max(b0, at), hi = std::min(b1, at + x.bytes);
      if (lo < hi) std::memcpy((char*)x.dst + (lo - at), (const char*)x.src + (lo - at), hi - lo);
      at += x.bytes;
    }
  };
  const size_t nt = copy_threads(total);
  const size_t per = (total / nt + 4095) / 4096 * 4096;
  std::vector<std::thread> th;
  for (size_t t = 1; t < nt; ++t) {
    // without a thread to be had, this one does the rest
    try {
      th.emplace_back(part, t * per, t + 1 == nt ? total : (t + 1) * per);
    } catch (const std::system_error&) {
      part(t * per, total);
      break;
    }
  }
  part(0, nt == 1 ? total : per);
  for (auto& x : th) x.join();
}

// ---------------------------------------------------------------- core ----
// Shared by sbg_full (dim 3) and sbg_projected / batch (dim 2).
// odd (dim 3, 4PCF only): the odd-parity Lambda, zeta4 receives Im of each coefficient
sbg_status measure(sbg_context* ctx, int dim, const void* field, sbg_dtype dtype, int n, const double* edges, int nb,
                   int lmax3, int lmax4, sbg_precision prec, unsigned flags, double* zeta3, double* zeta4,
                   bool odd = false) {
  const bool do3 = flags & SBG_3PCF, do4 = flags & SBG_4PCF;
  const long long ng = dim == 3 ? (long long)n * n * n : (long long)n * n;
  const int L = std::max(do3 ? lmax3 : 0, do4 ? lmax4 : 0);
  // number of (l, m>=0) groups in 3D, or m groups in 2D
  auto npair = [&](int l) { return dim == 3 ? (l + 1) * (l + 2) / 2 : l + 1; };
  const int ngroups = npair(L);
  const int ngroups4 = do4 ? npair(lmax4) : 0;
  const std::vector<double> e2 = snap_e2(edges, nb);
  TableGuard tables{ctx};
  const std::vector<double> vb = flags & SBG_NORMALIZED ? cell_counts(n, dim, e2, nb) : std::vector<double>();
  if (flags & SBG_NORMALIZED)
    for (int b = 0; b < nb; ++b)
      if (vb[b] == 0.0) return fail(ctx, SBG_ERR_EMPTY_BIN, "bin " + std::to_string(b) + " holds no cell");

  ctx->kev_used = false;
  ctx->nlaunch = 0;
  rec(ctx, 0);
  // ---- inputs ----
  const size_t esz = dtype == SBG_F64 ? 8 : 4;
  const void* d_in = field;
  if (!(flags & SBG_FIELD_ON_DEVICE)) {
    void* stg;
    ST(buf(ctx, "stage", ng * esz, &stg));
    CU(cudaMemcpyAsync(stg, field, ng * esz, cudaMemcpyHostToDevice, ctx->stream));
    d_in = stg;
  }
  float* d_delta;
  float2 *d_dhat, *d_tw;
  double *d_acc, *d_e2, *d_vb;
  ST(buf(ctx, "delta", ng * 4, (void**)&d_delta));
  ST(buf(ctx, "dhat", ng * 8, (void**)&d_dhat));
  ST(buf(ctx, "acc", 64, (void**)&d_acc));
  ST(geometry_tables(ctx, n, e2, vb, &d_tw, &d_e2, &d_vb));
  CU(cudaMemsetAsync(d_acc, 0, 64, ctx->stream));
  KL(launch_sum(d_in, dtype == SBG_F64, ng, d_acc, ctx->stream));
  KL(launch_convert(d_in, dtype == SBG_F64, ng, d_acc, (flags & SBG_SUBTRACT_MEAN) ? 1 : 0, d_delta, ctx->stream));
  rec(ctx, 1);
  // ---- delta-hat ----
  ST(fft_all(ctx, dim, n, -1, LOAD_REAL, d_delta, d_dhat, 1, d_tw));
  rec(ctx, 2);
  // ---- kernel spectra (plan) ----
  const std::string key = spectra_key(dim, n, L, e2);
  const size_t gbytes = (size_t)ngroups * nb * ng * 8;
  const double inv_ng = 1.0 / (double)ng;
  auto gen_group = [&](int g, float2* dst) -> sbg_status {
    if (dim == 3) {
      CU(cudaMemsetAsync(dst, 0, (size_t)nb * ng * 8, ctx->stream));
      int l = 0;
      while ((l + 1) * (l + 2) / 2 <= g) ++l;
      const int m = g - l * (l + 1) / 2;
      KL(launch_kgen3d(n, l, m, ylm_norm(l, m), d_e2, nb, inv_ng, dst, ctx->stream));
      // the kernels vanish beyond the last edge: prune the zero lines
      const int rmax = std::min(n / 2 - 1, (int)std::ceil(edges[nb]));
      ST(fft_all(ctx, 3, n, +1, LOAD_COMPLEX, dst, dst, nb, d_tw, rmax));
    } else {
      KL(launch_kgen2d(n, g, 1, d_e2, nb, inv_ng, dst, ctx->stream));
      ST(fft_all(ctx, 2, n, +1, LOAD_COMPLEX, dst, dst, nb, d_tw));
    }
    return SBG_OK;
  };
  bool cached = false;
  if (ctx->gcached && ctx->gkey == key) {
    cached = true;
  } else {
    // try to (re)build the full cache; fall back to per-group regeneration
    dev_free(ctx, ctx->gcache);
    ctx->gcached = false;
    size_t freeb = 0, totb = 0;
    cudaMemGetInfo(&freeb, &totb);
    const size_t a4bytes = (size_t)ngroups4 * nb * ng * 8;
    const bool fits = gbytes + a4bytes + (size_t)nb * ng * 8 + (1ull << 30) < freeb &&
                      (!ctx->budget || ctx->used + gbytes + a4bytes + (size_t)nb * ng * 8 <= ctx->budget);
    if (fits && dev_alloc(ctx, ctx->gcache, gbytes) == SBG_OK) {
      for (int g = 0; g < ngroups; ++g) ST(gen_group(g, (float2*)ctx->gcache.p + (size_t)g * nb * ng));
      ctx->gcached = true;
      ctx->gkey = key;
      cached = true;
    } else {
      ctx->err.clear();
    }
  }
  rec(ctx, 3);
  // ---- convolutions + 3PCF Gram ----
  float2* d_astore = nullptr;
  float2* d_group = nullptr;
  double* d_S = nullptr;
  const int nsingle = ngroups4 * nb;  // singles in the blocked coefficient store
  if (do4) ST(buf(ctx, "astore", (size_t)nsingle * ng * 8, (void**)&d_astore));
  const bool fused = dim == 3 && !cached;  // see below
  int per = 1;  // groups per launch
  ST(conv_buffer(ctx, nb, ngroups, ng * 8, &per, &d_group));
  if (!cached) per = 1;
  // the stored groups' transforms by kind when several groups fit
  const bool together = per > 1 && ngroups4 > 0;
  const ConvTable conv = conv_table(dim, nb, ngroups, ngroups4, together);
  FftXf* d_xf = nullptr;
  ST(conv_upload(ctx, conv, dim, nb, ngroups, ngroups4, together, &d_xf));
  float2* d_gtmp = nullptr;
  if (!cached) ST(buf(ctx, "gtmp", (size_t)nb * ng * 8, (void**)&d_gtmp));
  const int ngroups3 = do3 ? npair(lmax3) : 0;
  if (do3) {
    ST(buf(ctx, "S", (size_t)std::max(ngroups3, 1) * nb * nb * 16, (void**)&d_S));
    CU(cudaMemsetAsync(d_S, 0, (size_t)ngroups3 * nb * nb * 16, ctx->stream));
  }
  // split-BF16 / split-TF32: both combination steps run on the tensor cores,
  // whose kernels report a wait that ran out in this word (a batch clears it
  // once and reads it after its last field)
  const bool tcomb = prec != SBG_PREC_FP32;
  const int tf32 = prec == SBG_PREC_TF32X3 ? 1 : 0;
  int* d_err = nullptr;
  if (tcomb) {
    ST(buf(ctx, "err", 16, (void**)&d_err));
    if (!ctx->defer) CU(cudaMemsetAsync(d_err, 0, 16, ctx->stream));
  }
  // 3D groups without cached spectra: kernel generation fused with the forward
  // FFT and the spectral product fused between the forward and inverse z
  // transforms (sbg_fft_fused.cu); the lines of the kernel support are listed
  // once per call
  int* d_lines = nullptr;
  int nlines = 0, Rsup = 0;
  if (fused) {
    if (ctx->lines_key != std::make_pair(n, e2[nb])) {
      ctx->lines_key = {0, 0.0};
      std::vector<int> lines;
      for (int zi = 0; zi < n; ++zi)
        for (int yi = 0; yi < n; ++yi) {
          const double z = zi < n - zi ? zi : zi - n, y = yi < n - yi ? yi : yi - n;
          if (y * y + z * z <= e2[nb]) lines.push_back(zi * n + yi);
        }
      ctx->rsup = 0;
      while ((double)(ctx->rsup + 1) * (ctx->rsup + 1) <= e2[nb]) ++ctx->rsup;
      ctx->nlines = (int)lines.size();
      ST(buf(ctx, "klines", std::max<size_t>(lines.size(), 1) * 4, (void**)&d_lines));
      if (ctx->nlines)
        CU(cudaMemcpyAsync(d_lines, lines.data(), lines.size() * 4, cudaMemcpyHostToDevice, ctx->stream));
      ctx->lines_key = {n, e2[nb]};
    }
    nlines = ctx->nlines;
    Rsup = ctx->rsup;
    ST(buf(ctx, "klines", (size_t)std::max(nlines, 1) * 4, (void**)&d_lines));
  }
  // delta-weighted Grams of the groups [g0, g1) in one launch: from the blocked
  // store, or from the group buffer
  auto gram = [&](int g0, int g1, bool stored) -> sbg_status {
    g1 = std::min(g1, ngroups3);
    if (!do3 || g0 >= g1) return SBG_OK;
    double* Sg = d_S + (size_t)g0 * nb * nb * 2;
    const float2* src = stored ? d_astore : d_group;
    const int ns = stored ? nsingle : 0, s0 = stored ? g0 * nb : 0;
    if (tcomb)
      KL(launch_gram_tc(src, ng, nb, d_delta, Sg, ns, s0, tf32, d_err, ctx->nsm, ctx->wait_ns, ctx->stall, ctx->stream, 1,
                        0, g1 - g0));
    else
      KL(launch_gram3(src, ng, nb, d_delta, Sg, ns, s0, ctx->stream, 1, 0, g1 - g0));
    return SBG_OK;
  };
  if (fused) {
    for (int g = 0, l = 0; g < ngroups; ++g) {
      while ((l + 1) * (l + 2) / 2 <= g) ++l;
      const int m = g - l * (l + 1) / 2;
      const bool stored = g < ngroups4;
      const int nbatch = conv.first[g + 1] - conv.first[g];
      FusedGroup fg{};
      fg.l = l;
      fg.m = m;
      fg.nb = nb;
      fg.norm_scale = ylm_norm(l, m) * inv_ng;
      fg.e2 = d_e2;
      fg.e2nb = e2[nb];
      fg.lines = d_lines;
      fg.nlines = nlines;
      fg.R = Rsup;
      fg.npack = stored && m == 0 ? nb : 0;
      fg.tw = d_tw;
      fg.kbuf = d_gtmp;
      fg.dhat = d_dhat;
      fg.out = d_group;
      ctx->nlaunch += 2;  // passes A and B (pass C counted by KL)
      KL(launch_fused_group(n, fg, ctx->stream));
      // inverse y and x passes
      FftPass p{};
      p.twiddle = d_tw;
      p.batch = nbatch;
      p.bstride = ng;
      p.sign = +1;
      p.in = d_group;
      p.out = d_group;
      p.load = LOAD_COMPLEX;
      p.outer = n;
      p.inner = n;
      ST(tune_fft(ctx, n, p));
      KL(fft_axis_pass(n, p, ctx->stream));
      p.tl = 0;
      p.outer = (long long)n * n;
      p.inner = 1;
      if (stored) {
        p.out = d_astore;
        p.out_blocked = m == 0 ? 2 : 1;
        p.nsingle = nsingle;
        p.xf = d_xf + conv.first[g];
      }
      KL(fft_axis_pass(n, p, ctx->stream));
      if (!stored) ST(gram(g, g + 1, false));
    }
  } else {
    const float2* G = cached ? (const float2*)ctx->gcache.p : d_gtmp;
    int g0 = 0;
    if (together) {
      ST(conv_stored(ctx, dim, n, d_xf, conv, per * nb, G, d_dhat, d_tw, d_group, d_astore, nsingle));
      g0 = ngroups4;
    }
    // the others in order: several 2D groups per launch where the spectra are
    // cached, else one by one (3D: step by step like the fused path)
    for (int g1; g0 < ngroups; g0 = g1) {
      const bool stored = g0 < ngroups4;
      g1 = dim == 2 && !stored ? std::min(ngroups, g0 + per) : g0 + 1;
      const int t0 = conv.first[g0], t1 = conv.first[g1];
      const bool pairs = conv.real[g0];
      if (!cached) ST(gen_group(g0, d_gtmp));
      ST(conv_run(ctx, dim, n, d_xf, t0, t1, pairs ? LOAD_MUL2 : LOAD_MUL,
                  cached && !pairs ? G + (long long)g0 * nb * ng : G, cached ? 0 : g0 * nb, d_dhat, d_tw, d_group,
                  stored ? d_astore : nullptr, nsingle));
      if (!stored) ST(gram(g0, g1, false));
    }
  }
  ST(gram(0, ngroups4, true));
  rec(ctx, 4);
  rec(ctx, 5);
  // ---- 4PCF ----
  double* d_z4 = nullptr;
  if (do4) {
    const bool tc = tcomb;                          // split BF16 or split TF32 on the tensor cores
    const bool tf = tf32 != 0;
    ST(ensure_tables4(ctx, dim, nb, lmax4, tc, odd));
    Tables4& t = *ctx->t4;
    const int cplx = dim == 2 ? 1 : 0;
    // kernel output mode: 0 Re (3D even), 1 complex (2D), 2 Im only (3D odd)
    const int kmode = dim == 2 ? 1 : (odd ? 2 : 0);
    double* d_T;
    ST(buf(ctx, "T", (size_t)std::max<long long>(t.tcount, 1) * 8 * (cplx ? 2 : 1), (void**)&d_T));
    CU(cudaMemsetAsync(d_T, 0, (size_t)t.tcount * 8 * (cplx ? 2 : 1), ctx->stream));
    if (tc) {
      const int ntl = (int)t.tiles.size();
      const long long kblocks = ng / 32;
      // x-splits per tile: units = ntl * nsplit spread over the CTAs; the three
      // best by their wave fill are timed by the autotuner on the first call
      std::vector<std::pair<double, int>> fill;
      for (int k = 1; k <= 32 && k <= kblocks; ++k) {
        const long long units = (long long)ntl * k;
        const long long rounds = (units + ctx->nsm - 1) / ctx->nsm;
        fill.push_back({(double)units / (double)(rounds * ctx->nsm), k});
      }
      std::stable_sort(fill.begin(), fill.end(), [](const std::pair<double, int>& x, const std::pair<double, int>& y) {
        return x.first > y.first + 0.02;
      });
      std::vector<int> cands;
      for (size_t i = 0; i < fill.size() && cands.size() < 3; ++i) cands.push_back(fill[i].second);
      long long epochs = 4;
      for (int k : cands) {
        const long long units = (long long)ntl * k;
        const long long rounds = (units + ctx->nsm - 1) / ctx->nsm;
        const long long nk_unit = (kblocks + k - 1) / k;
        epochs = std::max(epochs, rounds * ((nk_unit + kTcEpoch - 1) / kTcEpoch) + 4);
      }
      int* d_cnt;
      ST(buf(ctx, "tccnt", (size_t)epochs * 4, (void**)&d_cnt));
      void* d_bimg;
      ST(buf(ctx, "bimg", (size_t)(ng / 32) * (size_t)t.img_stride * (tf ? 2 : 1), &d_bimg));
      auto tc4_run = [&](int nsplit, double* T, cudaEvent_t e0, cudaEvent_t e1) -> cudaError_t {
        cudaError_t e = cudaMemsetAsync(d_cnt, 0, (size_t)epochs * 4, ctx->stream);
        if (e != cudaSuccess) return e;
        return launch_tc4(d_astore, d_bimg, (const BGroup*)t.d_bgroups.p, (int)t.bgroups.size(), t.chunks_per_kb,
                          t.img_stride, d_delta, ng, (const Tile4*)t.d_tiles.p, ntl, (const Row4*)t.d_rows.p,
                          (const int*)t.d_cols.p, (const int*)t.d_uniq.p, nsingle, kmode, nsplit, T, d_cnt, d_err,
                          ctx->nsm, ctx->stream, e0, e1, tf ? 1 : 0, ctx->wait_ns, ctx->stall);
      };
      int best = cands[0];
      if (cands.size() > 1 && !ctx->stall) {
        char key[160];
        snprintf(key, sizeof key, "tc4/%d/%d/%d/%d/%d/%d/%d", dim, n, nb, lmax4, (int)prec, odd ? 1 : 0, ntl);
        double* d_Ts;
        ST(buf(ctx, "tuneT", (size_t)std::max<long long>(t.tcount, 1) * 8 * (cplx ? 2 : 1), (void**)&d_Ts));
        ST(autotune(ctx, key, cands, [&](int c) { return tc4_run(c, d_Ts, nullptr, nullptr); }, &best));
      }
      ctx->nlaunch += 1;  // bimage_kernel
      KL(tc4_run(best, d_T, ctx->kev[0], ctx->kev[1]));
      ctx->kev_used = true;
    } else {
      CU(cudaEventRecord(ctx->kev[0], ctx->stream));
      ctx->kev_used = true;
      int launches = 0;
      CU(launch_simt4(d_astore, ng, d_delta, (const Tile4*)t.d_tiles.p, t.simt, (const Row4*)t.d_rows.p,
                      (const int*)t.d_cols.p, (const int*)t.d_uniq.p, kmode, nsingle, d_T, ctx->nsm, ctx->stream,
                      &launches));
      ctx->nlaunch += launches;
      CU(cudaEventRecord(ctx->kev[1], ctx->stream));
    }
    ST(buf(ctx, "z4", (size_t)t.nout * 8 * (cplx ? 2 : 1), (void**)&d_z4));
    KL(launch_couple(d_T, cplx, (const int*)t.d_ptr.p, (const int*)t.d_idx.p, (const double*)t.d_coef.p, t.nout, d_z4,
                     ctx->stream));
    if (flags & SBG_NORMALIZED) {
      const long long nouter = t.nout / ((long long)nb * nb * nb);
      KL(launch_normalize(d_z4, nouter, nb, 4, cplx ? 2 : 1, d_acc, (double)ng, d_vb, ctx->stream));
    }
  }
  if (tcomb && !ctx->defer) {  // a batch reads the flag once, after its last field
    int* perr;
    ST(host_staging(ctx, 64, (void**)&perr));
    CU(cudaMemcpyAsync(perr, d_err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    CU(cudaStreamSynchronize(ctx->stream));
    const int herr = *perr;
    if (herr)
      return fail(ctx, SBG_ERR_TIMEOUT, "a tensor-core combination kernel gave up waiting (code " + std::to_string(herr) + ")");
  }
  rec(ctx, 6);
  // ---- 3PCF finish + downloads ----
  const int ncomp3 = dim == 3 ? 1 : 2;
  const size_t z3bytes = do3 ? (size_t)(lmax3 + 1) * nb * nb * 8 * ncomp3 : 0;
  const size_t z4bytes = do4 ? (size_t)ctx->t4->nout * 8 * (dim == 2 ? 2 : 1) : 0;
  const size_t z3off = 0, z4off = (z3bytes + 255) / 256 * 256;
  unsigned char* hst;
  if (ctx->defer) {
    if (z4off + z4bytes > ctx->slot_bytes) return fail(ctx, SBG_ERR_INTERNAL, "batch staging slot too small");
    hst = (unsigned char*)ctx->hpin + 64 + (size_t)ctx->cur * ctx->slot_bytes;
  } else {
    ST(host_staging(ctx, z4off + z4bytes + 64, (void**)&hst));
  }
  if (do3) {
    double* d_z3;
    const int nl = lmax3 + 1;
    ST(buf(ctx, "z3", z3bytes, (void**)&d_z3));
    KL(launch_finish3(d_S, dim == 3, lmax3, nb, d_z3, ctx->stream));
    if (flags & SBG_NORMALIZED) KL(launch_normalize(d_z3, nl, nb, 3, ncomp3, d_acc, (double)ng, d_vb, ctx->stream));
    CU(cudaMemcpyAsync(hst + z3off, d_z3, z3bytes, cudaMemcpyDeviceToHost, ctx->stream));
  }
  if (do4) CU(cudaMemcpyAsync(hst + z4off, d_z4, z4bytes, cudaMemcpyDeviceToHost, ctx->stream));
  rec(ctx, 7);
  if (ctx->defer) {
    sbg_context::Pending& pd = ctx->pend[ctx->cur];
    pd.live = true;
    pd.zeta3 = do3 ? zeta3 : nullptr;
    pd.zeta4 = do4 ? zeta4 : nullptr;
    pd.off3 = z3off;
    pd.off4 = z4off;
    pd.b3 = z3bytes;
    pd.b4 = z4bytes;
    pd.launches = ctx->nlaunch;
    pd.kev_used = ctx->kev_used;
    tables.ok = true;
    return SBG_OK;
  }
  ST(finish_timings(ctx));
  std::vector<HostCopy> copies;
  if (do3) copies.push_back({zeta3, hst + z3off, z3bytes});
  if (do4) copies.push_back({zeta4, hst + z4off, z4bytes});
  copy_out(copies);
  tables.ok = true;
  return SBG_OK;
}

// ------------------------------------------------------------------ slabs --
// Projected 3PCF / 4PCF of nfld fields of one shape, dtype and bin set, measured
// together (a slab): their points follow each other in every buffer, and every
// stage of the path (preprocessing, delta-hat, convolutions, Grams, the 4PCF
// contraction, couplings, finalisation) is one launch over all of them, the
// fields being one more batch dimension (Secs. 2.2 and 2.4, Algorithms 2, 4,
// 7, 8 per field, exactly as measure() computes them one field at a time).
// Outputs are staged in pinned slot `slot` (layout: z3 of every field, then z4
// of every field) and copied to the fields' arrays by slab_copy_out once the
// stream has passed ev_done.
struct SlabOut {
  const sbg_field2d* fields = nullptr;
  int nfld = 0;
  size_t z3b = 0, z4b = 0;  // bytes per field
  size_t off4 = 0;          // z4 block within the slot
  unsigned char* host = nullptr;
};

sbg_status measure_slab(sbg_context* ctx, const sbg_field2d* fields, int nfld, int n, const double* edges, int nb,
                        int mmax, sbg_precision prec, unsigned flags, unsigned char* hslot, SlabOut* out) {
  const bool do3 = flags & SBG_3PCF, do4 = flags & SBG_4PCF;
  const long long ng = (long long)n * n;
  const int ngroups = mmax + 1;
  const int ngroups4 = do4 ? mmax + 1 : 0;
  const std::vector<double> e2 = snap_e2(edges, nb);
  TableGuard tables{ctx};
  const std::vector<double> vb = flags & SBG_NORMALIZED ? cell_counts(n, 2, e2, nb) : std::vector<double>();
  if (flags & SBG_NORMALIZED)
    for (int b = 0; b < nb; ++b)
      if (vb[b] == 0.0) return fail(ctx, SBG_ERR_EMPTY_BIN, "bin " + std::to_string(b) + " holds no cell");
  const sbg_dtype dtype = fields[0].dtype;
  const size_t esz = dtype == SBG_F64 ? 8 : 4;
  const bool on_dev = flags & SBG_FIELD_ON_DEVICE;
  cudaStream_t st = ctx->stream;

  // ---- inputs: the fields one after another (device fields that already are
  // contiguous, e.g. slices of a cube, are read in place) ----
  rec(ctx, 0);
  const void* d_in = nullptr;
  bool contiguous = on_dev;
  for (int i = 1; i < nfld && contiguous; ++i)
    contiguous = (const unsigned char*)fields[i].field == (const unsigned char*)fields[0].field + (size_t)i * ng * esz;
  if (contiguous) {
    d_in = fields[0].field;
  } else {
    void* stg;
    ST(buf(ctx, "stage", (size_t)nfld * ng * esz, &stg));
    for (int i = 0; i < nfld; ++i)
      CU(cudaMemcpyAsync((unsigned char*)stg + (size_t)i * ng * esz, fields[i].field, ng * esz,
                         on_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, st));
    d_in = stg;
  }
  float* d_delta;
  float2 *d_dhat, *d_tw;
  double *d_acc, *d_e2, *d_vb;
  ST(buf(ctx, "delta", (size_t)nfld * ng * 4, (void**)&d_delta));
  ST(buf(ctx, "dhat", (size_t)nfld * ng * 8, (void**)&d_dhat));
  ST(buf(ctx, "acc", (size_t)std::max(64, 16 * nfld), (void**)&d_acc));
  ST(geometry_tables(ctx, n, e2, vb, &d_tw, &d_e2, &d_vb));
  CU(cudaMemsetAsync(d_acc, 0, (size_t)16 * nfld, st));
  KL(launch_sum(d_in, dtype == SBG_F64, ng, d_acc, st, nfld));
  KL(launch_convert(d_in, dtype == SBG_F64, ng, d_acc, (flags & SBG_SUBTRACT_MEAN) ? 1 : 0, d_delta, st, nfld));
  rec(ctx, 1);
  // ---- delta-hat of every field ----
  ST(fft_all(ctx, 2, n, -1, LOAD_REAL, d_delta, d_dhat, nfld, d_tw));
  rec(ctx, 2);
  // ---- kernel spectra (shared by the fields: one shape, one bin set) ----
  const std::string key = spectra_key(2, n, mmax, e2);
  const size_t gbytes = (size_t)ngroups * nb * ng * 8;
  const double inv_ng = 1.0 / (double)ng;
  auto gen_group = [&](int g, float2* dst) -> sbg_status {
    KL(launch_kgen2d(n, g, 1, d_e2, nb, inv_ng, dst, st));
    ST(fft_all(ctx, 2, n, +1, LOAD_COMPLEX, dst, dst, nb, d_tw));
    return SBG_OK;
  };
  const float2* gbase = nullptr;
  {
    auto& gc = ctx->g2cache;
    auto it = std::find_if(gc.begin(), gc.end(), [&](const std::pair<std::string, DevBuf>& e) { return e.first == key; });
    if (it != gc.end()) {
      std::rotate(gc.begin(), it, it + 1);
      gbase = (const float2*)gc.front().second.p;
    } else {
      // a new geometry: make room by evicting the least recently used ones if
      // the allocation fails (cudaFree waits for the work that reads them)
      DevBuf b;
      sbg_status sa = dev_alloc(ctx, b, gbytes);
      while (sa != SBG_OK && !gc.empty()) {
        ctx->err.clear();
        dev_free(ctx, gc.back().second);
        gc.pop_back();
        sa = dev_alloc(ctx, b, gbytes);
      }
      if (sa == SBG_OK) {
        for (int g = 0; g < ngroups; ++g) ST(gen_group(g, (float2*)b.p + (size_t)g * nb * ng));
        gc.insert(gc.begin(), {key, b});
        if ((int)gc.size() > sbg_context::kG2Cache) {
          dev_free(ctx, gc.back().second);
          gc.pop_back();
        }
        gbase = (const float2*)gc.front().second.p;
      } else {
        ctx->err.clear();  // regenerated per group below
      }
    }
  }
  const bool cached = gbase != nullptr;
  rec(ctx, 3);
  // ---- convolutions + 3PCF Grams of every field ----
  const int nsingle = ngroups4 * nb;
  const long long npts = (long long)nfld * ng;  // points of the slab
  float2* d_astore = nullptr;
  if (do4) ST(buf(ctx, "astore", (size_t)nsingle * npts * 8, (void**)&d_astore));
  float2* d_group;
  int per = 1;  // groups per launch
  ST(conv_buffer(ctx, nb, std::max(1, std::min(ngroups, 65535 / (nfld * nb))), nfld * ng * 8, &per, &d_group));
  if (!cached) per = 1;
  const bool together = do4 && per > 1;  // as in measure()
  const ConvTable conv = conv_table(2, nb, ngroups, ngroups4, together);
  FftXf* d_xf = nullptr;
  ST(conv_upload(ctx, conv, 2, nb, ngroups, ngroups4, together, &d_xf));
  float2* d_gtmp = nullptr;
  if (!cached) ST(buf(ctx, "gtmp", (size_t)nb * ng * 8, (void**)&d_gtmp));
  const int ngroups3 = do3 ? mmax + 1 : 0;
  const long long s_stride = (long long)std::max(ngroups3, 1) * nb * nb * 2;  // doubles of S per field
  double* d_S = nullptr;
  if (do3) {
    ST(buf(ctx, "S", (size_t)nfld * s_stride * 8, (void**)&d_S));
    CU(cudaMemsetAsync(d_S, 0, (size_t)nfld * s_stride * 8, st));
  }
  const bool tcomb = prec != SBG_PREC_FP32;
  const int tf32 = prec == SBG_PREC_TF32X3 ? 1 : 0;
  int* d_err = nullptr;
  if (tcomb) ST(buf(ctx, "err", 16, (void**)&d_err));  // cleared by the caller once per batch
  // (every group is stored, or none)
  auto gram = [&](int g0, int g1, bool stored) -> sbg_status {
    if (!do3 || g0 >= g1) return SBG_OK;
    double* Sg = d_S + (size_t)g0 * nb * nb * 2;
    const float2* src = stored ? d_astore : d_group;
    const int ns = stored ? nsingle : 0, s0 = stored ? g0 * nb : 0;
    if (tcomb)
      KL(launch_gram_tc(src, ng, nb, d_delta, Sg, ns, s0, tf32, d_err, ctx->nsm, ctx->wait_ns, ctx->stall, st, nfld,
                        s_stride, g1 - g0));
    else
      KL(launch_gram3(src, ng, nb, d_delta, Sg, ns, s0, st, nfld, s_stride, g1 - g0));
    return SBG_OK;
  };
  const float2* G = cached ? gbase : d_gtmp;
  int g0 = 0;
  if (together) {
    ST(conv_stored(ctx, 2, n, d_xf, conv, per * nb, G, d_dhat, d_tw, d_group, d_astore, nsingle, nfld));
    g0 = ngroups;
  }
  for (int g1; g0 < ngroups; g0 = g1) {
    g1 = do4 ? g0 + 1 : std::min(ngroups, g0 + per);
    const int t0 = conv.first[g0], t1 = conv.first[g1];
    const bool pairs = conv.real[g0];
    if (!cached) ST(gen_group(g0, d_gtmp));
    ST(conv_run(ctx, 2, n, d_xf, t0, t1, pairs ? LOAD_MUL2 : LOAD_MUL,
                cached && !pairs ? G + (long long)g0 * nb * ng : G, cached ? 0 : g0 * nb, d_dhat, d_tw, d_group, d_astore,
                nsingle, nfld));
    if (!do4) ST(gram(g0, g1, false));
  }
  if (do4) ST(gram(0, ngroups, true));
  rec(ctx, 4);
  rec(ctx, 5);
  // ---- 4PCF of every field ----
  double* d_z4 = nullptr;
  Tables4* t4 = nullptr;
  if (do4) {
    ST(ensure_tables4(ctx, 2, nb, mmax, tcomb, false));
    t4 = ctx->t4;
    Tables4& t = *t4;
    const long long tstride = std::max<long long>(t.tcount, 1);  // T entries per field (complex)
    double* d_T;
    ST(buf(ctx, "T", (size_t)nfld * tstride * 16, (void**)&d_T));
    CU(cudaMemsetAsync(d_T, 0, (size_t)nfld * tstride * 16, st));
    if (tcomb) {
      const int ntl = (int)t.tiles.size();
      const long long fkb = ng / 32;  // K-blocks of one field
      // x-splits per field: a power of two dividing its K-blocks, for the best
      // spread of the units over the CTAs
      // (the three best by their wave fill are timed by the autotuner on the
      // first slab of this size)
      std::vector<std::pair<double, int>> fill;
      for (int k = 1; k <= 16 && k <= fkb; k *= 2) {
        const long long units = (long long)ntl * nfld * k;
        const long long rounds = (units + ctx->nsm - 1) / ctx->nsm;
        fill.push_back({(double)units / (double)(rounds * ctx->nsm), k});
      }
      std::stable_sort(fill.begin(), fill.end(), [](const std::pair<double, int>& x, const std::pair<double, int>& y) {
        return x.first > y.first + 0.02;
      });
      std::vector<int> cands;
      for (size_t i = 0; i < fill.size() && cands.size() < 3; ++i) cands.push_back(fill[i].second);
      long long epochs = 4;
      for (int k : cands) {
        const long long units = (long long)ntl * nfld * k;
        const long long rounds = (units + ctx->nsm - 1) / ctx->nsm;
        epochs = std::max(epochs, rounds * ((fkb / k + kTcEpoch - 1) / kTcEpoch) + 4);
      }
      int* d_cnt;
      ST(buf(ctx, "tccnt", (size_t)epochs * 4, (void**)&d_cnt));
      void* d_bimg;
      ST(buf(ctx, "bimg", (size_t)(npts / 32) * (size_t)t.img_stride * (tf32 ? 2 : 1), &d_bimg));
      auto tc4_run = [&](int spf, double* T, cudaEvent_t e0, cudaEvent_t e1) -> cudaError_t {
        cudaError_t e = cudaMemsetAsync(d_cnt, 0, (size_t)epochs * 4, st);
        if (e != cudaSuccess) return e;
        return launch_tc4(d_astore, d_bimg, (const BGroup*)t.d_bgroups.p, (int)t.bgroups.size(), t.chunks_per_kb,
                          t.img_stride, d_delta, npts, (const Tile4*)t.d_tiles.p, ntl, (const Row4*)t.d_rows.p,
                          (const int*)t.d_cols.p, (const int*)t.d_uniq.p, nsingle, 1, nfld * spf, T, d_cnt, d_err,
                          ctx->nsm, st, e0, e1, tf32, ctx->wait_ns, ctx->stall, spf, tstride * 2);
      };
      int spf = cands[0];
      if (cands.size() > 1 && !ctx->stall) {
        char key[160];
        snprintf(key, sizeof key, "tc4slab/%d/%d/%d/%d/%d/%d", n, nb, mmax, (int)prec, ntl, nfld);
        double* d_Ts;
        ST(buf(ctx, "tuneT", (size_t)nfld * tstride * 16, (void**)&d_Ts));
        ST(autotune(ctx, key, cands, [&](int c) { return tc4_run(c, d_Ts, nullptr, nullptr); }, &spf));
      }
      ctx->nlaunch += 1;  // bimage_kernel
      KL(tc4_run(spf, d_T, ctx->kev[0], ctx->kev[1]));
      ctx->kev_used = true;
    } else {
      CU(cudaEventRecord(ctx->kev[0], st));
      ctx->kev_used = true;
      int launches = 0;
      CU(launch_simt4(d_astore, npts, d_delta, (const Tile4*)t.d_tiles.p, t.simt, (const Row4*)t.d_rows.p,
                      (const int*)t.d_cols.p, (const int*)t.d_uniq.p, 1, nsingle, d_T, ctx->nsm, st, &launches, nfld,
                      tstride * 2));
      ctx->nlaunch += launches;
      CU(cudaEventRecord(ctx->kev[1], st));
    }
    ST(buf(ctx, "z4", (size_t)nfld * t.nout * 16, (void**)&d_z4));
    KL(launch_couple(d_T, 1, (const int*)t.d_ptr.p, (const int*)t.d_idx.p, (const double*)t.d_coef.p, t.nout, d_z4, st,
                     nfld, tstride));
    if (flags & SBG_NORMALIZED) {
      const long long nouter = t.nout / ((long long)nb * nb * nb);
      KL(launch_normalize(d_z4, nouter, nb, 4, 2, d_acc, (double)ng, d_vb, st, nfld));
    }
  }
  rec(ctx, 6);
  // ---- 3PCF finish + downloads into the pinned slot ----
  const size_t z3b = do3 ? (size_t)(mmax + 1) * nb * nb * 16 : 0;
  const size_t z4b = do4 ? (size_t)t4->nout * 16 : 0;
  const size_t off4 = ((size_t)nfld * z3b + 255) / 256 * 256;
  if (do3) {
    double* d_z3;
    ST(buf(ctx, "z3", (size_t)nfld * z3b, (void**)&d_z3));
    KL(launch_finish3(d_S, 0, mmax, nb, d_z3, st, nfld, s_stride));
    if (flags & SBG_NORMALIZED) KL(launch_normalize(d_z3, mmax + 1, nb, 3, 2, d_acc, (double)ng, d_vb, st, nfld));
    CU(cudaMemcpyAsync(hslot, d_z3, (size_t)nfld * z3b, cudaMemcpyDeviceToHost, st));
  }
  if (do4) CU(cudaMemcpyAsync(hslot + off4, d_z4, (size_t)nfld * z4b, cudaMemcpyDeviceToHost, st));
  rec(ctx, 7);
  out->fields = fields;
  out->nfld = nfld;
  out->z3b = z3b;
  out->z4b = z4b;
  out->off4 = off4;
  out->host = hslot;
  tables.ok = true;
  return SBG_OK;
}

// Copies a slab's results from the pinned slot to the fields' arrays.
void slab_copy_out(const SlabOut& o) {
  std::vector<HostCopy> c;
  for (int i = 0; i < o.nfld; ++i) {
    if (o.z3b && o.fields[i].zeta3) c.push_back({o.fields[i].zeta3, o.host + (size_t)i * o.z3b, o.z3b});
    if (o.z4b && o.fields[i].zeta4) c.push_back({o.fields[i].zeta4, o.host + o.off4 + (size_t)i * o.z4b, o.z4b});
  }
  copy_out(c);
}

}  // namespace

// =================================================================== C ABI ==
extern "C" {

sbg_status sbg_create(int cuda_device, size_t hbm_budget_bytes, sbg_context** out) {
  if (!out) return SBG_ERR_INVALID_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
    cudaGetLastError();
    return SBG_ERR_CUDA;
  }
  if (cuda_device < 0 || cuda_device >= ndev) return SBG_ERR_INVALID_ARG;
  if (cudaSetDevice(cuda_device) != cudaSuccess) return SBG_ERR_CUDA;
  sbg_context* ctx = new sbg_context();
  ctx->device = cuda_device;
  ctx->budget = hbm_budget_bytes;
  cudaDeviceGetAttribute(&ctx->nsm, cudaDevAttrMultiProcessorCount, cuda_device);
  if (cudaStreamCreateWithFlags(&ctx->own, cudaStreamNonBlocking) != cudaSuccess) {
    delete ctx;
    return SBG_ERR_CUDA;
  }
  ctx->stream = ctx->own;
  for (int k = 0; k < 2; ++k) {
    for (int i = 0; i <= kStages; ++i) {
      if (cudaEventCreate(&ctx->evs[k][i]) != cudaSuccess) {
        sbg_destroy(ctx);
        return SBG_ERR_CUDA;
      }
    }
    for (int i = 0; i < 2; ++i) {
      if (cudaEventCreate(&ctx->kevs[k][i]) != cudaSuccess) {
        sbg_destroy(ctx);
        return SBG_ERR_CUDA;
      }
    }
  }
  *out = ctx;
  return SBG_OK;
}

void sbg_destroy(sbg_context* ctx) {
  if (!ctx) return;
  cudaSetDevice(ctx->device);
  if (ctx->stream) cudaStreamSynchronize(ctx->stream);
  for (auto& kv : ctx->bufs) dev_free(ctx, kv.second);
  dev_free(ctx, ctx->gcache);
  for (auto& kv : ctx->g2cache) dev_free(ctx, kv.second);
  ctx->g2cache.clear();
  for (auto& kv : ctx->t4cache) free_tables4(ctx, kv.second);
  ctx->t4cache.clear();
  ctx->t4 = nullptr;
  if (ctx->hpin) cudaFreeHost(ctx->hpin);
  for (int k = 0; k < 2; ++k) {
    for (int i = 0; i <= kStages; ++i)
      if (ctx->evs[k][i]) cudaEventDestroy(ctx->evs[k][i]);
    for (int i = 0; i < 2; ++i)
      if (ctx->kevs[k][i]) cudaEventDestroy(ctx->kevs[k][i]);
  }
  for (int i = 0; i < 2; ++i)
    if (ctx->tev[i]) cudaEventDestroy(ctx->tev[i]);
  if (ctx->own) cudaStreamDestroy(ctx->own);
  delete ctx;
}

sbg_status sbg_set_stream(sbg_context* ctx, void* cuda_stream) {
  if (!ctx) return SBG_ERR_INVALID_ARG;
  ctx->stream = cuda_stream ? (cudaStream_t)cuda_stream : ctx->own;
  return SBG_OK;
}

const char* sbg_status_string(sbg_status s) {
  switch (s) {
    case SBG_OK: return "SBG_OK";
    case SBG_ERR_INVALID_ARG: return "SBG_ERR_INVALID_ARG";
    case SBG_ERR_UNSUPPORTED_SHAPE: return "SBG_ERR_UNSUPPORTED_SHAPE";
    case SBG_ERR_BIN_RANGE: return "SBG_ERR_BIN_RANGE";
    case SBG_ERR_EMPTY_BIN: return "SBG_ERR_EMPTY_BIN";
    case SBG_ERR_OUT_OF_MEMORY: return "SBG_ERR_OUT_OF_MEMORY";
    case SBG_ERR_CUDA: return "SBG_ERR_CUDA";
    case SBG_ERR_TIMEOUT: return "SBG_ERR_TIMEOUT";
    case SBG_ERR_INTERNAL: return "SBG_ERR_INTERNAL";
  }
  return "SBG_UNKNOWN_STATUS";
}

const char* sbg_last_error(const sbg_context* ctx) { return ctx ? ctx->err.c_str() : "null context"; }

sbg_status sbg_lambda_count(int lmax, int* n_lambda) {
  if (!n_lambda || lmax < 0 || lmax > kMaxL3) return SBG_ERR_INVALID_ARG;
  int c = 0;
  for (int l1 = 0; l1 <= lmax; ++l1)
    for (int l2 = 0; l2 <= lmax; ++l2)
      for (int l3 = std::abs(l1 - l2); l3 <= std::min(l1 + l2, lmax); ++l3)
        if (!((l1 + l2 + l3) & 1)) ++c;
  *n_lambda = c;
  return SBG_OK;
}

sbg_status sbg_unique_bins(int nbins, int order, int* n_index, int* bins) {
  if (!n_index || nbins < 1 || nbins > kMaxBins || (order != 3 && order != 4)) return SBG_ERR_INVALID_ARG;
  int c = 0;
  for (int b1 = 0; b1 < nbins; ++b1)
    for (int b2 = b1 + 1; b2 < nbins; ++b2) {
      if (order == 3) {
        if (bins) {
          bins[2 * c] = b1;
          bins[2 * c + 1] = b2;
        }
        ++c;
        continue;
      }
      for (int b3 = b2 + 1; b3 < nbins; ++b3) {
        if (bins) {
          bins[3 * c] = b1;
          bins[3 * c + 1] = b2;
          bins[3 * c + 2] = b3;
        }
        ++c;
      }
    }
  *n_index = c;
  return SBG_OK;
}

sbg_status sbg_unique_gather(const double* zeta, long long nouter, int nbins, int order, int ncomp, double* out) {
  if (!zeta || !out || nouter < 0 || nbins < 1 || nbins > kMaxBins || (order != 3 && order != 4) ||
      (ncomp != 1 && ncomp != 2))
    return SBG_ERR_INVALID_ARG;
  const long long inner = order == 3 ? (long long)nbins * nbins : (long long)nbins * nbins * nbins;
  long long k = 0;
  for (long long o = 0; o < nouter; ++o) {
    const double* z = zeta + o * inner * ncomp;
    for (int b1 = 0; b1 < nbins; ++b1)
      for (int b2 = b1 + 1; b2 < nbins; ++b2) {
        if (order == 3) {
          for (int q = 0; q < ncomp; ++q) out[k++] = z[((long long)b1 * nbins + b2) * ncomp + q];
          continue;
        }
        for (int b3 = b2 + 1; b3 < nbins; ++b3)
          for (int q = 0; q < ncomp; ++q) out[k++] = z[(((long long)b1 * nbins + b2) * nbins + b3) * ncomp + q];
      }
  }
  return SBG_OK;
}

sbg_status sbg_lambda_odd_count(int lmax, int* n_lambda) {
  if (!n_lambda || lmax < 0 || lmax > kMaxL3) return SBG_ERR_INVALID_ARG;
  int c = 0;
  for (int l1 = 0; l1 <= lmax; ++l1)
    for (int l2 = 0; l2 <= lmax; ++l2)
      for (int l3 = std::abs(l1 - l2); l3 <= std::min(l1 + l2, lmax); ++l3)
        if ((l1 + l2 + l3) & 1) ++c;
  *n_lambda = c;
  return SBG_OK;
}

sbg_status sbg_lambda_odd_list(int lmax, int* l123) {
  if (!l123 || lmax < 0 || lmax > kMaxL3) return SBG_ERR_INVALID_ARG;
  int c = 0;
  for (int l1 = 0; l1 <= lmax; ++l1)
    for (int l2 = 0; l2 <= lmax; ++l2)
      for (int l3 = std::abs(l1 - l2); l3 <= std::min(l1 + l2, lmax); ++l3)
        if ((l1 + l2 + l3) & 1) {
          l123[3 * c] = l1;
          l123[3 * c + 1] = l2;
          l123[3 * c + 2] = l3;
          ++c;
        }
  return SBG_OK;
}

sbg_status sbg_lambda_list(int lmax, int* l123) {
  if (!l123 || lmax < 0 || lmax > kMaxL3) return SBG_ERR_INVALID_ARG;
  int c = 0;
  for (int l1 = 0; l1 <= lmax; ++l1)
    for (int l2 = 0; l2 <= lmax; ++l2)
      for (int l3 = std::abs(l1 - l2); l3 <= std::min(l1 + l2, lmax); ++l3)
        if (!((l1 + l2 + l3) & 1)) {
          l123[3 * c] = l1;
          l123[3 * c + 1] = l2;
          l123[3 * c + 2] = l3;
          ++c;
        }
  return SBG_OK;
}

sbg_status sbg_full(sbg_context* ctx, const void* field, sbg_dtype dtype, const int64_t shape[3], const double* edges,
                    int nbins, int lmax3, int lmax4, sbg_precision prec, unsigned flags, double* zeta3,
                    double* zeta4) {
  if (!ctx) return SBG_ERR_INVALID_ARG;
  ctx->err.clear();
  if (!field || !shape || !edges) return fail(ctx, SBG_ERR_INVALID_ARG, "null field, shape or edges");
  if (dtype != SBG_F32 && dtype != SBG_F64) return fail(ctx, SBG_ERR_INVALID_ARG, "dtype");
  if (prec != SBG_PREC_FP32 && prec != SBG_PREC_BF16X3 && prec != SBG_PREC_TF32X3)
    return fail(ctx, SBG_ERR_INVALID_ARG, "precision");
  if (flags & ~31u) return fail(ctx, SBG_ERR_INVALID_ARG, "unknown flag bits");
  if (!(flags & (SBG_3PCF | SBG_4PCF))) return fail(ctx, SBG_ERR_INVALID_ARG, "neither SBG_3PCF nor SBG_4PCF");
  if (nbins < 1 || nbins > kMaxBins) return fail(ctx, SBG_ERR_INVALID_ARG, "nbins must be 1..20");
  if ((flags & SBG_3PCF) && (lmax3 < 0 || lmax3 > kMaxL3 || !zeta3)) return fail(ctx, SBG_ERR_INVALID_ARG, "lmax3/zeta3");
  if ((flags & SBG_4PCF) && (lmax4 < 0 || lmax4 > kMaxL4 || !zeta4)) return fail(ctx, SBG_ERR_INVALID_ARG, "lmax4/zeta4");
  if (!(shape[0] == shape[1] && shape[1] == shape[2]) || !pow2_in(shape[0], 8, 512))
    return fail(ctx, SBG_ERR_UNSUPPORTED_SHAPE, "3D shape must be cubic with a power-of-two side in 8..512");
  const int n = (int)shape[0];
  ST(check_edges(ctx, edges, nbins, n));
  if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(ctx, SBG_ERR_CUDA, "cudaSetDevice");
  return measure(ctx, 3, field, dtype, n, edges, nbins, lmax3, lmax4, prec, flags, zeta3, zeta4);
}

sbg_status sbg_full_odd(sbg_context* ctx, const void* field, sbg_dtype dtype, const int64_t shape[3],
                        const double* edges, int nbins, int lmax4, sbg_precision prec, unsigned flags,
                        double* zeta4_odd) {
  if (!ctx) return SBG_ERR_INVALID_ARG;
  ctx->err.clear();
  if (!field || !shape || !edges || !zeta4_odd) return fail(ctx, SBG_ERR_INVALID_ARG, "null field, shape, edges or zeta4_odd");
  if (dtype != SBG_F32 && dtype != SBG_F64) return fail(ctx, SBG_ERR_INVALID_ARG, "dtype");
  if (prec != SBG_PREC_FP32 && prec != SBG_PREC_BF16X3 && prec != SBG_PREC_TF32X3)
    return fail(ctx, SBG_ERR_INVALID_ARG, "precision");
  if (flags & ~(unsigned)(SBG_NORMALIZED | SBG_SUBTRACT_MEAN | SBG_FIELD_ON_DEVICE))
    return fail(ctx, SBG_ERR_INVALID_ARG, "unknown flag bits");
  if (nbins < 1 || nbins > kMaxBins) return fail(ctx, SBG_ERR_INVALID_ARG, "nbins must be 1..20");
  if (lmax4 < 1 || lmax4 > kMaxL4) return fail(ctx, SBG_ERR_INVALID_ARG, "lmax4 must be 1..5 (odd Lambda need l >= 1)");
  if (!(shape[0] == shape[1] && shape[1] == shape[2]) || !pow2_in(shape[0], 8, 512))
    return fail(ctx, SBG_ERR_UNSUPPORTED_SHAPE, "3D shape must be cubic with a power-of-two side in 8..512");
  const int n = (int)shape[0];
  ST(check_edges(ctx, edges, nbins, n));
  if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(ctx, SBG_ERR_CUDA, "cudaSetDevice");
  return measure(ctx, 3, field, dtype, n, edges, nbins, 0, lmax4, prec, flags | SBG_4PCF, nullptr, zeta4_odd, true);
}

sbg_status sbg_projected(sbg_context* ctx, const void* field, sbg_dtype dtype, const int64_t shape[2],
                         const double* edges, int nbins, int mmax, sbg_precision prec, unsigned flags, double* zeta3,
                         double* zeta4) {
  if (!ctx) return SBG_ERR_INVALID_ARG;
  ctx->err.clear();
  if (!field || !shape || !edges) return fail(ctx, SBG_ERR_INVALID_ARG, "null field, shape or edges");
  if (dtype != SBG_F32 && dtype != SBG_F64) return fail(ctx, SBG_ERR_INVALID_ARG, "dtype");
  if (prec != SBG_PREC_FP32 && prec != SBG_PREC_BF16X3 && prec != SBG_PREC_TF32X3)
    return fail(ctx, SBG_ERR_INVALID_ARG, "precision");
  if (flags & ~31u) return fail(ctx, SBG_ERR_INVALID_ARG, "unknown flag bits");
  if (!(flags & (SBG_3PCF | SBG_4PCF))) return fail(ctx, SBG_ERR_INVALID_ARG, "neither SBG_3PCF nor SBG_4PCF");
  if (nbins < 1 || nbins > kMaxBins) return fail(ctx, SBG_ERR_INVALID_ARG, "nbins must be 1..20");
  if (mmax < 0 || mmax > kMaxM) return fail(ctx, SBG_ERR_INVALID_ARG, "mmax must be 0..10");
  if (((flags & SBG_3PCF) && !zeta3) || ((flags & SBG_4PCF) && !zeta4))
    return fail(ctx, SBG_ERR_INVALID_ARG, "null output for a requested statistic");
  if (shape[0] != shape[1] || !pow2_in(shape[0], 8, 1024))
    return fail(ctx, SBG_ERR_UNSUPPORTED_SHAPE, "2D shape must be square with a power-of-two side in 8..1024");
  const int n = (int)shape[0];
  ST(check_edges(ctx, edges, nbins, n));
  if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(ctx, SBG_ERR_CUDA, "cudaSetDevice");
  if (ctx->defer) return SBG_OK;  // checks only (a batch validates its fields first)
  return measure(ctx, 2, field, dtype, n, edges, nbins, mmax, mmax, prec, flags, zeta3, zeta4);
}

sbg_status sbg_projected_batch(sbg_context* ctx, const sbg_field2d* fields, int nfields, int nbins, int mmax,
                               sbg_precision prec, unsigned flags) {
  if (!ctx) return SBG_ERR_INVALID_ARG;
  ctx->err.clear();
  if (!fields || nfields < 1) return fail(ctx, SBG_ERR_INVALID_ARG, "fields/nfields");
  if (nbins < 1 || nbins > kMaxBins || mmax < 0) return fail(ctx, SBG_ERR_INVALID_ARG, "nbins/mmax");
  // every field is checked before any work is queued
  ctx->defer = true;
  for (int i = 0; i < nfields; ++i) {
    sbg_status s = sbg_projected(ctx, fields[i].field, fields[i].dtype, fields[i].shape, fields[i].edges, nbins, mmax,
                                 prec, flags, fields[i].zeta3, fields[i].zeta4);
    if (s != SBG_OK) {
      ctx->defer = false;
      ctx->err = "field " + std::to_string(i) + ": " + ctx->err;
      return s;
    }
  }
  ctx->defer = false;
  const bool do3 = flags & SBG_3PCF, do4 = flags & SBG_4PCF;
  const bool tcomb = prec != SBG_PREC_FP32;
  const int tf32 = prec == SBG_PREC_TF32X3 ? 1 : 0;
  // the 4PCF plan is shared by every field (one bin count, one order)
  if (do4) ST(ensure_tables4(ctx, 2, nbins, mmax, tcomb, false));
  const Tables4* t4 = do4 ? ctx->t4 : nullptr;
  const int nsingle = do4 ? (mmax + 1) * nbins : 0;
  const size_t z3b = do3 ? (size_t)(mmax + 1) * nbins * nbins * 16 : 0;
  const size_t z4b = do4 ? (size_t)t4->nout * 16 : 0;
  // Slabs: runs of consecutive fields with one shape, dtype and bin set, cut
  // so that a slab's buffers fit the device (or the context's budget), its
  // results a pinned staging slot of kSlotMax bytes, and its FFT batches the
  // grid's 65535 rows.
  constexpr size_t kSlotMax = 512ull << 20;
  size_t freeb = 0, totb = 0;
  cudaMemGetInfo(&freeb, &totb);
  size_t avail = (freeb > (4ull << 30) ? freeb - (4ull << 30) : freeb / 2) + ctx->used;
  if (ctx->budget) avail = std::min(avail, ctx->budget);
  avail = avail / 10 * 7;
  struct Slab {
    int i0, nf, n;
  };
  std::vector<Slab> slabs;
  auto same = [&](const sbg_field2d& a, const sbg_field2d& b) {
    if (a.dtype != b.dtype || a.shape[0] != b.shape[0]) return false;
    for (int k = 0; k <= nbins; ++k)
      if (a.edges[k] != b.edges[k]) return false;
    return true;
  };
  for (int i = 0; i < nfields;) {
    int j = i + 1;
    while (j < nfields && same(fields[i], fields[j])) ++j;
    const int n = (int)fields[i].shape[0];
    const size_t ng = (size_t)n * n;
    const size_t esz = fields[i].dtype == SBG_F64 ? 8 : 4;
    size_t per = ng * (esz + 4 + 8 + (size_t)nbins * 8) + 2 * z3b;
    if (do4) per += ng * ((size_t)nsingle * 8 + (size_t)(t4->img_stride + 31) / 32 * (tf32 ? 2 : 1)) +
                    (size_t)std::max<long long>(t4->tcount, 1) * 16 + 2 * z4b;
    int cap = (int)std::max<size_t>(1, avail / std::max<size_t>(per, 1));
    cap = std::min(cap, (int)std::max<size_t>(1, kSlotMax / std::max<size_t>(z3b + z4b, 1)));
    cap = std::min(cap, 65535 / nbins);
    for (int k = i; k < j; k += cap) slabs.push_back({k, std::min(cap, j - k), n});
    i = j;
  }
  size_t slot = 0;
  for (const Slab& sl : slabs) slot = std::max(slot, ((size_t)sl.nf * z3b + 255) / 256 * 256 + (size_t)sl.nf * z4b);
  slot = (slot + 255) / 256 * 256;
  unsigned char* hs;
  ST(host_staging(ctx, 64 + 2 * slot, (void**)&hs));
  int* d_err = nullptr;
  if (tcomb) {
    ST(buf(ctx, "err", 16, (void**)&d_err));
    CU(cudaMemsetAsync(d_err, 0, 16, ctx->stream));
  }
  // Slab c is queued in pinned slot c % 2 with event set c % 2; slab c - 1 is
  // completed (waited for, timed and copied out) after slab c is queued, so
  // the host's copies overlap the GPU's next slab.
  double acc[kStages] = {0};
  double kms = 0.0;
  long long nl = 0;
  SlabOut pend[2];
  bool live[2] = {false, false};
  bool kev_live[2] = {false, false};
  auto complete = [&](int sl) -> sbg_status {
    if (!live[sl]) return SBG_OK;
    live[sl] = false;
    CU(cudaEventSynchronize(ctx->evs[sl][kStages]));
    for (int k = 0; k < kStages; ++k) {
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, ctx->evs[sl][k], ctx->evs[sl][k + 1]) != cudaSuccess) {
        cudaGetLastError();
        ms = 0.f;
      }
      acc[k] += ms;
    }
    if (kev_live[sl]) {
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, ctx->kevs[sl][0], ctx->kevs[sl][1]) == cudaSuccess) kms += ms;
      else cudaGetLastError();
    }
    slab_copy_out(pend[sl]);
    return SBG_OK;
  };
  auto done = [&](sbg_status s) -> sbg_status {
    cudaStreamSynchronize(ctx->stream);
    ctx->ev = ctx->evs[0];
    ctx->kev = ctx->kevs[0];
    return s;
  };
  ctx->nlaunch = 0;
  for (size_t c = 0; c < slabs.size(); ++c) {
    const int sl = (int)(c & 1);
    ctx->ev = ctx->evs[sl];
    ctx->kev = ctx->kevs[sl];
    ctx->kev_used = false;
    const Slab& b = slabs[c];
    sbg_status s = measure_slab(ctx, fields + b.i0, b.nf, b.n, fields[b.i0].edges, nbins, mmax, prec, flags,
                                hs + 64 + (size_t)sl * slot, &pend[sl]);
    if (s != SBG_OK) {
      ctx->err = "fields " + std::to_string(b.i0) + ".." + std::to_string(b.i0 + b.nf - 1) + ": " + ctx->err;
      return done(s);
    }
    live[sl] = true;
    kev_live[sl] = ctx->kev_used;
    if (c > 0 && (s = complete(sl ^ 1)) != SBG_OK) return done(s);
  }
  sbg_status s = complete((int)((slabs.size() - 1) & 1));
  if (s != SBG_OK) return done(s);
  int herr = 0;
  if (tcomb) {
    int* perr = (int*)ctx->hpin;
    CU(cudaMemcpyAsync(perr, d_err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    done(SBG_OK);
    herr = *perr;
  } else {
    done(SBG_OK);
  }
  if (herr)
    return fail(ctx, SBG_ERR_TIMEOUT, "a tensor-core combination kernel gave up waiting (code " + std::to_string(herr) + ")");
  nl = ctx->nlaunch;
  for (int k = 0; k < kStages; ++k) ctx->timings[k] = acc[k];
  ctx->last_launches = nl;
  ctx->contraction_ms = kms;
  return SBG_OK;
}

sbg_status sbg_projected_slices(sbg_context* ctx, const void* cube, sbg_dtype dtype, const int64_t shape[3],
                                const double* edges, int nbins, int mmax, sbg_precision prec, unsigned flags,
                                double* zeta3, double* zeta4) {
  if (!ctx) return SBG_ERR_INVALID_ARG;
  ctx->err.clear();
  if (!cube || !shape || !edges) return fail(ctx, SBG_ERR_INVALID_ARG, "null cube, shape or edges");
  if (dtype != SBG_F32 && dtype != SBG_F64) return fail(ctx, SBG_ERR_INVALID_ARG, "dtype");
  if (shape[0] < 1 || shape[0] > 65536 || shape[1] < 1 || shape[2] < 1)
    return fail(ctx, SBG_ERR_UNSUPPORTED_SHAPE, "cube shape");
  if (((flags & SBG_3PCF) && !zeta3) || ((flags & SBG_4PCF) && !zeta4))
    return fail(ctx, SBG_ERR_INVALID_ARG, "zeta3/zeta4");
  // slice i = cube[i] (contiguous n1 x n2 block), outputs slice-major
  const size_t elem = dtype == SBG_F64 ? 8 : 4;
  const size_t w = 2 * (size_t)mmax + 1;
  const size_t s3 = (size_t)(mmax + 1) * nbins * nbins * 2, s4 = w * w * nbins * nbins * nbins * 2;
  std::vector<sbg_field2d> f((size_t)shape[0]);
  for (int64_t i = 0; i < shape[0]; ++i) {
    sbg_field2d& g = f[(size_t)i];
    g.field = (const unsigned char*)cube + (size_t)i * (size_t)shape[1] * (size_t)shape[2] * elem;
    g.dtype = dtype;
    g.shape[0] = shape[1];
    g.shape[1] = shape[2];
    g.edges = edges;
    g.zeta3 = (flags & SBG_3PCF) ? zeta3 + (size_t)i * s3 : nullptr;
    g.zeta4 = (flags & SBG_4PCF) ? zeta4 + (size_t)i * s4 : nullptr;
  }
  return sbg_projected_batch(ctx, f.data(), (int)shape[0], nbins, mmax, prec, flags);
}

sbg_status sbg_set_wait_limit(sbg_context* ctx, unsigned long long wait_ns, int test_stall) {
  if (!ctx) return SBG_ERR_INVALID_ARG;
  if (wait_ns == 0 || (test_stall != 0 && test_stall != 1)) return fail(ctx, SBG_ERR_INVALID_ARG, "bad wait limit");
  ctx->wait_ns = wait_ns;
  ctx->stall = test_stall;
  return SBG_OK;
}

sbg_status sbg_set_autotune(sbg_context* ctx, int enable) {
  if (!ctx) return SBG_ERR_INVALID_ARG;
  if (enable != 0 && enable != 1) return fail(ctx, SBG_ERR_INVALID_ARG, "enable must be 0 or 1");
  ctx->autotune_on = enable != 0;
  if (!ctx->autotune_on) ctx->tune.clear();
  return SBG_OK;
}

sbg_status sbg_autotune_report(const sbg_context* ctx, char* text, size_t len, size_t* needed) {
  if (!ctx) return SBG_ERR_INVALID_ARG;
  std::string r;
  for (const auto& kv : ctx->tune) r += kv.first + "=" + std::to_string(kv.second) + "\n";
  if (needed) *needed = r.size() + 1;
  if (text && len) {
    const size_t k = std::min(len - 1, r.size());
    std::memcpy(text, r.data(), k);
    text[k] = '\0';
  }
  return SBG_OK;
}

sbg_status sbg_last_timings(const sbg_context* ctx, double* ms_per_stage, int* n_stages) {
  if (!ctx || !ms_per_stage || !n_stages) return SBG_ERR_INVALID_ARG;
  for (int i = 0; i < kStages; ++i) ms_per_stage[i] = ctx->timings[i];
  ms_per_stage[kStages] = (double)ctx->last_launches;
  *n_stages = kStages + 1;
  return SBG_OK;
}

sbg_status sbg_last_contraction_ms(const sbg_context* ctx, double* ms) {
  if (!ctx || !ms) return SBG_ERR_INVALID_ARG;
  *ms = ctx->contraction_ms;
  return SBG_OK;
}

sbg_status sbg_plan4_info(int dim, int nbins, int lmax, sbg_precision prec, int odd, int* ntiles, int* nrows,
                          int* covering) {
  if ((dim != 2 && dim != 3) || nbins < 1 || nbins > kMaxBins || lmax < 0 || lmax > (dim == 3 ? kMaxL4 : kMaxM) ||
      (prec != SBG_PREC_FP32 && prec != SBG_PREC_BF16X3 && prec != SBG_PREC_TF32X3) || (odd != 0 && odd != 1) ||
      (odd && dim != 3))
    return SBG_ERR_INVALID_ARG;
  sbg_context host;  // receives the error text only: the tables stay on the host
  Tables4 t;
  const sbg_status s = build_tables4(&host, t, dim, nbins, lmax, prec != SBG_PREC_FP32, odd != 0, false);
  if (s != SBG_OK) return s;
  if (ntiles) *ntiles = (int)t.tiles.size();
  if (nrows) *nrows = (int)t.rows.size();
  if (covering) *covering = t.covering;
  return SBG_OK;
}

}  // extern "C"
