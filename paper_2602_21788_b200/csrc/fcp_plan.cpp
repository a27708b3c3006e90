// Host side of libfcp: the strategy planner (Sec. 4.4, Eq. 7, Algorithm 1) and the block plan that
// the kernels consume.  Plain C++, integers and doubles only; nothing here touches the GPU.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <functional>
#include <limits>
#include <memory>
#include <new>
#include <numeric>
#include <vector>

#include "fcp_plan.hpp"

namespace {
thread_local char g_err[512] = "";
}

void fcp_set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
}

extern "C" const char* fcp_last_error_message(void) { return g_err; }

extern "C" const char* fcp_status_string(int status) {
  switch (status) {
    case FCP_OK: return "FCP_OK";
    case FCP_ERR_INVALID_ARG: return "FCP_ERR_INVALID_ARG";
    case FCP_ERR_INFEASIBLE: return "FCP_ERR_INFEASIBLE";
    case FCP_ERR_UNSUPPORTED: return "FCP_ERR_UNSUPPORTED";
    case FCP_ERR_WORKSPACE: return "FCP_ERR_WORKSPACE";
    case FCP_ERR_CUDA: return "FCP_ERR_CUDA";
    case FCP_ERR_TIMEOUT: return "FCP_ERR_TIMEOUT";
    case FCP_ERR_NOT_UPLOADED: return "FCP_ERR_NOT_UPLOADED";
    case FCP_ERR_NO_MEMORY: return "FCP_ERR_NO_MEMORY";
    default: return "FCP_ERR_UNKNOWN";
  }
}

namespace {
// The two planners allocate by the size of the batch; no exception may leave a C entry point.
int no_memory(const char* call) {
  fcp_set_error("%s: the host's memory does not suffice for this batch", call);
  return FCP_ERR_NO_MEMORY;
}
}  // namespace

// ---------------------------------------------------------------------------------------------
// Strategy planner
// ---------------------------------------------------------------------------------------------
namespace {

struct GroupSums {  // sums over the sequences of one atomic group
  double quad = 0.0, lin = 0.0, tot = 0.0;
};

// T(G, d), Eq. 6: T_cp + T_cm - min(T_cpa, T_cma).  Eqs. 4-5 are written per group; the d ranks of
// a group share the compute terms, and ring communication only exists for d > 1.
double group_time(const GroupSums& g, int d, const fcp_cost_coeffs& c) {
  const double t_cpa = g.quad / d;
  const double t_cp = (g.quad + g.lin) / d + c.beta1;
  const double t_cm = d > 1 ? (c.alpha3 * g.tot) / c.v + c.beta2 : 0.0;
  const double t_cma = t_cm;
  return t_cp + t_cm - std::min(t_cpa, t_cma);
}

}  // namespace

extern "C" int fcp_plan_strategy(const int32_t* seqlens, int32_t B, int32_t N, double E,
                                 double M_token, double M_ms, const fcp_cost_coeffs* coeffs,
                                 int32_t* group_of, int32_t* cp_degree, int32_t* n_groups,
                                 double* makespan) try {
  if (!seqlens || !coeffs || B <= 0 || N <= 0 || !(E > M_ms) || !(M_token > 0.0) || !(coeffs->v > 0.0)) {
    fcp_set_error("fcp_plan_strategy: invalid argument");
    return FCP_ERR_INVALID_ARG;
  }
  if (N > FCP_MAX_DEGREE) {
    fcp_set_error("fcp_plan_strategy: N=%d exceeds FCP_MAX_DEGREE=%d", N, FCP_MAX_DEGREE);
    return FCP_ERR_UNSUPPORTED;
  }
  for (int i = 0; i < B; ++i)
    if (seqlens[i] <= 0) {
      fcp_set_error("fcp_plan_strategy: seqlens[%d]=%d", i, seqlens[i]);
      return FCP_ERR_INVALID_ARG;
    }

  // Stage 1: best-fit-decreasing.  Longest first (ties: lower index); a sequence goes to the open
  // group with the least remaining headroom that still holds it (ties: lowest group), otherwise it
  // opens a group of d_min = ceil(need / budget) ranks.
  const double budget = E - M_ms;
  std::vector<int> order(B);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return seqlens[a] > seqlens[b]; });
  std::vector<double> headroom;
  std::vector<int> dmin;
  std::vector<int> gof(B, 0);
  for (int i : order) {
    const double need = double(seqlens[i]) * M_token;
    int best = -1;
    for (int g = 0; g < (int)headroom.size(); ++g)
      if (headroom[g] >= need && (best < 0 || headroom[g] < headroom[best])) best = g;
    if (best < 0) {
      const int dm = std::max(1, (int)std::ceil(need / budget));
      headroom.push_back(dm * budget - need);
      dmin.push_back(dm);
      best = (int)headroom.size() - 1;
    } else {
      headroom[best] -= need;
    }
    gof[i] = best;
  }
  const int K = (int)dmin.size();
  long long need_ranks = 0;
  for (int d : dmin) need_ranks += d;
  if (need_ranks > N) {
    fcp_set_error("fcp_plan_strategy: minimum degrees need %lld ranks, only %d available", need_ranks, N);
    return FCP_ERR_INFEASIBLE;
  }

  // Per-group sums in sequence-index order.
  std::vector<GroupSums> sums(K);
  for (int i = 0; i < B; ++i) {
    const double L = double(seqlens[i]);
    const double eta = coeffs->eta ? coeffs->eta[i] : 0.0;
    GroupSums& g = sums[gof[i]];
    g.quad += coeffs->alpha1 * (1.0 + eta) * L * L;
    g.lin += coeffs->alpha2 * L;
    g.tot += L;
  }

  // Stage 2: the recurrence of Eq. 7, best[k][j] = min over d of max(best[k-1][j-d], T(G_k, d)), kept as two
  // rolling rows over j plus the arg-min of every (group, j) cell for the walk back.  A cell (k, j) is
  // reachable when the first k groups can have their minimum degrees (j >= lo[k]) and the remaining ones
  // still get theirs (j <= N - (need - lo[k])); d ranges over [d_min, j - lo[k-1]].  Ties keep the smallest
  // d (strict comparison, d ascending).  The answer is read at j = N: the strategy hands out every rank, as
  // the paper's text does ("backtrack from DP[K'][N]"; its case-study mixes add up to the rank count).
  // Because T(G, d) is not monotone in d once the ring term appears at d = 2, a plan that leaves ranks
  // idle could have a smaller makespan; that variant (min over j <= N) is not what the paper runs.
  const double INF = std::numeric_limits<double>::infinity();
  std::vector<int> lo(K + 1, 0);                 // lo[k] = sum of d_min over the first k groups
  for (int k = 0; k < K; ++k) lo[k + 1] = lo[k] + dmin[k];
  std::vector<double> prev(N + 1, INF), cur(N + 1, INF);
  std::vector<int> choice((size_t)K * (N + 1), 0);
  std::vector<double> tg(N + 1, 0.0);            // T(G_k, d) for the group at hand
  prev[0] = 0.0;
  for (int k = 0; k < K; ++k) {
    const int j_hi = N - ((int)need_ranks - lo[k + 1]);
    for (int d = dmin[k]; d <= j_hi - lo[k]; ++d) tg[d] = group_time(sums[k], d, *coeffs);
    std::fill(cur.begin(), cur.end(), INF);
    for (int j = lo[k + 1]; j <= j_hi; ++j) {
      double best = INF;
      int arg = 0;
      for (int d = dmin[k]; d <= j - lo[k]; ++d) {
        const double cand = std::max(prev[j - d], tg[d]);
        if (cand < best) {
          best = cand;
          arg = d;
        }
      }
      cur[j] = best;
      choice[(size_t)k * (N + 1) + j] = arg;
    }
    prev.swap(cur);
  }
  const double best_makespan = prev[N];
  std::vector<int> deg(K, 0);
  for (int k = K - 1, j = N; k >= 0; --k) {
    deg[k] = choice[(size_t)k * (N + 1) + j];
    j -= deg[k];
  }
  for (int i = 0; i < B; ++i) {
    if (group_of) group_of[i] = gof[i];
    if (cp_degree) cp_degree[i] = deg[gof[i]];
  }
  if (n_groups) *n_groups = K;
  if (makespan) *makespan = best_makespan;
  return FCP_OK;
} catch (const std::bad_alloc&) {
  return no_memory("fcp_plan_strategy");
}

// ---------------------------------------------------------------------------------------------
// Block plan
// ---------------------------------------------------------------------------------------------
namespace {

struct Pair {
  int32_t seq, rank, step, qc, kc, kind;
  bool operator<(const Pair& o) const {
    if (rank != o.rank) return rank < o.rank;
    if (step != o.step) return step < o.step;
    if (qc != o.qc) return qc < o.qc;
    return kc < o.kc;
  }
};

inline int ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

// Puts a unit list into execution order and describes it in work groups (fcp_plan.hpp).  Two things pull against each
// other.  Long units must come early, over all KV heads, or the last head's long units run alone at the end; and the
// CTAs that run together should share what one (sequence, KV head) keeps in L2: the K/V tiles of the forward pass, the
// dQ rows of the backward pass (reductions that miss the L2 run at less than half the speed).  So sequences go longest
// first, sequences whose data of one KV head fit kOrderBytes together form a group, as many KV heads as fit form a
// block, and within (group, block) the units go by cost.  Backward kernel, whole lists per KV head -> groups of 64 MB:
// 8K-token batch 341 -> 290 us, ragged 16K D = 64 225 -> 184 us, large batches unchanged.  Groups of 32 MB: 328 us, of
// 128 MB: 275 us but 128K bimodal batch +2 %; no limit (all heads by cost): 128K bimodal batch 93 -> 146 ms.
// The cheapest units of all sequences wait for the end, all KV heads together: they level out what the last block's
// long units leave uneven.  Half of the longest unit per SM is enough (simulated with measured unit times: 16K new
// batch 1421 us -> 1250 us for a mean of 1240, 8K batch 248 -> 226 for 220), at most 15 % of the work, and only where
// the longest unit is over a quarter of an SM's share: these units touch the ends of all sequences and share little (64K
// batch, 15 %: backward +2 % when they wait).  Measured: 8K step 501 -> 485 us, 16K new batch 2.50 -> 2.37 ms.
constexpr int64_t kOrderBytes = int64_t(64) << 20;
constexpr int64_t kOrderSms = FCP_PLAN_SMS;

// Stable sort of indexes by an ascending key of [0, n_keys), in two passes over the list.  The plan of a 16K-token batch of ten
// sequences, one of 8192 at degree 31 (1980 pairs, 1475 items, 1501 forward units), takes 145-160 us with it, 165-190 with std::stable_sort.
template <typename Key>
void sort_by_key(std::vector<int32_t>& order, size_t n_keys, Key key) {
  std::vector<int32_t> at(n_keys + 1, 0), out(order.size());
  for (int32_t i : order) ++at[key(i) + 1];
  for (size_t k = 1; k <= n_keys; ++k) at[k] += at[k - 1];
  for (int32_t i : order) out[at[key(i)]++] = i;
  order.swap(out);
}

void order_units(const std::vector<int32_t>& seq, const std::vector<int32_t>& cost, const int32_t* seqlens, int B,
                 int32_t heads, int64_t bytes_per_token, std::vector<int32_t>& order, std::vector<int32_t>& groups) {
  std::vector<int32_t> by_len(B), group_of(B), group_heads;
  std::iota(by_len.begin(), by_len.end(), 0);
  std::stable_sort(by_len.begin(), by_len.end(), [&](int a, int b) { return seqlens[a] > seqlens[b]; });
  int64_t bytes = 0;
  for (int i = 0; i < B; ++i) {
    const int64_t b = seqlens[by_len[i]] * bytes_per_token;
    if (i == 0 || bytes + b > kOrderBytes) {
      group_heads.push_back(1);
      bytes = 0;
    }
    bytes += b;
    group_of[by_len[i]] = (int32_t)group_heads.size() - 1;
    group_heads.back() = (int32_t)std::max<int64_t>(1, std::min<int64_t>(kOrderBytes / bytes, 1 << 16));
  }
  order.resize(seq.size());
  std::iota(order.begin(), order.end(), 0);
  std::vector<int32_t> unit_group(seq.size());
  for (size_t i = 0; i < seq.size(); ++i) unit_group[i] = group_of[seq[i]];
  const int32_t top = order.empty() ? 0 : *std::max_element(cost.begin(), cost.end());   // at most a sequence's tiles
  sort_by_key(order, (size_t)top + 1, [&](int32_t i) { return cost[i]; });
  {
    int64_t total = 0, late = 0;
    for (int32_t c : cost) total += c;
    const int64_t longest = kOrderSms * (order.empty() ? 0 : cost[order.back()]) / heads;   // on every SM, per KV head
    const int64_t most = 4 * longest > total ? std::min<int64_t>(longest / 2, total * 15 / 100) : 0;
    const int32_t last = (int32_t)group_heads.size();
    group_heads.push_back(1 << 16);
    for (int32_t i : order) {
      late += cost[i];
      if (late > most) break;
      unit_group[i] = last;
    }
  }
  std::iota(order.begin(), order.end(), 0);      // ties in list order, as the sort by cost leaves them
  sort_by_key(order, (size_t)top + 1, [&](int32_t i) { return top - cost[i]; });
  sort_by_key(order, group_heads.size(), [&](int32_t i) { return unit_group[i]; });
  for (size_t i = 0; i < order.size();) {
    size_t n = i;
    const int g = unit_group[order[i]];
    while (n < order.size() && unit_group[order[n]] == g) ++n;
    const int32_t row[FCP_WORK_GROUP_W] = {(int32_t)i, (int32_t)(n - i), group_heads[g], 0};
    groups.insert(groups.end(), row, row + FCP_WORK_GROUP_W);
    i = n;
  }
}

}  // namespace

// With fewer items than SMs every unit runs at once and the longest one is the launch.  Its two Q tiles as items of their
// own take a quarter less time, because a tile alone does not wait for the other one's turn in the MUFU and the tensor core;
// but with more than half as many units as SMs some SMs get a second item, which starts late, and the empty half of a unit
// with one tile holds up what comes behind it too.  Measured, whole against split (kernel, us; n units of sequences of L tokens):
//   D = 64:  L = 256, n = 74: 13.1, 12.8; n = 80: 13.2, 16.7; n = 144: 14.5, 17.7     L = 512, n = 80: equal; n = 144: 16.8, 18.9
//            L = 1024, n = 112: 23.0, 20.9; n = 144: 23.0, 23.1                       L = 2048, n = 144: 35.7, 32.2
//   D = 128: L = 256, n = 80: 14.8, 17.3; L = 1024, n = 112: 24.2, 22.9; n = 144: 24.8, 25.5; L = 2048, n = 144: 35.3, 34.8
// So both launches are played through, in quarters of the time of one key tile of a Q tile alone: a tile 4, a second item 12
// more (8 behind an empty half), a whole unit of two tiles 5 per key tile of the longer one and 6.  Over 224 measured lists of
// equal and unequal units this takes the slower launch, by over 3 %, once; always splitting does 62 times, by up to 30 %.
bool split_units(const std::vector<int32_t>& units, const std::vector<int32_t>& groups, int heads, int per, int sms) {
  const int64_t n_units = (int64_t)(units.size() / FCP_FWD_UNIT_W);
  if (n_units * heads * per >= sms) return false;
  std::vector<int64_t> busy;                     // when each SM is done (a heap, the earliest on top, once all have an item)
  int64_t split = 0, whole = 0;
  bool two = false;
  auto hand_out = [&](int64_t tiles) {
    const int64_t t = tiles > 0 ? 4 * tiles : 8;
    if ((int)busy.size() < sms) {
      busy.push_back(2 * t + (tiles > 0));       // lowest bit: the SM's last item was not an empty half
      std::push_heap(busy.begin(), busy.end(), std::greater<int64_t>());
    } else {
      std::pop_heap(busy.begin(), busy.end(), std::greater<int64_t>());
      busy.back() = 2 * (busy.back() / 2 + (busy.back() & 1 ? 12 : 0) + t) + (tiles > 0);
      std::push_heap(busy.begin(), busy.end(), std::greater<int64_t>());
    }
  };
  for (size_t g = 0; g < groups.size(); g += FCP_WORK_GROUP_W)
    for (int h0 = 0; h0 < heads; h0 += groups[g + WG_HEADS])                       // the order of WorkOrder::locate
      for (int32_t u = 0; u < groups[g + WG_N_UNITS]; ++u) {
        const int32_t* U = &units[(size_t)(groups[g + WG_FIRST] + u) * FCP_FWD_UNIT_W];
        const int32_t a = U[FU_NT_STAGE0], b = U[FU_NT_STAGE1], most = std::max(a, b);
        two = two || (a > 0 && b > 0);
        whole = std::max<int64_t>(whole, a > 0 && b > 0 ? 5 * most + 6 : 4 * most);
        for (int i = std::min(groups[g + WG_HEADS], heads - h0) * per; i > 0; --i) {
          hand_out(a);
          hand_out(b);
        }
      }
  for (int64_t t : busy)
    if (t & 1) split = std::max(split, t / 2);
  return two && split <= whole;
}

extern "C" int fcp_plan_blocks(const int32_t* seqlens, const int32_t* cp_degrees, int32_t B,
                               const fcp_params* params, fcp_plan** out) {
  return fcp_plan_blocks_spans(seqlens, cp_degrees, B, nullptr, nullptr, params, out);
}

extern "C" int fcp_plan_blocks_spans(const int32_t* seqlens, const int32_t* cp_degrees, int32_t B,
                                     const int32_t* span_offset, const int32_t* spans,
                                     const fcp_params* params, fcp_plan** out) try {
  if (!seqlens || !cp_degrees || !params || !out || B <= 0 || (span_offset && !spans && span_offset[B] > 0)) {
    fcp_set_error("fcp_plan_blocks: invalid argument");
    return FCP_ERR_INVALID_ARG;
  }
  *out = nullptr;
  if ((params->head_dim != 64 && params->head_dim != 128) || params->hq <= 0 || params->hkv <= 0 ||
      params->hq % params->hkv != 0) {
    fcp_set_error("fcp_plan_blocks: unsupported shape hq=%d hkv=%d head_dim=%d", params->hq, params->hkv,
                  params->head_dim);
    return FCP_ERR_UNSUPPORTED;
  }
  int64_t T = 0;
  int32_t max_len = 0;
  for (int b = 0; b < B; ++b) {
    if (seqlens[b] <= 0 || cp_degrees[b] <= 0) {
      fcp_set_error("fcp_plan_blocks: sequence %d has length %d, degree %d", b, seqlens[b], cp_degrees[b]);
      return FCP_ERR_INVALID_ARG;
    }
    if (cp_degrees[b] > FCP_MAX_DEGREE) {
      fcp_set_error("fcp_plan_blocks: degree %d > FCP_MAX_DEGREE", cp_degrees[b]);
      return FCP_ERR_UNSUPPORTED;
    }
    T += seqlens[b];
    max_len = std::max(max_len, seqlens[b]);
  }
  if (T >= (int64_t(1) << 31) - 2 * FCP_FWD_UNIT_ROWS) {
    fcp_set_error("fcp_plan_blocks: %lld tokens exceed the 2^31 limit", (long long)T);
    return FCP_ERR_INVALID_ARG;
  }

  std::unique_ptr<fcp_plan> owner(new fcp_plan());
  fcp_plan* const p = owner.get();
  p->params = *params;
  if (!(p->params.scale > 0.f)) p->params.scale = 1.0f / std::sqrt((float)params->head_dim);
  p->B = B;
  p->T = T;
  p->max_seqlen = max_len;
  p->cu_seqlens.assign(B + 1, 0);
  for (int b = 0; b < B; ++b) p->cu_seqlens[b + 1] = p->cu_seqlens[b] + seqlens[b];

  // Bidirectional spans: query t sees the keys before row_limit[t]; key t is seen from query
  // first_query[t] on (both in packed-token indices, both non-decreasing within a sequence).
  const bool has_spans = span_offset != nullptr && span_offset[B] > span_offset[0];
  if (has_spans) {
    p->span_offset.assign(span_offset, span_offset + B + 1);
    p->spans.assign(spans, spans + 2 * (size_t)span_offset[B]);
    p->row_limit.resize(T);
    p->first_query.resize(T);
    for (int64_t t = 0; t < T; ++t) {
      p->row_limit[t] = (int32_t)t + 1;
      p->first_query[t] = (int32_t)t;
    }
    for (int b = 0; b < B; ++b) {
      int32_t prev_end = 0;
      if (span_offset[b + 1] < span_offset[b]) {
        fcp_set_error("fcp_plan_blocks_spans: span_offset decreases at sequence %d", b);
        return FCP_ERR_INVALID_ARG;
      }
      for (int32_t i = span_offset[b]; i < span_offset[b + 1]; ++i) {
        const int32_t a = spans[2 * i], e = spans[2 * i + 1];
        if (a < prev_end || e <= a || e > seqlens[b]) {
          fcp_set_error("fcp_plan_blocks_spans: span [%d, %d) of sequence %d (length %d) is empty, out of range, "
                        "unsorted or overlaps the one before", a, e, b, seqlens[b]);
          return FCP_ERR_INVALID_ARG;
        }
        prev_end = e;
        const int32_t t0 = p->cu_seqlens[b];
        for (int32_t t = a; t < e; ++t) {
          p->row_limit[t0 + t] = t0 + e;
          p->first_query[t0 + t] = t0 + a;
        }
      }
    }
  }

  // Chunk bounds and pairs.
  p->chunk_offset.push_back(0);
  std::vector<Pair> pairs;
  {
    size_t n_pairs = 0;
    for (int b = 0; b < B; ++b) {                // a short sequence has one token in each of L chunks, the others are empty
      const size_t n = std::min(2 * cp_degrees[b], seqlens[b]);
      n_pairs += n * (n + 1) / 2;
    }
    pairs.reserve(n_pairs);
  }
  for (int b = 0; b < B; ++b) {
    const int64_t L = seqlens[b];
    const int d = cp_degrees[b];
    const int32_t t0 = p->cu_seqlens[b];
    const size_t base = p->chunk_bounds.size();
    for (int c = 0; c <= 2 * d; ++c) p->chunk_bounds.push_back(t0 + (int32_t)((int64_t)c * L / (2 * d)));
    p->chunk_offset.push_back((int32_t)p->chunk_bounds.size());
    auto nonempty = [&](int c) { return p->chunk_bounds[base + c + 1] > p->chunk_bounds[base + c]; };
    auto add = [&](int r, int s, int qc, int kc) {
      if (nonempty(qc) && nonempty(kc)) pairs.push_back(Pair{b, r, s, qc, kc, qc == kc ? 1 : 0});
    };
    const int last = 2 * d - 1;
    for (int r = 0; r < d; ++r) {
      if (!nonempty(r) && !nonempty(last - r)) continue;   // all but L ranks of a sequence of L < d tokens
      for (int s = 0; s < d; ++s) {              // the pairs of a step ascend as they are written here: r, j < d <= last - r, last - j
        const int j = r >= s ? r - s : r - s + d;   // rank whose K/V visits at this ring step
        if (s == 0) {
          add(r, s, r, r);
          add(r, s, last - r, r);
          add(r, s, last - r, last - r);
        } else if (j < r) {
          add(r, s, r, j);
          add(r, s, last - r, j);
        } else {
          add(r, s, last - r, j);
          add(r, s, last - r, last - j);
        }
      }
    }
  }
  p->pairs.resize(pairs.size() * 6);
  for (size_t i = 0; i < pairs.size(); ++i) {
    const Pair& x = pairs[i];
    const int32_t row[6] = {x.seq, x.rank, x.step, x.qc, x.kc, x.kind};
    std::copy(row, row + 6, &p->pairs[i * 6]);
  }
  // Block pairs above the chunk diagonal that a span makes necessary: (q_chunk, kv_chunk > q_chunk) such that
  // a span reaches into both.  The rank that owns q_chunk computes it when the owner of kv_chunk visits.
  if (has_spans) {
    for (int b = 0; b < B; ++b) {
      const int d = cp_degrees[b];
      const int32_t* cbp = &p->chunk_bounds[p->chunk_offset[b]];
      const int32_t t0 = cbp[0];
      std::vector<Pair> sp;
      auto owner = [&](int c) { return c < d ? c : 2 * d - 1 - c; };
      for (int qc = 0; qc < 2 * d; ++qc)
        for (int kc = qc + 1; kc < 2 * d; ++kc) {
          bool hit = false;
          for (int32_t i = span_offset[b]; i < span_offset[b + 1] && !hit; ++i) {
            const int32_t a = t0 + spans[2 * i], e = t0 + spans[2 * i + 1];
            hit = std::max(a, cbp[qc]) < std::min(e, cbp[qc + 1]) && std::max(a, cbp[kc]) < std::min(e, cbp[kc + 1]);
          }
          if (hit) {
            const int r = owner(qc);
            sp.push_back(Pair{b, r, ((r - owner(kc)) % d + d) % d, qc, kc, 2});
          }
        }
      std::sort(sp.begin(), sp.end());
      for (const Pair& x : sp) {
        const int32_t row[5] = {x.seq, x.rank, x.step, x.qc, x.kc};
        p->span_pairs.insert(p->span_pairs.end(), row, row + 5);
      }
    }
  }

  p->items.reserve(pairs.size() * 8);            // at most one per pair
  // Items: one per (seq, rank, step, q_chunk); slot = order of the step among the steps touching
  // that Q chunk; partial rows are laid out in item order.
  const int n_chunks_total = p->chunk_offset[B] - B;  // sum of 2d
  std::vector<int32_t> chunk_index0(B + 1, 0);        // global chunk index of chunk 0 of each sequence
  for (int b = 0; b < B; ++b) chunk_index0[b + 1] = chunk_index0[b] + 2 * cp_degrees[b];
  std::vector<std::vector<std::pair<int, int>>> chunk_items(n_chunks_total);  // (step, item index)
  int64_t row = 0;
  for (size_t i = 0; i < pairs.size();) {
    size_t n = 1;
    while (i + n < pairs.size() && pairs[i + n].seq == pairs[i].seq && pairs[i + n].rank == pairs[i].rank &&
           pairs[i + n].step == pairs[i].step && pairs[i + n].qc == pairs[i].qc)
      ++n;
    const Pair& x = pairs[i];
    const int item = (int)(p->items.size() / 8);
    const int32_t cb = p->chunk_offset[x.seq] + x.qc;
    const int32_t len = p->chunk_bounds[cb + 1] - p->chunk_bounds[cb];
    const int32_t rowv[8] = {x.seq, x.rank, x.step, x.qc, 0, (int32_t)row, (int32_t)n, (int32_t)i};
    p->items.insert(p->items.end(), rowv, rowv + 8);
    chunk_items[chunk_index0[x.seq] + x.qc].push_back({x.step, item});
    row += len;
    if (row >= (int64_t(1) << 31) - 2 * FCP_FWD_UNIT_ROWS) {
      fcp_set_error("fcp_plan_blocks: partial rows exceed the 2^31 limit");
      return FCP_ERR_INVALID_ARG;
    }
    i += n;
  }
  p->R = row;
  p->slot_offset.push_back(0);
  for (int c = 0; c < n_chunks_total; ++c) {
    auto& v = chunk_items[c];
    std::sort(v.begin(), v.end());
    for (size_t k = 0; k < v.size(); ++k) {
      p->items[(size_t)v[k].second * 8 + 4] = (int32_t)k;
      p->slot_rows.push_back(p->items[(size_t)v[k].second * 8 + 5]);
    }
    p->slot_offset.push_back((int32_t)p->slot_rows.size());
  }

  // ---- derived work lists (execution order; not part of the canonical tables) ----
  // Forward: an item's Q chunk is cut into units of two adjacent 128-row tiles.  KV ranges of an
  // item are its pairs in kv_chunk order, so a DIAG range (kv_chunk == q_chunk) is always last.
  struct FU { int32_t f[FCP_FWD_UNIT_W]; };
  std::vector<FU> fus;
  std::vector<int32_t> fu_seq;
  const int64_t kv_token_bytes = (int64_t)params->head_dim * 4;                                   // K and V, bf16
  const int64_t dq_token_bytes = (int64_t)params->head_dim * 4 * (params->hq / params->hkv);      // fp32 dQ rows
  auto emit_fwd = [&](const std::vector<FU>& units, const std::vector<int32_t>& seq, std::vector<int32_t>& rows,
                      std::vector<int32_t>& groups) {
    std::vector<int32_t> cost, order;
    cost.reserve(units.size());
    for (const FU& u : units) cost.push_back(u.f[FU_NT_STAGE0] + u.f[FU_NT_STAGE1]);
    order_units(seq, cost, seqlens, B, params->hkv, kv_token_bytes, order, groups);
    rows.resize(units.size() * FCP_FWD_UNIT_W);
    for (size_t i = 0; i < order.size(); ++i) std::copy(units[order[i]].f, units[order[i]].f + FCP_FWD_UNIT_W, &rows[i * FCP_FWD_UNIT_W]);
  };
  const int n_items = (int)(p->items.size() / 8);
  fus.reserve(n_items);
  fu_seq.reserve(n_items);
  for (int it = 0; it < n_items; ++it) {
    const int32_t* I = &p->items[(size_t)it * 8];
    const int b = I[0], qc = I[3], np = I[6], fp = I[7];
    const int32_t* cbp = &p->chunk_bounds[p->chunk_offset[b]];
    const int32_t q0 = cbp[qc], q1 = cbp[qc + 1];
    int32_t kb[2] = {0, 0}, ke[2] = {0, 0}, kd[2] = {0, 0};
    for (int r = 0; r < np; ++r) {
      const Pair& x = pairs[fp + r];
      kb[r] = cbp[x.kc];
      ke[r] = cbp[x.kc + 1];
      kd[r] = x.kind;
    }
    const int last = np - 1;
    const int nt_first = np == 2 ? ceil_div(ke[0] - kb[0], FCP_TILE) : 0;
    for (int32_t off = 0; off < q1 - q0; off += FCP_FWD_UNIT_ROWS) {
      FU u{};
      const int32_t rows = std::min<int32_t>(FCP_FWD_UNIT_ROWS, q1 - q0 - off);
      u.f[FU_Q_ROW0] = q0 + off;
      u.f[FU_Q_ROWS] = rows;
      u.f[FU_PART_ROW0] = I[5] + off;
      u.f[FU_N_RANGES] = np;
      u.f[FU_KV0_BEGIN] = kb[0]; u.f[FU_KV0_END] = ke[0]; u.f[FU_KV0_DIAG] = kd[0];
      u.f[FU_KV1_BEGIN] = kb[1]; u.f[FU_KV1_END] = ke[1]; u.f[FU_KV1_DIAG] = kd[1];
      for (int s = 0; s < 2; ++s) {
        const int32_t rs = std::min<int32_t>(FCP_TILE, rows - s * FCP_TILE);
        int nt = 0;
        if (rs > 0) {
          if (kd[last]) nt = ceil_div((int64_t)off + s * FCP_TILE + rs, FCP_TILE);  // keys up to the last row
          else nt = ceil_div(ke[last] - kb[last], FCP_TILE);
          nt += nt_first;
        }
        u.f[FU_NT_STAGE0 + s] = nt;
      }
      u.f[FU_NT_RANGE0] = np == 2 ? nt_first : 0x7fffffff;
      u.f[FU_ITEM] = it;
      {
        const int ci = chunk_index0[b] + qc;   // a Q chunk with one slot needs no merge
        u.f[FU_SINGLE_SLOT] = p->slot_offset[ci + 1] - p->slot_offset[ci] == 1;
      }
      fus.push_back(u);
      fu_seq.push_back(b);
    }
  }
  emit_fwd(fus, fu_seq, p->fwd_units, p->fwd_groups);
  p->fwd_split = split_units(p->fwd_units, p->fwd_groups, params->hkv, params->hq / params->hkv, FCP_PLAN_SMS);

  // Fused forward (merge on the fly): all items of a Q chunk run on one CTA, so the KV ranges of the
  // chunk's block pairs are swept in one online softmax and no partial leaves the SM.  The pairs of a
  // Q chunk are every chunk with tokens before it and the DIAG pair of the chunk itself; every key
  // before the chunk precedes every row of it, so one DIAG range from the sequence start describes
  // them exactly, and the chunks of a sequence are one run of rows, tiled in units of two Q tiles
  // from its start: no tile is cut at a chunk edge.  Inside a span a row sees keys up to the span's end.
  {
    std::vector<FU> gus;
    std::vector<int32_t> gu_seq;
    for (int b = 0; b < B; ++b) {
      const int32_t t0 = p->cu_seqlens[b], t1 = p->cu_seqlens[b + 1];
      for (int32_t row0 = t0; row0 < t1; row0 += FCP_FWD_UNIT_ROWS) {
        FU u{};
        const int32_t rows = std::min<int32_t>(FCP_FWD_UNIT_ROWS, t1 - row0);
        u.f[FU_Q_ROW0] = row0;
        u.f[FU_Q_ROWS] = rows;
        u.f[FU_N_RANGES] = 1;
        u.f[FU_KV0_BEGIN] = t0; u.f[FU_KV0_END] = t1; u.f[FU_KV0_DIAG] = 1;
        for (int s = 0; s < 2; ++s) {
          const int32_t rs = std::min<int32_t>(FCP_TILE, rows - s * FCP_TILE);
          if (rs <= 0) continue;
          // key tiles up to the last key the stage's last row sees (row limits do not decrease along a sequence)
          const int32_t last_row = row0 + s * FCP_TILE + rs - 1;
          u.f[FU_NT_STAGE0 + s] = ceil_div((has_spans ? p->row_limit[last_row] : last_row + 1) - t0, FCP_TILE);
        }
        u.f[FU_NT_RANGE0] = 0x7fffffff;
        u.f[FU_ITEM] = -1;
        u.f[FU_SINGLE_SLOT] = 1;
        gus.push_back(u);
        gu_seq.push_back(b);
      }
    }
    emit_fwd(gus, gu_seq, p->fused_units, p->fused_groups);
    p->fused_split = split_units(p->fused_units, p->fused_groups, params->hkv, params->hq / params->hkv, FCP_PLAN_SMS);
  }

  // Backward: one unit per 128-key tile; it visits the Q rows of all block pairs whose kv_chunk holds
  // its keys, that is of its own chunk (DIAG) and of every later one: one DIAG range from the chunk
  // start to the sequence end.  So the key tiles are cut from the start of the sequence instead of
  // from each chunk start (a key tile may then span two KV chunks; the causal mask only depends on
  // token positions): neither key tiles nor query tiles are cut at chunk edges, and a query tile has
  // the same rows for every key tile, by which the dQ accumulator is laid out.
  {
    std::vector<int32_t> seq, cost;
    for (int b = 0; b < B; ++b) {
      const int32_t t0 = p->cu_seqlens[b], t1 = p->cu_seqlens[b + 1];
      const int32_t rowq[FCP_BWD_QRANGE_W] = {t0, t1, 1, 0};
      p->bwd_qranges.insert(p->bwd_qranges.end(), rowq, rowq + FCP_BWD_QRANGE_W);
      for (int32_t k0 = t0, t = 0; k0 < t1; k0 += FCP_TILE, ++t) {
        const int32_t rows = std::min<int32_t>(FCP_TILE, t1 - k0);
        // Q tiles run from T_FIRST on; those before T_MASK_END hold (query, key) pairs the mask removes.  Causal: the tile on
        // the diagonal only.  With spans a tile is first seen where its first key is (earlier than the tile's own position
        // when that key lies inside a span).
        const int32_t t_first = has_spans ? (p->first_query[k0] - t0) / FCP_TILE : t;
        const int32_t t_mask_end = has_spans ? ceil_div(p->first_query[k0 + rows - 1] - t0, FCP_TILE) : t + 1;
        const int32_t tiles = ceil_div(t1 - t0, FCP_TILE) - t_first;
        int32_t u[FCP_BWD_UNIT_W] = {};
        u[BU_KV_ROW0] = k0;
        u[BU_KV_ROWS] = rows;
        u[BU_FIRST_QRANGE] = b;
        u[BU_N_QRANGES] = 1;
        u[BU_T_FIRST] = t_first;
        u[BU_COST] = tiles;
        u[BU_SEQ] = b;
        u[BU_T_MASK_END] = t_mask_end;
        p->bwd_units.insert(p->bwd_units.end(), u, u + FCP_BWD_UNIT_W);
        seq.push_back(b);
        cost.push_back(tiles);
      }
    }
    order_units(seq, cost, seqlens, B, params->hkv, dq_token_bytes, p->bwd_work, p->bwd_groups);
  }

  // Merge: runs of up to FCP_MERGE_TOKENS tokens inside one chunk.  Chunks with two or more slots
  // come first: a forward pass that writes the single-slot chunks straight to the output only needs
  // the first n_merge_multi units merged.
  for (int pass = 0; pass < 2; ++pass) {
    for (int b = 0; b < B; ++b) {
      const int32_t* cbp = &p->chunk_bounds[p->chunk_offset[b]];
      for (int c = 0; c < 2 * cp_degrees[b]; ++c) {
        const int ci = chunk_index0[b] + c;
        const bool single = p->slot_offset[ci + 1] - p->slot_offset[ci] <= 1;
        if (single != (pass == 1)) continue;
        for (int32_t t = cbp[c]; t < cbp[c + 1]; t += FCP_MERGE_TOKENS) {
          const int32_t rowm[4] = {t, std::min<int32_t>(FCP_MERGE_TOKENS, cbp[c + 1] - t), ci, cbp[c]};
          p->merge_units.insert(p->merge_units.end(), rowm, rowm + 4);
        }
      }
    }
    if (pass == 0) p->n_merge_multi = (int32_t)(p->merge_units.size() / FCP_MERGE_UNIT_W);
  }
  *out = owner.release();
  return FCP_OK;
} catch (const std::bad_alloc&) {
  return no_memory("fcp_plan_blocks");
}

extern "C" int fcp_span_mask_efficiency(int32_t length, const int32_t* spans, int32_t n_spans, double* eta) {
  if (length <= 0 || !eta || n_spans < 0 || (n_spans > 0 && !spans)) {
    fcp_set_error("fcp_span_mask_efficiency: invalid argument");
    return FCP_ERR_INVALID_ARG;
  }
  // a span of m tokens adds the m(m-1)/2 pairs above its diagonal to the L(L+1)/2 causal ones
  double extra = 0.0;
  int32_t prev_end = 0;
  for (int i = 0; i < n_spans; ++i) {
    const int32_t a = spans[2 * i], e = spans[2 * i + 1];
    if (a < prev_end || e <= a || e > length) {
      fcp_set_error("fcp_span_mask_efficiency: span [%d, %d) is empty, out of range, unsorted or overlapping", a, e);
      return FCP_ERR_INVALID_ARG;
    }
    prev_end = e;
    const double m = double(e - a);
    extra += m * (m - 1.0) / 2.0;
  }
  *eta = extra / (double(length) * (double(length) + 1.0) / 2.0);
  return FCP_OK;
}

extern "C" int fcp_plan_get(const fcp_plan* plan, int32_t which, const int32_t** host_ptr, int64_t* count) {
  if (!plan || !host_ptr || !count) return FCP_ERR_INVALID_ARG;
  const std::vector<int32_t>* v = nullptr;
  switch (which) {
    case FCP_TABLE_CU_SEQLENS: v = &plan->cu_seqlens; break;
    case FCP_TABLE_CHUNK_OFFSET: v = &plan->chunk_offset; break;
    case FCP_TABLE_CHUNK_BOUNDS: v = &plan->chunk_bounds; break;
    case FCP_TABLE_PAIRS: v = &plan->pairs; break;
    case FCP_TABLE_ITEMS: v = &plan->items; break;
    case FCP_TABLE_SLOT_OFFSET: v = &plan->slot_offset; break;
    case FCP_TABLE_SLOT_ROWS: v = &plan->slot_rows; break;
    case FCP_TABLE_FWD_UNITS: v = &plan->fwd_units; break;
    case FCP_TABLE_BWD_UNITS: v = &plan->bwd_units; break;
    case FCP_TABLE_BWD_QRANGES: v = &plan->bwd_qranges; break;
    case FCP_TABLE_MERGE_UNITS: v = &plan->merge_units; break;
    case FCP_TABLE_BWD_WORK: v = &plan->bwd_work; break;
    case FCP_TABLE_FUSED_UNITS: v = &plan->fused_units; break;
    case FCP_TABLE_ROW_LIMIT: v = &plan->row_limit; break;
    case FCP_TABLE_FIRST_QUERY: v = &plan->first_query; break;
    case FCP_TABLE_FWD_GROUPS: v = &plan->fwd_groups; break;
    case FCP_TABLE_FUSED_GROUPS: v = &plan->fused_groups; break;
    case FCP_TABLE_BWD_GROUPS: v = &plan->bwd_groups; break;
    case FCP_TABLE_SPAN_PAIRS: v = &plan->span_pairs; break;
    default: fcp_set_error("fcp_plan_get: unknown table %d", which); return FCP_ERR_INVALID_ARG;
  }
  *host_ptr = v->data();
  *count = (int64_t)v->size();
  return FCP_OK;
}

extern "C" int fcp_plan_info(const fcp_plan* plan, int32_t which, int64_t* value) {
  if (!plan || !value) return FCP_ERR_INVALID_ARG;
  switch (which) {
    case 0: *value = plan->T; break;
    case 1: *value = plan->R; break;
    case 2: *value = (int64_t)plan->pairs.size() / 6; break;
    case 3: *value = (int64_t)plan->items.size() / 8; break;
    case 4: *value = (int64_t)plan->fwd_units.size() / FCP_FWD_UNIT_W; break;
    case 5: *value = (int64_t)plan->bwd_units.size() / FCP_BWD_UNIT_W; break;
    case 6: *value = (int64_t)plan->merge_units.size() / FCP_MERGE_UNIT_W; break;
    case 7: *value = plan->B; break;
    case 8: *value = plan->n_merge_multi; break;
    case 9: *value = (int64_t)plan->fused_units.size() / FCP_FWD_UNIT_W; break;
    case 10: *value = plan->fused_split; break;
    default: return FCP_ERR_INVALID_ARG;
  }
  return FCP_OK;
}
