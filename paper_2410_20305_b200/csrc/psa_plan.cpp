// Host planner: block-sparsity tile map of the prefix-sharing mask with packing
// (Algorithm 3), built once per step and reused by every layer (Section 3.1).
//
// Tiles are 128 x 128 and aligned to each sample's first token, so that within a
// sample query tile i and key tile j cover local rows [128 i, 128 i + 128) and
// [128 j, 128 j + 128).  In local coordinates (cs = P, rs = P + C, len = P+C+R)
// the mask is:  kv <= q  and not (q >= rs and cs <= kv < rs).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <numeric>
#include <utility>
#include <vector>

#include "psa_internal.h"

namespace psa {

BwdWorkspace bwd_workspace_layout(int64_t T, int Hq, int d) {
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  BwdWorkspace w{};
  int64_t Tpad = (T + kTile - 1) / kTile * kTile + kTile;
  w.dq_accum_off = 0;
  w.dq_accum_bytes = up(size_t(T) * Hq * d * sizeof(float));
  w.delta_off = w.dq_accum_off + w.dq_accum_bytes;
  w.delta_bytes = up(size_t(Hq) * Tpad * sizeof(float));
  w.total = w.delta_off + w.delta_bytes;
  return w;
}

namespace {

// Classification of tile pair (i, j) of one sample.  Returns 0 = dropped,
// 1 = live and full, 2 = live and needs masking.  `bwd` also requires the rows
// past the sample's end (ragged last query tile) to be masked.
int classify(int i, int j, int len, int cs, int rs, bool bwd) {
  if (j > i) return 0;
  const int q0 = i * kTile, q1 = std::min(q0 + kTile, len);  // valid query rows
  const int k0 = j * kTile, k1 = std::min(k0 + kTile, len);  // valid key rows
  if (j == i) return 2;  // the diagonal tile always holds the row's own key
  // j < i: causality holds for every pair.  Forbidden rectangle: q >= rs, cs <= kv < rs.
  const bool rows_all_rejected = q0 >= rs;
  const bool rows_some_rejected = q1 > rs;        // q1 - 1 >= rs
  const bool keys_all_chosen = k0 >= cs && k1 <= rs;
  const bool keys_some_chosen = k1 > cs && k0 < rs;
  if (rows_all_rejected && keys_all_chosen) return 0;
  bool partial = rows_some_rejected && keys_some_chosen;
  if (bwd && q0 + kTile > len) partial = true;
  return partial ? 2 : 1;
}

// A query tile is PRECISE when one of its rows sees fewer than 128 keys.  Such rows
// have large probabilities, whose bf16 rounding dominates the error of dK and dV;
// the kernels carry P and dS of these tiles as a sum of two bf16 terms.
bool precise_rows(int i, int len, int cs, int rs) {
  if (i == 0) return true;                          // row 0 sees one key
  const int q0 = i * kTile, q1 = std::min(q0 + kTile, len);
  const int q = std::max(q0, rs);                   // first rejected row of the tile, if any
  return q < q1 && cs + (q - rs + 1) < kTile;       // it sees the prompt and q - rs + 1 own keys
}

// Work items that a CTA of the forward takes.  Two pay the CTA's fixed costs once for both; one each spreads the items
// over more of the CTAs that the chip holds at a time (two per SM), and a launch lasts at least as long as its longest
// CTA.  In key tiles, with 3.5 for an item's fixed costs: two, where the share of a resident CTA is at least 94 % of two
// longest items.  Over 300 packs drawn from long prompts, short samples, single samples (450 to 2400 items) the rule is
// 0.18 % behind the better of the two, more than 2 % in 11 of them and 7 % in one; a line at 1184 items is 0.56 % behind,
// more than 2 % in 27 and 13 % in one.  (A simulation of both launches: 0.10 %, more than 2 % in 6; not worth its time.)
// us with one / two:
//   3876 tokens, 32/8 heads of 128, lists of 2.5 (1152 items) 43.8 / 40.6    8158, 16 of 64, 2.8 (1136) 36.7 / 32.6
//   858 tokens, 32/8 of 128, 2.6 (256) 14.0 / 21.4           7763, 8/2 of 128, lists of 1 to 24 (496) 48.3 / 82.4
//   16629, 8/2 of 128, 1 to 36 (1080) 100.1 / 129.0    21996, 8/2 of 128, 1 to 32 (1416) 114.8 / 124.2
//   5061, 32/8 of 128 (1312) 100.4 / 96.6              31041, 32/8 of 128 (7904) 1019 / 965
void items_per_cta(const psa_plan_t* p, int n_sm, PlanPart* part) {
  if (part->n_q_tiles == 0) return;
  const TileRec* tiles = p->q_tiles.data() + part->q_tile0;
  int64_t work = 0;
  for (int32_t i = 0; i < part->n_q_tiles; ++i) work += (2 * tiles[i].list_cnt + 7) * int64_t(p->Hq);
  const int64_t two_longest = 2 * (2 * int64_t(tiles[0].list_cnt) + 7);
  part->fwd_items_per_cta = work * 100 >= 94 * 2 * int64_t(n_sm) * two_longest ? 2 : 1;
}

// List scheduling on `n` slots: every pair goes to the slot that is free first.
struct Slots {
  std::vector<int64_t> free_at;   // a heap, earliest first
  std::vector<int64_t> scratch;
  int64_t end = 0;                // when the last pair so far ends
  bool sorted = true;             // free_at ascends as a whole

  explicit Slots(size_t n = 0) : free_at(n, 0) {}

  void take(int64_t cost) {
    const size_t n = free_at.size();
    const int64_t t = free_at[0] + cost;   // the earliest slot takes the pair and sinks to its new place
    end = std::max(end, t);
    size_t i = 0;
    for (size_t k = 1; k < n; k = 2 * i + 1) {
      if (k + 1 < n && free_at[k + 1] < free_at[k]) ++k;
      if (free_at[k] >= t) break;
      free_at[i] = free_at[k];
      i = k;
    }
    free_at[i] = t;
    sorted = false;
  }

  // `count` pairs of one cost.  Many at a time: the slots that are taken ascend, and so do their new times, so that the next
  // one is the smaller head of two ascending rows.
  void take_equal(int32_t count, int64_t cost) {
    if (count < 32) {
      for (; count > 0; --count) take(cost);
      return;
    }
    if (!sorted) std::sort(free_at.begin(), free_at.end());
    sorted = true;
    const size_t n = free_at.size();
    scratch.resize(size_t(count) + n);
    int64_t* const taken = scratch.data();
    size_t i = 0, j = 0;
    for (size_t k = 0; k < size_t(count); ++k)
      taken[k] = cost + (i < n && (j == k || free_at[i] <= taken[j]) ? free_at[i++] : taken[j++]);
    end = std::max(end, taken[count - 1]);
    std::merge(free_at.begin() + i, free_at.end(), taken + j, taken + count, taken + count);
    std::copy(taken + count, taken + count + n, free_at.begin());
  }
};

// Launch order of the backward for the samples [s0, s1), appended to the plan's list, and the number of CTAs that share
// the iterations of one (key tile, kv head) pair.
//
// Order: every CTA adds its dQ contributions into the fp32 accumulator rows of its sample and query-head group, so CTAs
// that share those rows are launched together: the rows then stay in L2 while they are being updated.  Samples with
// the most work first, then kv head, then the sample's key tiles, longest list first.  That can leave a ragged tail, so
// the end of the order is handed out longest first: the last wave and a bit (115 % of one pair per SM), or, where the
// whole accumulator stays in L2 anyway, 30 %, 50 % or all of it, whichever a list-scheduling simulation finds shortest.
// It has to be 1.5 % shorter than the grouped order.  us of the whole backward with the last 0 / 5 / 10 / 20 / 30 / 100 %
// longest first (before: 30 %, where that was 5 % shorter in the simulation):
//   31041 tokens, 32/8 heads of 128 (13 waves)  2398 / 2352 / 2366 / 2458 / 2512 / 2598
//   19431, 32/8 of 128 (8)    1039 / 1031 / 1015 / 1028 / 1046 / 1107     16215, 32/8 of 128 (7)  892 / 893 / 871 / 850 / 864 / 930
//   7727, 32/8 of 128 (3.7)   226 / 224 / 223 / 218 / 211 / 227           accumulators of 19 to 42 MB:
//   4952, 8/8 of 128 (2.2)    109 / 110 / 106 / 101 / 96 / 91             5465, 32/8 of 64 (2.4)  223 / 222 / 217 / 204 / 191 / 166
//
// The simulation costs no more than the order is worth to a step that plans for itself (psa_plan and psa_plan_destroy on
// the host, us: 7965 tokens, 16/16 heads of 64, 242 -> 50; 31041, 32/8 of 128, 290 -> 154): the shares have the grouped order's start in
// common, which is simulated once, and a sorted end is runs of equal pairs; sorting and simulating the order for each share
// was the difference.
void order_backward(psa_plan_t* p, const std::vector<std::vector<int32_t>>& tiles_of, int s0, int s1, int n_sm,
                    PlanPart* part) {
  struct Pair {
    int32_t tile, kv_head, len;   // key tile record, kv head, length of the tile's list
  };
  std::vector<int64_t> work(s1 - s0, 0);
  size_t n_pairs = 0;
  for (int s = s0; s < s1; ++s) {
    for (int32_t t : tiles_of[s]) work[s - s0] += p->kv_tiles[t].list_cnt;
    n_pairs += tiles_of[s].size() * size_t(p->Hkv);
  }
  std::vector<int> order(s1 - s0);
  std::iota(order.begin(), order.end(), s0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return work[a - s0] > work[b - s0]; });
  std::vector<Pair> pairs;   // grouped, until the end of this function
  pairs.reserve(n_pairs);
  int64_t total_work = 0, squares = 0;
  int32_t longest = 0;
  for (int s : order)
    for (int hk = 0; hk < p->Hkv; ++hk)
      for (int32_t t : tiles_of[s]) {
        const int32_t n = p->kv_tiles[t].list_cnt;
        pairs.push_back(Pair{t, hk, n});
        total_work += n;
        squares += int64_t(n) * n;
        longest = std::max(longest, n);
      }
  part->bwd_long_lists = total_work > 0 && squares >= kLongLists * total_work;
  const int64_t iter_ns = p->d == 128 ? 2050 : 1600, fixed_ns = p->d == 128 ? 8000 : 7000, combine_ns = 3000;
  const int64_t group = p->Hq / p->Hkv;
  auto alone = [&](int32_t n) { return n * group * iter_ns + fixed_ns; };

  // First pair of the longest-first end that holds the last `permille` of the work.
  auto end_of = [&](int64_t permille) {
    int64_t acc = 0;
    size_t at = 0;
    while (at < pairs.size() && acc * 1000 < total_work * (1000 - permille)) acc += pairs[at++].len;
    return at;
  };
  size_t sorted_from = pairs.size();
  int64_t best = 0;
  const bool whole = part == &p->whole;
  if (pairs.size() <= size_t(n_sm)) {
    best = alone(longest);
  } else if (whole) {
    // Candidates: first pairs of the sorted ends, in the order in which they are preferred.
    size_t candidates[4], n_candidates = 0;
    const bool in_l2 = int64_t(p->T) * p->Hq * p->d * 4 <= (int64_t(64) << 20);
    const int64_t wave = std::min<int64_t>(1000, 1150 * int64_t(n_sm) / int64_t(pairs.size()));
    candidates[n_candidates++] = end_of(wave);
    if (in_l2)
      for (int64_t permille : {300, 500, 1000}) candidates[n_candidates++] = end_of(permille);
    // One pass over the grouped order, which stops at every candidate's start to keep the slots as they are there.
    Slots slots(n_sm), at_start[4];
    for (size_t i = 0; i < pairs.size(); ++i) {
      for (size_t c = 0; c < n_candidates; ++c)
        if (candidates[c] == i) at_start[c] = slots;
      slots.take(alone(pairs[i].len));
    }
    best = slots.end;
    // No order is shorter than the mean load or the longest pair.
    const int64_t least = std::max((total_work * group * iter_ns + int64_t(pairs.size()) * fixed_ns) / n_sm, alone(longest));
    int64_t shortest = best * 985 / 1000;
    std::vector<int32_t> of_length(longest + 1);
    for (size_t c = 0; c < n_candidates && least < shortest; ++c) {
      if (candidates[c] == pairs.size()) continue;
      std::fill(of_length.begin(), of_length.end(), 0);
      for (size_t i = candidates[c]; i < pairs.size(); ++i) ++of_length[pairs[i].len];
      for (int32_t n = longest; n > 0; --n) at_start[c].take_equal(of_length[n], alone(n));
      const int64_t t = at_start[c].end;
      if (t >= shortest) continue;
      shortest = best = t;
      sorted_from = candidates[c];
    }
  }
  // CTAs per pair: where the pairs are few, the longest of them lasts longer than the rest of the chip is busy.  Sharing
  // a pair costs each of its CTAs the fixed part of a CTA and the reduction over the cluster, so it only pays below two
  // pairs per SM.  Of 148 SMs clusters of 2, 4 and 8 reach 148, 132 and 120.  us of the whole backward, split 1 / 2 / 4 / 8:
  //   436 tokens, 8/2 heads of 128 (8 pairs)        53 / 37 / 25 / 24     1814 tokens, 8/2 of 64 (34)      62 / 38 / 26 / 40
  //   3160 tokens, 8/2 heads of 64 (50)             261 / 108 / 59 / 82   11799 tokens, 8/2 of 128 (186)   818 / 645 / 660 / 794
  //   16700 tokens, 8/2 heads of 128 (262)          1383 / 1262 / 1374 / 1482 in short runs, 1376 / 1389 in long ones,
  //   where the power limit sets the clock: a prediction of less than 10 % is not worth it.
  //   5061 tokens, 32/8 heads of 128 (328)          264 / 270 / 354 / 575
  if (!whole) {
    part->bwd_split = p->whole.bwd_split;   // dk and dv are summed in the same order, and come out the same, as for the whole
  } else if (pairs.size() <= 2 * size_t(n_sm)) {
    // Pairs that share their iterations are few, and handed out longest first as a whole (2008 tokens, 32/8 heads of 128,
    // 145 -> 103 us; 2436 tokens, 32/8 of 64, 151 -> 110), also where the simulation has the grouped order 2 % shorter (1429
    // tokens, 32/8 of 128, 82.4 against 86.5; 2299, 32/8 of 64, 65.6 against 69.2).  What sharing takes is judged by the
    // shorter of the two simulated times, although one order is launched: by the launched order's alone four CTAs become two
    // in 73 of 40000 packs, which takes 0.96 to 1.25 times as long, 1.08 in the middle (4400 tokens, 8/2 of 64, 59 -> 70).
    // Where only the sorted order makes sharing worth while, lists of less than 20 iterations have to gain a quarter, which
    // errs on the side of one CTA per pair: of 518 packs of up to 296 pairs the choice differs from 10 % throughout on two
    // (1375 tokens, 32/8 of 128, 69.6 us with one CTA, 51.3 with two; 1682 tokens, 8/8 of 128, 45.3 and 39.0).
    const int64_t need = longest * group >= 20 ? 90 : 75;
    std::vector<int32_t> of_length(longest + 1, 0);
    for (const Pair& c : pairs) ++of_length[c.len];
    for (int split : {2, 4, 8}) {
      const size_t n_slots = std::max(1, split == 2 ? n_sm / 2 : (split == 4 ? n_sm * 33 / 148 : n_sm * 15 / 148));
      auto shared = [&](int32_t n) { return (n * group + split - 1) / split * iter_ns + fixed_ns + combine_ns; };
      int64_t grouped = shared(longest), sorted = grouped;
      if (pairs.size() > n_slots) {
        Slots in_turn(n_slots), longest_first(n_slots);
        for (const Pair& c : pairs) in_turn.take(shared(c.len));
        for (int32_t n = longest; n > 0; --n) longest_first.take_equal(of_length[n], shared(n));
        grouped = in_turn.end;
        sorted = longest_first.end;
      }
      if (grouped * 100 < best * 90 || sorted * 100 < best * need) {
        best = std::min(grouped, sorted);
        part->bwd_split = split;
      }
    }
    if (part->bwd_split > 1) sorted_from = 0;
  }
  part->cta0 = int32_t(p->bwd_cta_map.size() / 2);
  part->n_ctas = int32_t(pairs.size());
  std::stable_sort(pairs.begin() + sorted_from, pairs.end(), [](const Pair& a, const Pair& b) { return a.len > b.len; });
  p->bwd_cta_map.reserve(p->bwd_cta_map.size() + pairs.size() * 2);
  for (const Pair& c : pairs) {
    p->bwd_cta_map.push_back(c.tile);
    p->bwd_cta_map.push_back(c.kv_head);
  }
}

}  // namespace
}  // namespace psa

using psa::kTile;
using psa::TileRec;

extern "C" const char* psa_status_string(psa_status_t s) {
  switch (s) {
    case PSA_OK: return "ok";
    case PSA_ERR_INVALID_ARG: return "invalid argument";
    case PSA_ERR_INCONSISTENT_LENGTHS: return "cu_seqlens inconsistent with prefix/chosen/rejected lengths";
    case PSA_ERR_UNSUPPORTED: return "unsupported configuration";
    case PSA_ERR_ALIGNMENT: return "device pointer not 16-byte aligned";
    case PSA_ERR_CUDA: return "CUDA call failed";
    case PSA_ERR_DEVICE_STATUS: return "kernel reported bad data";
    case PSA_ERR_TIMEOUT: return "bounded device wait expired";
  }
  return "unknown status";
}

extern "C" psa_status_t psa_plan(const int32_t* cu_seqlens, const int32_t* prefix_len,
                                 const int32_t* chosen_len, const int32_t* rejected_len,
                                 int32_t n_samples, int32_t n_q_heads, int32_t n_kv_heads,
                                 int32_t head_dim, float softmax_scale, int32_t flags,
                                 void* stream, psa_plan_t** out) {
  if (!out) return PSA_ERR_INVALID_ARG;
  *out = nullptr;
  if (n_samples < 0 || !cu_seqlens) return PSA_ERR_INVALID_ARG;
  if (n_samples > 0 && (!prefix_len || !chosen_len || !rejected_len)) return PSA_ERR_INVALID_ARG;
  if (n_q_heads <= 0 || n_kv_heads <= 0) return PSA_ERR_INVALID_ARG;
  if (flags & ~PSA_PLAN_HOST_ONLY) return PSA_ERR_INVALID_ARG;
  if (n_q_heads % n_kv_heads != 0) return PSA_ERR_UNSUPPORTED;
  if (head_dim != 64 && head_dim != 128) return PSA_ERR_UNSUPPORTED;
  if (cu_seqlens[0] != 0) return PSA_ERR_INCONSISTENT_LENGTHS;
  for (int s = 0; s < n_samples; ++s) {
    if (prefix_len[s] < 0 || chosen_len[s] < 0 || rejected_len[s] < 0) return PSA_ERR_INVALID_ARG;
    int64_t tot = int64_t(prefix_len[s]) + chosen_len[s] + rejected_len[s];
    if (int64_t(cu_seqlens[s + 1]) - cu_seqlens[s] != tot) return PSA_ERR_INCONSISTENT_LENGTHS;
  }
  // Row indices, and row*heads products used for grid sizes, stay in int32.
  if (int64_t(cu_seqlens[n_samples]) > (int64_t(1) << 30)) return PSA_ERR_UNSUPPORTED;

  psa_plan_t* p = new (std::nothrow) psa_plan_t;
  if (!p) return PSA_ERR_INVALID_ARG;
  p->n_samples = n_samples;
  p->T = cu_seqlens[n_samples];
  p->Hq = n_q_heads;
  p->Hkv = n_kv_heads;
  p->d = head_dim;
  p->scale = softmax_scale > 0.f ? softmax_scale : 1.0f / std::sqrt(float(head_dim));

  for (int s = 0; s < n_samples; ++s) {
    const int P = prefix_len[s], C = chosen_len[s], R = rejected_len[s];
    const int len = P + C + R, cs = P, rs = P + C, ds = cu_seqlens[s];
    p->useful_pairs += int64_t(P + C) * (P + C + 1) / 2 + int64_t(R) * P + int64_t(R) * (R + 1) / 2;
    const int nt = (len + kTile - 1) / kTile;
    for (int i = 0; i < nt; ++i) {  // forward: query tile i, its key tiles in ascending order
      TileRec r{ds + i * kTile, ds, i * kTile, len, cs, rs, int32_t(p->fwd_entries.size()), 0};
      for (int j = 0; j <= i; ++j) {
        int c = psa::classify(i, j, len, cs, rs, false);
        if (!c) continue;
        p->fwd_entries.push_back((j << 2) | (int(psa::precise_rows(i, len, cs, rs)) << 1) | (c == 2));
        ++r.list_cnt;
        ++p->live_tiles;
        p->partial_tiles += (c == 2);
      }
      p->q_tiles.push_back(r);
    }
    for (int j = 0; j < nt; ++j) {  // transposed: key tile j, its query tiles in ascending order
      TileRec r{ds + j * kTile, ds, j * kTile, len, cs, rs, int32_t(p->bwd_entries.size()), 0};
      for (int i = j; i < nt; ++i) {
        int c = psa::classify(i, j, len, cs, rs, true);
        if (!c) continue;
        p->bwd_entries.push_back((i << 2) | (int(psa::precise_rows(i, len, cs, rs)) << 1) | (c == 2));
        ++r.list_cnt;
      }
      p->kv_tiles.push_back(r);
    }
    // Rejected rows past the first query tile that see fewer than kFewKeys keys (only a sample
    // with a prompt shorter than that has any).
    for (int q = std::max(rs, kTile); q < len && P + (q - rs + 1) < psa::kFewKeys; ++q)
      p->few_key_rows.push_back(psa::FewKeyRow{ds + q, ds, P, ds + rs});
  }
  // Longest list first: the hardware hands out CTAs in index order, so the long
  // work items start early and the short ones fill the tail.
  auto longest_first = [](const TileRec& a, const TileRec& b) { return a.list_cnt > b.list_cnt; };
  std::stable_sort(p->q_tiles.begin(), p->q_tiles.end(), longest_first);
  std::stable_sort(p->kv_tiles.begin(), p->kv_tiles.end(), longest_first);
  p->bwd_workspace_bytes = psa::bwd_workspace_layout(p->T, p->Hq, p->d).total;
  {
    int n_sm = 148;
    if (!(flags & PSA_PLAN_HOST_ONLY)) {
      int dev = 0, v = 0;
      if (cudaGetDevice(&dev) == cudaSuccess &&
          cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
        n_sm = v;
    }
    p->n_sm = n_sm;
    // Key tiles of every sample, longest list first.
    std::vector<std::vector<int32_t>> tiles_of(n_samples);
    for (size_t t = 0; t < p->kv_tiles.size(); ++t) {
      // the sample is found from its start row (cu_seqlens is increasing over non-empty samples)
      const int32_t ds = p->kv_tiles[t].ds;
      int s = int(std::upper_bound(cu_seqlens, cu_seqlens + n_samples + 1, ds) - cu_seqlens) - 1;
      while (s + 1 < n_samples && cu_seqlens[s + 1] == ds) ++s;   // skip zero-length samples
      tiles_of[s].push_back(int32_t(t));
    }
    p->whole.row1 = p->T;
    p->whole.n_q_tiles = int32_t(p->q_tiles.size());
    p->whole.n_few = int32_t(p->few_key_rows.size());
    psa::items_per_cta(p, n_sm, &p->whole);
    psa::order_backward(p, tiles_of, 0, n_samples, n_sm, &p->whole);

    // Parts for psa_step_host: runs of whole samples of about a sixth of the pack (4 to 24 differ by 5 %; with more
    // parts the copies get too short for the link) and of at least 2 MB of q, which the link takes 40 us for.  A
    // smaller pack has none: its copies take less time than the overlap costs the host.
    const int64_t row_bytes = int64_t(p->Hq) * p->d * 2, least_bytes = int64_t(2) << 20;
    const int64_t least = std::max(int64_t(p->T) / 6, (least_bytes + row_bytes - 1) / row_bytes);
    std::vector<int> first{0};   // first sample of each part
    for (int s = 0; s < n_samples; ++s)
      if (cu_seqlens[s + 1] - cu_seqlens[first.back()] >= least || s + 1 == n_samples) first.push_back(s + 1);
    if (first.size() > 2) {
      const size_t n_whole = p->q_tiles.size();
      for (size_t i = 0; i + 1 < first.size(); ++i) {
        psa::PlanPart w;
        w.row0 = cu_seqlens[first[i]];
        w.row1 = cu_seqlens[first[i + 1]];
        if (w.row1 == w.row0) continue;
        w.q_tile0 = int32_t(p->q_tiles.size());
        for (size_t t = 0; t < n_whole; ++t) {   // (still longest list first)
          const TileRec r = p->q_tiles[t];
          if (r.row0 >= w.row0 && r.row0 < w.row1) p->q_tiles.push_back(r);
        }
        w.n_q_tiles = int32_t(p->q_tiles.size()) - w.q_tile0;
        const int32_t n_few = int32_t(p->few_key_rows.size());
        while (w.few0 < n_few && p->few_key_rows[w.few0].row < w.row0) ++w.few0;
        while (w.few0 + w.n_few < n_few && p->few_key_rows[w.few0 + w.n_few].row < w.row1) ++w.n_few;
        psa::items_per_cta(p, n_sm, &w);
        psa::order_backward(p, tiles_of, first[i], first[i + 1], n_sm, &w);
        p->parts.push_back(w);
      }
    } else if (int64_t(p->T) * row_bytes >= least_bytes) {
      p->parts.push_back(p->whole);
    }
  }

  if (!(flags & PSA_PLAN_HOST_ONLY)) {
    psa_status_t st = psa_plan_upload(p, stream);
    if (st != PSA_OK) {
      delete p;
      return st;
    }
  }
  *out = p;
  return PSA_OK;
}

namespace {
// Process-wide cache of plan blobs.  An entry is a device allocation, a pinned staging buffer of
// the same size and two events: `copied` (the last upload has been read out of the staging buffer)
// and `last_use` (every kernel that read the device blob under its previous owner has finished).
struct BlobEntry {
  int device = -1;
  void* dptr = nullptr;
  void* hptr = nullptr;
  size_t capacity = 0;
  cudaEvent_t copied = nullptr, last_use = nullptr;
  bool last_use_valid = false;
};
constexpr size_t kBlobCacheMax = 16;
std::mutex g_blob_mutex;
std::vector<BlobEntry> g_blob_cache;

void free_entry(BlobEntry& e) {
  if (e.dptr) cudaFree(e.dptr);
  if (e.hptr) cudaFreeHost(e.hptr);
  if (e.copied) cudaEventDestroy(e.copied);
  if (e.last_use) cudaEventDestroy(e.last_use);
  e = BlobEntry{};
}

bool take_entry(int device, size_t bytes, BlobEntry* out) {
  {
    std::lock_guard<std::mutex> lock(g_blob_mutex);
    int best = -1;
    for (size_t i = 0; i < g_blob_cache.size(); ++i) {
      const BlobEntry& e = g_blob_cache[i];
      if (e.device == device && e.capacity >= bytes && (best < 0 || e.capacity < g_blob_cache[best].capacity))
        best = int(i);
    }
    if (best >= 0) {
      *out = g_blob_cache[best];
      g_blob_cache.erase(g_blob_cache.begin() + best);
      return true;
    }
  }
  BlobEntry e;
  e.device = device;
  e.capacity = (bytes + 65535) / 65536 * 65536;   // round up so that plans of similar size share entries
  if (cudaMalloc(&e.dptr, e.capacity) != cudaSuccess || cudaMallocHost(&e.hptr, e.capacity) != cudaSuccess ||
      cudaEventCreateWithFlags(&e.copied, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&e.last_use, cudaEventDisableTiming) != cudaSuccess) {
    free_entry(e);
    return false;
  }
  *out = e;
  return true;
}

void give_entry(BlobEntry e) {
  {
    std::lock_guard<std::mutex> lock(g_blob_mutex);
    if (g_blob_cache.size() < kBlobCacheMax) {
      g_blob_cache.push_back(e);
      return;
    }
  }
  if (e.last_use_valid) cudaEventSynchronize(e.last_use);
  free_entry(e);
}
}  // namespace

extern "C" psa_status_t psa_plan_upload(psa_plan_t* p, void* stream) {
  if (!p) return PSA_ERR_INVALID_ARG;
  if (p->d_blob) return PSA_OK;
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t b0 = up(p->q_tiles.size() * sizeof(TileRec));
  const size_t b1 = up(p->kv_tiles.size() * sizeof(TileRec));
  const size_t b2 = up(p->fwd_entries.size() * sizeof(int32_t));
  const size_t b3 = up(p->bwd_entries.size() * sizeof(int32_t));
  const size_t b4 = up(p->bwd_cta_map.size() * sizeof(int32_t));
  const size_t b5 = up(p->few_key_rows.size() * sizeof(psa::FewKeyRow));
  const size_t total = b0 + b1 + b2 + b3 + b4 + b5 + 256;
  if (cudaGetDevice(&p->device) != cudaSuccess) return PSA_ERR_CUDA;
  if (!p->parts.empty()) psa::make_host_pipes(p->device);   // here, so that psa_step_host creates nothing
  BlobEntry e;
  if (!take_entry(p->device, total, &e)) return PSA_ERR_CUDA;
  const cudaStream_t st = cudaStream_t(stream);
  // The staging buffer may still be feeding the previous owner's upload (not in steady state: that
  // copy was enqueued a whole step ago), and the device blob may still be read by the previous
  // owner's kernels: the new upload is ordered after them on the device, without a host wait.
  bool ok = cudaEventSynchronize(e.copied) == cudaSuccess;
  if (ok && e.last_use_valid) ok = cudaStreamWaitEvent(st, e.last_use, 0) == cudaSuccess;
  if (ok) {
    char* host = static_cast<char*>(e.hptr);
    std::memcpy(host, p->q_tiles.data(), p->q_tiles.size() * sizeof(TileRec));
    std::memcpy(host + b0, p->kv_tiles.data(), p->kv_tiles.size() * sizeof(TileRec));
    std::memcpy(host + b0 + b1, p->fwd_entries.data(), p->fwd_entries.size() * sizeof(int32_t));
    std::memcpy(host + b0 + b1 + b2, p->bwd_entries.data(), p->bwd_entries.size() * sizeof(int32_t));
    std::memcpy(host + b0 + b1 + b2 + b3, p->bwd_cta_map.data(), p->bwd_cta_map.size() * sizeof(int32_t));
    std::memcpy(host + b0 + b1 + b2 + b3 + b4, p->few_key_rows.data(), p->few_key_rows.size() * sizeof(psa::FewKeyRow));
    ok = cudaMemcpyAsync(e.dptr, e.hptr, total, cudaMemcpyHostToDevice, st) == cudaSuccess &&
         cudaEventRecord(e.copied, st) == cudaSuccess;
  }
  if (!ok) {
    cudaDeviceSynchronize();
    free_entry(e);
    return PSA_ERR_CUDA;
  }
  char* b = static_cast<char*>(e.dptr);
  p->d_blob = e.dptr;
  p->h_stage = e.hptr;
  p->blob_capacity = e.capacity;
  p->ev_copied = e.copied;
  p->ev_last_use = e.last_use;
  p->used_streams.clear();
  p->used_streams.push_back(stream);   // the upload itself
  p->d_q_tiles = reinterpret_cast<const TileRec*>(b);
  p->d_kv_tiles = reinterpret_cast<const TileRec*>(b + b0);
  p->d_fwd_entries = reinterpret_cast<const int32_t*>(b + b0 + b1);
  p->d_bwd_entries = reinterpret_cast<const int32_t*>(b + b0 + b1 + b2);
  p->d_bwd_cta_map = reinterpret_cast<const int32_t*>(b + b0 + b1 + b2 + b3);
  p->d_few_key_rows = reinterpret_cast<const psa::FewKeyRow*>(b + b0 + b1 + b2 + b3 + b4);
  return PSA_OK;
}

namespace psa {
void note_plan_use(const psa_plan_t* plan, void* stream) {
  std::lock_guard<std::mutex> lock(plan->used_mutex);
  for (void* s : plan->used_streams)
    if (s == stream) return;
  // used_streams[0] is the upload's stream; any other stream has to see the uploaded blob first
  if (plan->ev_copied) cudaStreamWaitEvent(cudaStream_t(stream), cudaEvent_t(plan->ev_copied), 0);
  plan->used_streams.push_back(stream);
}
}  // namespace psa

extern "C" psa_status_t psa_plan_destroy(psa_plan_t* p) {
  if (!p) return PSA_OK;
  psa_status_t st = PSA_OK;
  if (p->d_blob) {
    // Hand the blob back.  Its next owner must not overwrite it before the kernels enqueued under
    // this plan have run: one event, recorded in turn on every stream that used the plan (each
    // stream first waits for the previous recording, so the last recording covers them all).
    BlobEntry e;
    e.device = p->device;
    e.dptr = p->d_blob;
    e.hptr = p->h_stage;
    e.capacity = p->blob_capacity;
    e.copied = cudaEvent_t(p->ev_copied);
    e.last_use = cudaEvent_t(p->ev_last_use);
    int cur = -1;
    bool ok = cudaGetDevice(&cur) == cudaSuccess && (cur == p->device || cudaSetDevice(p->device) == cudaSuccess);
    bool first = true;
    for (void* s : p->used_streams) {
      if (!ok) break;
      if (!first) ok = cudaStreamWaitEvent(cudaStream_t(s), e.last_use, 0) == cudaSuccess;
      if (ok) ok = cudaEventRecord(e.last_use, cudaStream_t(s)) == cudaSuccess;
      first = false;
    }
    if (!ok) {   // a stream is gone or the context is in trouble: fall back to a full wait
      cudaGetLastError();
      if (cudaDeviceSynchronize() != cudaSuccess) st = PSA_ERR_CUDA;
      e.last_use_valid = false;
    } else {
      e.last_use_valid = true;
    }
    if (cur >= 0 && cur != p->device) cudaSetDevice(cur);
    give_entry(e);
  }
  delete p;
  return st;
}

extern "C" psa_status_t psa_plan_stats(const psa_plan_t* p, int64_t* total_tokens, int64_t* useful_pairs,
                                       int64_t* live_tiles, int64_t* partial_tiles,
                                       size_t* bwd_workspace_bytes) {
  if (!p) return PSA_ERR_INVALID_ARG;
  if (total_tokens) *total_tokens = p->T;
  if (useful_pairs) *useful_pairs = p->useful_pairs;
  if (live_tiles) *live_tiles = p->live_tiles;
  if (partial_tiles) *partial_tiles = p->partial_tiles;
  if (bwd_workspace_bytes) *bwd_workspace_bytes = p->bwd_workspace_bytes;
  return PSA_OK;
}

extern "C" psa_status_t psa_plan_counts(const psa_plan_t* p, int32_t direction, int32_t* n_tiles,
                                        int32_t* n_entries) {
  if (!p || (direction != 0 && direction != 1)) return PSA_ERR_INVALID_ARG;
  const auto& entries = direction ? p->bwd_entries : p->fwd_entries;
  if (n_tiles) *n_tiles = direction ? int32_t(p->kv_tiles.size()) : p->whole.n_q_tiles;
  if (n_entries) *n_entries = int32_t(entries.size());
  return PSA_OK;
}

extern "C" psa_status_t psa_plan_launch(const psa_plan_t* p, int32_t* fwd_items_per_cta, int32_t* bwd_ctas_per_pair) {
  if (!p) return PSA_ERR_INVALID_ARG;
  if (fwd_items_per_cta) *fwd_items_per_cta = p->whole.fwd_items_per_cta;
  if (bwd_ctas_per_pair) *bwd_ctas_per_pair = p->whole.bwd_split;
  return PSA_OK;
}

extern "C" psa_status_t psa_plan_export(const psa_plan_t* p, int32_t direction, int32_t* tiles,
                                        int32_t* entries) {
  if (!p || (direction != 0 && direction != 1) || !tiles || !entries) return PSA_ERR_INVALID_ARG;
  const auto& t = direction ? p->kv_tiles : p->q_tiles;
  const auto& e = direction ? p->bwd_entries : p->fwd_entries;
  const size_t n = direction ? t.size() : size_t(p->whole.n_q_tiles);
  if (n) std::memcpy(tiles, t.data(), n * sizeof(TileRec));
  if (!e.empty()) std::memcpy(entries, e.data(), e.size() * sizeof(int32_t));
  return PSA_OK;
}

// First-fit-decreasing packing (Section 3.2 / 4.3.2).  The "first bin with room" query is
// answered by a max segment tree over the bins' free space: O(n log n) for n units.
extern "C" psa_status_t psa_pack_ffd(const int32_t* unit_len, int32_t n_units, int32_t capacity,
                                     int32_t* bin_of_unit, int32_t* n_bins) {
  if (n_units < 0 || capacity <= 0 || !n_bins || (n_units > 0 && (!unit_len || !bin_of_unit)))
    return PSA_ERR_INVALID_ARG;
  for (int i = 0; i < n_units; ++i) {
    if (unit_len[i] < 0) return PSA_ERR_INVALID_ARG;
    if (unit_len[i] > capacity) return PSA_ERR_UNSUPPORTED;
  }
  std::vector<int32_t> order(n_units);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return unit_len[a] > unit_len[b]; });
  int leaves = 1;
  while (leaves < std::max(n_units, 1)) leaves <<= 1;
  std::vector<int32_t> tree(2 * leaves, 0);   // free space of bin b at tree[leaves + b]; unopened bins hold 0
  int32_t opened = 0;
  auto update = [&](int b, int32_t v) {
    int node = leaves + b;
    tree[node] = v;
    for (node >>= 1; node >= 1; node >>= 1) tree[node] = std::max(tree[2 * node], tree[2 * node + 1]);
  };
  for (int32_t u : order) {
    const int32_t len = unit_len[u];
    int b;
    if (opened > 0 && tree[1] >= len) {
      int node = 1;
      while (node < leaves) node = tree[2 * node] >= len ? 2 * node : 2 * node + 1;   // leftmost bin with room
      b = node - leaves;
    } else {
      b = opened++;
      update(b, capacity);
    }
    update(b, tree[leaves + b] - len);
    bin_of_unit[u] = b;
  }
  *n_bins = opened;
  return PSA_OK;
}
