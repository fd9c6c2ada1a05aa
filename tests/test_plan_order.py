"""The launch order of the backward and the number of CTAs per pair, read out of the plan and compared with the rules of
psa_plan.cpp written down plainly: whole orders sorted and simulated one by one."""
import heapq
import os
import subprocess

import pytest

from paper_2410_20305_b200 import binding as B
from paper_2410_20305_b200 import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 148

READER = r"""
#include <cstdio>
#include <vector>
#include "psa_internal.h"
int main() {
  int n, hq, hkv, d;
  while (scanf("%d %d %d %d", &n, &hq, &hkv, &d) == 4) {
    std::vector<int32_t> cu(n + 1, 0), len[3];
    for (auto& l : len) l.resize(n);
    for (int i = 0; i < n; ++i) {
      for (auto& l : len) if (scanf("%d", &l[i]) != 1) return 1;
      cu[i + 1] = cu[i] + len[0][i] + len[1][i] + len[2][i];
    }
    psa_plan_t* p = nullptr;
    if (psa_plan(cu.data(), len[0].data(), len[1].data(), len[2].data(), n, hq, hkv, d, 0.f, PSA_PLAN_HOST_ONLY, nullptr, &p) != PSA_OK) return 2;
    std::vector<psa::PlanPart> parts = p->parts;
    parts.insert(parts.begin(), p->whole);
    printf("%zu %zu\n", p->kv_tiles.size(), parts.size());
    for (auto& t : p->kv_tiles) printf("%d %d\n", t.ds, t.list_cnt);
    for (auto& w : parts) {
      printf("%d %d %d %d %d\n", w.row0, w.row1, w.n_ctas, w.bwd_split, w.bwd_long_lists);
      for (int i = 0; i < 2 * w.n_ctas; ++i) printf("%d ", p->bwd_cta_map[2 * w.cta0 + i]);
      printf("\n");
    }
    psa_plan_destroy(p);
  }
}
"""


@pytest.fixture(scope="module")
def reader(tmp_path_factory):
    B.load_library()
    at = tmp_path_factory.mktemp("order")
    (at / "reader.cpp").write_text(READER)
    pkg = os.path.join(ROOT, "paper_2410_20305_b200")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(pkg, "csrc"), str(at / "reader.cpp"),
                    "-o", str(at / "reader"), os.path.join(pkg, "libpsa.so"), "-Wl,-rpath," + pkg], check=True)
    return str(at / "reader")


def _read(reader, pack):
    """key tiles [(first row of the sample, list length)], parts [(row0, row1, split, long, [(tile, kv head)])]"""
    lengths = [x for l in (pack.prefix_len, pack.chosen_len, pack.rejected_len) for x in l]
    n = pack.n_samples
    text = "%d %d %d %d\n" % (n, pack.n_q_heads, pack.n_kv_heads, pack.head_dim)
    text += " ".join(str(lengths[i + n * k]) for i in range(n) for k in range(3))
    out = list(map(int, subprocess.run([reader], input=text, capture_output=True, text=True, check=True).stdout.split()))
    out = iter(out)
    n_tiles, n_parts = next(out), next(out)
    tiles = [(next(out), next(out)) for _ in range(n_tiles)]
    parts = []
    for _ in range(n_parts):
        row0, row1, n_ctas, split, long = (next(out) for _ in range(5))
        parts.append((row0, row1, split, long, [(next(out), next(out)) for _ in range(n_ctas)]))
    return tiles, parts


def _makespan(lengths, slots, cost):
    free = [0] * slots
    end = 0
    for n in lengths:
        t = heapq.heappop(free) + cost(n)
        end = max(end, t)
        heapq.heappush(free, t)
    return end


def _grouped(tiles, row0, row1, n_kv_heads):
    samples = {}
    for i, (ds, n) in enumerate(tiles):
        if row0 <= ds < row1:
            samples.setdefault(ds, []).append(i)
    by_work = sorted(sorted(samples), key=lambda ds: -sum(tiles[i][1] for i in samples[ds]))
    return [(i, hk) for ds in by_work for hk in range(n_kv_heads) for i in samples[ds]]


def _tail_sorted(order, tiles, permille):
    total, acc, at = sum(tiles[i][1] for i, _ in order), 0, 0
    while at < len(order) and acc * 1000 < total * (1000 - permille):
        acc += tiles[order[at][0]][1]
        at += 1
    return order[:at] + sorted(order[at:], key=lambda c: -tiles[c[0]][1])


def _rule(pack, tiles):
    """The whole pack's order and split."""
    group = pack.n_q_heads // pack.n_kv_heads
    per_iteration, fixed = (2050, 8000) if pack.head_dim == 128 else (1600, 7000)
    alone = lambda n: n * group * per_iteration + fixed
    of = lambda order: [tiles[i][1] for i, _ in order]
    grouped = _grouped(tiles, 0, pack.total_tokens, pack.n_kv_heads)
    order, best = grouped, _makespan(of(grouped), SMS, alone)
    if len(grouped) > SMS:
        wave = min(1000, 1150 * SMS // len(grouped))
        in_l2 = pack.total_tokens * pack.n_q_heads * pack.head_dim * 4 <= 64 << 20
        shortest = best * 985 // 1000
        for permille in (wave, 300, 500, 1000) if in_l2 else (wave,):
            o = _tail_sorted(grouped, tiles, permille)
            t = _makespan(of(o), SMS, alone)
            if t < shortest:
                shortest = best = t
                order = o
    split = 1
    if len(grouped) <= 2 * SMS:
        longest_first = _tail_sorted(grouped, tiles, 1000)
        need = 90 if max(of(grouped)) * group >= 20 else 75
        for s, slots in ((2, 74), (4, 33), (8, 15)):
            shared = lambda n: -(-n * group // s) * per_iteration + fixed + 3000
            t, t_sorted = (_makespan(of(o), slots, shared) for o in (grouped, longest_first))
            if t * 100 < best * 90 or t_sorted * 100 < best * need:
                best, split = min(t, t_sorted), s
        if split > 1:
            order = longest_first
    return order, split


def _packs():
    yield wl.config_pack(0)
    # clusters for which the grouped order is the shorter one in the simulation
    yield wl.pack_from_lengths("turn-a", [(29, 141, 19), (2, 21, 13), (292, 82, 38), (173, 50, 18), (251, 41, 84), (427, 132, 103)], 32, 8, 128)
    yield wl.pack_from_lengths("turn-b", [(745, 43, 198), (550, 32, 183), (126, 35, 45), (121, 139, 119)], 32, 8, 64)
    yield wl.pack_from_lengths("empty", [(0, 0, 0)], 4, 2, 64)
    for heads in ((32, 8, 128), (16, 16, 64), (8, 2, 128), (8, 2, 64), (32, 8, 64), (8, 8, 128)):
        for seed, (n, longest) in enumerate([(1, 900), (2, 2500), (5, 700), (9, 1500), (30, 200), (12, 60)]):
            yield wl.random_pack(200 + seed, n, longest, *heads)
        yield wl.pack_from_lengths("one", [(7000, 300, 411)], *heads)


@pytest.mark.parametrize("pack", list(_packs()), ids=lambda p: "%s-%d-%d-%d" % (p.name, p.n_q_heads, p.n_kv_heads, p.head_dim))
def test_order_and_split_follow_the_rules(reader, pack):
    tiles, parts = _read(reader, pack)
    order, split = _rule(pack, tiles) if tiles else ([], 1)
    for k, (row0, row1, s, long, got) in enumerate(parts):
        grouped = _grouped(tiles, row0, row1, pack.n_kv_heads)
        assert sorted(got) == sorted(grouped)
        assert s == split
        assert got == (order if (row0, row1) == (0, pack.total_tokens) else grouped), k
        n = [tiles[i][1] for i, _ in grouped]
        assert bool(long) == (sum(x * x for x in n) >= 43 * sum(n) > 0)


@pytest.mark.parametrize("lengths,heads,split,kept", [
    ([(3000, 300, 301), (900, 200, 252)], (8, 8, 128), 1, "less than half"),
    ([(2600, 500, 200), (1500, 300, 420), (300, 90, 77)], (32, 8, 128), 1, "about half"),
    ([(1500, 300, 209)], (32, 8, 128), 2, "none"),
    ([(700, 130, 60), (1, 0, 1), (250, 129, 128)], (16, 16, 64), 1, "none")])
def test_packs_of_the_gradient_test_take_the_orders_that_they_are_there_for(reader, lengths, heads, split, kept):
    """How much of the grouped order is left at the start (tests/test_gpu_bwd_order.py)."""
    pack = wl.pack_from_lengths("order", lengths, *heads)
    tiles, parts = _read(reader, pack)
    grouped, got = _grouped(tiles, 0, pack.total_tokens, pack.n_kv_heads), parts[0][4]
    same = next((i for i, (a, b) in enumerate(zip(grouped, got)) if a != b), len(got)) / len(got)
    assert parts[0][2] == split
    assert {"about half": 0.4 < same < 0.6, "less than half": same < 0.5, "none": same < 0.1}[kept], same
    lists = [tiles[i][1] for i, _ in got[int(same * len(got)) + 1:]]
    assert lists == sorted(lists, reverse=True)
