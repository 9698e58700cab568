"""The rule that sends a call to the batch kernels (batch_fits in csrc/batch.cuh): where it says yes, no CTA's share of the
runs' row blocks touches more runs than the CTA's list holds.  The rule is compiled by itself and compared with the shares that
the plan would deal out, worked out here one by one; no GPU."""
import os
import random
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAX_SEGS, MAX_TASKS, RUN, CHUNK, FIXED = 40, 640, 8, 2048, 12

PROGRAM = r"""
#include <cstdio>
#include "batch.cuh"
int main() {
  slicemoe_shape s = {};
  int T, sms;
  while (std::scanf("%d %d %d %d %d %d %d", &s.hidden, &s.inter, &s.top_k, &s.n_shared, &s.shared_inter, &T, &sms) == 7)
    std::printf("%d %d\n", slicemoe::batch_fits(&s, s.n_shared, T, sms) ? 1 : 0, slicemoe::kBMaxSegs);
}
"""


def _rule(tmp_path, rows):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2512_12990_b200", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, r)) for r in rows), text=True, capture_output=True, check=True).stdout
    got = [tuple(map(int, line.split())) for line in out.splitlines()]
    assert all(segs == MAX_SEGS for _, segs in got)
    return [bool(fits) for fits, _ in got]


def _block_cost(n, highs):
    return (4 if highs else 2) + (1 if n <= 2 else 2) * (2 if 0 < highs < n else 1)


def _most_touched(row, runs):
    """Most runs that a share touches in either projection; runs: (pairs, those at both slices)."""
    hidden, inter, k, n_shared, shared_inter, T, sms = row
    parts = -(-T // RUN)
    segs = [[], []]
    for n, highs, width in [(n, h, inter) for n, h in runs] + [(min(T, RUN),) * 2 + (shared_inter,)] * (n_shared * parts):
        c = _block_cost(n, highs)
        segs[0].append((2 * c * (hidden // 128) + FIXED, width // 16))
        for c0 in range(0, width, CHUNK):
            segs[1].append((c * (min(CHUNK, width - c0) // 128) + FIXED, hidden // 16))
    most = 0
    for phase in segs:
        total = sum(c * u for c, u in phase)
        touched, at = [0] * sms, 0
        for cost, units in phase:
            # the CTA whose window a row block's start lies in
            ctas = {(at + i * cost) * sms // total for i in {0, units - 1} | set(range(0, units, max(1, total // (sms * cost))))}
            for c in ctas:
                touched[c] += 1
            at += cost * units
        most = max(most, max(touched))
    return most, max(len(p) for p in segs)


def _rows(rng, count, sms):
    rows = []
    while len(rows) < count:
        hidden, inter, k = 128 * rng.randint(1, 32), 128 * rng.choice([1, 1, 2, 3, 5, 11, 17]), rng.randint(1, 16)
        n_shared = rng.randint(0, 4)
        shared_inter = 128 * rng.randint(1, 40) if n_shared else 0
        if k * inter + n_shared * shared_inter <= 12288:
            rows.append((hidden, inter, k, n_shared, shared_inter, rng.randint(4, 16), sms))
    return rows


def test_shares_that_the_rule_admits_fit_the_list(tmp_path):
    rng = random.Random(3)
    rows = _rows(rng, 150, 148) + _rows(rng, 150, 12) + _rows(rng, 150, 4)
    refused = too_many = 0
    for row, fits in zip(rows, _rule(tmp_path, rows)):
        pairs = row[2] * row[5]
        assert fits or row[6] < 148, "a whole device takes every layer"
        refused += not fits
        for kind in range(3):
            if kind == 0:                      # all experts distinct, mostly from the MSB slice
                runs = [(1, int(rng.random() < 0.2)) for _ in range(pairs)]
            elif kind == 1:                    # cheap runs side by side, then dear ones
                runs = [(1, 0)] * (pairs // 2) + [(1, 1)] * (pairs - pairs // 2)
            else:
                runs, left = [], pairs
                while left:
                    n = min(left, rng.randint(1, RUN))
                    runs.append((n, rng.randint(0, n)))
                    left -= n
            most, tasks = _most_touched(row, runs)
            too_many += most > MAX_SEGS
            if fits:
                assert most <= MAX_SEGS and tasks <= MAX_TASKS, (row, kind, most, tasks)
    assert refused and too_many, "the ranges reach beyond the list"
