"""How the batch-1 decode kernel deals its gate/up tasks (csrc/decode_schedule.cuh), compiled by itself and gone through task by
task; and the hand-over of the rows that its two phases share.  No GPU."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_12990_b200", "csrc")
GROUPS, CHUNK, SMS = 4, 2048, 148

PROGRAM = r"""
#include <cstdio>
#include "decode_schedule.cuh"
using namespace slicemoe;
int main() {
  int nshared, nboth, nmsb, P;  // tasks: of the shared experts, from both slices (with those), MSB-only; CTAs
  while (std::scanf("%d %d %d %d", &nshared, &nboth, &nmsb, &P) == 4)
    for (int c = 0; c < P; ++c) {
      Deal d;
      const int count_s = dealt(nshared, c, P);
      for (int n = 0; n < count_s; ++n) {  // as the roles see them before the plan stands: nothing of `d` is set
        const TaskPlace p(n + 1, n);
        std::printf("s %d %d %d %d %d %d\n", c, n, d.ordinal(count_s, n, c, P), p.producer, p.group(), p.round());
      }
      d.set(nboth, nmsb, c, P);
      for (int n = 0; n < d.count1; ++n) {
        const TaskPlace p(d.count_both, n);
        std::printf("t %d %d %d %d %d %d\n", c, n, d.ordinal(count_s, n, c, P), p.producer, p.group(), p.round());
      }
    }
}
"""


@pytest.fixture(scope="module")
def schedule(tmp_path_factory):
    d = tmp_path_factory.mktemp("schedule")
    (d / "s.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "s.cpp"), "-o", str(d / "s")], check=True)

    def run(nshared, nboth, nmsb, P=SMS):
        """[(n, ordinal, producer, group, round)] per CTA, and the same of the tasks known before the plan."""
        out = subprocess.run([str(d / "s")], input=f"{nshared} {nboth} {nmsb} {P}", text=True, capture_output=True, check=True).stdout
        tasks, early = [[] for _ in range(P)], [[] for _ in range(P)]
        for line in out.splitlines():
            kind, c, *rest = line.split()
            (tasks if kind == "t" else early)[int(c)].append(tuple(map(int, rest)))
        return tasks, early
    return run


COUNTS = [  # shared, both-slice (with those), MSB-only
    (0, 0, 0), (0, 0, 1), (0, 1, 0), (0, 8, 8), (0, 80, 80), (0, 296, 296), (8, 304, 296), (176, 440, 264), (352, 352, 264), (0, 128, 256), (256, 256, 128),
    (0, 147, 1), (0, 148, 147), (0, 149, 600), (0, 443, 3), (136, 496, 216), (768, 768, 0), (0, 0, 768)]


@pytest.mark.parametrize("nshared,nboth,nmsb", COUNTS)
@pytest.mark.parametrize("P", [SMS, 20, 3])
def test_every_task_once_and_in_order(schedule, nshared, nboth, nmsb, P):
    tasks, early = schedule(nshared, nboth, nmsb, P)
    assert sorted(t[1] for cta in tasks for t in cta) == list(range(nboth + nmsb))
    cost = []
    for cta, ahead in zip(tasks, early):
        assert cta[:len(ahead)] == ahead, "what is requested ahead of the plan is what the plan says"
        assert all(o < nshared for _, o, *_ in ahead) and all(o >= nshared for _, o, *_ in cta[len(ahead):])
        both = [t for t in cta if t[1] < nboth]
        assert both == cta[:len(both)], "both-slice tasks come first"
        assert [t[1] for t in both] == sorted(t[1] for t in both)
        for group in range(GROUPS):
            mine = [t for t in cta if t[3] == group]
            assert [t[4] for t in mine] == list(range(len(mine))), "a group's rounds follow one another"
            assert all(t[2] == group % 2 for t in mine)
        for producer in range(2):  # the producer's two groups in turn
            mine = [t[3] // 2 for t in cta if t[2] == producer]
            assert mine == [i % 2 for i in range(len(mine))]
        cost.append(2 * len(both) + len(cta) - len(both))
    assert max(cost) - min(cost) <= 2, "the CTAs differ by a task"


def _tasks(hidden, inter, k, n_both, shared_inter):
    return shared_inter // 16, shared_inter // 16 + n_both * inter // 16, (k - n_both) * inter // 16


# hidden, inter, top_k, both-slice entries, shared inter; CTAs in which a group that has a task has no chunk of the first output
# rows, with another group's both-slice task not after it in the CTA's order
HANDOVER = [((2048, 2048, 3, 1, 0), 68), ((2560, 2048, 1, 0, 4096), 40)]


@pytest.mark.parametrize("shape,ctas", HANDOVER)
def test_rows_of_a_group_without_down_chunks(schedule, shape, ctas):
    """A group's rows of partial sums: in gate/up a group waits, before it writes round r, for the epilogue warp to have taken round
    r - 1; that leaves its last round.  The epilogue takes the tasks in the CTA's order, so it may still be at another group's task
    when this group, which has no chunk of the down projection to wait for, writes its (zero) share of the first output rows.
    These shapes have such groups; so the two phases' rows are apart."""
    hidden, inter, k, n_both, shared_inter = shape
    chunks = k * -(-inter // CHUNK) + (-(-shared_inter // CHUNK) if shared_inter else 0)
    assert chunks < GROUPS
    exposed = 0
    tasks, _ = schedule(*_tasks(*shape))
    for c, cta in enumerate(tasks):
        if c >= hidden // 16:
            continue  # no output rows: nothing is written in phase 2
        last = {t[3]: t[0] for t in cta}  # a group's last task
        exposed += any(g >= chunks and any(t[0] < n and t[3] != g for t in cta) for g, n in last.items())
    assert exposed == ctas

    source = open(os.path.join(CSRC, "decode.cu")).read()
    consumer = source[source.index("__device__ void consumer_loop"):source.index("__device__ void epilogue_loop")]
    gate_up, down = consumer[:consumer.index("// ---- phase 2")], consumer[consumer.index("// ---- phase 2"):]
    written = [re.findall(r"(\w+)\[warp \* 16 \+ lr\.r\] =", part) for part in (gate_up, down)]
    assert written == [["partial"], ["partial2"]]
    at = {name: int(size) for name, size in re.findall(r"constexpr int \w+ = (partial2?) \+ kConsumerWarps \* 16 \* (?:2 \* )?(4);", source)}
    assert set(at) == {"partial", "partial2"}, "each has storage of its own"
