// How the batch-1 decode kernel (decode.cu) deals its gate/up tasks to the CTAs of a grid and to the warps of a CTA.  Plain integer
// arithmetic that the host compiles too: tests/test_host_decode_schedule.py goes through it task by task.
#pragma once

#ifndef SM_HD
#ifdef __CUDACC__
#define SM_HD __host__ __device__
#else
#define SM_HD
#endif
#endif

namespace slicemoe {

constexpr int kGroups = 4;     // consumer groups of a CTA
constexpr int kProducers = 2;  // producer warps of a CTA

// How many of n things, dealt to P CTAs one by one, go to CTA c.
SM_HD inline int dealt(int n, int c, int P) { return n > c ? (n - c + P - 1) / P : 0; }

// CTA c's share of nboth both-slice tasks and, behind them in number, nmsb MSB-only ones, half as long.  Both-slice tasks go to CTA
// o mod P; of the MSB-only ones, the `light` CTAs short of a both-slice task get two first, and the rest is dealt out: the CTAs
// differ by a task at most.
struct Deal {
  int count_both, count1;                      // tasks from both slices, tasks in all
  int light, count_light, ord_light, ord_rest;  // its MSB-only tasks: see ordinal()

  SM_HD void set(int nboth, int nmsb, int c, int P) {
    const int q = nboth / P, r = nboth - q * P;
    light = r ? P - r : 0;
    const int first = nmsb < 2 * light ? nmsb : 2 * light, rest = nmsb - first;
    const int at = c - r, rest_q = rest / P;  // (the two divisions of this chain)
    count_both = q + (c < r ? 1 : 0);
    count_light = at >= 0 ? (at < first ? 1 : 0) + (at + light < first ? 1 : 0) : 0;
    count1 = count_both + count_light + rest_q + (c < rest - rest_q * P ? 1 : 0);
    ord_light = nboth + at;
    ord_rest = nboth + first + c;
  }
  // The number in the grid of the CTA's task n.  (The first count_s, of the shared experts, are known before set() has run.)
  SM_HD int ordinal(int count_s, int n, int c, int P) const {
    if (n < count_s || n < count_both) return c + n * P;
    n -= count_both;
    return n < count_light ? ord_light + n * light : ord_rest + (n - count_light) * P;
  }
};

// Which producer a task goes to and which of that producer's tasks it is; the producer's groups take its tasks in turn.  The
// tasks of both slices alternate; where their number is odd, the first two of the MSB-only ones, half as long, go to the
// producer that got one less, the rest alternates again.
struct TaskPlace {
  int producer, turn;
  SM_HD TaskPlace(int count_both, int n) {
    const int k = n - count_both;  // among the MSB-only tasks
    if (k >= 0 && (count_both & 1)) {
      producer = k < 2 ? 1 : k & 1;
      turn = (count_both >> 1) + (k < 2 ? k : producer ? 2 + ((k - 2) >> 1) : 1 + ((k - 2) >> 1));
    } else {
      producer = n & 1;
      turn = n >> 1;
    }
  }
  SM_HD int group() const { return producer + kProducers * (turn & 1); }
  SM_HD int round() const { return turn >> 1; }  // which of its group's tasks it is
};
static_assert(kProducers == 2 && kGroups == 4, "two groups to a producer");

}  // namespace slicemoe
