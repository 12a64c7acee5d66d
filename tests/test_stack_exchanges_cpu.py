"""The exchanges inside a cluster of the persistent layer kernel, checked without a GPU: nothing but the exchanges themselves
keeps a fast rank from writing where a slow one still reads, so for the shared-memory plan of every shape the order in
which each table is written and read has to follow from what a rank has received."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1811_03115_b200", "csrc")
RANKS = 8

# prints, for every shape and variant that one sequence may get, where the tables lie that ranks write into one another
PLANS = r"""
#include <cstdio>
#include "stack_plan.hpp"
int main() {
  using namespace bpd;
  for (int d : {256, 512, 1024})
    for (int units : {128, 256})
      for (int rows = 1; rows <= fused::kMaxRows; ++rows)
        for (int lean : {0, 1, 2, 3}) {
          Config c;
          memset(&c, 0, sizeof(c));
          c.dtype = 1; c.d = d; c.H = d / fused::kDH; c.d_ff = units * c.H; c.n_dec = 6; c.k_model = rows;
          stack::Layout L;
          const bool split = lean == 2 || lean == 3;
          const int long_seq = lean == 2 || lean == 0, cross = split ? 8 : 40;
          if (!stack_plan(c, rows, 1, 16, cross, long_seq, lean, 232448 - 2048, &L)) continue;
          const int NT = rows > 8 ? 2 : 1, RP = 8 * NT, UPR = units / fused::kC;
          const int chunk = std::max(NT * 3 * fused::kDH * 4, UPR * RP * 4);
          printf("%d %d %d %d  %d %d  %d %d  %d %d  %d %d\n", d, units, rows, lean, L.inbox, fused::kC * chunk, L.lvl2,
                 (int)(fused::kC * rows * stack::kState * 4), L.hid, fused::kC * 2 * RP * UPR * 2, L.stats, fused::kC * fused::kMaxRows * 8);
        }
  printf("rows\n");
  for (int rows = 1; rows <= fused::kMaxRows; ++rows)
    for (int c = 0; c < fused::kC; ++c) printf("%d %d\n", stack::row_bytes_sent(c, rows, 512), stack::row_bytes_awaited(c, rows, 512));
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    tmp = tmp_path_factory.mktemp("plans")
    (tmp / "plans.cu").write_text(PLANS)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC, "-o", str(tmp / "plans"), str(tmp / "plans.cu")], check=True)
    out = subprocess.run([str(tmp / "plans")], check=True, capture_output=True, text=True).stdout
    shapes, sent = ([[int(v) for v in line.split()] for line in part.splitlines() if line] for part in out.split("rows"))
    assert shapes and len(sent) == 16 * RANKS
    return shapes, [sent[i:i + RANKS] for i in range(0, len(sent), RANKS)]


def _faults(exchanges):
    """exchanges: (tables written at the receiver, tables read there afterwards, ranks that send).  The order of things per rank:
    send m, wait for m, read, send m + 1.  known[c][r]: the latest exchange of which c knows that r has sent its part, hence
    has finished its reads after the one before.  Returns what a rank may overwrite too early."""
    found = set()
    known = [[-1] * RANKS for _ in range(RANKS)]        # two barriers alternate: r must have passed exchange m - 2
    overlap = lambda a, b: a[0] < b[0] + b[1] and b[0] < a[0] + a[1]
    for m, (writes, _, senders) in enumerate(exchanges):
        for c in senders:
            for r in range(RANKS):
                if r == c:
                    continue
                if m >= 2 and known[c][r] < m - 1:
                    found.add((m, m - 2))
                for q in range(m):
                    for w in writes:
                        for t in exchanges[q][1]:
                            if overlap(w, t) and known[c][r] < q + 1:
                                found.add((m, q))
        for c in range(RANKS):
            known[c][c] = m
        before = [row[:] for row in known]
        for c in range(RANKS):
            for s in senders:
                known[c] = [max(a, b) for a, b in zip(known[c], before[s])]
    return found


def test_no_rank_overwrites_what_another_still_reads(plans):
    for d, units, rows, lean, *at in plans[0]:
        inbox, states, hidden, stats = zip(at[0::2], at[1::2])
        every = range(RANKS)
        with_rows = [c for c in every if plans[1][rows - 1][c][0] > 0]
        partials, finish = ((inbox, stats), (inbox, stats), every), ((hidden,), (hidden,), every)
        share, some = ((states,), (states,), every), ((), (), with_rows)
        if lean in (2, 3):        # keys, values and queries, then states, in both attentions
            layer = [partials, some, share, partials, some, share, partials, finish]
        else:                     # keys, values and queries, finished rows (or states), finished rows
            layer = [partials, some, share if lean == 0 else some, partials, some, partials, finish]
        assert not _faults(layer * 3), (d, units, rows, lean)


def test_an_exchange_of_rows_awaits_what_is_sent(plans):
    for sent in plans[1]:
        for c in range(RANKS):
            assert sent[c][0] > 0 and sent[c][1] == sum(n for n, _ in sent) - sent[c][0]
