"""The host arithmetic that splits the rows of sweeps over the CTAs (csrc/lbm_schedule.h), built with the
host compiler: shared lists of a batch hold every row of every strip once, whatever the cases, and segment
lengths are those of a search over every number of segments."""
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_09431_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "lbm_schedule.h"
struct Item { int case_id, x0, y0, y1; };
// reads "rs slots cap strips", then the rows of each strip; prints the shares and their items
// with an argument: "ny strips resident rs fill", prints the segment length
int main(int argc, char **) {
  if (argc > 1) {
    int ny, strips, resident, step, fill;
    while (std::scanf("%d %d %d %d %d", &ny, &strips, &resident, &step, &fill) == 5)
      std::printf("%d\n", lbm::choose_segment(ny, strips, resident, step, fill));
    return 0;
  }
  int rs, slots, n;
  unsigned long long cap;
  while (std::scanf("%d %d %llu %d", &rs, &slots, &cap, &n) == 4) {
    std::vector<Item> strips, out;
    for (int i = 0; i < n; ++i) {
      int rows;
      if (std::scanf("%d", &rows) != 1) return 1;
      strips.push_back({i, 7 * i, 0, rows});
    }
    const int shares = lbm::share_out(strips, rs, slots, (size_t)cap, &out);
    std::printf("%d %d", shares, (int)(shares ? out.size() : 0));
    if (shares)
      for (const Item &w : out) std::printf(" %d %d %d %d", w.case_id, w.x0, w.y0, w.y1);
    std::printf("\n");
  }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("schedule")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")],
                   check=True)

    def call(queries, *arguments):
        if arguments:
            text = "\n".join(" ".join(map(str, q)) for q in queries)
            out = subprocess.run([str(d / "main"), *arguments], input=text, capture_output=True, text=True, check=True)
            return [int(line) for line in out.stdout.splitlines()]
        text = "\n".join(" ".join(map(str, (rs, slots, cap, len(rows), *rows))) for rs, slots, cap, rows in queries)
        out = subprocess.run([str(d / "main")], input=text, capture_output=True, text=True, check=True).stdout
        return [list(map(int, line.split())) for line in out.splitlines()]

    return call


def queries():
    r = random.Random(5)
    fixed = [[200] * 2] * 1 + [[3], [8], [9, 7, 500], [640] * 30 + [97] * 10, [200] * 512, [1] * 400, [100000, 3]]
    for rows in fixed:
        for rs, slots in ((2, 304), (2, 1), (2, 456), (4, 152)):
            yield rs, slots, 10 ** 9, rows
    for _ in range(300):
        rows = [r.choice((3, 8, r.randint(3, 30), r.randint(3, 700))) for _ in range(r.randint(1, 60))]
        yield r.choice((1, 2, 4, 8)), r.randint(1, 500), r.choice((10 ** 9, sum(-(-v // 8) for v in rows))), rows


def test_shared_lists_hold_every_row_once(run):
    asked = list(queries())
    pieces_most, padded = 0, 0
    for (rs, slots, cap, rows), (shares, count, *flat) in zip(asked, run(asked)):
        if shares == 0:
            assert count == 0
            continue
        items = [flat[4 * i:4 * i + 4] for i in range(count)]
        assert shares <= slots and count <= cap and count % shares == 0
        seen = {i: [] for i in range(len(rows))}
        fill = 3 * rs + rs * -(-6 // rs)
        cost = [0] * shares
        pieces = [0] * shares
        for k, (case, x0, y0, y1) in enumerate(items):
            if y1 <= y0:
                padded += 1
                continue
            assert x0 == 7 * case and y0 % rs == 0 and (y1 - y0 >= 8 or y0 == 0 and y1 == rows[case])
            seen[case].append((y0, y1))
            cost[k % shares] += y1 - y0 + fill
            pieces[k % shares] += 1
        for case, spans in seen.items():
            spans.sort()
            assert spans[0][0] == 0 and spans[-1][1] == rows[case]
            assert all(a[1] == b[0] for a, b in zip(spans, spans[1:]))
        pieces_most = max(pieces_most, max(pieces))
        # no share above the mean by more than a piece's fill and the rounding of its ends
        assert max(cost) <= (sum(rows) + fill * len(rows)) / slots + 2 * fill + 16 + 2 * rs
    assert pieces_most > 2 and padded > 0  # the cases reach several pieces a share, and lists with empty items


def test_lists_that_do_not_fit_are_refused(run):
    assert run([(2, 1, 2, [20, 20, 20])]) == [[0, 0]]


def segment(ny, strips, resident, rs, fill):
    best = None
    for nseg in range(1, -(-ny // rs) + 1):
        length = -(-(-(-ny // nseg)) // rs) * rs
        if -(-ny // length) != nseg:
            continue  # rounding merged two segments
        cost = -(-strips * nseg // resident) * (length + fill)
        if best is None or cost < best[0]:
            best = cost, length
    return best[1] if best else ny


def test_segment_length_is_the_best_of_all(run):
    r = random.Random(9)
    asked = []
    for _ in range(4000):
        rs = r.choice((1, 2, 3, 4, 6, 8))
        ny = r.choice((r.randint(3, 40), r.randint(3, 700), r.randint(3, 3000)))
        strips = r.choice((1, r.randint(1, 40), r.randint(1, 3000)))
        asked.append((ny, strips, r.choice((152, 304, 456, 760, r.randint(1, 50))), rs, 3 * rs + rs * -(-6 // rs)))
    for q, got in zip(asked, run(asked, "segments")):
        assert got == segment(*q), q
