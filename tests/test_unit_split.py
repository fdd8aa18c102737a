"""How the CTAs of a column tile share the rows of a product or the hidden units
of a cell (csrc/unit_split.h), on the host: whatever the order of the block
sizes, no CTA is given much more than the mean."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1911_08020_gb300 import build as darb_build

MAIN = r"""
#include "unit_split.h"
#include <cstdio>
#include <thread>
#include <vector>
int main() {
    long rows, gates, members;
    if (std::scanf("%ld %ld %ld", &rows, &gates, &members) != 3) return 1;
    std::vector<int64_t> prefix(1, 0);
    for (long r = 0, c; r < rows; ++r) {
        if (std::scanf("%ld", &c) != 1) return 1;
        prefix.push_back(prefix.back() + c);
    }
    darb::UnitSplits splits;
    splits.set(prefix.data(), rows / gates, int(gates));
    const darb::UnitSplit *seen[8];
    std::vector<std::thread> threads;   // any thread may be the first to ask
    for (int i = 0; i < 8; ++i)
        threads.emplace_back([&, i] {
            static thread_local darb::UnitSplit local;
            seen[i] = &splits.get(int(members), local);
        });
    for (auto &t : threads) t.join();
    for (int i = 1; i < 8; ++i) if (seen[i] != seen[0]) return 2;
    const darb::UnitSplit &s = *seen[0];
    std::printf("%ld %d %ld %d %d\n", long(s.by_cost.busiest), s.by_cost.most_units, long(s.equal.busiest),
                s.equal.most_units, int(s.prefer_by_cost));
    for (long q = 0; q <= members; ++q) std::printf("%d ", s.start[q]);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("split")
    (d / "main.cc").write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", darb_build.CSRC, str(d / "main.cc"), "-o",
                    str(d / "main")], check=True)
    return os.path.join(d, "main")


def _split(program, cost, gates, members):
    r = subprocess.run([program], input=f"{len(cost)} {gates} {members}\n" + " ".join(map(str, cost)),
                       capture_output=True, text=True)
    assert r.returncode == 0, r.returncode
    head, starts = r.stdout.split("\n")
    return (*map(int, head.split()), np.array(starts.split(), np.int64))


def _costs(order, rows, cols):
    """Chunks of each row, and one more: `order` of its block sizes."""
    g = np.random.default_rng(5)
    m = {"tenth": np.r_[np.full(rows // 10, 4), np.full(rows - rows // 10, 64)],
         "tenth_last": np.r_[np.full(rows - rows // 10, 64), np.full(rows // 10, 4)],
         "half": np.r_[np.full(rows // 2, 8), np.full(rows - rows // 2, 64)],
         "sorted": np.sort(g.choice([8, 16, 32, 64], rows)),
         "mixed": g.choice([8, 16, 32, 64], rows),
         "equal": np.full(rows, 16),
         "extreme": np.r_[np.full(1, 1), np.full(rows - 1, 256)]}[order]
    return -(-(-(-cols // m)) // 8) + 1


@pytest.mark.parametrize("gates", [1, 4])
@pytest.mark.parametrize("members", [1, 19, 152])
@pytest.mark.parametrize("rows,cols", [(160, 300), (1024, 1024), (4096, 9216)])
@pytest.mark.parametrize("order", ["tenth", "tenth_last", "half", "sorted", "mixed", "equal", "extreme"])
def test_no_member_has_much_more_than_the_mean(program, order, rows, cols, members, gates):
    by_row = np.concatenate([np.random.default_rng(q).permutation(_costs("mixed", rows, cols)) if q else
                             _costs(order, rows, cols) for q in range(gates)])
    busiest, most, equal, most_equal, prefer, start = _split(program, by_row, gates, members)
    cost = by_row.reshape(gates, rows).sum(axis=0)   # of a unit: row u of every gate
    assert start[0] == 0 and start[-1] == rows and np.all(np.diff(start) >= 1)
    assert most == np.diff(start).max()
    assert busiest == np.add.reduceat(cost, start[:-1]).max()
    even = np.arange(members + 1) * rows // members
    assert equal == np.add.reduceat(cost, even[:-1]).max()
    assert most_equal == np.diff(even).max()
    assert bool(prefer) == (busiest < 0.95 * equal)
    # a range ends within half a unit of its share, but for the units left to later members
    if rows >= 4 * members and order != "extreme":
        assert busiest <= cost.sum() / members + cost.max()
    if gates == 1 and order == "equal":
        assert not prefer
    if gates == 1 and order in ("tenth", "half") and rows == 4096 and members > 1:
        assert prefer and busiest < 0.7 * equal
