"""When the members of a graph ensemble start (psc_batch_plan.h): host arithmetic,
compiled here and checked for the sizes the rule has to be right at."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MB = 1 << 20
BUDGET = 320 * MB
BYTES = {32: 2 * MB, 64: 15 * MB, 96: 50 * MB, 128: 119 * MB, 192: 390 * MB, 256: 940 * MB, 512: 7400 * MB,
         1024: 59000 * MB}

MAIN = """
#include <cstdio>
#include "psc_batch_plan.h"
int main() {
  std::vector<psc::PlanMember> m;
  long long b;
  int N;
  while (std::scanf("%lld %d", &b, &N) == 2) m.push_back(psc::PlanMember{(size_t)b, N});
  for (const auto& s : psc::batch_plan(m)) {
    std::printf("%d %d %d", s.member, s.share, (int)s.crowd);
    for (int a : s.after) std::printf(" %d", a);
    std::printf("\\n");
  }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("plan")
    (d / "main.cpp").write_text(MAIN)
    subprocess.check_call([cc, "-std=c++17", "-I" + os.path.join(ROOT, "paper_2012_04838_gb300", "csrc"),
                           str(d / "main.cpp"), "-o", str(d / "plan")])

    def run(sizes):
        text = "".join("%d %d\n" % (BYTES[N], N) for N in sizes)
        out = subprocess.run([str(d / "plan")], input=text, stdout=subprocess.PIPE, check=True, text=True).stdout
        rows = [[int(v) for v in line.split()] for line in out.splitlines()]
        return [(r[0], r[1], bool(r[2]), r[3:]) for r in rows]  # member, share, crowd, after

    return run


@pytest.mark.parametrize("sizes", [[64], [256], [512], [1024], [192] * 2, [192] * 4, [256] * 3, [512] * 2, [128] * 3,
                                   [96] * 8, [256] + [64] * 8, [192] + [64] * 8, [1024, 64]])
def test_few_members_start_together(plan, sizes):
    for member, share, crowd, after in plan(sizes):
        assert after == []
        assert share == len(sizes)
        # a member alone, and a grid that fills the chip, keep the variants measured for them
        if len(sizes) == 1 or sizes[member] >= 512:
            assert not crowd


@pytest.mark.parametrize("sizes", [[64] * 48 + [96] * 12 + [128] * 3, [64] * 64 + [96] * 16 + [128] * 4, [96] * 40,
                                   [256] + [64] * 60, [256] * 2 + [192] * 2 + [128] * 2 + [96] * 2 + [64] * 2,
                                   [1024] * 9])
def test_many_members_within_the_budget(plan, sizes):
    rows = plan(sizes)
    assert sorted(r[0] for r in rows) == list(range(len(sizes)))
    cost = [min(BYTES[N], BUDGET // 4) for N in sizes]
    started, over = [], set()
    for member, share, crowd, after in rows:
        assert set(after) <= set(started)  # only what has been started is waited for
        over |= set(after)
        started.append(member)
        under_way = [i for i in started if i not in over]
        assert sum(cost[i] for i in under_way) <= BUDGET
        assert 1 <= share <= len(sizes)
        assert crowd == (sizes[member] < 512)
    assert over  # the budget does hold members back
    # however large, four members may run side by side
    assert all(r[3] == [] for r in rows[:4])


def test_a_member_above_the_budget_leaves_room_for_small_ones(plan):
    first = {r[0]: r for r in plan([256] + [64] * 60)}
    beside = [i for i in range(1, 61) if first[i][3] == []]
    assert len(beside) >= 8
