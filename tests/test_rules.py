"""The query loops' arithmetic rules (csrc/lb_rules.h), compiled alone: no GPU."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1711_00231_gb300", "csrc")


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    """call(expression) -> its value, from a C++ program that includes the rules."""
    d = tmp_path_factory.mktemp("rules")

    def run(*exprs):
        src = d / "rules.cpp"
        body = "".join(f'  printf("%llu\\n", (unsigned long long)({e}));\n' for e in exprs)
        src.write_text(f'#include <stdio.h>\n#include "lb_rules.h"\nusing namespace lbk;\nint main() {{\n{body}}}\n')
        exe = d / "rules"
        subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)])
        return [int(x) for x in subprocess.check_output([str(exe)]).split()]

    return run


def test_iteration_cap_never_below_the_vertices(call):
    # twice the vertices and some more, also where that passes 32 bits
    ns = [1, 2, 1000, 1 << 30, (1 << 31) - 100, (1 << 31) - 33, (1 << 31) - 2, (1 << 31) - 1]
    for n, k in zip(ns, call(*[f"threshold_levels({n}ll)" for n in ns])):
        assert k == min(2 * n + 66, 0xFFFFFFF0) and k > n


def test_work_left_at_the_iteration_cap_is_an_error(call):
    goes_on, done, cut = 0, 1, 2
    cases = [((0, 0, 5, 10), done), ((0, 0, 11, 10), done), ((1, 0, 10, 10), goes_on), ((1, 0, 11, 10), cut),
             ((0, 1, 10, 10), goes_on), ((0, 1, 11, 10), cut), ((1, 1, 11, 10), cut)]
    got = call(*["level_end({}, {}, {}u, {}u)".format(*args) for args, _ in cases])
    assert got == [want for _, want in cases]


def test_an_empty_list_is_no_iteration(call):
    assert call("level_after(7u, 0u)", "level_after(7u, 1u)", "level_after(7u, 4000000000u)") == [7, 8, 8]


def test_threshold_needs_a_growing_front(call):
    grid = [4 * (k + 1) for k in range(2000)]  # lists of a grid: longer by a little every iteration
    rand = [1 << k for k in range(18)] + [400000, 300000, 120000, 50000] + [40000 - 2000 * k for k in range(19)]
    exprs, want = [], []
    for lists, grows in ((grid, True), (rand, False)):
        for k in range(32, len(lists)):
            exprs.append(f"front_grows({lists[k]}ull, {k + 1}u, {sum(lists[:k + 1])}ull)")
            want.append(int(grows))
    assert call(*exprs) == want


def test_interval_widens_while_its_pull_costs_more_than_its_lists(call):
    big = 1 << 30
    cases = [  # delta, reads, lists, edges, least -> width
        ((8, 0, 8, 8 * 3000, 0), 8),            # cheap pull, lists of middle length: as it is
        ((8, 2048 * 8, 8, 8 * 3000, 0), 8),
        ((8, 2048 * 8 + 1, 8, 8 * 3000, 0), 16),  # the pull outweighs the lists
        ((8, 100000, 8, 8 * 3000, 0), 16),
        ((8, 100000, 8, 8 * 6000, 0), 16),      # also when the lists are long
        ((8, 2048 * 2, 8, 8 * 6000, 0), 8),     # narrower would soon be too costly
        ((8, 2048 * 2 - 1, 8, 8 * 6000, 0), 4),
        ((8, 0, 8, 8 * 1000, 0), 16),           # short lists
        ((8, 0, 8, 8 * 3000, 8 * 3000 + 1), 16),  # fewer edges than asked
        ((8, 0, 8, 8 * 6000, 2 * 6000), 8),
        ((1, 0, 8, 8 * 6000, 0), 1),
        ((big, 1 << 40, 8, 8, 0), big),
    ]
    got = call(*["next_width({}u, {}ull, {}u, {}ull, {}ull, 8192u, {}u)".format(*a, big) for a, _ in cases])
    assert got == [w for _, w in cases]
