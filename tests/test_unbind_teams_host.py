"""The rule that shares the self-boundness check's larger groups among CTAs, compiled for
the host: in a launch of any number of CTAs every group finds a team that takes it."""
import subprocess
from pathlib import Path

import pytest

import paper_2501_10622_gb300 as pkg

CSRC = Path(pkg.__file__).parent / "csrc"


def _run(tmp_path, body):
    """The lines that `body`, a main's statements, prints."""
    src = tmp_path / "t.cpp"
    src.write_text('#include <cstdio>\n#include "unbind_teams.cuh"\nusing namespace cwthf;\n'
                   "int main() {\n" + body + "\n}\n")
    subprocess.run(["g++", "-std=c++17", "-I", str(CSRC), str(src), "-o", str(tmp_path / "t")], check=True)
    return subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]


@pytest.mark.parametrize("want", [8, 64])
def test_a_team_fits_any_launch(tmp_path, want):
    out = _run(tmp_path, f'for (int c = 1; c <= 1024; c++) printf("%d\\n", ub_team_ctas({want}, c));')
    assert [int(x) for x in out] == [min(want, c) for c in range(1, 1025)]


def _ways(tmp_path, kind, cases):
    body = "".join(f'printf("%d\\n", ub_{kind}_way({n}ll, {total}ll, {ctas}));\n' for n, total, ctas in cases)
    return [int(x) for x in _run(tmp_path, body)]


def test_few_groups_take_many_ctas_and_many_take_few(tmp_path):
    sizes = [int(x) for x in _run(tmp_path, 'for (int w = 0; w < kUbWays; w++) printf("%d\\n", ub_team_size(w));')]
    assert sizes == [1024, 128, 64, 8, 4, 2, 1]
    n, count = [2049, 4000, 5000, 40000, 65536], [1, 38, 100, 300, 2000]
    cases = [(a, a * c, 304) for a in n for c in count]
    for (a, total, ctas), way in zip(cases, _ways(tmp_path, "medium", cases)):
        assert sizes[way] == max(s for s in (1, 2, 4, 8) if s <= max(1, ctas * a // total, a // 4096)), (a, total)
    big = [(1 << 20, 1 << 20, 304), (131072, 131072, 304), (70000, 70000, 304), (300000, 600000, 304),
           (300000, 900000, 304), (65537, 1 << 30, 304)]
    assert [sizes[w] for w in _ways(tmp_path, "big", big)] == [128, 128, 64, 128, 64, 64]


@pytest.mark.parametrize("ctas", [1, 5, 8, 40, 64, 152, 304, 1024])
def test_ways_of_any_launch(tmp_path, ctas):
    # shares and products stay in range, and the teams' control words are enough for the launch
    sizes = [2049, 65536, 65537, 1 << 20]
    cases = [(n, t, ctas) for n in sizes for t in (n, 2 ** 31 - 1)]
    ways = _ways(tmp_path, "medium", cases) + _ways(tmp_path, "big", cases)
    assert all(3 <= w <= 6 for w in ways[:len(cases)]) and all(w in (1, 2) for w in ways[len(cases):])
    out = _run(tmp_path, f"""for (int w = 0; w < kUbWays; w++) {{
        int size = ub_team_ctas(ub_team_size(w), {ctas});
        printf("%d\\n", {ctas} / size <= ub_first_team(w + 1) - ub_first_team(w) || size < ub_team_size(w));
    }}""")
    assert out == ["1"] * 7
