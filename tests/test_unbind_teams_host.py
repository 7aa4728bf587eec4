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
    src.write_text('#include <cstdio>\n#include "unbind_teams.cuh"\nusing namespace cwthf;\nint main() {\n' + body + "\n}\n")
    subprocess.run(["g++", "-std=c++17", "-I", str(CSRC), str(src), "-o", str(tmp_path / "t")], check=True)
    return subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]


@pytest.mark.parametrize("want", [8, 64])
def test_a_team_fits_any_launch(tmp_path, want):
    out = _run(tmp_path, f'for (int c = 1; c <= 1024; c++) printf("%d\\n", ub_team_ctas({want}, c));')
    assert [int(x) for x in out] == [min(want, c) for c in range(1, 1025)]
