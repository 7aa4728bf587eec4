"""What programmatic launches ask of every kernel's source (its blocks may start while the
kernel before it still writes): the wait comes first, and no pointer parameter is read-only
and __restrict__, which would tell the compiler that the data never change while the kernel
is resident and so let a load pass the wait or stay in a cache that it does not refresh."""
import re
from pathlib import Path

import paper_2501_10622_gb300 as pkg

SOURCES = sorted((Path(pkg.__file__).parent / "csrc").glob("*.cu*"))


def _kernels():
    """(file, name, parameters, body's beginning) of every kernel."""
    for path in SOURCES:
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", path.read_text(), flags=re.S)
        for m in re.finditer(r"__global__[^{;]*?(\w+)\s*\(((?:[^(){}]|\([^(){}]*\))*)\)\s*\{([^;]*;)", text):
            yield path.name, m.group(1), m.group(2), m.group(3).strip()


def test_every_kernel_is_seen():
    n = sum(len(re.findall(r"__global__", re.sub(r"//[^\n]*", "", p.read_text()))) for p in SOURCES)
    assert n == len(list(_kernels())) > 40


def test_the_wait_is_the_first_statement():
    assert not [k[:2] for k in _kernels() if k[3] != "pdl_wait();"]


def test_no_input_is_declared_unchanging():
    bad = [(f, name) for f, name, params, _ in _kernels()
           for p in params.split(",") if re.search(r"\bconst\b[^*]*\*\s*__restrict__", p)]
    assert not bad, bad
