"""Integration's kernels may start before their predecessor has finished, so what
the predecessor writes must not be read through the read-only path, which wants
data that is constant while the kernel lives: neither by __ldg nor through a
pointer that is const and __restrict__ (the compiler then takes that path).
Read from the source: nothing observable tells the two apart."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_1905_02082_gb300", "csrc", "rf_integrate.cu")

# kernel -> inputs that its predecessor may write (k_frustum's: the caller's)
WRITTEN = {"k_frustum": ["mask", "T", "n_blocks"], "k_cull": ["tilemax"], "k_integrate": ["cand"], "k_nbr_fixup": []}


@pytest.fixture(scope="module")
def source():
    with open(SOURCE) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_every_programmatic_launch_is_listed(source):
    launched = set(re.findall(r"launch_after\(\s*vol,[^;]*?(k_\w+)", source))
    assert launched == set(WRITTEN)


@pytest.mark.parametrize("kernel", sorted(WRITTEN))
def test_predecessors_data_is_read_by_ordinary_loads(source, kernel):
    params = re.search(r"__global__[^;{]*?\b" + kernel + r"\(([^)]*)\)", source).group(1)
    for name in WRITTEN[kernel]:
        decl = [p for p in params.split(",") if re.search(r"\b" + name + r"$", p.strip())]
        assert len(decl) == 1 and "__restrict__" not in decl[0]
        assert not re.search(r"__ldg\(\s*" + name + r"\b", source)
    # the blocks inserted by k_integrate, looked up by k_nbr_fixup
    assert all(m == "<false>" for m in re.findall(r"\bhash_find(<\w+>)?\(", source))
