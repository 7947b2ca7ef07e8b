"""How many RVEs the engine advances at once: read from its header and evaluated on the CPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1504_07499_gb300", "csrc")


@pytest.fixture(scope="module")
def branches(tmp_path_factory):
    d = tmp_path_factory.mktemp("branches")
    (d / "b.cpp").write_text('#include <cstdio>\n#include <cstdlib>\n#include "hmg_branches.h"\n'
                             "int main(int, char** v) {\n"
                             '    std::printf("%zu\\n", hmg::side_branches(strtoull(v[1], 0, 10), strtoull(v[2], 0, 10)));\n}\n')
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "b.cpp"), "-o", str(d / "b")], check=True)
    return lambda Ns: int(subprocess.run([str(d / "b"), str(len(Ns)), str(sum(72 * n ** 3 for n in Ns))],
                                         capture_output=True, text=True, check=True).stdout)


@pytest.mark.parametrize("Ns,want", [([16] * 48, 16), ([8], 16), ([32] * 24, 16), ([48] * 12, 8), ([64] * 12, 3),
                                     ([64] * 5 + [96] * 4 + [128] * 3, 3), ([512], 3), ([16] * 8 + [32] * 8 + [48] * 8, 16),
                                     ([], 3)])
def test_small_grids_take_more_branches(branches, Ns, want):
    assert branches(Ns) == want
