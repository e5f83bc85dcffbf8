"""The pinned host memory that a server asks for (csrc/cg_serve.h), compiled for the
host: the admission budget's bytes, no more than 1 GiB, in whole units."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2207_04350_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("serve")
    (d / "serve.cpp").write_text('#include <cstdio>\n#include <cstdlib>\n#include "cg_serve.h"\n'
                                 "int main(int, char** a) {\n"
                                 '  std::printf("%zu", cg::pinned_result_bytes(std::strtoull(a[1], nullptr, 10)));\n}\n')
    exe = str(d / "serve")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", exe, str(d / "serve.cpp")], check=True)
    return exe


@pytest.mark.parametrize("budget,pinned", [
    (1, 0), (65535, 0), (65536, 65536), ((16 << 20) + 1, 16 << 20), ((1 << 30) - 1, (1 << 30) - 65536),
    (1 << 30, 1 << 30), (150 << 30, 1 << 30), ((1 << 64) - 1, 1 << 30)])
def test_pinned_memory_follows_the_budget(program, budget, pinned):
    assert int(subprocess.run([program, str(budget)], capture_output=True, text=True, check=True).stdout) == pinned
