"""Host logic of the matrix-instruction products' lists (csrc/hm_lists.h, build_mm_lists),
compiled with the host compiler and walked as the kernels walk them: index bounds, load
alignment, every T pair written once, and the sums of both stages equal to the blocks'
products in exact integers.  A damaged list set must fail."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2307_03968_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("mm_lists") / "mm_lists_check")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror", "-fsanitize=address,undefined", "-I", CSRC,
                    "-o", exe, os.path.join(HERE, "mm_lists_check.cpp")], check=True)
    return exe


@pytest.mark.parametrize("mode,target,ok", [(0, 608, True), (0, 8, True), (1, 608, True), (2, 100, True), (3, 608, True),
                                            (4, 608, True), (5, 608, False)])
@pytest.mark.parametrize("seed", [1, 2])
def test_lists_give_the_products(checker, seed, mode, target, ok):
    p = subprocess.run([checker, str(seed), str(mode), str(target)], capture_output=True, text=True)
    assert (p.returncode == 0) == ok and p.stdout.startswith("ok" if ok else "FAIL"), p.stdout + p.stderr
