"""The shape codes that choose an unrolled tensor kernel (csrc/tensor_shapes.h,
compiled here as plain C++): over every node the library accepts (children of
1 term up, at most 13 output terms), sorted as the launchers sort them, a code
stands for exactly that node's terms, and no node without a compiled kernel has
one. ckks_tensor takes single polynomials, so nodes of one term count too."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "paper_2601_15401_gb300/csrc/tensor_shapes.h"
#include <cstdio>
using namespace ckks;
int main() {
    for (int a = 1; a <= 13; ++a)
        for (int b = 1; b <= a; ++b) {
            printf("2 %d %d 0 %d\n", a, b, tensor_fixed_code(2, a, b, 0));
            for (int c = 1; c <= b; ++c) printf("3 %d %d %d %d\n", a, b, c, tensor_fixed_code(3, a, b, c));
        }
    for (int a = 1; a <= 13; ++a) printf("1 %d 0 0 %d\n", a, tensor_fixed_code(1, a, 0, 0));
    printf("4 2 2 2 %d\n", tensor_fixed_code(4, 2, 2, 2));
    printf("small %d\n", kTensorSmallCode);
    for (int i = 0; i < kTensorShapeCount; ++i)
        printf("shape %d %d %d\n", kTensorShapes[i].a, kTensorShapes[i].b, kTensorShapes[i].c);
}
"""


def test_a_code_stands_for_exactly_its_terms(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "codes.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "codes"
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", ROOT, "-o", str(exe), str(src)], check=True)
    lines = [x.split() for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n") if x]
    shapes = [tuple(map(int, x[1:])) for x in lines if x[0] == "shape"]
    small = int(next(x[1] for x in lines if x[0] == "small"))
    assert len(set(shapes)) == len(shapes)
    assert [max(s) <= 3 for s in shapes] == [i >= small for i in range(len(shapes))]
    for x in lines:
        if x[0] in ("shape", "small"):
            continue
        m, a, b, c, code = map(int, x)
        if m in (2, 3) and (a, b, c) in shapes:
            assert code == shapes.index((a, b, c)), x
            assert all(t >= 2 for t in (a, b, c)[:m])   # kernels for ciphertexts and larger tuples only
        else:
            assert code == -1, x
