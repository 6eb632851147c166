"""The kernels of the two-level preconditioner's coarse space on their own
(tests/gpu/coarse_main.cu, linked against the library)."""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build
    lib = build.build()
    out = str(tmp_path_factory.mktemp("coarse") / "coarse_main")
    subprocess.check_call([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "-cudart", "shared", "-I", build.CSRC, "-I",
                           os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "gpu", "coarse_main.cu"), lib,
                           "-Xlinker", "-rpath=" + os.path.dirname(lib), "-o", out])
    return out


def _run(exe, *args):
    return float(subprocess.check_output([exe, *[str(a) for a in args]], text=True, timeout=120))


def _corner_leaves(dim, top):
    """A level-2 grid refined towards the box corner to level `top`, Morton order."""
    lev, anc = [], []

    def visit(level, a):
        s = 1 << (top - level)
        if level < 2 or (level < top and all(x == 0 for x in a)):
            for c in range(1 << dim):
                visit(level + 1, [x + ((c >> d) & 1) * s // 2 for d, x in enumerate(a)])
        else:
            lev.append(level)
            anc.append(a)

    visit(0, [0] * dim)
    return np.array(lev, np.uint8), np.array(anc, np.uint32)


@pytest.mark.parametrize("entries", [1, 7, 63, 64, 65, 127, 1000, 1024])
def test_sums_of_the_operator_build(exe, entries):
    assert _run(exe, "gather", entries) <= 1.0


@pytest.mark.parametrize("entries", [1, 8, 31, 32, 33, 125, 1000, 1024])
def test_sums_of_the_restriction(exe, entries):
    assert _run(exe, "restrict", entries) <= 1.0


@pytest.mark.parametrize("pieces", [1, 7, 8, 9, 100])
def test_sum_of_the_pieces(exe, pieces):
    assert _run(exe, "pieces", pieces) <= 1.0


# 2D products are floats down to 12 levels below the coarse grid, 3D ones to 8
@pytest.mark.parametrize("dim,top", [(2, 8), (2, 13), (2, 15), (2, 20), (3, 6), (3, 9), (3, 11), (3, 20)])
def test_restriction_is_the_transpose_of_the_prolongation(exe, tmp_path, dim, top):
    lev, anc = _corner_leaves(dim, top)
    path = str(tmp_path / "leaves.bin")
    with open(path, "wb") as f:
        f.write(np.int64(len(lev)).tobytes() + np.int32(dim).tobytes() + np.int32(top).tobytes() + lev.tobytes() + anc.tobytes())
    assert _run(exe, "weights", path, 1) <= 1.0
