"""A refused kernel launch fails the solve that made it, whichever launch it is, and leaves nothing
behind: the next solve succeeds and builds its graph anew.  The library runs on a fake CUDA
runtime on the host (launch_errors.cpp): no GPU, and none of the launches is a bad one."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HP_ERR_CUDA = "-4"


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import paper_1909_03948_gb300.hp as hp
    from paper_1909_03948_gb300 import build
    if not os.path.exists(hp.LIB_PATH):
        build.build()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime_api.h")):
        pytest.skip("no host compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("fake") / "launch_errors")
    lib = os.path.join(cuda, "lib64")
    subprocess.run(["g++", "-std=c++17", "-O1", "-rdynamic", "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "launch_errors.cpp"), "-o", exe,
                    hp.LIB_PATH, "-Wl,-rpath," + os.path.dirname(hp.LIB_PATH), "-Wl,-rpath," + lib, "-L" + lib],
                   check=True)

    def go(*args):
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout + r.stderr
        return [line.split() for line in r.stdout.splitlines()]
    return go


# levels run as legs (2D, for blocks and for one column), with a one-CTA coarse end (3D), a
# whole PCG in one CTA, and as per-level kernels (3D)
@pytest.mark.parametrize("dim,N,cols", [(2, 128, 5), (2, 128, 1), (2, 72, 5), (3, 24, 5), (2, 32, 3), (3, 32, 5)])
def test_every_refused_launch_fails_its_solve(run, dim, N, cols):
    head, *rows = run(dim, N, cols, 0)
    count = int(head[1])
    assert head[0] == "launches" and len(rows) == count > 0
    assert [r[1:] for r in rows] == [[HP_ERR_CUDA, "0", str(count)]] * count, rows


@pytest.mark.parametrize("dim,N,cols", [(3, 24, 5), (2, 32, 3)])
def test_refused_kernel_attribute_fails_the_solve(run, dim, N, cols):
    assert run(dim, N, cols, 1) == [["attribute", "1", HP_ERR_CUDA, "0"]]
