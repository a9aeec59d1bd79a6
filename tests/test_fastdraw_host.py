"""The closed-form draw against 64-bit running sums, on the host: where a row is
usable its answers are those of the sums, and it answers nearly always, so the
draws that the GPU tests compare do take it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N = 20_000


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("fastdraw") / "fastdraw_host")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2603_01122_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fastdraw_host.cu"), "-o", exe], check=True)

    def run(cases):
        text = "".join(f"{K} {kappa} {share} {seed} {n}\n" for K, kappa, share, seed, n in cases)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [[float(v) for v in line.split()] for line in out.splitlines()]

    return run


@pytest.mark.parametrize("K", [16, 20, 23, 36, 64])
def test_answers_are_those_of_the_sums(check, K):
    """Every answer is the heading of the sums, with u anywhere and with u next to
    a boundary; most draws get one (one in some thousands is left open up to
    |kappa| = 2, one in 45 at 3, where the table's start is coarse)."""
    cases = [(K, kappa, share, 7 + i, N) for i, kappa in enumerate((-3.0, -1.0, 0.0, 0.02, 0.5, 1.5, 2.999))
             for share in (1e-4, 0.1, 0.5, 1.0)]
    for case, (usable, open_uniform, open_edge, wrong, tol) in zip(cases, check(cases)):
        assert usable and wrong == 0, case
        assert open_uniform < 0.1 * N and open_edge > 0.3 * N, (case, open_uniform, open_edge, tol)


def test_no_row_beyond_the_usable_kappa(check):
    assert [r[0] for r in check([(36, k, 0.5, 1, 10) for k in (3.1, -3.1, 100.0, float("inf"), float("nan"))])] == [0] * 5
