"""The library's host code around its kernels, compiled into small check programs that run on
the CPU with a stand-in for the CUDA runtime (fake_runtime.cuh)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1801_10277_gb300", "csrc")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    """check(program, *arguments): tests/<program>.cu compiled once and run with no GPU visible."""
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    where, built = tmp_path_factory.mktemp("checks"), {}

    def run(program, *args):
        if program not in built:
            exe = str(where / program)
            r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode",
                                "arch=compute_103a,code=compute_103a", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                                "-I", HERE, os.path.join(HERE, program + ".cu"), "-o", exe],
                               capture_output=True, text=True)
            assert r.returncode == 0, r.stdout + r.stderr
            built[program] = exe
        r = subprocess.run([built[program], *map(str, args)], capture_output=True, text=True, timeout=300,
                           env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout

    return run


def test_a_failed_launch_leaves_no_ready_flags(check):
    check("item_launch_check", "flags")


def test_a_second_device_gets_its_own_set_up(check):
    check("item_launch_check", "devices")


def test_trust_region_shared_memory_alignment(check):
    check("fit_layout_check")


@pytest.mark.parametrize("schedule", ["colour", "cyclades"])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32only"])
def test_device_memory_of_a_fit(check, precision, schedule):
    check("fit_memory_check", precision, schedule)


def test_device_memory_of_a_problem(check):
    check("api_check", "memory")


def test_a_new_problem_is_settled(check):
    check("api_check", "settled")


def test_autotune_times_the_map_passes_that_run(check):
    check("api_check", "autotune")


def test_order_of_multiply_covered_pixels(check):
    check("cover_order_check")


def test_hessian_sums_match_the_pixel_frame(check):
    """As accurate as the pixel-frame formulas in the same type: at most twice their worst error of
    a quantity's scale (and 1e-6, or that many rounding units in FP64, for none at all).  A wrong
    index or a dropped term gives order one."""
    rows = {tuple(line.split()[:2]): tuple(map(float, line.split()[2:]))
            for line in check("base_sums_check").splitlines()}
    assert len(rows) == 10
    for (kind, name), (kernel, formulas) in rows.items():
        assert kernel <= 2.0 * formulas + 1e-6 * (1.0 if kind == "float" else 2.0 ** -29), (kind, name, kernel, formulas)
