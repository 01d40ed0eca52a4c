"""The layout of a launch, checked on the host with the kernels' own functions, and device functions by themselves."""
import os
import subprocess

import pytest

from paper_1912_00167_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def _host_program(tmp_path, name):
    build.build()
    exe = str(tmp_path / name)
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-std=c++17", "-gencode",
                           "arch=compute_100a,code=sm_100a", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                           "-o", exe, os.path.join(HERE, name + ".cu"), build.LIB, "-Xlinker", "-rpath=" + build.PKG])
    return exe


def test_rows_that_are_read_without_a_look_at_the_row_exist(tmp_path):
    """Every group of every block, those without a tile too: no row, next row or bootstrap value beyond the tensors."""
    done = subprocess.run([_host_program(tmp_path, "geometry_check")], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout


def test_a_stage_is_handed_back_behind_the_whole_warps_reads():
    """Lanes other than the one that arrives copy bytes of a stage: the one place that arrives at an "empty" barrier has
    the warp's barrier in front of the arrival, and both kernels hand their stages back through it."""
    read = lambda name: open(os.path.join(build.CSRC, name)).read()
    body = read("impact_flat.cuh").split("void hand_back_stage(")[1].split("\n}")[0]
    assert 0 <= body.find("__syncwarp();") < body.find("mbarrier.arrive")
    for name in ("impact_categorical.cuh", "impact_gaussian.cu"):
        arrivals = [line for line in read(name).splitlines() if "empty_bar[" in line and "init" not in line and "test" not in line]
        uses = [line for line in arrivals if "__shared__" not in line]
        assert uses and all("hand_back_stage(" in line for line in uses), uses


def test_launches_that_take_a_companion(tmp_path):
    done = subprocess.run([_host_program(tmp_path, "companion_check")], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout


def test_every_wide_row_has_its_lanes(tmp_path):
    done = subprocess.run([_host_program(tmp_path, "wide_check")], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout


def test_bytes_outside_one_range_are_not_read_in_place(tmp_path):
    """A kernel reads host memory only where all of it lies in one pinned range: the arithmetic of that."""
    done = subprocess.run([_host_program(tmp_path, "pinned_check")], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout


def test_the_host_finds_the_state_that_the_last_step_left(tmp_path):
    done = subprocess.run([_host_program(tmp_path, "ring_check")], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout


@pytest.mark.gpu
def test_what_counts_as_one_pinned_range(tmp_path):
    """Allocations and registrations, and two registrations with a hole between them (pointers only, nothing is read)."""
    done = subprocess.run([_host_program(tmp_path, "pinned_check"), "driver"], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout + done.stderr


@pytest.mark.gpu
def test_a_wait_that_gives_up_raises_the_error_word(tmp_path):
    """Waits for a value that nothing ever brings return after their limit and say so in the workspace's error word."""
    done = subprocess.run([_host_program(tmp_path, "wait_check")], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout + done.stderr


@pytest.mark.gpu
def test_a_ring_step_whose_wait_gives_up_leaves_a_whole_batch(tmp_path):
    """...and a handle that is told so goes on."""
    done = subprocess.run([_host_program(tmp_path, "ring_check"), "steps"], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout + done.stderr


@pytest.mark.gpu
def test_what_comes_after_a_tile_has_the_same_bits_wherever_it_is_found(tmp_path):
    """Values published or not, near or far."""
    done = subprocess.run([_host_program(tmp_path, "lookback_check")], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout + done.stderr


@pytest.mark.gpu
def test_the_reciprocal_is_as_good_as_a_rounded_one(tmp_path):
    done = subprocess.run([_host_program(tmp_path, "reciprocal_check")], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout + done.stderr
