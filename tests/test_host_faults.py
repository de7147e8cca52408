"""The host code of the library (csrc/lbm_axi.cu, csrc/lbm_batch.cu) driven on
the CPU over a CUDA runtime that only keeps books (tests/fake_cuda.cpp): what it
launches after an allocation has failed, under a caller's stream capture, and
on device memory that is too short."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1512_01977_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    exe = str(tmp_path_factory.mktemp("host") / "host_faults")
    srcs = [os.path.join(CSRC, f) for f in ("lbm_axi.cu", "lbm_batch.cu", "lbm_tiles.cu", "eos_host.cu")]
    cmd = ["g++", "-std=c++17", "-O1", "-x", "c++", "-I", cuda, "-I", os.path.join(ROOT, "include"), "-I", CSRC, *srcs,
           os.path.join(ROOT, "tests", "fake_cuda.cpp"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def _run(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (what, r.returncode, r.stderr)


@pytest.mark.parametrize("what", ["retune_device_warps", "retune_host_warps", "retune_host_many",
                                  "retune_device_phases", "retune_host_fp64"])
def test_batch_keeps_its_plan_when_a_new_one_fails(program, what):
    _run(program, what)


@pytest.mark.parametrize("what", ["capture32", "capture64"])
def test_steps_can_be_captured(program, what):
    _run(program, what)


@pytest.mark.parametrize("what", ["short32", "short64"])
def test_fields_are_not_written_past_an_allocation(program, what):
    _run(program, what)


@pytest.mark.parametrize("what", ["create_phases", "create_fp64", "create_warps", "create_ctas"])
def test_creation_reports_that_memory_ran_out(program, what):
    _run(program, what)


def test_a_step_of_a_large_batch_is_one_launch(program):
    _run(program, "launches")


def test_forms_go_by_whole_tiles(program):
    _run(program, "forms")


def test_steps_on_the_legacy_stream(program):
    _run(program, "legacy_stream")


def test_plan_of_the_warp_march(program):
    _run(program, "warp_plan")
