"""The C API's launch order on the host: capi.cpp built with the host compiler against a
fake CUDA runtime and fake launches (tests/capi_probe.cpp), which record for every
launch the launches that are sure to have finished before it."""
import os
import shutil
import subprocess

import pytest

from test_plan_host import CSRC, ROOT, _cuda_include


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    cxx, inc = shutil.which("g++") or shutil.which("c++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("host C++ compiler or CUDA headers not found")
    exe = str(tmp_path_factory.mktemp("capi") / "capi_probe")
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-I", inc, "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    os.path.join(ROOT, "tests", "capi_probe.cpp"), os.path.join(CSRC, "pass_plan.cpp"), "-o", exe],
                   check=True, capture_output=True, text=True)
    env = {k: v for k, v in os.environ.items() if not k.startswith("RPIV_")}

    def run(text, extra_env=None):
        out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True, env={**env, **(extra_env or {})})
        return [[int(x) for x in line.split()] for line in out.stdout.strip().split("\n")]
    return run


FRAMES = {0: "256 256", 1: "3341 630"}  # host frames: 4.2 MB per pair, a part each


@pytest.mark.parametrize("host", [0, 1])
@pytest.mark.parametrize("n", [2, 4, 15, 16, 17, 33, 64])
def test_predictors_in_other_parts_outputs_are_read_before_they_are_written(probe, n, host):
    shifts = sorted({0, 1, n // 2, n - 1})
    res = probe("".join(f"batch {FRAMES[host]} {n} {host} {k}\n" for k in shifts))
    for shift, (status, parts, unordered, _) in zip(shifts, res):
        assert status == 0 and unordered == 0, (shift, parts)
        if shift and n > 1 and (host or n >= 16):
            assert parts == 1  # some pair's predictor lies in another part's outputs


@pytest.mark.parametrize("host", [0, 1])
def test_calls_whose_parts_do_not_conflict_stay_in_parts(probe, host):
    # predictors in memory of their own, and in the pair's own outputs
    for shift in (-1, 0):
        res = probe("".join(f"batch {FRAMES[host]} {n} {host} {shift}\n" for n in (1, 4, 16, 33)))
        assert [r[:2] for r in res] == [[0, p] for p in ((1, 4, 4, 4) if host else (1, 1, 2, 2))]


@pytest.mark.parametrize("setting", ["0", "1"])
def test_parts_can_be_turned_off(probe, setting):
    text = "".join(f"batch {FRAMES[host]} {n} {host} -1\n" for host in (0, 1) for n in (4, 16, 33))
    assert [r[1] for r in probe(text, {"RPIV_SPLIT_BATCH": setting})] == [1] * 6
    assert [r[1] for r in probe(text, {"RPIV_SPLIT_BATCH": "4"})] == [1, 2, 4, 4, 4, 4]


def test_a_score_workspace_that_could_not_be_initialised_is_not_used(probe):
    # three calls, the first one's initialisation fails (status CUDA); per call: status,
    # initialisations done, evaluations launched
    assert probe("adjoint\n") == [[4, 0, 0, 0, 1, 1, 0, 1, 2]]


def test_only_later_parts_uploads_make_room_for_passes(probe):
    # the first part's upload runs before any pass, with the device to itself
    res = probe("".join(f"batch {FRAMES[1]} {n} 1 -1\n" for n in (1, 2, 4, 33)))
    assert [r[3] for r in res] == [r[1] - 1 for r in res] == [0, 1, 3, 3]


def test_parts_too_small_to_be_cut_upload_side_by_side(probe):
    # 17 frames of 0.2 MB: two parts, neither of which waits for the other's upload or makes room for it
    assert probe("batch 519 403 17 1 -1\n") == [[0, 2, 0, 0]]
