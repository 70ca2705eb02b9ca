"""The host runtime's bookkeeping on the CPU: tests/helpers/host_runtime.cpp links the
runtime against a CUDA whose device memory is host memory and whose copies and
launches are only noted."""
import os
import subprocess

import pytest

from paper_2104_10073_gb300 import build, zmc

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    build.build()  # writes the header with the run-time compiled sources
    exe = str(tmp_path_factory.mktemp("host") / "host_runtime")
    csrc = os.path.join(ROOT, "paper_2104_10073_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "include"),
                    "-I", csrc, "-I", os.path.join(ROOT, "paper_2104_10073_gb300", "_build"),
                    "-I", "/usr/local/cuda/include",
                    os.path.join(ROOT, "tests", "helpers", "host_runtime.cpp"),
                    *[os.path.join(csrc, f"zmc_{s}.cpp")
                      for s in ("runtime", "tune", "pool", "polyroots")],
                    "-o", exe, "-ldl"], check=True)

    def call(*args):
        out = subprocess.run([exe, *args], capture_output=True, text=True, check=True, timeout=60)
        return out.stdout.splitlines()

    return call


def test_copies_join_only_what_is_consecutive(run):
    assert run("upload_gap") == ["0 160", "2048 522"]


def test_user_call_leaves_a_plan_between_its_tables_alone(run):
    assert run("udf_next_to_plan") == ["0 0"]


@pytest.mark.parametrize("context", ["two_tables", "two_serving_tables"])
def test_a_plans_scratch_takes_no_room_from_a_later_table(run, context):
    assert run(context) == ["1 1"]


def test_taking_scratch_back_makes_records_and_writes_no_result(run):
    assert run("scratch_taken_after_sampling") == ["1", "records split 1000"]


@pytest.mark.parametrize("rows,taken,whole", [(1000, 1, 1), (100000, 0, 0)])
def test_no_more_scratch_is_taken_back_than_makes_room(run, rows, taken, whole):
    assert run("scratch_taken_from", str(rows)) == [str(taken), str(whole)]


def test_a_cuda_error_while_scratch_is_taken_back_is_reported(run):
    assert run("scratch_cannot_be_taken") == [str(zmc.ZMC_ECUDA)] * 2


def test_scratch_comes_back_when_there_is_room_again(run):
    assert run("scratch_comes_back") == ["1000 0 1000"]


def test_a_callers_graph_of_the_sampling_stage_resets_the_counters(run):
    assert run("captured_by_a_caller") == [
        "memset; batched 2 split 1000; ",
        "finish split 1000; ",
        "memset; batched 2 split 1000; ",  # the graph may have been replayed in between
        "device sync; records split 1000; "]


def test_geometry_tuner_times_what_runs_and_leaves_small_launches_spread(run):
    # one row of 7 chunks, the last of 160 samples: 56 units, one warp per block and SM
    assert run("tuned_geometry") == ["batched 2 split 2432", "0 56 32 2"]


def test_split_rule(run):
    """Resident warps 2432: nothing beyond the lines near two and four warps per scheduler,
    half a wave of equal chunks above one unless the work ends on two warps per scheduler
    or fits one wave, a wave of unlike ones, and no constant."""
    assert run("split_rule") == ["1 851 0 0 1217 1629 0 0 1216 1216 ",
                                 "1 972 0 0 1217 1945 0 0 1216 1216 ",
                                 "1216 1216 0 0 1216 1216 1216 0 1216",
                                 "0 2000 2432 0"]
