"""Host logic of the solver on recorded launches (CPU): tests/launch_trace.cu runs the C ABI
with every launch and runtime call replaced by a recording stand-in."""
import re
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent


@pytest.fixture(scope="module")
def trace(tmp_path_factory):
    from paper_2402_09996_gb300 import build_lib

    exe = tmp_path_factory.mktemp("trace") / "launch_trace"
    subprocess.run([build_lib._nvcc(), "-std=c++17", "-O1", "-w", *build_lib.ARCH, "-I", str(ROOT / "include"),
                    "-o", str(exe), str(ROOT / "tests" / "launch_trace.cu")], check=True)

    def run(*args):
        out = subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True, text=True).stdout
        return re.search(r"-- begin\n(.*)-- end 0\n", out, re.S).group(1).splitlines()

    return run


@pytest.mark.parametrize("scenario", ["step_host", "step_graph", "group"])
def test_no_pass_goes_by_a_flag_that_its_own_launch_writes(trace, scenario):
    """The inverse y pass sets IterStatus::done (its side work) while its other CTAs start, so
    they go by another flag of the record; the forward one goes by done."""
    lines = [re.search(r"sign=(-?\d) kind=(\d) goes_by=(\w+)", t).groups() for t in trace(scenario) if t.startswith("line")]
    assert {("-1", "1"), ("1", "2")} == {t[:2] for t in lines}
    for sign, _, flag in lines:
        assert flag == ("done" if sign == "-1" else "status")


def test_material_tables_are_complete_when_the_call_returns(trace):
    """The handle's default stream is the calling thread's, so a step from another thread does
    not wait for work that rve_set_material leaves in flight."""
    calls = trace("material")
    assert "rate_table" in calls and calls[-1] == "sync"


def test_autotuner_times_the_pass_that_runs(trace):
    """The widths of the y tile are timed on the forward pass with its side work (an extra row
    of CTAs), which is what an iteration launches."""
    lines = [re.search(r"sign=(-?\d) kind=(\d) goes_by=(\w+) HC=(\d+) grid=\d+,(\d+) nz=(\d+)", t).groups()
             for t in trace("tune") if t.startswith("line")]
    first = next(k for k, t in enumerate(lines) if t[0] == "1")  # the first inverse pass
    tuned = lines[: first - 1]
    assert len({t[3] for t in tuned}) == 5
    assert all(t[1] == "1" and int(t[4]) == int(t[5]) + 1 for t in tuned)
