"""Host-side checks of the rule that picks the way of a checkpoint to device memory, compiled from
the solver's header: one launch on the device, or copies."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def answers(tmp_path, body):
    src, exe = tmp_path / "r.cpp", tmp_path / "r"
    src.write_text('#include <cstdio>\n#include <initializer_list>\n#include "lbs_internal.h"\n'
                   "using namespace lbs;\nint main() {\n" + body + "\nreturn 0; }\n")
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1702_01335_gb300", "csrc"), str(src),
                           "-o", str(exe)])
    return subprocess.check_output([str(exe)]).decode().split()


def test_gathering_launch_needs_the_solvers_device_to_be_current(tmp_path):
    """Memory of the solver's device with that device current: the launch.  Another device current
    (a launch on the solver's stream would fail, a copy does not), another device's memory, or
    memory of no device: the copies."""
    got = answers(tmp_path, """
    for (int solver : {0, 1})
        for (int device : {-1, 0, 1})
            for (int current : {-1, 0, 1}) {
                GatherTarget t;
                t.device = device;
                t.current = current;
                std::printf("%d ", gather_allowed(t, solver));
            }""")
    want = [d == s and c == s for s in (0, 1) for d in (-1, 0, 1) for c in (-1, 0, 1)]
    assert [g == "1" for g in got] == want and sum(want) == 2
