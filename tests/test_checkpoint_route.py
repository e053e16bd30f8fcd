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
                t.bytes = 1 << 20;
                std::printf("%d ", gather_allowed(t, solver, 1 << 20));
            }""")
    want = [d == s and c == s for s in (0, 1) for d in (-1, 0, 1) for c in (-1, 0, 1)]
    assert [g == "1" for g in got] == want and sum(want) == 2


def test_gathering_launch_needs_an_allocation_that_holds_the_state(tmp_path):
    """A destination whose allocation ends before the state does is left to the copies, which
    refuse it; the kernel would write past it.  Nothing is known of memory that a query failed for."""
    got = answers(tmp_path, """
    for (size_t bytes : {size_t(0), size_t(599), size_t(600), size_t(601), size_t(1) << 40}) {
        GatherTarget t;
        t.device = t.current = 0;
        t.bytes = bytes;
        std::printf("%d ", gather_allowed(t, 0, 600));
    }
    std::printf("%d ", gather_allowed(GatherTarget(), 0, 0));""")
    assert got == ["0", "0", "1", "1", "1", "0"]
