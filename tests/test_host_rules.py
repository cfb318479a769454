"""The C ABI's host-side decisions (csrc/host_rules.cuh), compiled by the host compiler
and run without a GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2002_12160_gb300", "csrc")


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """Compile a main() over the rules, run it with arguments, return its words."""
    d = tmp_path_factory.mktemp("rules")

    def go(name, body, *args):
        exe = d / name
        if not exe.exists():
            src = d / (name + ".cpp")
            src.write_text('#include <cstdio>\n#include <cstdlib>\n#include <cstring>\n#include "host_rules.cuh"\nusing namespace ih;\n'
                           "int main(int argc, char **argv) {\n(void)argc;\n" + body + "\nreturn 0;\n}\n")
            subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)])
        return subprocess.check_output([str(exe), *map(str, args)], text=True).split()

    return go


TOUCH = """
CallerArray a;
a.kind = !strcmp(argv[1], "device") ? CallerArray::kDevice : !strcmp(argv[1], "managed") ? CallerArray::kManaged : CallerArray::kOther;
a.device = atoi(argv[2]);
a.at = strtoull(argv[3], 0, 0); a.bytes = strtoull(argv[4], 0, 0);
a.base = strtoull(argv[5], 0, 0); a.size = strtoull(argv[6], 0, 0);
printf("%d", (int)kernel_may_touch(a, atoi(argv[7]), atoi(argv[8]), atoi(argv[9])));
"""
M = 2 ** 64 - 1


@pytest.mark.parametrize("kind,device,at,bytes_,base,size,handle,current,stream,want", [
    ("device", 0, 4096, 64, 4096, 64, 0, 0, 0, 1),        # the whole allocation
    ("device", 0, 4100, 60, 4096, 64, 0, 0, 0, 1),        # its tail
    ("device", 1, 4096, 64, 4096, 64, 1, 1, 1, 1),
    ("managed", -1, 4096, 64, 4096, 64, 0, 0, 0, 1),      # managed memory is every device's
    ("device", 0, 4096, 64, 4096, 64, 0, 1, 0, 0),        # another device current
    ("device", 0, 4096, 64, 4096, 64, 0, 1, 1, 0),        # ... and its default stream
    ("device", 0, 4096, 64, 4096, 64, 0, 0, 1, 0),        # another device's stream
    ("managed", -1, 4096, 64, 4096, 64, 0, 1, 1, 0),
    ("device", 1, 4096, 64, 4096, 64, 0, 0, 0, 0),        # a peer's memory
    ("host", 0, 4096, 64, 4096, 64, 0, 0, 0, 0),          # host memory, pinned or not
    ("device", 0, 4096, 65, 4096, 64, 0, 0, 0, 0),        # past the allocation's end
    ("device", 0, 4100, 64, 4096, 64, 0, 0, 0, 0),
    ("device", 0, 4095, 4, 4096, 64, 0, 0, 0, 0),         # before its start
    ("device", 0, 4096, M, 4096, 64, 0, 0, 0, 0),         # sums that wrap
    ("device", 0, M - 3, 4, 4096, 64, 0, 0, 0, 0),
    ("device", 0, 4096, 4, 0, 0, 0, 0, 0, 0),             # an allocation that is not known
])
def test_a_read_back_launches_only_where_a_kernel_may_touch_the_array(run, kind, device, at, bytes_, base, size, handle,
                                                                      current, stream, want):
    assert run("touch", TOUCH, kind, device, at, bytes_, base, size, handle, current, stream) == [str(want)]


# calls of horizon H and checkpoint interval K over a device with `avail` floats free:
# what each takes, and how often memory was asked for in all
SEGMENTS = """
size_t held = 0, refused = (size_t)-1;
int asked = 0;
for (int i = 1; i + 4 < argc; i += 5) {
    const int H = atoi(argv[i]), K = atoi(argv[i + 1]);
    const size_t budget = strtoull(argv[i + 2], 0, 0), avail = strtoull(argv[i + 3], 0, 0);
    if (!strcmp(argv[i + 4], "reset")) refused = (size_t)-1;
    bool failed = false;
    const int k = longer_segment(H, K, budget, held, refused, failed, [&](int k) { return (size_t)k * 100; },
                                 [&](size_t f) {
                                     ++asked;
                                     if (!strcmp(argv[i + 4], "fail")) return Reserve::kFailed;
                                     if (f > avail / 2) return Reserve::kNoMemory;
                                     held = f;
                                     return Reserve::kDone;
                                 });
    printf("%d:%d:%d ", k, asked, (int)failed);
}
"""
BIG = 10 ** 9


@pytest.mark.parametrize("calls,want", [
    # the whole horizon when it fits, without asking again
    ([(30, 10, BIG, BIG, "-")] * 2, ["30:1:0", "30:1:0"]),
    # the budget decides: 15, then none above K
    ([(30, 10, 2000, BIG, "-"), (30, 10, 1400, BIG, "-")], ["15:1:0", "0:1:0"]),
    # the free memory decides; more of it changes nothing until the budget is set again
    ([(30, 10, BIG, 3200, "-"), (30, 10, BIG, 0, "-"), (30, 10, BIG, BIG, "-"), (30, 10, BIG, BIG, "reset")],
     ["15:2:0", "15:2:0", "15:2:0", "30:3:0"]),
    # nothing fits: asked once for each length, then never
    ([(30, 2, BIG, 100, "-"), (30, 2, BIG, 100, "-"), (30, 2, BIG, BIG, "-")], ["0:8:0", "0:8:0", "0:8:0"]),
    # a smaller need than the refused one is still tried
    ([(30, 10, BIG, 2400, "-"), (11, 10, BIG, 2400, "-")], ["0:2:0", "11:3:0"]),
    # an error ends the call
    ([(30, 10, BIG, BIG, "fail")], ["0:1:1"]),
    # no longer one than the horizon, none at all when K is the horizon
    ([(10, 10, BIG, BIG, "-"), (1, 1, BIG, BIG, "-")], ["0:0:0", "0:0:0"]),
])
def test_the_adjoints_segments_settle(run, calls, want):
    assert run("segments", SEGMENTS, *[v for c in calls for v in c]) == want
