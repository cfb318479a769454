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
