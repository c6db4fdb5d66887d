"""Workspaces that hold parts (the adjoint's partial traces, the velocity gradient's partial sums) where an
allocation is refused: a fake allocator with a limit, and one that fails for another reason."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1204_1225_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "kh_room.h"

enum Status { OK, NO_ROOM, BROKEN };

int main(int argc, char** argv)
{
    int parts = std::atoi(argv[1]), limit = std::atoi(argv[2]), calls = 0;   // limit < 0: another failure
    const Status e = kh::grow_parts(parts, NO_ROOM, [&](int n) {
        ++calls;
        return limit < 0 ? BROKEN : n <= limit ? OK : NO_ROOM;
    });
    std::printf("%d %d %d\n", (int)e, parts, calls);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("grow")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I" + CSRC, str(d / "p.cpp"), "-o", str(d / "p")], check=True)
    return str(d / "p")


@pytest.mark.parametrize("parts, limit, status, got, calls", [
    (1, 1, 0, 1, 1), (19, 32, 0, 19, 1), (19, 18, 0, 10, 2), (19, 9, 0, 5, 3), (32, 1, 0, 1, 6), (2, 1, 0, 1, 2),
    (32, 0, 1, 1, 6), (1, 0, 1, 1, 1), (8, -1, 2, 8, 1)])
def test_fewer_parts_where_there_is_no_room(program, parts, limit, status, got, calls):
    out = subprocess.run([program, str(parts), str(limit)], check=True, capture_output=True, text=True).stdout
    assert [int(x) for x in out.split()] == [status, got, calls]
