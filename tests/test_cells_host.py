"""Host-side rules of the cells, compiled from their header: no GPU needed."""

import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_08838_b200", "csrc")


def run_cpp(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <cstdio>\n#include "sd2_cells.hpp"\nusing namespace sd2;\nint main() {\n%s\nreturn 0; }\n' % body)
    subprocess.run(["g++", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


def test_weights_of_another_gpu_are_not_read_in_place(tmp_path):
    cases = [("kPlaceDevice", 0, 0, 0, 1), ("kPlaceDevice", 1, 1, 0, 1),      # the handle's own GPU
             ("kPlaceDevice", 1, 0, 0, 0), ("kPlaceDevice", 0, 1, 0, 0),      # another one: by way of a copy
             ("kPlaceManaged", 1, 0, 0, 1), ("kPlaceHost", 0, 0, 0, 0), ("kPlaceHost", -1, 0, 0, 0),
             ("kPlaceDevice", 0, 0, 1, 0), ("kPlaceManaged", 0, 0, 1, 0)]     # an odd address
    body = "".join('std::printf("%%d ", (int)readable_in_place(%s, %d, %d, (const void*)(uintptr_t)%d, 2));'
                   % (p, owner, device, 4096 + shift) for p, owner, device, shift, _ in cases)
    assert [int(v) for v in run_cpp(tmp_path, body)] == [c[-1] for c in cases]
