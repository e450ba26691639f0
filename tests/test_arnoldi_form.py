"""The Arnoldi step's form by the room a device has: on a part of one, no cluster or grid that it cannot hold."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = """
#include <cstdio>
#include <cstdlib>
#include "arnoldi_form.cuh"
int main(int, char **a) {
  const vie::ArnoldiRoom room{atoi(a[3]), atoi(a[4])};
  printf("%d", vie::arnoldi_one_launch(atoi(a[1]), atoi(a[2]), room));
}
"""


@pytest.fixture(scope="module")
def one_launch(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("form")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "form")
    subprocess.run(["g++", "-x", "c++", str(d / "main.cpp"), "-I", os.path.join(ROOT, "paper_1610_00835_gb300", "csrc"),
                    "-o", exe], check=True)
    return lambda *v: subprocess.run([exe, *map(str, v)], check=True, capture_output=True, text=True).stdout == "1"


# blocks, right-hand sides, largest cluster, CTAs resident
@pytest.mark.parametrize("blocks,R,cluster,resident,want", [
    (1, 1, 0, 1, True), (1, 64, 0, 1, True),            # one block waits for nobody
    (16, 1, 16, 608, True), (16, 1, 8, 608, False),     # a cluster of 16
    (16, 64, 8, 608, True), (9, 64, 8, 608, False), (16, 64, 0, 608, False),  # 8 with two blocks a CTA
    (304, 1, 16, 608, True), (304, 1, 16, 304, True), (304, 1, 16, 303, False), (17, 1, 0, 16, False),
    (17, 2, 16, 608, False),
])
def test_one_launch_only_where_there_is_room(one_launch, blocks, R, cluster, resident, want):
    assert one_launch(blocks, R, cluster, resident) is want
