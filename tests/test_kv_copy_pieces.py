"""The launches of a K/V import or export (csrc/pieces.h), with a launch function that fails at a chosen piece: the call
waits for the pieces before it and returns that piece's error."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_07423_b200", "csrc")

PROGRAM = r"""
#include "pieces.h"
#include <cstdio>
#include <cstdlib>
int main(int, char** v) {   // pos0 n_pos max_pages failing_piece(-1: none) wait_result
    const int pos0 = atoi(v[1]), n_pos = atoi(v[2]), max_pages = atoi(v[3]), fail = atoi(v[4]), result = atoi(v[5]);
    int piece = 0;
    const int r = syn::for_pieces(pos0, n_pos, 16, max_pages,
        [&](int at, int n, int64_t done) { printf("%d:%d:%d ", at, n, (int)done); return piece++ == fail ? -8 : 0; },
        [&] { printf("wait "); return result; });
    printf("%d\n", r);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("pieces")
    (d / "main.cpp").write_text(PROGRAM)
    subprocess.check_call([gxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")])
    return str(d / "main")


@pytest.mark.parametrize("args,want", [
    ("5 20 4 -1 0", "5:20:0 wait 0"),
    ("5 200 4 -1 0", "5:59:0 64:64:59 128:64:123 192:13:187 wait 0"),
    ("0 128 4 -1 -8", "0:64:0 64:64:64 wait -8"),
    ("0 200 4 0 0", "0:64:0 wait -8"),
    ("0 200 4 1 0", "0:64:0 64:64:64 wait -8"),       # the first piece is in flight when the second fails
    ("0 200 4 1 -10", "0:64:0 64:64:64 wait -8"),
])
def test_a_failed_piece_is_reported_after_the_wait(program, args, want):
    assert subprocess.check_output([program, *args.split()], text=True).strip() == want
