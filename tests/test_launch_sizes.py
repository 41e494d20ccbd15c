"""Launch sizes and rules (csrc/osscir_launch.h), from the host helpers that the launchers
use (a small program compiled here; no GPU).  The tile-view pairs of 8192 x 8192 pixels
pass 2^31 at 8192 views and 2^32 above 16384; a grid counts as small by the device's own
SMs, also where its product does not fit in 32 bits."""
import subprocess

import pytest

from paper_1801_06263_gb300 import build

SOURCE = """
#include <cstdio>
#include <cstdlib>
#include "osscir_launch.h"
int main(int, char** a) {
    const size_t s = osscir::bt_spans(atoi(a[1]), atoi(a[2]));
    printf("%zu %u", s, osscir::thread_blocks(s, 256));
    for (int per = 1; per < 4; ++per) printf(" %d", (int)osscir::few_blocks(dim3(atoi(a[1]), atoi(a[2])), per, 100));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("launch_sizes")
    (d / "p.cu").write_text(SOURCE)
    out = str(d / "p")
    subprocess.run([build._nvcc(), "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-o", out, str(d / "p.cu")],
                   check=True, capture_output=True)
    return out


@pytest.mark.parametrize("n,views", [(1, 1), (256, 512), (8191, 8192), (8192, 8192), (8192, 16385), (8192, 100000)])
def test_span_pass_covers_every_tile_and_view(program, n, views):
    spans, blocks = map(int, subprocess.run([program, str(n), str(views)], check=True, capture_output=True,
                                            text=True).stdout.split()[:2])
    want = ((n + 15) // 16) ** 2 * views
    assert spans == want and blocks == (want + 255) // 256 < 2 ** 31


@pytest.mark.parametrize("x,y", [(1, 1), (10, 10), (101, 1), (10, 20), (3, 67), (20, 15), (7, 43), (1 << 20, 1 << 12)])
def test_few_blocks_follows_the_sm_count(program, x, y):
    got = subprocess.run([program, str(x), str(y)], check=True, capture_output=True, text=True).stdout.split()[2:]
    assert [int(v) for v in got] == [int(x * y <= per * 100) for per in (1, 2, 3)]
