"""Index arithmetic of the row kernels' copies, compiled for the host."""
import subprocess

from paper_2208_09267_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "step_row.cuh"
int main() {
  int ny;
  unsigned row_bytes;
  while (scanf("%d %u", &ny, &row_bytes) == 2) printf("%lld\n", lbm::plane_span(ny, row_bytes));
}
"""


def test_wrapped_rows_of_large_planes_keep_their_distance(tmp_path):
    """A plane's rows wrap around over its whole span, at 2^32 bytes and past
    them: rows of 8 to 248 cells of 2, 4 bytes, up to the 2^31 - 1 cells that the
    row kernels take."""
    (tmp_path / "span.cu").write_text(PROGRAM)
    exe = str(tmp_path / "span")
    subprocess.run([build.nvcc()] + build.ARCH + build.COMMON + ["-o", exe, str(tmp_path / "span.cu")], check=True,
                   capture_output=True, text=True)
    sizes = [(ny, nxp * elem) for nxp in (8, 128, 248) for elem in (2, 4)
             for ny in (1, 2 ** 20, 2 ** 32 // (nxp * elem) - 1, 2 ** 32 // (nxp * elem) + 1, (2 ** 31 - 1) // nxp)
             if ny * nxp < 2 ** 31]
    out = subprocess.run([exe], input="\n".join(f"{a} {b}" for a, b in sizes), check=True, capture_output=True, text=True)
    assert [int(v) for v in out.stdout.split()] == [a * b for a, b in sizes]
