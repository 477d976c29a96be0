"""The nodes that the quadratic deposit's columns add to, over every row segment
of small grids (the narrowest accepted is three cells): the kernel's own index
function, compiled for the host, gives for each the node that two modulos give,
and so none outside the grid."""
import subprocess

from paper_2509_11100_gb300 import build

SOURCE = r"""
#include "common.cuh"
#include <cstdio>
int main()
{
    long wrong = 0, seen = 0;
    for (int nx = 3; nx <= 70; ++nx)
        for (int ny = 3; ny <= 6; ++ny)
            for (int uw = 8; uw <= 32; uw *= 2)
                for (int i0 = 0; i0 < nx; i0 += uw) {
                    const int cn = uw < nx - i0 ? uw : nx - i0;
                    for (int j = 0; j < ny; ++j)
                        for (int cl = 0; cl < cn + 3; ++cl)
                            for (int place = 0; place < 12; ++place, ++seen) {
                                const int col = (i0 + cl - 1 + (place >> 2) + nx) % nx, row = (j - 1 + (place & 3) + ny) % ny;
                                wrong += relsim::column_node_q(i0 + cl, j, place, nx, ny) != row * nx + col;
                            }
                }
    std::printf("%ld %ld\n", seen, wrong);
}
"""


def test_column_nodes_lie_in_the_grid(tmp_path):
    src, exe = tmp_path / "columns.cu", tmp_path / "columns"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc()] + build.ARCH + build.NVFLAGS + [str(src), "-o", str(exe)], check=True)
    seen, wrong = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert seen > 1e5 and wrong == 0
