"""Host-side checks of the stage kernel's shared-memory layout, compiled from the headers that
the kernels include (nvcc, no GPU)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# for every layout the launchers know and the smallest tiles and velocity sets that the solver
# accepts: the CTA's dynamic shared memory against what the folded-in finalisation lays over it
SRC = r"""
#include <cstdio>
#include "kernels.cuh"
using namespace lbs;
template <typename T>
static void check(int layout)
{
    const int KC = layout_columns(layout), es = sizeof(T), as = sizeof(typename Acc<T>::type);
    const bool grouped = layout & kGrouped;
    for (int Qx = 1; Qx <= 4; ++Qx)
        for (int Qy = grouped ? 4 : 1; Qy <= 8; Qy += grouped ? 4 : 1)
            for (int Qz = 1; Qz <= 4; ++Qz)
                for (int zn = 3; zn <= 6; ++zn) {
                    const int nzm = (KC - 1) / (Qx * Qy) + 1 < Qz ? (KC - 1) / (Qx * Qy) + 1 : Qz;
                    const StageSmem L = stage_smem(zn, KC, factor_stride(Qx, Qy, nzm, grouped, es), es, as,
                                                   rec_stride_of(Qx, Qy, Qz), grouped, layout & kZSplit ? 4 : 1);
                    std::printf("%d %d %d %d %d %d %zu %zu\n", es, layout, Qx, Qy, Qz, zn, L.total,
                                sizeof(FinShared<T, 4>));
                }
}
int main()
{
    for (int V : {1, 2, 4, 4 | kGrouped}) check<float>(V), check<double>(V);
    for (int V : {1 | kZSplit, 4 | kGrouped | kZSplit}) check<double>(V);
    return 0;
}
"""


def test_folded_finalisation_fits_the_stage_kernels_shared_memory(tmp_path):
    """The finalisation folded into the stage kernel (fuse = 1) lays its cell group over the CTA's
    dynamic shared memory: it fits in every layout, down to one node per axis and tiles of three
    cells."""
    from paper_1702_01335_gb300 import build as B
    src, exe = tmp_path / "layout.cu", tmp_path / "layout"
    src.write_text(SRC)
    subprocess.check_call([B.NVCC] + B.ARCH + ["-std=c++17", "-I" + B.CSRC, str(src), "-o", str(exe)])
    rows = [tuple(map(int, r.split())) for r in subprocess.check_output([str(exe)]).decode().splitlines()]
    assert len(rows) == 2 * (3 * 128 * 4 + 32 * 4) + 128 * 4 + 32 * 4
    short = [r for r in rows if r[6] < r[7]]
    assert not short, short
