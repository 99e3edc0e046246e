"""Places of the FFT axes' twiddle tables (csrc/fv_tables.cuh), compiled for the host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "fv_tables.cuh"
#include <cstdio>
#include <cstdlib>
// argv: M fixed, M fixed, ...; prints "offset first" per axis and the total (a fixed axis has M + 7 extra elements)
int main(int argc, char **argv)
{
    fv::TableMap map;
    std::map<int, size_t> at;
    for (int i = 1; i + 1 < argc; i += 2) at[i] = map.place(atoi(argv[i]), atoi(argv[i + 1]), atoi(argv[i]) + 7);
    for (int i = 1; i + 1 < argc; i += 2)
        printf("%zu %d\n", at[i], (int)map.take(atoi(argv[i]), atoi(argv[i + 1])));
    printf("%zu\n", map.total());
}
"""


def test_axes_share_tables_only_with_their_like(tmp_path):
    src = tmp_path / "tables.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "tables"
    subprocess.run(["g++", "-std=c++17", "-I" + os.path.join(ROOT, "paper_2506_02130_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    # two channels: x and y with compile-time lengths, the up axis general; y of the second channel has the length of
    # the first one's up axis
    axes = [(640, 1), (320, 1), (400, 0), (1280, 1), (400, 1), (640, 0), (640, 1), (400, 0)]
    out = subprocess.run([str(exe)] + [str(v) for a in axes for v in a], check=True, capture_output=True,
                         text=True).stdout.split("\n")
    got = [tuple(int(v) for v in line.split()) for line in out[:len(axes)]]
    total = int(out[len(axes)])
    spans = {}
    for (M, fixed), (at, first) in zip(axes, got):
        assert ((M, fixed) not in spans) == first           # one axis fills each table
        assert spans.setdefault((M, fixed), at) == at
    used = sorted((at, at + M + (M + 7 if fixed else 0)) for (M, fixed), at in spans.items())
    assert used[0][0] == 0 and used[-1][1] == total
    assert all(a[1] == b[0] for a, b in zip(used, used[1:]))
