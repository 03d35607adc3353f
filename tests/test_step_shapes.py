"""Work split and tile of the D2Q9 and D2Q16 steps by grid size: the rule itself, compiled
for the host from the kernels' header, over grids of every shape and parts of several SM
counts."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
SRC = r"""
#include "pond_q16.cuh"
#include <cstdio>
#include <cstdlib>
using namespace pond;
int main(int argc, char **argv)
{
    for (int k = 1; k + 6 < argc; k += 7) {
        int a[7];
        for (int j = 0; j < 7; ++j) a[j] = atoi(argv[k + j]);
        const StepShape s = step_shape(a[0], a[1], a[2], a[3], a[4], a[5], a[6]);
        const bool split = s.lanes == 16;
        const size_t m = !a[0] ? (a[1] ? q16_smem_bytes<float>(s.tx, s.ty) : q16_smem_bytes<double>(s.tx, s.ty))
                               : (a[1] ? step_smem_bytes(s.tx, s.ty, split, Slot<float>::stride, 4)
                                       : step_smem_bytes(s.tx, s.ty, split, Slot<double>::stride, 8));
        std::printf("%d %d %d %lld %zu\n", s.lanes, s.tx, s.ty, s.blocks(a[2], a[3]), m);
    }
    // the wider halo (FP64): every stencil it serves (floors -2 .. 1, four nodes from the floor
    // less one) lies within the staged rows and columns, and the slots within a block's memory
    for (int nodes = 12; nodes <= STEP_NB; nodes += nodes == 12 ? 20 : nodes)
        for (int tx = 1; tx <= nodes; ++tx) {
            const int ty = nodes / tx, h = widest_halo(tx, ty, 8), wt = tx + 2 * h, n = step_slots(tx, ty, h);
            const int first = h * wt + h, last = (ty - 1 + h) * wt + tx - 1 + h;
            if (tx * ty != nodes) continue;
            if ((nodes < STEP_NB || tx == 16) != (h == HALO_FAR) && tx != 8) return 1;
            if (widest_halo(tx, ty, 4) != HALO) return 1;
            if (first + (1 - h - 1) * (wt + 1) < 0 || last + (h - 2 + 2) * (wt + 1) >= n) return 2;
            const size_t m = step_smem_bytes(tx, ty, nodes == 12, Slot<double>::stride, 8);
            // two resident blocks on the tiles of large grids
            if (m + 2048 > 227 * 1024 || (tx == 16 && 2 * (m + 2048) > 228 * 1024)) return 3;
        }
    std::printf("%d %d\n", STEP_THREADS, SPLIT_NB);
}
"""
SIZES = [1, 2, 3, 4, 5, 7, 8, 12, 15, 16, 17, 33, 64, 90, 128, 300, 1000, 2048, 4097, 20000]


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("shapes")
    (d / "shapes.cu").write_text(SRC)
    subprocess.check_call([NVCC, "-std=c++17", "-O1", "-gencode=arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "paper_2002_09217_gb300", "csrc"), "-o", str(d / "shapes"), str(d / "shapes.cu")])

    def run(queries):
        out = []
        for k in range(0, len(queries), 2000):
            args = [str(int(v)) for q in queries[k:k + 2000] for v in q]
            lines = subprocess.check_output([str(d / "shapes")] + args, text=True).split("\n")[:-1]
            assert lines[-1] == "128 12"      # threads of a block; nodes of a block with nine lanes each
            out += [tuple(map(int, x.split())) for x in lines[:-1]]
        return out
    return run


def test_every_tile_fits_its_block_and_covers_the_grid(shapes):
    q = [(d2q9, mixed, nx, ny, lanes, tx, sms) for d2q9 in (0, 1) for mixed in (0, 1) for nx in SIZES for ny in SIZES
         for lanes in (0, 8, 16) for tx in (0, 1, 2, 4, 8, 16) for sms in (152,) if nx * ny <= 4000000]
    for (d2q9, mixed, nx, ny, lanes, opt, _), (split, tx, ty, blocks, smem) in zip(q, shapes(q)):
        assert tx >= 1 and ty >= 1
        assert tx * ty == 12 if split == 16 else tx * ty in (32, 64, 128)
        assert blocks * tx * ty >= nx * ny
        assert smem + 2048 <= 227 * 1024
        if not d2q9:
            assert split == 8
        elif lanes == 16 or (lanes == 8 and mixed):
            assert split == lanes                  # the caller's choice (8 in FP64: by size)
        if opt:
            assert tx == ({8: 6, 16: 12}.get(opt, opt) if split == 16 else opt)


@pytest.mark.parametrize("sms", [20, 152, 304])
def test_transposed_grids_take_as_many_turns(shapes, sms):
    """A grid of few columns is tiled as well as the same grid on its side: it needs no more
    than twice the turns of its blocks on the SMs."""
    q, t = [], []
    for d2q9 in (0, 1):
        for mixed in (0, 1):
            for a in (1, 2, 3, 4, 5, 8, 9):
                for b in (64, 300, 2048, 4097, 20000, 300000):
                    q.append((d2q9, mixed, a, b, 0, 0, sms))
                    t.append((d2q9, mixed, b, a, 0, 0, sms))
    for x, tall, wide in zip(q, shapes(q), shapes(t)):
        if tall[0] != wide[0]:
            continue                               # near the line of the nine lanes: 4 x 3 tiles do not transpose
        assert -(-tall[3] // sms) <= 2 * -(-wide[3] // sms), (x, tall, wide)


def test_the_lines_of_the_rule_follow_the_sm_count(shapes):
    def lanes_of(mixed, nx, ny, sms):
        return shapes([(1, mixed, nx, ny, 0, 0, sms)])[0]
    for sms in (76, 152):
        # nine lanes: 4 x 3 tiles, two blocks an SM (mixed) and five (FP64)
        assert lanes_of(1, 4 * sms, 6, sms)[0] == 16 and lanes_of(1, 4 * sms + 1, 6, sms)[0] == 8
        assert lanes_of(0, 4 * sms, 15, sms)[0] == 16 and lanes_of(0, 4 * sms + 1, 15, sms)[0] == 8
        # strips: tiles of 32, then 64 nodes while that is one block an SM
        for n in (1, 2, 4):
            for nodes in (32, 64):
                w = nodes // n
                last = sms * w
                if nodes == 32 and n == 1:
                    assert lanes_of(1, last, 1, sms)[0] == 8
                for nx, ny in ((last, n), (n, last)):
                    lanes, tx, ty, blocks, _ = lanes_of(1, nx, ny, sms)
                    assert (lanes, (tx, ty) if ny == n else (ty, tx), blocks) == (8, (w, n), sms)
            assert lanes_of(1, sms * 64 // n + 1, n, sms)[1:3] == (128 // n, n)
        # no strip
        assert lanes_of(1, sms * 8, 5, sms)[1:3] == (16, 8)
