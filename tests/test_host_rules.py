"""The rules of csrc/lbm_host_rules.h, compiled by the host compiler (no GPU)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1412_7228_gb300", "csrc")


def ask(tmp_path, body):
    """The numbers that a program with this body of main() prints."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "ask.cpp"
    src.write_text('#include <cstdio>\n#include <initializer_list>\n#include "lbm_host_rules.h"\nint main() {\n%s\nreturn 0; }\n' % body)
    exe = tmp_path / "ask"
    r = subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    return [int(v) for v in out.split()]


def test_arrays_off_their_values_alignment_are_left_to_the_copies(tmp_path):
    got = ask(tmp_path, """
        for (size_t size : {4, 8})
            for (uintptr_t off = 0; off < 17; ++off)
                printf("%d ", lbm::in_place({0x7f0000001000 + off, 100 * size}, size, {0x7f0000000000, 1 << 20}));
    """)
    assert got == [int(off % size == 0) for size in (4, 8) for off in range(17)]


def test_arrays_beyond_one_mapped_range_are_left_to_the_copies(tmp_path):
    """Ranges of 0x10000 bytes at 0x20000 and, unmapped pages between them, at
    0x40000; also one that ends with the address space."""
    got = ask(tmp_path, """
        const lbm::Span first = {0x20000, 0x10000}, last = {~uintptr_t(0) - 0xffff, 0xffff};
        printf("%d %d %d ", lbm::in_place({0x20000, 0x10000}, 4, first), lbm::in_place({0x2fffc, 4}, 4, first),
               lbm::in_place({0x23000, 0x1000}, 8, first));
        printf("%d %d %d %d ", lbm::in_place({0x20000, 0x10004}, 4, first), lbm::in_place({0x2f000, 0x12000}, 4, first),
               lbm::in_place({0x1f000, 0x2000}, 4, first), lbm::in_place({0x40000, 4}, 4, first));
        printf("%d %d %d ", lbm::in_place({last.at, 0xfffc}, 4, last), lbm::in_place({last.at + 0x8000, ~size_t(3)}, 4, last),
               lbm::in_place({0x20000, 4}, 4, {0, 0}));
    """)
    assert got == [1, 1, 1, 0, 0, 0, 0, 1, 0, 0]


SHAPES = "const lbm::ClusterShape s[4] = {{64, 4}, {64, 8}, {64, 16}, {128, 8}};"   # as in lbm_cluster.cu, FP32


def test_a_lattice_takes_the_first_cluster_that_the_device_can_hold(tmp_path):
    """64^2 in 16, 8 or 4 CTAs; a refusal of one leaves the next."""
    got = ask(tmp_path, SHAPES + """
        for (int most : {16, 15, 8, 7, 4, 3})
            printf("%d ", lbm::pick_cluster(s, 4, 64, 64, [&](int k) { return s[k].ctas(64) <= most; }));
        printf("%d %d ", lbm::pick_cluster(s, 4, 65, 64, [&](int k) { return s[k].ctas(64) <= 8; }),
               lbm::pick_cluster(s, 4, 65, 64, [&](int k) { return s[k].ctas(64) <= 7; }));
    """)
    assert got == [0, 1, 1, 2, 2, -1, 3, -1]


def test_the_lattices_that_fit_a_cluster(tmp_path):
    """FP32: up to 64 x 256 or 128 x 128, the last strip of 4, 8 or 16 rows (8 beyond
    64 wide) at least two rows high."""
    sizes = [(nx, ny) for nx in (1, 2, 64, 65, 128, 129) for ny in range(2, 260)]
    got = ask(tmp_path, SHAPES + """
        for (int nx : {1, 2, 64, 65, 128, 129})
            for (int ny = 2; ny < 260; ++ny) printf("%d ", lbm::pick_cluster(s, 4, nx, ny, [](int) { return true; }));
    """)
    for (nx, ny), k in zip(sizes, got):
        fits = [(bx, by) for bx, by in ((64, 4), (64, 8), (64, 16), (128, 8))
                if 2 <= nx <= bx and ny <= 16 * by and (ny % by == 0 or ny % by >= 2)]
        assert (k >= 0) == bool(fits), (nx, ny)
        if fits:
            assert ((64, 4), (64, 8), (64, 16), (128, 8))[k] == fits[0]


W, M, N = (128, 16), (64, 16), (32, 16)


@pytest.mark.parametrize("fp64,n,nx,ny,tile", [
    # one FP32 lattice: by its nodes, and wide ones of few rows
    (0, 1, 2, 2, N), (0, 1, 1000, 900, N), (0, 1, 1531, 1117, M), (0, 1, 4096, 4096, W), (0, 1, 50000, 12, W),
    (0, 1, 1 << 20, 1 << 20, W),
    # FP32 batches: full 128 x 16 tiles or not, few of them, large lattices, one tile wide, few rows
    (0, 60, 128, 128, W), (0, 8, 128, 128, N), (0, 15, 256, 256, W), (0, 8, 300, 300, N), (0, 4, 512, 512, M),
    (0, 60, 70, 70, W), (0, 100, 96, 96, N), (0, 300, 64, 64, M), (0, 1000, 128, 4, N), (0, 60, 256, 256, W),
    # FP64
    (1, 6, 128, 4, (16, 8)), (1, 200, 128, 4, (32, 8)), (1, 2000, 128, 4, (32, 8)), (1, 1, 400, 400, (16, 8)),
    (1, 1, 512, 512, (32, 8)), (1, 1, 600, 600, (16, 8)), (1, 1, 1024, 1024, (32, 32)), (1, 1, 65536, 16, (32, 8)),
    (1, 1, 100, 10000, (16, 8)), (1, 195, 128, 8, (32, 8)), (1, 1, 1 << 20, 1 << 20, (32, 32))])
def test_the_tile_a_context_starts_with(tmp_path, fp64, n, nx, ny, tile):
    """The faster of the tiles on both sides of each line of the rule (the
    times stand beside it)."""
    got = ask(tmp_path, """
        static int nx[2000], ny[2000];
        for (int i = 0; i < %d; ++i) { nx[i] = %d; ny[i] = %d; }
        const lbm::StartTile t = lbm::start_tile(%d, %d, nx, ny);
        printf("%%d %%d ", t.bx, t.by);
    """ % (n, nx, ny, fp64, n))
    assert tuple(got) == tile
