"""Host checks of the two-stage pass table (``csrc/croft_two_stage.h``): every entry factorises its
length into radices that have a butterfly, and its tile fits the launch and shared-memory limits it
names; and of the plane pass's rule (``csrc/croft_plane_pass.h``): the edges of what it takes, and that
every plane has a kernel and fits (CPU only)."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2002_04896_gb300", "csrc")
RADICES = {2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32}

PROGRAM = r"""
#include <cstdio>
#include "croft_two_stage.h"
static void put(char k, int n, const CroftTwo& t, bool row) {
    if (t.r1) std::printf("%c %d %d %d %d %d %d %d %d %d\n", k, n, t.r1, t.t, t.w, t.minb, t.stage, t.ld, t.ctas, croft_two_smem(t, n, row));
}
int main() {
    for (int n = 1; n <= 5000; ++n) {
        put('s', n, croft_two_col(n, false), false);
        put('l', n, croft_two_col(n, true), false);
        put('r', n, croft_two_row(n), true);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("two")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    out = subprocess.run([str(d / "t")], check=True, capture_output=True, text=True).stdout
    return [(a[0], *map(int, a[1:])) for a in (line.split() for line in out.splitlines())]


def test_entries_fit(table):
    assert len(table) > 100
    for kind, n, r1, t, w, minb, stage, ld, ctas, smem in table:
        r2 = n // r1
        assert r1 * r2 == n and r1 in RADICES and r2 in RADICES, (kind, n)
        threads = w * t
        assert threads * minb <= 2048 and threads <= 1024, (kind, n, threads, minb)
        # registers of the launch bound hold the points of the larger butterfly
        assert min(255, 65536 // (threads * minb)) >= 2 * max(r1, r2), (kind, n)
        assert minb * (smem + 1024) <= 227 * 1024, (kind, n, smem, minb)
        if kind == "r":
            assert ld >= r2 * (r1 + (r1 % 2 == 0)) - (r1 % 2 == 0), (n, ld)
        else:
            assert w % 8 == 0, (kind, n, w)  # rows of at least 64 bytes
        # two CTAs share a tile: each takes half of the butterflies of either stage, from global twiddles
        assert ctas == 1 or (ctas == 2 and kind != "r" and stage == 0 and smem == r2 * ((r1 + 1) // 2) * w * 8)


PLANE_PROGRAM = r"""
#include <cstdio>
#include "croft_plane_pass.h"
int main() {
    const int sms[2] = {152, 148};
    for (int s : sms)
        for (int conv = 0; conv < 2; ++conv)
            for (int nx = 1; nx <= 1200; ++nx)
                for (int ny = 1; ny <= 140; ++ny)
                    for (int nz = 1; nz <= 140; ++nz)
                        if (croft_plane_pass_rule(nx, ny, nz, s, conv != 0))
                            std::printf("%d %d %d %d %d %d %d %d %d\n", s, conv, nx, ny, nz, croft_plane_r1y(ny), croft_plane_r1z(nz),
                                        croft_plane_smem(ny, nz), croft_plane_threads(nx, ny, nz, s));
    return 0;
}
"""


def test_plane_rule_edges(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    (tmp_path / "p.cpp").write_text(PLANE_PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(tmp_path / "p.cpp"), "-o", str(tmp_path / "p")], check=True)
    out = subprocess.run([str(tmp_path / "p")], check=True, capture_output=True, text=True).stdout
    rows = [tuple(map(int, line.split())) for line in out.splitlines()]
    took = {r[:5] for r in rows}
    for _, _, nx, ny, nz, r1y, r1z, smem, threads in rows:
        assert r1y in RADICES and r1z in RADICES and ny % r1y == 0 and nz % r1z == 0 and max(ny // r1y, nz // r1z) <= 25
        assert smem <= 99 * 1024 and threads in (128, 256, 512), (nx, ny, nz)
        assert ny * nz <= 4800 and nx * ny * nz <= 4 * 1024 * 1024
    assert {r[4] for r in rows} == {32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 125}
    # the number of planes up to which small planes are taken (two SMs of three) or rows of 32 points (five of six), and from
    # which the longer planes are, follows the device
    for sms, few, rows32, many in ((152, 101, 126, 456), (148, 98, 123, 444)):
        t, c = (sms, 0), (sms, 1)  # transforms, convolutions
        assert t + (few, 48, 48) in took and t + (few + 1, 48, 48) not in took and t + (few, 50, 48) not in took
        assert t + (few, 64, 54) in took and t + (few, 72, 54) not in took and t + (18, 54, 54) not in took and t + (few, 36, 72) not in took
        assert c + (few, 64, 64) in took and c + (few + 1, 64, 64) not in took and c + (few + 1, 48, 64) in took
        assert t + (rows32, 128, 32) in took and t + (rows32 + 1, 128, 32) not in took and c + (rows32 + 1, 128, 32) in took
        assert t + (many, 90, 50) in took and t + (many - 1, 90, 50) not in took and c + (many - 1, 90, 50) in took
        assert t + (1, 36, 60) in took and t + (1, 48, 40) not in took and t + (1, 32, 48) in took


def test_half_tiles_follow_the_sm_count(tmp_path):
    """complex128 half tiles: taken exactly where the fullest of the device's SMs then has fewer pencils."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    (tmp_path / "h.cpp").write_text("""
#include <cstdio>
#include "croft_sched.h"
int main() {
    const int sms[3] = {152, 148, 1};
    for (int s : sms)
        for (int n = 1; n <= 20000; n += 37) std::printf("%d %d %d\\n", s, n, (int)croft_half_tiles64(n, 16, s));
    std::printf("0 0 %d\\n", (int)croft_half_tiles64(100, 16, 0) + (int)croft_half_tiles64(100, 15, 152));
    return 0;
}
""")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h")], check=True)
    out = subprocess.run([str(tmp_path / "h")], check=True, capture_output=True, text=True).stdout
    rows = [tuple(map(int, line.split())) for line in out.splitlines()]
    assert rows[-1] == (0, 0, 0)
    for s, n, half in rows[:-1]:
        assert half == (-(-(-(-n // 8)) // s) * 8 < -(-(-(-n // 16)) // s) * 16), (s, n)
    assert [r[2] for r in rows if r[0] == 152] != [r[2] for r in rows if r[0] == 148]
