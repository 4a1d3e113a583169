"""Launch shapes of the solvers, on the host: what the rules choose has to fit
the SM (228 KB of shared memory, 1 KB of it reserved per block) as often as
the shape says, for every restart length."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include "kp_ctx.h"
// lines "N m mixed wmin hmax one_size count one_launch windows threads blocks cluster cluster_blocks" -> the shape
int main() {
  int N, m, mixed, wmin, hmax, one, count, launch, win, bt, mb, cs, cb;
  while (scanf("%d %d %d %d %d %d %d %d %d %d %d %d %d", &N, &m, &mixed, &wmin, &hmax, &one, &count, &launch, &win,
               &bt, &mb, &cs, &cb) == 13) {
    kp_ctx c;
    kp_options_default(&c.opt);
    c.opt.block_threads = bt;
    c.opt.blocks_per_sm = mb;
    c.opt.cluster_size = cs;
    c.opt.cluster_blocks_per_sm = cb;
    c.sms = 152;
    c.smem_optin = 227 * 1024;
    kp::Shape s;
    const int st = kp::gmres_shape(&c, N, m, &s, mixed, wmin, hmax, one, count, launch, win);
    printf("%d %d %d %d %d %zu %d %d\n", st, s.ept, s.nt, s.S, s.minb, s.smem, s.cs, (int)s.reg);
  }
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    if not shutil.which("nvcc"):
        pytest.skip("no nvcc")
    from paper_2511_17634_gb300 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("shapes")
    (d / "driver.cu").write_text(DRIVER)
    exe = str(d / "driver")
    subprocess.run(["nvcc", *build.ARCH, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", build.CSRC,
                    str(d / "driver.cu"), lib, "-o", exe, "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)

    def run(rows):
        text = "\n".join(" ".join(str(int(v)) for v in r) for r in rows)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        keys = ("status", "ept", "nt", "S", "minb", "smem", "cs", "reg")
        return [dict(zip(keys, map(int, line.split()))) for line in out.splitlines()]
    return run


def _fits(s):
    return s["minb"] * (s["smem"] + 1024) <= 228 * 1024


def test_fp64_blocks_share_an_sm_as_the_shape_says(shapes):
    # the rule's shapes (one system, one per SM, two, more; one launch) and the
    # shapes on request, every restart length
    rows = [(1024, m, 0, 32, 32, 1, count, launch, 0, 0, 0, 0, 0)
            for m in range(1, 65) for count in (1, 152, 153, 304, 305, 456, 2000) for launch in (0, 1)]
    rows += [(1024, m, 0, 32, 32, 1, 500, 0, 0, bt, mb, 0, 0)
             for m in range(1, 65) for bt, mb in ((256, 2), (256, 3), (128, 2), (128, 3), (128, 4), (64, 4))]
    for r, s in zip(rows, shapes(rows)):
        assert s["status"] == 0 and _fits(s), (r, s)
        assert (s["nt"] * s["ept"]) == 1024 and 1 <= s["S"] <= r[1] + 1


def test_fp64_blocks_of_a_window_keep_their_sm_while_few_would_share_it(shapes):
    # more than one system per SM up to one and a half: no second block beside
    # the first wherever the restart length has that many vectors; then two
    rows = [(1024, m, 0, 32, 32, 1, count, 0, 1, 0, 0, 0, 0) for m in range(16, 65) for count in (152, 153, 228, 229, 304)]
    for r, s in zip(rows, shapes(rows)):
        assert s["status"] == 0 and s["minb"] == 2
        assert _fits(s) != (152 < r[6] <= 228), (r, s)


def test_mixed_grid_is_what_its_kernel_keeps_resident(shapes):
    # full CTAs of 4096 points: three of them per SM are compiled for one and
    # four CTAs per system, two for two
    rows = [(n, m, 1, W, H, 1, 2000, 1, 0, 0, 0, 0, 0) for m in range(1, 65)
            for n, H, W in ((4096, 64, 64), (8192, 64, 128), (8192, 128, 64), (16384, 128, 128))]
    for r, s in zip(rows, shapes(rows)):
        assert s["status"] == 0 and s["reg"] and s["ept"] == 16 and s["S"] >= 3
        assert (s["cs"], s["minb"]) == {4096: (0, 3), 8192: (2, 2), 16384: (4, 3)}[r[0]]
        if r[1] <= 40:
            assert _fits(s), (r, s)


def test_autotuner_can_choose_what_the_solver_would(shapes):
    # the automatic shape, and every shape that a march's rule comes to
    from paper_2511_17634_gb300 import autotune
    assert (0, 0) in autotune.SHAPE_CANDIDATES
    rows = [(1024, 40, 0, 32, 32, 1, count, 0, win, 0, 0, 0, 0) for count in (4, 152, 153, 230, 304, 305, 5000) for win in (0, 1)]
    for s in shapes(rows):
        assert (s["nt"], s["minb"]) in autotune.SHAPE_CANDIDATES, s
