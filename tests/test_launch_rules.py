"""The rules of launch shapes (csrc/launch_rules.h), compiled for the host."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2505_13390_gb300", "csrc")


def run_host(tmp_path, body):
    """Output lines of a C++ program around `body` with the rules included."""
    if not shutil.which("g++"):
        pytest.skip("g++ not found")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <stdio.h>\n#include <initializer_list>\n#include <thread>\n#include <vector>\n#include "launch_rules.h"\n'
                   "using namespace mg;\nint main() {\n" + body + "\n}\n")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")


def launch(kernel, source):
    """The launch configuration of `kernel` in a source file."""
    return re.search(kernel + r"<<<(.*?)>>>", open(os.path.join(CSRC, source)).read(), re.S)[1]


def test_near_kernel_sweep_covers_every_row(tmp_path):
    """One warp takes 4 to 32 rows and does not loop: 2^20 blocks of 128 rows
    would stop at row 134,217,728."""
    assert launch("k_nk_sweep<R>", "setup.cu").startswith("blocks_covering(h->m, R * kNkWarps)")
    out = run_host(tmp_path, """
  for (long long n : {1LL, 31LL, 128LL, 129LL, (1LL << 27), (1LL << 27) + 1, (1LL << 31) - 1})
    printf("%lld %d\\n", n, blocks_covering(n, 128));""")
    for n, b in (map(int, line.split()) for line in out if line):
        assert 1 <= b < 2 ** 31 and 128 * (b - 1) < n <= 128 * b


def test_settings_are_made_on_each_device(tmp_path):
    """A kernel's shared-memory limit belongs to the device it was set on: every
    device has it made once, again after a failure, and once under threads."""
    body = open(os.path.join(CSRC, "setup.cu")).read()
    body = body[body.index("mgpbd_status galerkin_smem_limits()"):]
    assert "OncePerDevice" in body[:body.index("\n}\n")]
    out = run_host(tmp_path, """
  OncePerDevice once;
  int made[3] = {0, 0, 0}, bad = 0;
  auto use = [&](int d) { return once(d, [&] { made[d]++; return 0; }); };
  bool ok = use(0) == 0 && use(1) == 0 && use(0) == 0;
  ok = ok && once(2, [&] { bad++; return -6; }) == -6 && use(2) == 0 && use(2) == 0;
  OncePerDevice shared;
  int n = 0;
  std::vector<std::thread> ts;
  for (int k = 0; k < 8; ++k) ts.emplace_back([&] { shared(k % 2, [&] { n++; return 0; }); });
  for (auto &t : ts) t.join();
  printf("%d %d %d %d %d %d\\n", ok, made[0], made[1], made[2], bad, n);""")
    assert out[0] == "1 1 1 1 1 2"


def test_partials_never_exceed_their_room(tmp_path):
    """The grid of every kernel that leaves one partial per block goes through
    the rule, which holds on a part of any number of SMs."""
    out = run_host(tmp_path, """
  for (long long blocks : {0LL, 1LL, 4095LL, 4096LL, 4097LL, 1LL << 40})
    for (long long resident : {1LL, 2432LL, 4096LL, 100000LL})
      printf("%lld %lld %d\\n", blocks, resident, partial_blocks(blocks, resident));
  printf("%d\\n", kPartials);""")
    room = int(out[24])
    for blocks, resident, got in (map(int, line.split()) for line in out[:24]):
        assert got == max(1, min(blocks, resident, room))
    for name in ("solve.cu", "mfree.cu"):
        src = open(os.path.join(CSRC, name)).read()
        # kernels of kDotThreads are those that leave partials
        assert not re.search(r"wave_blocks\([^;]*kDotThreads\)", src), name
    assert "&h->partials, kPartials + 16" in open(os.path.join(CSRC, "api.cu")).read()


@pytest.mark.gpu
def test_near_kernel_beyond_two_to_the_27_rows():
    """A chain of 2^27 + 3,000 rows whose rows are dead (both ends pinned) but
    for the last 2,500: one sweep x - omega D^-1 A x on those, from the start
    that a setup without sweeps leaves."""
    import numpy as np
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available() or torch.cuda.mem_get_info()[0] < 80 << 30:
        pytest.skip("needs a CUDA device with 80 GB free")
    from paper_2505_13390_gb300.meshgen import Mesh, default_params
    from paper_2505_13390_gb300.mgpbd import Solver
    rows, live = (1 << 27) + 3000, 2500
    x = np.zeros((rows + 1, 3))
    x[:, 0] = 0.01 * np.arange(rows + 1)
    w = np.zeros(rows + 1)
    w[-live:] = 1.0
    e = np.empty((rows, 2), np.int32)
    e[:, 0] = np.arange(rows)
    e[:, 1] = e[:, 0] + 1
    mesh = Mesh("long", x, w, e, np.zeros((0, 4), np.int32), np.full(rows, 1e-6), x, np.zeros_like(x))
    vec = {}
    for sweeps in (0, 1):
        g = Solver(mesh, default_params(nk_sweeps=sweeps, nk_omega=0.5, coarse_max=2000, max_levels=3))
        g.begin_frame()
        g.eval_assemble()
        g.setup()
        if not sweeps:
            ptr, col, val = (a[-n:].cpu().numpy() for a, n in zip(g.matrix(0, device=True), (2901, 10000, 10000)))
        vec[sweeps] = g.level_agg(0)[4]
        g.close()
        torch.cuda.empty_cache()
    first, shift = rows - 2900, ptr[-1] - 10000
    for i in range(first, rows):
        a, b = ptr[i - first] - shift, ptr[i - first + 1] - shift
        want = vec[0][i] - 0.5 * (val[a:b] @ vec[0][col[a:b]]) / val[b - 1]
        # three products per row, each below 2 max |x| (|A_ij| <= 2 A_ii here)
        assert abs(vec[1][i] - want) <= 1e-14 * np.abs(vec[0][first:]).max(), i
