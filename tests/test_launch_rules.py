"""Launch rules of the kernels (plain C++ headers, compiled here with the host compiler)."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_13929_gb300", "csrc")
SOURCE = r"""
#include "spmc_plan.h"
#include "spnn_plan.h"
extern "C" int pass_steps(int option, double mus, double porosity) { return spmc::pass_steps(option, mus, porosity); }
extern "C" int staged_bricks(int want, size_t own, int resident) { return spmc::staged_bricks(want, own, resident); }
extern "C" unsigned ring_budget(long long tiles, int grid_n, int ksteps, int sms, int scatter, int alone, int option_kb) {
    return spnn::ring_budget(tiles, grid_n, ksteps, sms, scatter, alone, option_kb);
}
extern "C" int slab_depth(int bx, int by, long long columns, int D, int n, int kc_total, int sms) {
    return spnn::slab_shape(bx, by, columns, D, n, kc_total, sms).zp;
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rules")
    src, lib = d / "rules.cpp", d / "rules.so"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(lib), str(src)], check=True)
    r = ctypes.CDLL(str(lib))
    r.pass_steps.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double]
    r.staged_bricks.argtypes = [ctypes.c_int, ctypes.c_size_t, ctypes.c_int]
    r.ring_budget.argtypes = [ctypes.c_longlong] + [ctypes.c_int] * 6
    r.slab_depth.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong] + [ctypes.c_int] * 4
    r.ring_budget.restype = ctypes.c_uint
    return r


@pytest.mark.parametrize("option", [1, 3, 8, 16, 29, 64])
@pytest.mark.parametrize("mus,porosity", [(0.5, 0.70), (2.0, 0.5), (0.5, 0.90), (0.0, 0.9), (0.3, 1.0)])
def test_a_pass_length_that_was_set_is_taken(rules, option, mus, porosity):
    assert rules.pass_steps(option, mus, porosity) == option


def test_automatic_pass_length_follows_the_optics(rules):
    assert rules.pass_steps(0, 0.5, 0.70) == 4          # an interaction every 10 steps
    assert rules.pass_steps(0, 0.5, 0.90) == 8          # every 30
    assert rules.pass_steps(0, 0.0, 0.5) == 8


@pytest.mark.parametrize("own", [4352, 20736, 21760, 42000])
@pytest.mark.parametrize("resident", [3, 4, 8])
@pytest.mark.parametrize("want", [0, 1, 512, 2048, 5000, 8192, 12288, 20000, 28512])
def test_staged_bricks_keep_the_resident_ctas(rules, want, own, resident):
    """The slab shrinks by the kernel's own shared memory instead of costing a CTA per SM."""
    per_sm, per_cta, reserved, bare = 228 * 1024, 227 * 1024, 1024, 4352
    n = rules.staged_bricks(want, own, resident)
    before = max(1, min(resident, per_sm // (8 * want + bare + reserved)))
    assert 0 <= n <= want
    assert 8 * n + own <= per_cta
    if n:
        assert min(resident, per_sm // (8 * n + own + reserved)) >= before
        assert n == want or 8 * (n + 1) + own > min(per_cta, per_sm // before - reserved)


def test_staged_bricks_at_scratch_limits(rules):
    assert rules.staged_bricks(28513, 21760, 4) == 28513      # over 227 KB beside the tallies: refused by the launch
    assert rules.staged_bricks(20000, 0, 4) == 20000          # a kernel without shared memory of its own
    assert rules.staged_bricks(-1, 21760, 4) == -1


@pytest.mark.parametrize("tiles,grid_n,ksteps,scatter,alone,kb", [
    (4, 1, 9, 0, 0, 200), (32, 1, 9, 0, 0, 200), (304, 1, 9, 0, 0, 200), (305, 1, 9, 0, 0, 110), (152, 2, 9, 0, 0, 200),
    (153, 2, 1, 0, 0, 110),
    # N tiles count: up 256 -> 128 from 8^3 at batch 64 is 256 boxes x 8 N tiles; scatter
    # epilogues keep two CTAs per SM however few tiles there are ...
    (256, 8, 4, 0, 0, 110), (256, 8, 4, 1, 0, 110), (4, 8, 4, 1, 0, 110), (32, 4, 2, 1, 0, 110), (128, 2, 1, 1, 0, 110),
    (256, 4, 1, 1, 0, 110), (256, 1, 1, 1, 0, 110),
    # ... except where the first of two N tiles would leave the second few CTAs
    (253, 2, 1, 1, 0, 110), (254, 2, 1, 1, 0, 200), (256, 2, 2, 1, 0, 200), (303, 2, 1, 1, 0, 200),
    (304, 2, 1, 1, 0, 110), (256, 2, 3, 1, 0, 110),
    (4, 1, 9, 0, 1, 220), (5000, 1, 9, 0, 1, 220), (5000, 1, 1, 1, 1, 220),
])
def test_ring_budget_counts_output_tiles(rules, tiles, grid_n, ksteps, scatter, alone, kb):
    assert rules.ring_budget(tiles, grid_n, ksteps, 152, scatter, alone, 0) == kb * 1024
    assert rules.ring_budget(tiles, grid_n, ksteps, 152, scatter, alone, 90) == 90 * 1024


def _slab(rules, B, D, H, W, cin, cout):
    """Box depth of the z-walk on 152 SMs and boxes per CTA."""
    bx = min(W, 32)
    by = 128 // bx
    assert H >= by                                            # one-plane tiles
    columns = (W // bx) * (H // by) * B
    zp = rules.slab_depth(bx, by, columns, D, cout, cin // 8, 152)
    return zp, columns * (D // zp) / 152 if zp else 0


def test_slab_cases_reach_every_depth_with_reused_buffers(rules):
    from test_gpu_surrogate_slab_depths import CASES
    reached = set()
    for *shape, depth in CASES:
        zp, boxes = _slab(rules, *shape)
        assert zp == depth, shape
        if boxes > 2:
            reached.add((shape[-1], zp))
    assert reached == {(16, 2), (16, 4), (16, 8), (16, 16), (32, 2), (32, 4), (32, 8), (64, 2), (64, 4)}


@pytest.mark.parametrize("n,cin,fits", [(16, 16, True), (32, 64, True), (32, 80, False), (64, 32, True), (64, 48, False),
                                        (48, 16, False), (128, 16, False), (8, 16, False)])
def test_slab_takes_only_what_fits(rules, n, cin, fits):
    assert (rules.slab_depth(32, 4, 64, 32, n, cin // 8, 152) > 0) == fits
    assert rules.slab_depth(32, 4, 64, 1, n, cin // 8, 152) == 0          # no depth to walk
