"""Passes of 1 to 64 voxel steps give the same tallies bit for bit.

A lane takes the plain step form for a whole pass unless the path cap or the
iteration limit could fall inside it; a cap or limit of a few dozen steps puts
that change of form inside the longer passes.  Dilute optics (an interaction
every 30 steps or more), where passes run long, and dense ones, both tallies and
both lateral faces, single runs and one-launch batches."""
import numpy as np
import pytest

from paper_2604_13929_gb300 import inputs

pytestmark = pytest.mark.gpu

RAW = ("raw_R", "raw_T", "raw_A", "raw_gated", "raw_lost", "raw_gain", "raw_hist", "raw_depth",
       "raw_sum_w", "raw_sum_wP", "raw_sum_wP2", "batch_photons")
COUNTS = ("launched", "interactions", "scatters", "rr_survive", "rr_kill", "exit_R", "exit_T",
          "gated_n", "steps", "solid_steps")


@pytest.fixture(scope="module")
def spmc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_13929_gb300 import build
    build.build()
    from paper_2604_13929_gb300 import spmc as s
    return s


def _run(spmc, problem, n, **opt):
    sim = spmc.Simulation(*problem, **opt)
    sim.run(n, 29)
    out = sim.tallies(check=False), sim.raw_field() if opt.get("tally_field", 1) else None
    sim.close()
    return out


def _assert_same(a, b, what):
    for k in RAW:
        assert np.array_equal(a[0][k], b[0][k]), (what, k)
    for k in COUNTS:
        assert a[0][k] == b[0][k], (what, k)
    assert a[1] is None or np.array_equal(a[1], b[1]), what


@pytest.mark.parametrize("mu_s,phi", [(0.3, 0.95), (1.5, 0.6)])
@pytest.mark.parametrize("field,mirror", [(1, 0), (0, 0), (1, 1), (0, 1)])
@pytest.mark.parametrize("limit", [{}, {"path_cap": 20.3}, {"iter_limit": 37}])
def test_pass_lengths_agree(spmc, mu_s, phi, field, mirror, limit):
    problem = (inputs.random_mask((37, 22, 18), phi, 5), mu_s, 0.01, 0.6)
    opt = dict(limit, tally_field=field, lateral_bc=mirror)
    base = _run(spmc, problem, 30000, steps_per_pass=1, **opt)
    if limit:
        assert base[0]["gated_n"] > 0
    _assert_same(base, _run(spmc, problem, 30000, **opt), "automatic")
    for length in (4, 8, 29, 64):
        _assert_same(base, _run(spmc, problem, 30000, steps_per_pass=length, **opt), length)


@pytest.mark.parametrize("length", [None, 1, 29, 64])
def test_batched_pass_lengths_agree(spmc, length):
    problems = [(inputs.random_mask((40, 24, 24), 0.95, 1), 0.3, 0.01, 0.6),
                (inputs.random_mask((20, 16, 12), 0.6, 2), 1.5, 0.02, 0.2),
                (inputs.random_mask((33, 9, 10), 0.9, 3), 0.05, 0.002, 0.9)]
    n = [20000, 9000, 15000]
    with spmc.Batch(problems, path_cap=55.7, **({} if length is None else {"steps_per_pass": length})) as b:
        b.run(n, 29)
        for i, problem in enumerate(problems):
            ref = _run(spmc, problem, n[i], steps_per_pass=1, path_cap=55.7)
            _assert_same(ref, (b.tallies(i), b.raw_field(i)), (i, length))


@pytest.mark.parametrize("field", [1, 0])
@pytest.mark.parametrize("threads", [64, 256])
def test_staged_bricks_agree(spmc, field, threads):
    """Staging the entry slab of the mask, as many bricks as fit, changes no result."""
    problem = (inputs.random_mask((96, 92, 100), 0.9, 5), 0.3, 0.01, 0.6)
    base = _run(spmc, problem, 20000, tally_field=field, threads=threads)
    for bricks in (-1, 1, 2048, 12288, 28000):
        _assert_same(base, _run(spmc, problem, 20000, tally_field=field, threads=threads, smem_bricks=bricks), bricks)


def test_pass_length_change_between_graph_replays(spmc):
    """Setting the pass length rebuilds the problem table and the captured graph; photon ids go on."""
    problems = [(inputs.random_mask((40, 24, 24), 0.95, 1), 0.3, 0.01, 0.6),
                (inputs.random_mask((20, 16, 12), 0.6, 2), 1.5, 0.02, 0.2)]
    n = [9000, 5000]
    with spmc.Batch(problems, graph=1) as b:
        assert b.get_option("steps_per_pass") == 8
        for length in (None, None, 29, 29, 1):
            if length:
                b.set_option("steps_per_pass", length)
                assert b.get_option("steps_per_pass") == length
            b.run(n, 29)
        for i, problem in enumerate(problems):
            ref = _run(spmc, problem, 5 * n[i], steps_per_pass=1)
            _assert_same(ref, (b.tallies(i), b.raw_field(i)), i)
