"""All builds of the FP32 transport kernel round alike.

A run that records photons takes the general build (64-bit voxel addresses,
unwrapped positions, lateral faces decided at run time); its tallies must equal
those of the build without records, which production runs take, bit for bit, and
its records must add up to them.  So must the batched builds."""
import numpy as np
import pytest

from paper_2604_13929_gb300 import inputs

pytestmark = pytest.mark.gpu

RAW = ("raw_R", "raw_T", "raw_A", "raw_gated", "raw_lost", "raw_gain", "raw_hist", "raw_depth",
       "raw_sum_w", "raw_sum_wP", "raw_sum_wP2", "batch_photons")
COUNTS = ("launched", "interactions", "scatters", "rr_survive", "rr_kill", "exit_R", "exit_T",
          "gated_n", "steps", "solid_steps")
# shape, porosity, mu_s, mu_a, g, options: dilute and dense, isotropic and forward, odd sizes and
# a few voxels wide, roulette often, absorption beyond the short series, a path cap
CASES = [((37, 22, 18), 0.95, 0.3, 0.01, 0.6, {}), ((24, 40, 31), 0.6, 1.5, 0.02, 0.0, {}),
         ((64, 3, 5), 0.8, 0.5, 0.005, 0.9, {}), ((20, 16, 12), 0.5, 2.0, 0.05, -0.4, {"rr_weight": 0.3}),
         ((16, 17, 33), 0.7, 0.5, 0.3, 0.7, {}), ((48, 12, 12), 0.9, 0.4, 0.004, 0.8, {"path_cap": 60.5})]


@pytest.fixture(scope="module")
def spmc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_13929_gb300 import build
    build.build()
    from paper_2604_13929_gb300 import spmc as s
    return s


def _problem(case):
    shape, phi, mu_s, mu_a, g, _ = case
    return inputs.random_mask(shape, phi, 7), mu_s, mu_a, g


def _assert_same(a, b, what):
    for k in RAW:
        assert np.array_equal(a[k], b[k]), (what, k)
    for k in COUNTS:
        assert a[k] == b[k], (what, k)


@pytest.mark.parametrize("field,mirror", [(1, 0), (0, 0), (1, 1), (0, 1)])
@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("n_rec", [1, 30000])
def test_run_with_records_equals_run_without(spmc, case, field, mirror, n_rec):
    n, opt = 30000, dict(case[5], tally_field=field, lateral_bc=mirror)
    plain, rec = (spmc.Simulation(*_problem(case), **opt, **extra) for extra in ({}, {"records": n_rec}))
    plain.run(n, 41)
    rec.run(n, 41)
    a, b = plain.tallies(check=False), rec.tallies(check=False)
    _assert_same(a, b, "records")
    if field:
        assert np.array_equal(plain.raw_field(), rec.raw_field())
    if n_rec == n:
        _, ints, _ = rec.records(n)                   # interactions, steps, how it ended, roulette survivals
        assert ints[:, 0].sum() == a["interactions"] and ints[:, 1].sum() == a["steps"]
        assert [int((ints[:, 2] == k).sum()) for k in (1, 2, 3, 4)] == [
            a[k] for k in ("exit_R", "exit_T", "rr_kill", "gated_n")]
        assert ints[:, 3].sum() == a["rr_survive"]
    plain.close()
    rec.close()


@pytest.mark.parametrize("mirror", [0, 1])
def test_batched_builds_equal_single_runs(spmc, mirror):
    with spmc.Batch([_problem(c) for c in CASES], lateral_bc=mirror, rr_weight=0.01) as b:
        b.run([8000 + 1111 * i for i in range(len(CASES))], 43)
        for i, case in enumerate(CASES):
            sim = spmc.Simulation(*_problem(case), lateral_bc=mirror, rr_weight=0.01)
            sim.run(8000 + 1111 * i, 43)
            _assert_same(b.tallies(i), sim.tallies(check=False), i)
            assert np.array_equal(b.raw_field(i), sim.raw_field())
            sim.close()


def test_path_moment_sums_carry(spmc):
    """Straight flights through a pore column of 11863283 voxels: two photons of a lane
    already overflow 64 bits of the second moment, all lanes of a block end together, and
    the sums must be the exact 128-bit integers."""
    nz, n = 11863283, 256 * 3
    sim = spmc.Simulation(np.ones((nz, 1, 1), dtype=np.uint8), 0.5, 0.005, 0.7, tally_field=0, blocks=1)
    sim.run(n, 3)
    t = sim.tallies()
    path = np.float32(nz)
    words = lambda v: [v % 2 ** 64, v >> 64]                                      # noqa: E731
    assert t["exit_T"] == n
    assert [int(x) for x in t["raw_sum_wP"]] == words(n * int(path) * 2 ** 32)
    assert [int(x) for x in t["raw_sum_wP2"]] == words(n * int(path * path) * 2 ** 16)
    sim.close()
