"""Batched launches whose voxel fields form several groups equal separate runs.

Warps stay with a problem until it runs out, then take another of its group of
problems (fields of at most 96 MB together), then the next group.  Five volumes
of 160^3 and one small one (33.6 MB a field: groups of two) with uneven photon
counts, zero among them, and claims that leave some warps without a chunk."""
import numpy as np
import pytest

from paper_2604_13929_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts,chunk", [([30000, 0, 500, 45000, 20000, 9000], 128), ([40, 1, 0, 0, 3000, 17], 32)])
def test_groups_equal_separate_runs(counts, chunk):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_13929_gb300 import build
    build.build()
    from paper_2604_13929_gb300 import spmc
    sizes = [160, 160, 160, 160, 160, 24]
    problems = [(inputs.random_mask((n,) * 3, 0.6 + 0.05 * i, i), 0.3 + 0.2 * i, 0.01, 0.15 * i)
                for i, n in enumerate(sizes)]
    with spmc.Batch(problems, batch_chunk=chunk) as b:
        b.run(counts, 13)
        b.run(counts, 13)
        for i, pr in enumerate(problems):
            sim = spmc.Simulation(*pr)
            sim.run(2 * counts[i], 13)
            t, ref = b.tallies(i), sim.tallies(check=False)
            for k in ("raw_R", "raw_T", "raw_A", "raw_hist", "raw_depth", "raw_sum_w", "raw_sum_wP2", "batch_photons"):
                assert np.array_equal(t[k], ref[k]), (i, k)
            for k in ("launched", "interactions", "scatters", "exit_R", "exit_T", "steps", "solid_steps"):
                assert t[k] == ref[k], (i, k)
            assert np.array_equal(b.raw_field(i), sim.raw_field())
            sim.close()
