"""Aperture records summed by one and by eight threads: radii with too few rows for eight splits and
with many, aperture counts around a block's, against the oracle (bounds of test_gpu_map_direct)."""
import numpy as np
import pytest

from test_gpu_map_direct import check, est, run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ap", [1, 15, 16, 17, 129])
def test_apertures_with_few_and_many_splits(torch_cuda, oracle, est, n_ap):  # noqa: F811
    rng = np.random.default_rng(n_ap)
    n, side = 3000, 40.0
    pos, sh, w = rng.uniform(0, side, (n, 2)), rng.normal(0, 0.3, (n, 2)), rng.uniform(0.5, 1.5, n)
    thetas = [0.5, 4.0]  # 16 or so and 128 rows of cells
    centres = [rng.uniform(0, side, (n_ap, 2)) for _ in thetas]
    mom, rec = run(torch_cuda, est, pos, sh, w, thetas, centres)
    check(oracle, pos, sh, w, thetas, centres, mom, rec)
