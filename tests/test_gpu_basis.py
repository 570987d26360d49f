"""The contraction through the independent sums (families F0..F3 and FW): sizes at the edges of
its register tiles, row tiles and column groups, against the oracle.

Tolerances are those of the parity tests (1e-10 for FP64, 1e-4 for the mixed forms, floor-relative;
FP32 with the floor of the uncorrected terms): the independent sums take the same products in the
same arithmetic, only grouped by multipole index."""
import numpy as np
import pytest

from metric import empty_slabs, rel_err
from test_gpu_parity import TOL, run_gpu, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(1, 5), (3, 0), (4, 1), (5, 2), (7, 3), (8, 1), (9, 2), (11, 1), (12, 2), (13, 1), (16, 1)]


def _case(nb, seed=31, n=150):
    rng = np.random.default_rng(seed + nb)
    pos = rng.uniform(0, 12, (n, 2))
    return pos, rng.normal(0, 0.3, pos.shape), rng.uniform(0.5, 1.5, n), np.geomspace(0.5, 7.0, nb + 1)


@pytest.mark.parametrize("prec,nb,nmax", [(p, nb, N) for p in ("fp64", "fp32", "f16x3") for nb, N in
                                          SHAPES + ([] if p == "f16x3" else [(17, 1), (24, 0), (25, 1), (32, 1)])
                                          + ([(2, 9), (6, 4), (10, 5), (14, 2), (15, 1)] if p == "f16x3" else [])])
def test_matches_oracle(torch_cuda, oracle, prec, nb, nmax):  # noqa: F811
    pos, sh, w, edges = _case(nb)
    ref = oracle.measure(pos, sh, w, edges, nmax)
    got = run_gpu(torch_cuda, pos, sh, w, edges, nmax, prec)
    unc = oracle.measure(pos, sh, w, edges, nmax, corrections=False) if prec == "fp32" else None
    assert rel_err(got, ref, unc, empty_slabs(pos, edges)).max() < TOL[prec]


@pytest.mark.parametrize("prec", ["fp64", "fp32", "f16x3"])
def test_alternating_output_slots(torch_cuda, prec):  # noqa: F811
    """Catalogues that alternate between two output slots add up in each slot as they do alone."""
    from paper_2509_07974_gb300 import ext4pcf
    torch, nb, nmax = torch_cuda, 5, 2
    cats = [_case(nb, seed=60 + k, n=60 + 20 * k) for k in range(4)]
    edges = cats[0][3]
    pos, sh, w = (np.concatenate([c[k] for c in cats]) for k in range(3))
    offs = np.concatenate([[0], np.cumsum([len(c[2]) for c in cats])]).astype(np.int64)
    slots = np.array([1, 0, 1, 0], dtype=np.int32)
    dev = torch.device("cuda:0")
    t = [torch.tensor(a, device=dev) for a in (pos, sh, w)]
    est = ext4pcf.Estimator(0, prec)
    ups = torch.zeros(ext4pcf.Estimator.ups_shape(nb, nmax, 2), dtype=torch.float64, device=dev)
    ext4pcf.ext4pcf_measure_batch(est.ctx, *t, len(w), edges, nb, nmax, offs, 4, slots, 2, None, ups)
    got = torch.view_as_complex(ups).cpu().numpy()
    est.close()
    alone = [run_gpu(torch, c[0], c[1], c[2], edges, nmax, prec) for c in cats]
    for s in (0, 1):
        want = sum(alone[k] for k in range(4) if slots[k] == s)
        assert rel_err(got[s], want).max() < TOL[prec]
