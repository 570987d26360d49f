"""The third-order contraction at the edges of its blocks: one bin and the most, n_max = 0 and the
largest, sums that fill no, one and several blocks, waves with a remainder, against the oracle's
brute force over triplets of distinct galaxies.

Bound: FP64 sums of at most n terms whose factors are sums of at most n phases of power 2 n_max + 3:
(2 n_max + 3 + 3 n) 2^-50 of the sum of the terms' magnitudes."""
import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nmax,nb,n,wave", [(0, 1, 40, 0), (0, 32, 90, 33), (1, 11, 70, 64), (3, 10, 70, 0),
                                            (2, 23, 70, 32), (40, 2, 40, 0)])
def test_third_order_at_block_edges(torch_cuda, oracle, nmax, nb, n, wave):  # noqa: F811
    from paper_2509_07974_gb300 import ext4pcf
    torch = torch_cuda
    rng = np.random.default_rng(nb + nmax)
    pos, sh, w = rng.uniform(0, 6.0, (n, 2)), rng.normal(0, 0.3, (n, 2)), rng.uniform(0.5, 1.5, n)
    edges = np.geomspace(0.3, 5.0, nb + 1)
    dev = torch.device("cuda:0")
    t = [torch.tensor(a, dtype=torch.float64, device=dev) for a in (pos, sh, w)]
    ups = torch.zeros((5, 2 * nmax + 1, nb, nb, 2), dtype=torch.float64, device=dev)
    est = ext4pcf.Estimator(0, "fp64", wave_centres=wave)
    ext4pcf.ext4pcf_measure3(est.ctx, *t, n, edges, nb, nmax, ups)
    torch.cuda.synchronize()
    got = torch.view_as_complex(ups).cpu().numpy()
    est.close()
    ref = oracle.bruteforce_multipoles(3, pos, sh, w, edges, nmax, distinct=True)
    r2 = ((pos[:, None] - pos[None]) ** 2).sum(-1)
    inside = [(r2 >= a * a) & (r2 < b * b) for a, b in zip(edges[:-1], edges[1:])]
    big = np.maximum(w, w * np.hypot(*sh.T))
    s = np.array([m @ big for m in inside])
    lim = (2 * nmax + 3 + 3 * n) * 2.0 ** -50 * np.einsum("i,ai,bi->ab", big, s, s)
    assert (np.abs(got - ref) <= lim).all(), (np.abs(got - ref) / np.maximum(lim, 1e-300)).max()
