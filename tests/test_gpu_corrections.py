"""Multiple-counting sums of few bins: FP32 partial sums of the mixed forms run over few centres.

512 centres on one spot see two galaxies of opposite shear at one place (their multipoles cancel, so the
contraction is exactly zero in their bin, and only the terms of a galaxy counted twice are left) and a
third galaxy.  In turns of 16 a centre's shear is 1, fourteen times 2^-27, and -1: added up in FP32 with
one of the large ones, the small ones are lost, and the large ones cancel.  Runs of k centres lose at most
2 (k - 1) of the fourteen; k is at most 1, 3 and 7 for 2, 4 and 6 bins.  What else rounds: two record entries of
powers <= 2 n_max + 6 = 10, (2 m + 16) 2^-23 each, and three products, 80 2^-23 in all."""
import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "f16x3"])
@pytest.mark.parametrize("nb,run", [(2, 1), (3, 3), (4, 3), (5, 7), (6, 7)])
def test_small_terms_survive_next_to_large_ones(torch_cuda, prec, nb, run):  # noqa: F811
    from paper_2509_07974_gb300 import ext4pcf
    torch, nmax, small = torch_cuda, 2, 2.0 ** -27
    edges = np.geomspace(1.0, 8.0, nb + 1)
    bm, bo = 0, nb - 1
    r = np.sqrt(edges[:-1] * edges[1:])
    ang = np.array([0.7, 0.7, 2.1])
    rad = np.array([r[bm], r[bm], r[bo]])
    pos = np.concatenate([np.zeros((512, 2)), np.stack([rad * np.cos(ang), rad * np.sin(ang)], 1)])
    sh = np.zeros((515, 2))
    sh[:512, 0] = np.tile(np.r_[1.0, np.full(14, small), -1.0], 32)
    sh[512:] = [[0.6, -0.35], [-0.6, 0.35], [0.25, 0.4]]
    mask = np.r_[np.ones(512), np.zeros(3)].astype(np.uint8)
    dev = torch.device("cuda:0")
    est = ext4pcf.Estimator(0, prec)
    ups = est.measure(*(torch.tensor(a, device=dev) for a in (pos, sh, np.ones(515))), edges, nmax, centre_mask=mask)
    got = torch.view_as_complex(ups).cpu().numpy()[0]
    est.close()
    x, u = sh[512:, 0] + 1j * sh[512:, 1], np.exp(1j * ang)
    total = sh[:512, 0].sum()
    for mu in range(8):
        t = ext4pcf.ext4pcf_nth_order_factors(4, mu)[2:].reshape(3, 5)
        for n2 in range(-nmax, nmax + 1):
            for n3 in range(-nmax, nmax + 1):
                f = []
                for _, conj, a2, a3, b in t:
                    v = x * u ** (a2 * n2 + a3 * n3 + b)
                    f.append(v.conj() if conj else v)
                for third in range(3):
                    i, j = [k for k in range(3) if k != third]
                    want = -total * (f[i][:2] * f[j][:2]).sum() * f[third][2]
                    bins = [bm, bm, bm]
                    bins[third] = bo
                    err = abs(got[mu, n2 + nmax, n3 + nmax, bins[0], bins[1], bins[2]] - want)
                    lim = 2 * (run - 1) / 14 + 80 * 2.0 ** -23
                    assert err <= lim * abs(want), (mu, n2, n3, bins, err / abs(want))
