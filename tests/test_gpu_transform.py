"""The real-space and aperture transforms at the edges of their tiles: odd, even and single angular
bins (a bin that is its own mirror or not), one tile and its remainders, few and many aperture
radii, more triples than one chunk, against the oracle, for multipoles without any symmetry.

Bounds: FP64 throughout.  A bin count or component sums (2 n_max + 1)^2 products, so Gamma N within
16 (2 n_max + 1) 2^-52 of the sum of their magnitudes, and Gamma within that over the smallest count.
The aperture integral loses what its polynomial and the sum over bins cancel, at most 1e6 here: 1e-9
of the largest of its eight components."""
import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [(0, 1, 1, 1), (0, 2, 2, 3), (1, 2, 16, 8), (2, 2, 17, 9), (5, 3, 31, 5), (3, 1, 48, 64), (20, 1, 65, 24),
         (40, 1, 33, 2)]


def _multipoles(N, nb, seed):
    rng = np.random.default_rng(seed)
    nn = 2 * N + 1
    u = rng.normal(size=(9, nn, nn, nb, nb, nb)) + 1j * rng.normal(size=(9, nn, nn, nb, nb, nb))
    u[8] /= nn * nn
    u[8, N, N] += 4.0 * np.pi  # the counts stay well away from 0
    if nb > 1:
        u[:, :, :, 1, 0, 1] = 0  # an empty triple
    return u


def _device(torch, u):
    return torch.tensor(np.stack([u.real, u.imag], axis=-1), device="cuda:0")


@pytest.mark.parametrize("N,nb,nphi,n_ap", CASES)
def test_transforms_at_tile_edges(torch_cuda, oracle, N, nb, nphi, n_ap):  # noqa: F811
    from paper_2509_07974_gb300 import ext4pcf
    u = _multipoles(N, nb, 100 * N + nphi)
    edges, ap = np.geomspace(1.0, 9.0, nb + 1), np.geomspace(1.0, 12.0, n_ap)
    gam_o, nrm_o = oracle.to_real_space(u, nphi)
    m4_o, eb_o, _ = oracle.map4(u, edges, nphi, ap)
    est = ext4pcf.Estimator(0, "fp64")
    d = _device(torch_cuda, u)
    gam, nrm = est.to_real_space(d, nphi)
    m4, eb, _ = est.to_map4(d, edges, nphi, ap)
    tiny, _, _ = est.to_map4(d * 2.0 ** -1000, edges, nphi, ap)  # Gamma is a ratio
    torch_cuda.cuda.synchronize()
    est.close()
    lim = 16 * (2 * N + 1) * 2.0 ** -52 * np.abs(u).sum(axis=(1, 2)) / nphi ** 2
    err_n = np.abs(nrm.cpu().numpy() - nrm_o).max(axis=(-1, -2))
    assert (err_n <= lim[8]).all(), (err_n / lim[8]).max()
    g = torch_cuda.view_as_complex(gam).cpu().numpy()
    count = np.abs(nrm_o).min(axis=(-1, -2))
    err_g = np.abs(g - gam_o).max(axis=(-1, -2))
    full = count > 0
    assert (err_g[:, ~full] == 0).all()
    bound = (lim[:8] + lim[8] * np.abs(gam_o).max(axis=(-1, -2)))[:, full] / count[full]
    assert (err_g[:, full] <= bound).all(), (err_g[:, full] / bound).max()
    for got, ref in ((m4, m4_o.reshape(-1)), (tiny, m4_o.reshape(-1)), (eb, eb_o)):
        got, ref = np.asarray(got).reshape(n_ap, -1), np.asarray(ref).reshape(n_ap, -1)
        if np.iscomplexobj(ref):
            ref = np.stack([ref.real, ref.imag], axis=-1).reshape(n_ap, -1)
        if np.iscomplexobj(got):
            got = np.stack([got.real, got.imag], axis=-1).reshape(n_ap, -1)
        scale = np.abs(ref).max(axis=1, keepdims=True)
        assert (np.abs(got - ref) <= 1e-9 * scale).all(), (np.abs(got - ref) / scale).max()


def test_map4_over_more_than_one_chunk(torch_cuda, oracle):  # noqa: F811
    from paper_2509_07974_gb300 import ext4pcf
    nb, nphi, ap = 2, 520, [4.0]  # eight triples, seven to a chunk
    u, edges = _multipoles(1, nb, 3), np.geomspace(1.0, 9.0, nb + 1)
    m4_o, _, _ = oracle.map4(u, edges, nphi, ap)
    est = ext4pcf.Estimator(0, "fp64")
    m4, _, _ = est.to_map4(_device(torch_cuda, u), edges, nphi, ap)
    est.close()
    got = np.asarray(m4).reshape(-1)
    got = got if np.iscomplexobj(got) else got[0::2] + 1j * got[1::2]
    assert np.abs(got - m4_o[0]).max() <= 1e-9 * np.abs(m4_o).max()
