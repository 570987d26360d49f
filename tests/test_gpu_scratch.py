"""Device memory that a call takes for its multiple-counting sums."""
import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _catalogue(torch, n):
    rng = np.random.default_rng(n)
    return [torch.tensor(a, device="cuda:0") for a in (rng.uniform(0, 10, (n, 2)), rng.normal(0, 0.3, (n, 2)), np.ones(n))]


def _taken(torch, call):
    """Bytes that a fresh context holds after its first call (the kernels have been loaded before)."""
    from paper_2509_07974_gb300 import ext4pcf
    used = []
    for _ in range(2):
        est = ext4pcf.Estimator(0, "fp32")
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        call(est)
        torch.cuda.synchronize()
        used.append(before - torch.cuda.mem_get_info()[0])
        est.close()
    return used[1]


def test_records_take_no_memory_for_sums_they_do_not_form(torch_cuda):  # noqa: F811
    """n_max = 23, 32 bins: a record is 87 KB, one copy of the sums 10.3 MB and 16 of them 165 MB."""
    from paper_2509_07974_gb300 import ext4pcf
    torch, nb, nmax, n = torch_cuda, 32, 23, 100
    cat, edges, centres = _catalogue(torch, n), np.geomspace(0.3, 5.0, nb + 1), np.arange(4, dtype=np.int64)
    rec = torch.zeros((4, ext4pcf.record_layout(nb, nmax)["rec"], 2), dtype=torch.float64, device="cuda:0")
    took = _taken(torch, lambda est: ext4pcf.ext4pcf_multipoles(est.ctx, *cat, n, edges, nb, nmax, centres, 4, rec))
    assert took < 64 << 20, took


def test_slots_share_the_sums_of_the_forms_that_take_them_in_turn(torch_cuda):  # noqa: F811
    """The FP32 form has one slot's sums at a time: eight slots take no more than one (16 copies of 0.55
    MB a slot before; allocations round up to 2 MB each, some forty of them)."""
    torch, nb, nmax, n = torch_cuda, 16, 4, 800
    cat, edges = _catalogue(torch, n), np.geomspace(0.3, 5.0, nb + 1)
    from paper_2509_07974_gb300 import ext4pcf
    offs, took = np.arange(9, dtype=np.int64) * 100, {}
    for n_out in (1, 8):
        ups = torch.zeros(ext4pcf.Estimator.ups_shape(nb, nmax, n_out), dtype=torch.float64, device="cuda:0")
        slots = np.arange(8, dtype=np.int32) % n_out
        took[n_out] = _taken(torch, lambda est: ext4pcf.ext4pcf_measure_batch(
            est.ctx, *cat, n, edges, nb, nmax, offs, 8, slots, n_out, None, ups))
    assert took[8] <= took[1] + (16 << 20), took


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-5), ("f16x3", 1e-5), ("3xtf32", 1e-5)])
def test_xi_of_alternating_slots(torch_cuda, prec, tol):  # noqa: F811
    """The xi accumulators of four catalogues in two slots, in turn, against the pair sums written out: sums
    of FP32 records, (2 m + 16) 2^-23 of the absolute sum with m <= 4 (3e-6), in FP64 2^-52."""
    from paper_2509_07974_gb300 import ext4pcf
    torch, nb, n = torch_cuda, 3, 120
    rng, edges = np.random.default_rng(9), np.geomspace(0.4, 4.0, nb + 1)
    pos, sh, w = rng.uniform(0, 8, (4 * n, 2)), rng.normal(0, 0.3, (4 * n, 2)), rng.uniform(0.5, 1.5, 4 * n)
    offs, slots = np.arange(5, dtype=np.int64) * n, np.array([1, 0, 1, 0], dtype=np.int32)
    ups = torch.zeros(ext4pcf.Estimator.ups_shape(nb, 2, 2), dtype=torch.float64, device="cuda:0")
    xi = torch.zeros((2, nb, 3, 2), dtype=torch.float64, device="cuda:0")
    est = ext4pcf.Estimator(0, prec)
    t = [torch.tensor(a, device="cuda:0") for a in (pos, sh, w)]
    ext4pcf.ext4pcf_measure_batch(est.ctx, *t, 4 * n, edges, nb, 2, offs, 4, slots, 2, None, ups, xi)
    got = torch.view_as_complex(xi).cpu().numpy()
    est.close()
    want, size = np.zeros((2, nb, 3), complex), np.zeros((2, nb, 3))
    for k in range(4):
        s = slice(k * n, (k + 1) * n)
        d = pos[s][None] - pos[s][:, None]
        r2, u = (d ** 2).sum(-1), np.exp(1j * np.arctan2(d[..., 1], d[..., 0]))
        x, ww = w[s] * (sh[s, 0] + 1j * sh[s, 1]), w[s]
        for b in range(nb):
            m = (r2 >= edges[b] ** 2) & (r2 < edges[b + 1] ** 2)
            for q, v in enumerate((x.conj()[:, None] * x[None], x[:, None] * x[None] * u ** -4, ww[:, None] * ww[None])):
                want[slots[k], b, q] += v[m].sum()
                size[slots[k], b, q] += np.abs(v[m]).sum()
    assert (np.abs(got - want) <= tol * size).all(), np.abs(got - want).max()
