"""Which kernel of the FP32 gather takes a centre (ext4pcf_sector_centres), and the places where the two
meet: tree passes that add into the records of dense catalogues, waves that hold dense and sparse catalogues, and
more centres than the sector kernel has blocks, over catalogues of different cells."""
import numpy as np
import pytest

from metric import rel_err
from test_gpu_parity import TOL, torch_cuda  # noqa: F401
from test_gpu_tree import _check as check_tree

pytestmark = pytest.mark.gpu


def _catalogue(n, side, seed):
    rng = np.random.default_rng(seed)
    return rng.uniform(0, side, (n, 2)), rng.normal(0, 0.3, (n, 2)), rng.uniform(0.5, 1.5, n)


def _records(torch, prec, cat, edges, nmax, centres, **tree):
    """Records of the centres and how many of them went through sectors."""
    from paper_2509_07974_gb300 import ext4pcf
    ctx = ext4pcf.ext4pcf_create(ext4pcf.Config(
        device=0, stream=torch.cuda.current_stream().cuda_stream, precision=ext4pcf.PRECISION[prec], deterministic=1, **tree))
    nb, lay = len(edges) - 1, ext4pcf.record_layout(len(edges) - 1, nmax)
    out = np.zeros((len(centres), lay["rec"], 2))
    t = [torch.tensor(a, device="cuda:0") for a in cat]
    ext4pcf.ext4pcf_multipoles(ctx, *t, len(cat[2]), edges, nb, nmax, centres, len(centres), out)
    taken = ext4pcf.ext4pcf_sector_centres(ctx)
    ext4pcf.ext4pcf_destroy(ctx)
    return out[..., 0] + 1j * out[..., 1], taken


def _within_rounding(torch, cat, edges, nmax, centres, got):
    """FP32 records against the FP64 form's, bound as in test_gpu_gather_sector: (2 m + 16 + t m) 2^-23 of the
    sum of the absolute weights (the records at power 0 of the same galaxies with real shears |gamma|)."""
    from paper_2509_07974_gb300 import ext4pcf
    ref, taken = _records(torch, "fp64", cat, edges, nmax, centres)
    assert taken == 0
    size = np.stack([np.hypot(*cat[1].T), np.zeros(len(cat[2]))], 1)
    size, _ = _records(torch, "fp64", (cat[0], size, cat[2]), edges, nmax, centres)
    nb, lay = len(edges) - 1, ext4pcf.record_layout(len(edges) - 1, nmax)
    turn = 2 ** 0.5 * edges[-1] / edges[:-1]
    for name in ("G", "W", "XX", "XA", "WW"):
        off, first, cnt = lay[name]
        m = np.abs(np.arange(first, first + cnt))[:, None]
        total = size[:, off - first * nb: off + (1 - first) * nb].real  # power 0
        err = np.abs(got - ref)[:, off: off + cnt * nb].reshape(-1, cnt, nb)
        assert (err <= (2 * m + 16 + turn * m) * 2.0 ** -23 * total[:, None, :]).all(), name


@pytest.mark.parametrize("nmax,nb,n,side,dense", [
    (20, 10, 9000, 10.0, True), (20, 10, 4000, 10.0, False), (30, 6, 5000, 10.0, True), (30, 6, 2500, 10.0, False),
    (40, 5, 4000, 10.0, True), (12, 10, 15000, 10.0, False), (6, 2, 120000, 10.0, False)])
def test_dense_catalogues_go_through_sectors(torch_cuda, nmax, nb, n, side, dense):  # noqa: F811
    """Every galaxy within reach, well past the line or well below it."""
    cat, edges = _catalogue(n, side, nmax + nb), np.geomspace(0.1, 0.7 * side, nb + 1)
    centres = np.arange(7, dtype=np.int64) * (n // 7)
    _, taken = _records(torch_cuda, "fp32", cat, edges, nmax, centres)
    assert taken == (len(centres) if dense else 0)


@pytest.mark.parametrize("nmax,nb,n,inner", [(21, 10, 60000, 0.05), (24, 10, 20000, 0.05), (30, 10, 9000, 0.05),
                                             (40, 10, 9000, 0.05), (18, 6, 29000, 0.3), (20, 12, 28000, 0.05)])
def test_narrow_bins_stay_with_the_power_sums(torch_cuda, nmax, nb, n, inner):  # noqa: F811
    """Many pairs in bins without sectors: the sector kernel was 3 to 18% slower there."""
    cat, edges = _catalogue(n, 10.0, nmax + nb), np.geomspace(7.0 * inner, 7.0, nb + 1)
    _, taken = _records(torch_cuda, "fp32", cat, edges, nmax, np.arange(7, dtype=np.int64))
    assert taken == 0


@pytest.mark.parametrize("nmax,n", [(7, 100000), (8, 45000), (9, 29000)])
def test_lowest_orders_of_the_sectors(torch_cuda, nmax, n):  # noqa: F811
    cat, edges = _catalogue(n, 10.0, nmax), np.geomspace(0.1, 7.0, 5)
    centres = np.arange(12, dtype=np.int64) * (n // 12)
    got, taken = _records(torch_cuda, "fp32", cat, edges, nmax, centres)
    assert taken == 12
    _within_rounding(torch_cuda, cat, edges, nmax, centres, got)


@pytest.mark.parametrize("nmax,nb,n", [(20, 9, 11000), (30, 6, 9000)])
def test_more_centres_than_blocks(torch_cuda, nmax, nb, n):  # noqa: F811
    cat, edges = _catalogue(n, 12.0, n), np.geomspace(0.1, 8.4, nb + 1)
    centres = np.random.default_rng(1).choice(n, 400, replace=False).astype(np.int64)
    got, taken = _records(torch_cuda, "fp32", cat, edges, nmax, centres)
    assert taken == 400
    _within_rounding(torch_cuda, cat, edges, nmax, centres, got)


@pytest.mark.parametrize("nmax,nb,n", [(20, 8, 60000), (30, 7, 50000)])
def test_tree_passes_add_into_the_records(torch_cuda, nmax, nb, n):  # noqa: F811
    """Cells of 1/16 and 1/8: the galaxies and both reduced catalogues are dense, every pass has bins
    without width, and the later two add.  Bound of the tree tests (2e-6 of the largest value)."""
    from oracle import tree
    from paper_2509_07974_gb300 import ext4pcf
    cat, edges = _catalogue(n, 16.0, n), np.geomspace(0.3, 11.0, nb + 1)
    levels = tree.bin_levels(edges, 0.0625, 2, 48.0)
    assert set(levels.tolist()) == {0, 1, 2}
    centres = np.arange(6, dtype=np.int64) * (n // 6)
    got, taken = _records(torch_cuda, "fp32", cat, edges, nmax, centres, tree_delta1=0.0625, tree_levels=2,
                          tree_rmin=48.0)
    assert taken == 3 * len(centres)
    lay = ext4pcf.record_layout(nb, nmax)
    G, W = (got[:, lay[k][0]: lay[k][0] + lay[k][2] * nb].reshape(len(centres), -1, nb) for k in ("G", "W"))
    refs = [_tree_centre(tree, cat, c, edges, levels, lay["G"][1], 2 * nmax, 0.0625) for c in centres]
    check_tree(G, W, lay["G"][1], np.stack([r[0] for r in refs]), np.stack([r[1] for r in refs]), nmax, 2e-6)


def _tree_centre(tree, cat, c, edges, levels, lo, hi, delta1):
    """oracle.tree.neighbour_multipoles for one centre."""
    pos, sh, w = cat
    cats = {0: (pos, w * (sh[:, 0] + 1j * sh[:, 1]), w)}
    for d in (1, 2):
        cats[d] = tree.reduced_catalogue(pos, sh, w, 2.0 ** (d - 1) * delta1, pos.min(axis=0))
    n = np.arange(lo, hi + 1)
    out = np.zeros((2, len(n), len(edges) - 1), complex)
    for b in range(len(edges) - 1):
        p, x, ww = cats[levels[b]]
        d = p - pos[c]
        r2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]
        s = (r2 >= edges[b] * edges[b]) & (r2 < edges[b + 1] * edges[b + 1])
        u = np.exp(1j * np.outer(n, np.arctan2(d[s, 1], d[s, 0])))
        out[0, :, b], out[1, :, b] = u @ x[s], u @ ww[s]
    return out


def test_one_wave_of_dense_and_sparse_catalogues(torch_cuda):  # noqa: F811
    """Seven catalogues in one split-FP16 wave, dense and sparse in turn, of different cells (each catalogue's
    grid follows its extent), 60 centres each; every one against the FP64 form."""
    from paper_2509_07974_gb300 import ext4pcf
    torch, nmax, nb = torch_cuda, 20, 6
    edges = np.geomspace(0.2, 7.0, nb + 1)
    shape = [(9000, 9.0), (700, 14.0), (12000, 11.0), (3000, 30.0), (30000, 18.0), (300, 6.0), (8000, 6.0)]
    cats = [_catalogue(n, side, k) for k, (n, side) in enumerate(shape)]
    pos, sh, w = (np.concatenate([c[k] for c in cats]) for k in range(3))
    offs = np.concatenate([[0], np.cumsum([len(c[2]) for c in cats])]).astype(np.int64)
    mask = np.zeros(len(w), np.uint8)
    rng = np.random.default_rng(5)
    for k in range(len(shape)):
        mask[offs[k] + rng.choice(shape[k][0], 60, replace=False)] = 1
    t = [torch.tensor(a, device="cuda:0") for a in (pos, sh, w)]
    got = {}
    for prec in ("fp64", "f16x3"):
        est = ext4pcf.Estimator(0, prec)
        ups, st = est.measure(*t, edges, nmax, cat_offsets=offs, centre_mask=mask, want_stats=True)
        got[prec] = torch.view_as_complex(ups).cpu().numpy()
        assert ext4pcf.ext4pcf_sector_centres(est.ctx) == (0 if prec == "fp64" else 4 * 60)
        est.close()
        assert prec == "fp64" or st["waves"] == 1
    for k in range(len(shape)):
        own = slice(offs[k], offs[k + 1])
        empty = _empty(pos[own], mask[own], edges)
        assert rel_err(got["f16x3"][k], got["fp64"][k], empty=empty).max() < TOL["f16x3"], k


def _empty(pos, mask, edges):
    """metric.empty_slabs for the centres of a mask."""
    nb = len(edges) - 1
    tri = np.array(np.meshgrid(*[np.arange(nb)] * 3, indexing="ij")).reshape(3, -1).T
    need = np.stack([(tri == b).sum(axis=1) for b in range(nb)], axis=1)
    full = np.zeros(len(tri), bool)
    for c in np.flatnonzero(mask):
        d = pos - pos[c]
        r2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]
        n = np.array([((r2 >= edges[b] ** 2) & (r2 < edges[b + 1] ** 2)).sum() for b in range(nb)])
        full |= (n[None, :] >= need).all(axis=1)
    return ~full.reshape(nb, nb, nb)
