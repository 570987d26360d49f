"""The neighbour records of dense catalogues (angular sectors), against the sums written out in numpy:
both orders of the sector moments, one bin and many, bins with and without sectors, more pairs in
the latter than are set aside at a time, all galaxies on one line (at the edge of two sectors), centres at the
field's edge and corners.

Bound: as for the power-by-power sums (2 m + 16) 2^-23 sum |weight| for the power m, and what the
rounding of the in-cell offsets (cells no wider than r_max) turns a pair at the bin's inner edge r:
m sqrt(2) (r_max / r) 2^-23."""
import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(pos, sh, w, edges, nmax, centres, got, lay):
    e2, x = edges * edges, w * (sh[:, 0] + 1j * sh[:, 1])
    weight = {"G": x, "W": w, "XX": x * x, "XA": np.abs(x) ** 2, "WW": w * w}
    for i, c in enumerate(centres):
        d = pos - pos[c]
        r2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]
        for b in range(len(edges) - 1):
            s = (r2 >= e2[b]) & (r2 < e2[b + 1])
            turn = 2 ** 0.5 * edges[-1] / edges[b]
            u = np.exp(1j * np.outer(np.arange(2 * nmax + 7), np.arctan2(d[s, 1], d[s, 0])))
            for name, wt in weight.items():
                off, first, cnt = lay[name]
                p = wt[s]
                up, dn = u @ p, u.conj() @ p
                for k in range(cnt):
                    m = first + k
                    ref = up[m] if m >= 0 else dn[-m]
                    lim = (2 * abs(m) + 16 + turn * abs(m)) * 2.0 ** -23 * np.abs(p).sum()
                    err = abs(got[i, off + k * (len(edges) - 1) + b] - ref)
                    assert err <= lim, (name, m, b, i, err / max(lim, 1e-300))
            u1, xs = np.exp(1j * np.arctan2(d[s, 1], d[s, 0])), x[s]
            tr = [xs ** 3 * u1.conj() ** 8, xs ** 3 * u1.conj() ** 4, xs ** 2 * xs.conj() * u1.conj() ** 4,
                  xs ** 2 * xs.conj(), w[s] ** 3 + 0j]
            for k, v in enumerate(tr):
                err = abs(got[i, lay["TR"][0] + k * (len(edges) - 1) + b] - v.sum())
                assert err <= (40 + 8 * turn) * 2.0 ** -23 * np.abs(v).sum(), ("TR", k, b, i)


@pytest.mark.parametrize("nmax,nb,n,side,shape", [
    (9, 3, 45000, 20.0, "box"), (12, 4, 20000, 12.0, "line"), (20, 1, 7000, 9.0, "box"), (20, 10, 15000, 20.0, "box"),
    (20, 8, 16000, 20.0, "clump"), (21, 7, 9300, 14.0, "box"), (30, 12, 14000, 14.0, "box"),
    (40, 5, 8000, 12.0, "clump")])
def test_dense_records_match_the_written_out_sums(torch_cuda, nmax, nb, n, side, shape):  # noqa: F811
    from paper_2509_07974_gb300 import ext4pcf
    torch = torch_cuda
    rng = np.random.default_rng(n + nmax)
    pos = rng.uniform(0, side, (n, 2))
    if shape == "line":  # every direction falls into two sectors, at their common edges' angle
        pos[:, 1] = pos[:, 0] * np.tan(np.pi * 5 / 64)
    elif shape == "clump":  # more pairs in the inner bins than are set aside
        pos[: n // 2] = side / 3 + rng.normal(0, 0.1, (n // 2, 2))
    pos[:4] = [[0, 0], [side, side], [0, side], [side / 2, side / 2]]
    sh, w = rng.normal(0, 0.3, (n, 2)), rng.uniform(0.5, 1.5, n)
    edges = np.geomspace(0.1, 0.7 * side, nb + 1)
    centres = np.concatenate([np.arange(4), rng.choice(n, 8, replace=False)]).astype(np.int64)
    lay = ext4pcf.record_layout(nb, nmax)
    dev = torch.device("cuda:0")
    t = [torch.tensor(a, device=dev) for a in (pos, sh, w)]
    rec = torch.zeros((len(centres), lay["rec"], 2), dtype=torch.float64, device=dev)
    est = ext4pcf.Estimator(0, "fp32")  # takes every number of bins
    ext4pcf.ext4pcf_multipoles(est.ctx, *t, n, edges, nb, nmax, centres, len(centres), rec)
    got = torch.view_as_complex(rec).cpu().numpy()
    est.close()
    _check(pos, sh, w, edges, nmax, centres, got, lay)
