"""The neighbour records (ext4pcf_multipoles) at the edges of the gather's power blocks: every
block size and count, bins from empty to crowded, centres at the field's edge and corners, against
the sums written out in numpy.

Bound: a power u^m carries the rounding of u (the coordinate difference, the inverse square root
and a product: three roundings a component) m times, and a sum of n weights rounds with its partial
sums: (2 m + 16) 2^-23 sum |weight| in FP32, the same with 2^-52 in FP64."""
import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def _reference(pos, x, w, centres, edges, nmax):
    """Per centre and bin: sums of the seven weights times u^m and their absolute sums."""
    e2, out = edges * edges, []
    m = np.arange(2 * nmax + 7)
    for c in centres:
        d = pos - pos[c]
        r2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]
        row = []
        for b in range(len(edges) - 1):
            s = (r2 >= e2[b]) & (r2 < e2[b + 1])
            u = np.exp(1j * np.outer(m, np.arctan2(d[s, 1], d[s, 0])))
            row.append((u, x[s], w[s]))
        out.append(row)
    return out


@pytest.mark.parametrize("prec", ["f16x3", "fp64"])
@pytest.mark.parametrize("nmax", [0, 1, 3, 4, 5, 9, 12, 13, 17, 20, 28, 29, 33, 36, 40])
def test_records_match_the_written_out_sums(torch_cuda, prec, nmax):  # noqa: F811
    from paper_2509_07974_gb300 import ext4pcf
    torch = torch_cuda
    rng = np.random.default_rng(nmax)
    n, edges = 700, np.array([0.2, 0.21, 0.9, 2.5, 6.0])  # the first bin is all but empty
    pos = rng.uniform(0, 20, (n, 2))
    pos[:4] = [[0, 0], [20, 20], [0, 20], [10, 10]]
    sh, w = rng.normal(0, 0.3, (n, 2)), rng.uniform(0.5, 1.5, n)
    centres = np.concatenate([np.arange(8), rng.choice(n, 12, replace=False)]).astype(np.int64)
    lay = ext4pcf.record_layout(4, nmax)
    dev = torch.device("cuda:0")
    t = [torch.tensor(a, device=dev) for a in (pos, sh, w)]
    rec = torch.zeros((len(centres), lay["rec"], 2), dtype=torch.float64, device=dev)
    est = ext4pcf.Estimator(0, prec)
    ext4pcf.ext4pcf_multipoles(est.ctx, *t, n, edges, 4, nmax, centres, len(centres), rec)
    got = torch.view_as_complex(rec).cpu().numpy()
    est.close()
    eps = 2.0 ** (-52 if prec == "fp64" else -23)
    x = w * (sh[:, 0] + 1j * sh[:, 1])
    power = lambda u, m: u[m] if m >= 0 else u[-m].conj()  # noqa: E731
    for i, row in enumerate(_reference(pos, x, w, centres, edges, nmax)):
        for b, (u, xs, ws) in enumerate(row):
            weight = {"G": xs, "W": ws, "XX": xs * xs, "XA": np.abs(xs) ** 2, "WW": ws * ws}
            for name, wt in weight.items():
                off, first, cnt = lay[name]
                for k in range(cnt):
                    m = first + k
                    err = abs(got[i, off + k * 4 + b] - (wt * power(u, m)).sum())
                    assert err <= (2 * abs(m) + 16) * eps * np.abs(wt).sum(), (name, m, b, i)
            tr = [xs ** 3 * power(u, 0) * np.conj(u[4]) ** 2, xs ** 3 * np.conj(u[4]), xs ** 2 * xs.conj() * np.conj(u[4]),
                  xs ** 2 * xs.conj(), ws ** 3 + 0j]
            for k, v in enumerate(tr):
                err = abs(got[i, lay["TR"][0] + k * 4 + b] - v.sum())
                assert err <= 40 * eps * np.abs(v).sum(), ("TR", k, b, i)
