"""The work that users of this library have it do, as cases to be timed: whole calls of the
public entry points (``Estimator`` and the functions of ``paper_2509_07974_gb300.ext4pcf``) over
the range of sizes, precisions and options they are used with.

Catalogues are Gaussian-random-field mocks (power-law spectrum, Kaiser-Squires shear, shape noise
0.26 per component, weights U[0.5, 1.5]) at the densities of the repository's workloads, 5 to 8
galaxies per arcmin^2, drawn on the GPU from the seed alone.

The mixed precisions compute in 32 bits or less and only collect their sums in 64-bit buffers, so
their results are handed on as 32-bit values, the way a program stores or plots them; the 64-bit
form's results stay 64-bit.

``exact`` restates every path in 64 bits with plain torch operations, from the paper's
definitions: dense distances, one power of e^{i phi} at a time, one matrix product per multipole
pair.
"""
import math

import numpy as np
import torch

from paper_2509_07974_gb300 import ext4pcf

DEV = "cuda:0"
DENSITY = 5.56  # galaxies per arcmin^2 where a case does not say otherwise


def listed():
    return [
        # the smallest calls: the 2000-galaxy parity workload, in the default precision of
        # Estimator and in the mixed precision of the large runs (launches and latency count)
        _measure("small_fp64", "fp64", 2000, 60.0, 1.0, 30.0, 8, 10, 0),
        _measure("small_f16x3", "f16x3", 2000, 60.0, 1.0, 30.0, 8, 10, 0),
        # a whole field at the main workload's density, bins and multipoles, every galaxy a
        # centre: what a measurement on one mock does
        _measure("field_f16x3", "f16x3", 200_000, 190.0, 0.5, 40.0, 10, 20, 0),
        # 64-bit reference run on a sample of centres, the check of a mixed run
        _measure("sample_fp64", "fp64", 100_003, 134.0, 0.5, 40.0, 10, 20, 1000),
        # ragged sizes in the other mixed precisions
        _measure("field_3xtf32", "3xtf32", 24_001, 65.0, 0.7, 21.0, 7, 13, 0),
        _measure("sample_fp32", "fp32", 60_000, 104.0, 0.5, 40.0, 9, 16, 1500),
        # uneven mocks in one call, a sample of centres in each (pinned host mask)
        _batch("mocks_f16x3", 6, 40_000, 400_000, 0.5, 60.0, 12, 20, 512, False),
        # overlapping patches of one survey into one output, high multipoles, the distant
        # bins from reduced catalogues (the tree approximation at the paper's setting)
        _batch("survey_tree_f16x3", 4, 500_000, 700_000, 0.5, 120.0, 12, 30, 256, True),
        # the neighbour multipoles alone, for a user's own contraction
        {"name": "multipoles_fp32", "kind": "multipoles", "precision": "f16x3", "n": 100_000, "side": 134.0,
         "lo": 0.6, "hi": 33.0, "nb": 7, "nmax": 15, "centres": 3001},
        # three-point multipoles of a field
        {"name": "third_order_field", "kind": "third", "precision": "f16x3", "n": 50_000, "side": 95.0,
         "lo": 0.5, "hi": 40.0, "nb": 10, "nmax": 20},
        # direct aperture statistics over the radii of the repository's comparison
        {"name": "direct_map", "kind": "direct", "precision": "f16x3", "n": 1_000_000, "side": 424.0,
         "t_lo": 1.0, "t_hi": 32.0, "n_theta": 12},
        # aperture measures of a measured 4PCF: 129 angular bins, 24 radii (the main workload's)
        {"name": "map4_aperture", "kind": "map4", "lo": 0.5, "hi": 40.0, "nb": 10, "nmax": 20, "nphi": 129,
         "n_ap": 24},
    ]


def _measure(name, precision, n, side, lo, hi, nb, nmax, centres):
    """centres: 0 every galaxy, else a device-resident mask with that many."""
    return {"name": name, "kind": "measure", "precision": precision, "n": n, "side": side, "lo": lo, "hi": hi,
            "nb": nb, "nmax": nmax, "centres": centres}


def _batch(name, n_cat, n_lo, n_hi, lo, hi, nb, nmax, centres, tree):
    return {"name": name, "kind": "batch", "precision": "f16x3", "n_cat": n_cat, "n_lo": n_lo, "n_hi": n_hi,
            "lo": lo, "hi": hi, "nb": nb, "nmax": nmax, "centres": centres, "tree": tree}


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["measure"] * 5 + ["batch"] * 2 + ["multipoles", "third", "direct", "map4", "real"])
    if kind in ("map4", "real"):
        nb, nmax, nphi = rng.randint(3, 10), rng.randint(4, 20), int(_log(rng, 16, 130))
        c = {"kind": kind, "lo": round(rng.uniform(0.5, 1.0), 3), "hi": round(rng.uniform(20.0, 40.0), 2), "nb": nb,
             "nmax": nmax, "nphi": nphi}
        if kind == "map4":
            c["n_ap"] = rng.randint(3, 24)
        else:  # the stored real-space arrays stay within about a gigabyte
            c["nphi"] = max(8, min(nphi, int(math.sqrt(8e6 / nb ** 3))))
        return c
    if kind == "direct":
        n = int(_log(rng, 3000, 1_000_000))
        side = math.sqrt(n / rng.uniform(5.0, 8.0))
        t_hi = min(32.0, side / 10.0)
        return {"kind": kind, "precision": "f16x3", "n": n, "side": round(side, 3), "t_lo": round(min(1.0, t_hi / 2), 3),
                "t_hi": round(t_hi, 3), "n_theta": rng.randint(2, 12)}
    nb, nmax = rng.randint(4, 12), rng.randint(5, 20)
    if kind == "batch":
        tree = rng.random() < 0.4
        n_hi = int(_log(rng, 20_000, 400_000))
        return _unnamed(_batch("", rng.randint(2, 9), max(2000, n_hi // rng.randint(2, 8)), n_hi,
                               round(rng.uniform(0.5, 0.8), 3), round(rng.uniform(30.0, 60.0), 2), nb, nmax,
                               int(_log(rng, 40, 700)), tree))
    n = int(_log(rng, 1500, 200_000))
    side = math.sqrt(n / rng.uniform(5.0, 8.0))
    lo, hi = round(rng.uniform(0.5, 1.0), 3), round(min(rng.uniform(15.0, 40.0), side / 2.0), 3)
    c = {"kind": kind, "precision": "f16x3", "n": n, "side": round(side, 3), "lo": lo, "hi": hi, "nb": nb, "nmax": nmax}
    if kind == "third":
        c["n"] = min(n, 50_000)
        c["side"] = round(math.sqrt(c["n"] / n) * side, 3)
        c["hi"] = round(min(hi, c["side"] / 2.0), 3)
        return c
    if kind == "multipoles":
        c["precision"] = rng.choice(["f16x3", "f16x3", "fp64"])
        c["centres"] = min(n, int(_log(rng, 100, 600 if c["precision"] == "fp64" else 6000)))
        return c
    c["precision"] = rng.choice(["f16x3", "f16x3", "f16x3", "fp64", "fp64", "3xtf32", "bf16x3", "tf32", "fp32"])
    # centres a pass of a few tenths of a second has room for: the 64-bit and plain 32-bit forms
    # run on the CUDA cores
    most = _cost_centres(c, {"fp64": 2.5e11, "fp32": 2e12}.get(c["precision"], 1e13))
    some = int(_log(rng, 50, max(60, most)))
    c["centres"] = 0 if n <= some else some
    return c


def _unnamed(c):
    return {k: v for k, v in c.items() if k != "name"}


def _pair_flops(c):
    return 100 * c["nmax"] + 160


def _contraction_flops(c):
    return 9 * (2 * c["nmax"] + 1) ** 2 * c["nb"] ** 3 * 8


def _pairs_per_centre(c):
    return c["n"] / c["side"] ** 2 * math.pi * (c["hi"] ** 2 - c["lo"] ** 2)


def _cost_centres(c, flops):
    return int(flops / (_contraction_flops(c) + _pairs_per_centre(c) * _pair_flops(c)))


# ---------------------------------------------------------------------------------- inputs
def _shear_field(grid, gen):
    """Kaiser-Squires shear of a convergence field with P(l) ~ l^-1.2, pixel rms 0.02."""
    white = torch.randn(grid, grid, generator=gen, device=DEV, dtype=torch.float64)
    k = torch.fft.fftfreq(grid, device=DEV, dtype=torch.float64)
    k1, k2 = torch.meshgrid(k, k, indexing="xy")
    ksq = k1 * k1 + k2 * k2
    ksq[0, 0] = 1.0
    amp = ksq ** -0.3
    amp[0, 0] = 0.0
    kap = torch.fft.fft2(white) * amp
    kap = kap * (0.02 / torch.fft.ifft2(kap).real.std())
    return torch.fft.ifft2(kap * torch.complex((k1 * k1 - k2 * k2) / ksq, 2 * k1 * k2 / ksq))


def _catalogue(n, side, gen, grid=512):
    g = _shear_field(grid, gen)
    pos = torch.rand(n, 2, generator=gen, device=DEV, dtype=torch.float64) * side
    i = (pos * (grid / side)).long().clamp_(0, grid - 1)
    shear = torch.view_as_real(g[i[:, 1], i[:, 0]]).contiguous()
    shear += 0.26 * torch.randn(n, 2, generator=gen, device=DEV, dtype=torch.float64)
    w = 0.5 + torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    return pos, shear, w


def _edges(c):
    return np.geomspace(c["lo"], c["hi"], c["nb"] + 1)


def _multipoles_of_a_field(c, gen):
    """An Upsilon as a measurement leaves it: N_n dominated by its n = 0 term (the neighbours'
    directions are nearly uniform), the components a decaying spectrum far below it."""
    nb, nn, e = c["nb"], 2 * c["nmax"] + 1, torch.as_tensor(_edges(c), device=DEV)
    area = math.pi * (e[1:] ** 2 - e[:-1] ** 2) * DENSITY
    count = 1e5 * area[:, None, None] * area[None, :, None] * area[None, None, :]
    noise = torch.randn(9, nn, nn, nb, nb, nb, 2, generator=gen, device=DEV, dtype=torch.float64)
    ups = torch.view_as_complex(noise)
    n = torch.arange(nn, device=DEV) - c["nmax"]
    damp = 1.0 / (1.0 + (n[:, None] + 2.0).abs() + (n[None, :] - 1.0).abs())
    ups[:8] *= 1e-4 * damp[None, :, :, None, None, None]
    ups[8] = (0.5 * 0.05 / nn) * (ups[8] + ups[8].flip(0, 1).conj())
    ups[8, c["nmax"], c["nmax"]] = 1.0
    ups *= count
    xi = torch.randn(nb, 3, 2, generator=gen, device=DEV, dtype=torch.float64) * 1e-4
    xi[:, 2, 0] = 1.0
    return torch.view_as_real(ups).contiguous(), (xi * area[:, None, None] * 1e5).contiguous()


def _lattice(c):
    """Aperture radii and their centres: a square lattice of spacing theta, 4 theta inside."""
    th = np.geomspace(c["t_lo"], c["t_hi"], c["n_theta"])
    return th, [ext4pcf.aperture_lattice((0.0, 0.0, c["side"], c["side"]), float(t), float(t)) for t in th]


class _Context:
    """A context with the tree approximation at the paper's setting, kept by the program."""

    def __init__(self, tree):
        cfg = ext4pcf.Config(device=0, stream=torch.cuda.current_stream().cuda_stream, deterministic=1,
                             precision=ext4pcf.PRECISION["f16x3"])
        if tree:
            cfg.tree_delta1, cfg.tree_levels, cfg.tree_rmin = 0.5, 3, 40.0
        self.ctx = ext4pcf.ext4pcf_create(cfg)

    def __del__(self):
        ext4pcf.ext4pcf_destroy(self.ctx)


def prepare(case, seed):
    c = case
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed * 7919 + 17)
    s = {"case": c, "edges": None}
    if c["kind"] in ("map4", "real"):
        s["ups"], s["xi"] = _multipoles_of_a_field(c, gen)
        s["est"] = ext4pcf.Estimator(0, "fp64")
        s["edges"] = _edges(c)
        if c["kind"] == "map4":
            s["radii"] = np.geomspace(1.0, 32.0, c["n_ap"])
        return s
    if c["kind"] == "direct":
        s["cat"] = _catalogue(c["n"], c["side"], gen)
        s["thetas"], cen = _lattice(c)
        s["centres"] = [torch.as_tensor(x, device=DEV) for x in cen]
        s["est"] = ext4pcf.Estimator(0, c["precision"])
        return s
    s["edges"] = _edges(c)
    if c["kind"] == "batch":
        k = np.arange(c["n_cat"])
        n = np.rint(c["n_lo"] + (c["n_hi"] - c["n_lo"]) * ((k * 0.618034) % 1.0)).astype(np.int64)
        parts, masks = [], []
        for nk in n.tolist():
            side = math.sqrt(nk / 7.0 if c["tree"] else nk / 6.5)
            pos, sh, w = _catalogue(nk, side, gen)
            # the centres: a sample of the patch's core (tree) or of the whole mock
            inner = (pos - 0.5 * side).abs().amax(1) < (0.25 * side if c["tree"] else side)
            pick = torch.nonzero(inner).flatten()
            pick = pick[torch.randperm(pick.numel(), generator=gen, device=DEV)[:c["centres"]]]
            m = torch.zeros(nk, dtype=torch.uint8, device=DEV)
            m[pick] = 1
            parts.append((pos, sh, w))
            masks.append(m)
        s["cat"] = tuple(torch.cat(x).contiguous() for x in zip(*parts))
        s["mask"] = torch.cat(masks).cpu().pin_memory()
        s["offsets"] = np.concatenate([[0], np.cumsum(n)])
        s["slots"] = np.zeros(c["n_cat"], dtype=np.int32) if c["tree"] else None
        s["n_out"] = 1 if c["tree"] else c["n_cat"]
        s["ctx"] = _Context(c["tree"])
        return s
    s["cat"] = _catalogue(c["n"], c["side"], gen)
    s["est"] = ext4pcf.Estimator(0, c["precision"])
    if c["kind"] == "measure":
        s["mask"] = None
        if c["centres"]:
            s["mask"] = torch.zeros(c["n"], dtype=torch.uint8, device=DEV)
            s["mask"][torch.randperm(c["n"], generator=gen, device=DEV)[:c["centres"]]] = 1
    if c["kind"] == "multipoles":
        pick = torch.randperm(c["n"], generator=gen, device=DEV)[:c["centres"]]
        s["centres"] = np.ascontiguousarray(pick.cpu().numpy().astype(np.int64))
    return s


# ------------------------------------------------------------------------------------- run
def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "map4":
        m4, eb, disc = s["est"].to_map4(s["ups"], s["edges"], c["nphi"], s["radii"], s["xi"])
        return {"m4": m4, "eb": eb, "disc": disc}
    if kind == "real":
        gamma, norm = s["est"].to_real_space(s["ups"], c["nphi"])
        return {"gamma": gamma, "norm": norm}
    pos, shear, w = s["cat"]
    if kind == "direct":
        moments, records = s["est"].map_direct(pos, shear, w, s["thetas"], s["centres"], want_records=True)
        return {"moments": moments.float(), "records": records.float()}
    keep = (lambda t: t) if c["precision"] == "fp64" else (lambda t: t.float())
    nb, nmax = c["nb"], c["nmax"]
    if kind == "measure":
        xi = torch.zeros(1, nb, 3, 2, dtype=torch.float64, device=DEV)
        ups = s["est"].measure(pos, shear, w, s["edges"], nmax, centre_mask=s["mask"], xi_acc=xi)
        return {"upsilon": keep(ups), "xi": keep(xi)}
    if kind == "batch":
        n_out = s["n_out"]
        ups = torch.zeros(ext4pcf.Estimator.ups_shape(nb, nmax, n_out), dtype=torch.float64, device=DEV)
        xi = torch.zeros(n_out, nb, 3, 2, dtype=torch.float64, device=DEV)
        ext4pcf.ext4pcf_measure_batch(s["ctx"].ctx, pos, shear, w, w.numel(), s["edges"], nb, nmax, s["offsets"],
                                      c["n_cat"], s["slots"], n_out, s["mask"], ups, xi)
        return {"upsilon": keep(ups), "xi": keep(xi)}
    if kind == "multipoles":
        rec = torch.zeros(c["centres"], ext4pcf.record_layout(nb, nmax)["rec"], 2, dtype=torch.float64, device=DEV)
        ext4pcf.ext4pcf_multipoles(s["est"].ctx, pos, shear, w, w.numel(), s["edges"], nb, nmax, s["centres"],
                                   c["centres"], rec)
        return {"records": keep(rec)}
    ups3 = torch.zeros(5, 2 * nmax + 1, nb, nb, 2, dtype=torch.float64, device=DEV)
    ext4pcf.ext4pcf_measure3(s["est"].ctx, pos, shear, w, w.numel(), s["edges"], nb, nmax, ups3)
    return {"upsilon3": keep(ups3)}


# ------------------------------------------------------------------------------------ work
def work(case):
    c = case
    kind = c["kind"]
    if kind in ("map4", "real"):
        # separable angular sums of nine components, and for the aperture measures the 28
        # polynomial coefficients of the eight components folded with every radius
        nn, tri, ph = 2 * c["nmax"] + 1, c["nb"] ** 3, c["nphi"]
        ups = 9 * nn * nn * tri * 16
        flops = tri * 9 * 2.0 * (nn * nn * ph + nn * ph * ph)  # the parities of both angles used
        if kind == "real":
            return {"bytes": ups + tri * ph * ph * 8 * 17, "flops": flops}
        return {"bytes": ups, "flops": flops + tri * ph * ph * 28 * 4.0 * c["n_ap"]}
    if kind == "direct":
        pairs, n_ap = 0.0, 0
        for t, cen in zip(*_lattice(c)):
            n_ap += len(cen)
            pairs += len(cen) * c["n"] / c["side"] ** 2 * math.pi * 16.0 * t * t
        return {"bytes": c["n"] * 40 + n_ap * 80, "flops": float(pairs * 30)}
    nn, nb = 2 * c["nmax"] + 1, c["nb"]
    rec = nb * (14 * c["nmax"] + 18)
    if kind == "batch":
        n_mean = 0.5 * (c["n_lo"] + c["n_hi"])
        n, cen = c["n_cat"] * n_mean, c["n_cat"] * c["centres"]
        rho = 7.0 if c["tree"] else 6.5
        side = math.sqrt(n_mean / rho)
        hi = min(c["hi"], side)
        per = rho * math.pi * hi * hi
        if c["tree"]:  # one reduced galaxy per cell of 1' in the outer bins
            per = rho * math.pi * min(hi, 20.0) ** 2 + math.pi * hi * hi
        out = (1 if c["tree"] else c["n_cat"]) * 9 * nn * nn * nb ** 3 * 16
    else:
        n, per = c["n"], _pairs_per_centre(c)
        cen = c.get("centres", 0) or n
        out = {"measure": 9 * nn * nn * nb ** 3 * 16, "multipoles": cen * rec * 16, "third": 5 * nn * nb * nb * 16}[kind]
    flops = cen * per * (100 * c["nmax"] + 160)
    if kind in ("measure", "batch"):  # a sixth of the ordered triples are independent
        flops += cen * 9 * nn * nn * nb ** 3 * 8 / 6
    if kind == "third":
        flops += cen * 5 * nn * nb * nb * 8 / 2
    return {"bytes": n * 40 + out, "flops": flops}


# ----------------------------------------------------------------------------------- exact
# factors of the components, (centre, A(Theta1; s), B(Theta2; n2), C(Theta3; n3)): the centre
# factor x, x^* or w; a factor (kind, sign, offset) is sum_j t_j u_j^(sign v + offset) with t the
# neighbours' x ("x"), x^* ("c") or w ("w"), u = e^{i phi}, v the index s = n2 + n3, n2 or n3
_FACTORS = [
    ("x", ("x", 1, -3), ("x", -1, -2), ("x", -1, -3)),
    ("c", ("x", 1, -1), ("x", -1, -2), ("x", -1, -1)),
    ("x", ("c", 1, 1), ("x", -1, -2), ("x", -1, -3)),
    ("x", ("x", 1, -3), ("c", -1, 2), ("x", -1, -3)),
    ("x", ("x", 1, -3), ("x", -1, -2), ("c", -1, 1)),
    ("c", ("c", 1, 3), ("x", -1, -2), ("x", -1, -1)),
    ("c", ("x", 1, -1), ("c", -1, 2), ("x", -1, -1)),
    ("c", ("x", 1, -1), ("x", -1, -2), ("c", -1, 3)),
    ("w", ("w", 1, 0), ("w", -1, 0), ("w", -1, 0)),
]
# the same for the 3PCF: (centre, F1(Theta1; n), F2(Theta2; n)), every component with a factor -1
_FACTORS3 = [
    ("x", ("x", 1, -3), ("x", -1, -3)),
    ("c", ("x", 1, -1), ("x", -1, -1)),
    ("x", ("c", 1, 1), ("x", -1, -3)),
    ("x", ("x", 1, -3), ("c", -1, 1)),
    ("w", ("w", 1, 0), ("w", -1, 0)),
]


def _sums(cen, pos, x, w, e2, nmax):
    """Per centre, bin and weight the sums of weight * u^m, m = 0 .. 2 nmax + 6: complex
    [C][nb][7][M], weights Re x, Im x, Re x^2, Im x^2, w, |x|^2, w^2; and u^0, u^4, u^8 sums of the
    triple weights [C][nb][5]."""
    C, n, nb, M = cen.shape[0], pos.shape[0], e2.numel() - 1, 2 * nmax + 7
    out = torch.zeros(C, nb, 7, M, dtype=torch.complex128, device=DEV)
    tri = torch.zeros(C, nb, 5, dtype=torch.complex128, device=DEV)
    step = max(1, min(C, int(4e7 // max(n, 1)), 512))
    for a in range(0, C, step):
        k = min(step, C - a)
        dx = pos[None, :, 0] - cen[a:a + k, None, 0]
        dy = pos[None, :, 1] - cen[a:a + k, None, 1]
        r2 = dx * dx + dy * dy
        ci, j = torch.nonzero((r2 >= e2[0]) & (r2 < e2[-1]), as_tuple=True)
        r2 = r2[ci, j]
        key = ci * nb + torch.bucketize(r2, e2, right=True) - 1
        key, order = torch.sort(key, stable=True)
        ci, j, r2 = ci[order], j[order], r2[order]
        u = torch.complex(dx[ci, j], dy[ci, j]) / torch.sqrt(r2)
        del dx, dy
        lengths = torch.bincount(key, minlength=k * nb)
        xj, wj = x[j], w[j]
        x2, xa = xj * xj, (xj * xj.conj()).real
        wt = torch.stack([xj.real, xj.imag, x2.real, x2.imag, wj, xa, wj * wj], 1)

        def total(v):
            flat = v.reshape(v.shape[0], -1)
            return torch.segment_reduce(flat, "sum", lengths=lengths, axis=0, unsafe=True)

        p = torch.ones_like(u)
        for m in range(M):
            out[a:a + k, :, :, m] = torch.view_as_complex(total(torch.view_as_real(wt * p[:, None])).reshape(k, nb, 7, 2))
            p = p * u
        u4 = u.conj() ** 4
        t5 = torch.stack([x2 * xj * u4 * u4, x2 * xj * u4, xa * xj * u4, xa * xj, (wj ** 3).to(u.dtype)], 1)
        tri[a:a + k] = torch.view_as_complex(total(torch.view_as_real(t5)).reshape(k, nb, 5, 2))
    return out, tri


class _Records:
    """The neighbour sums of a set of centres as functions of the power."""

    def __init__(self, sums, tri):
        self.s, self.tri = sums, tri

    def _pair(self, q, m):  # sum (weight q + i weight q+1) u^m
        a, b = self.s[:, :, q, abs(m)], self.s[:, :, q + 1, abs(m)]
        return a + 1j * b if m >= 0 else a.conj() + 1j * b.conj()

    def get(self, kind, m):
        """kind "x", "c" (x^*), "w", "xx" (x^2), "xa" (|x|^2), "ww": [C][nb]."""
        if kind == "x":
            return self._pair(0, m)
        if kind == "c":
            return self._pair(0, -m).conj()
        if kind == "xx":
            return self._pair(2, m)
        v = self.s[:, :, {"w": 4, "xa": 5, "ww": 6}[kind], abs(m)]
        return v if m >= 0 else v.conj()

    def factor(self, f, v):
        return self.get(f[0], f[1] * v + f[2])

    def same(self, f, vf, g, vg):
        """Sum over one neighbour of both factors' terms."""
        kind = {"xx": "xx", "xc": "xa", "cx": "xa", "ww": "ww"}[f[0] + g[0]]
        return self.get(kind, f[1] * vf + f[2] + g[1] * vg + g[2])


def _records(cen, pos, shear, w, edges, nmax):
    e2 = torch.as_tensor(edges * edges, device=DEV)
    return _Records(*_sums(cen, pos, w * torch.view_as_complex(shear), w, e2, nmax))


def _tree_records(cen, pos, shear, w, edges, nmax):
    """As _records, each bin from its level: the coarsest of the cells 0.5', 1', 2' with
    Theta_lo / side >= 40, else the galaxies."""
    x, nb = w * torch.view_as_complex(shear), len(edges) - 1
    level = [max([0] + [d for d in (1, 2, 3) if edges[b] / (0.5 * 2.0 ** (d - 1)) >= 40.0]) for b in range(nb)]
    s = torch.zeros(cen.shape[0], nb, 7, 2 * nmax + 7, dtype=torch.complex128, device=DEV)
    t = torch.zeros(cen.shape[0], nb, 5, dtype=torch.complex128, device=DEV)
    for d in sorted(set(level)):
        b = [k for k in range(nb) if level[k] == d]
        p, q, v = pos, x, w
        if d:
            cell = ((pos - pos.amin(0)) * (1.0 / (0.5 * 2.0 ** (d - 1)))).floor().long()
            _, inv = torch.unique(cell[:, 1] * 100_000 + cell[:, 0], return_inverse=True)
            m = int(inv.max()) + 1

            def add(val):
                return torch.zeros((m,) + val.shape[1:], dtype=val.dtype, device=DEV).index_add_(0, inv, val)

            v = add(w)
            p, q = add(pos * w[:, None]) / v[:, None], add(x)
        e = edges[b[0]:b[-1] + 2]
        s[:, b], t[:, b] = _sums(cen, p, q, v, torch.as_tensor(e * e, device=DEV), nmax)
    return _Records(s, t)


def _upsilon(R, x, w, nmax):
    """Corrected multipoles of the centres (x, w), [9][nn][nn][nb][nb][nb] complex."""
    nb, nn = R.s.shape[1], 2 * nmax + 1
    idx = range(-nmax, nmax + 1)
    eye = torch.eye(nb, dtype=torch.float64, device=DEV)
    d12, d13, d23 = eye[:, :, None], eye[:, None, :], eye[None, :, :]
    ups = torch.zeros(9, nn, nn, nb, nb, nb, dtype=torch.complex128, device=DEV)
    centre = {"x": x, "c": x.conj(), "w": w.to(x.dtype)}
    for mu, (t, A, B, C) in enumerate(_FACTORS):
        t = centre[t][:, None]
        Cn = torch.stack([R.factor(C, v) for v in idx])  # [nn][C][nb]
        As = {s: R.factor(A, s) for s in range(-2 * nmax, 2 * nmax + 1)}
        T12 = [(t * R.same(A, v, B, 0)).T @ R.factor(C, v) for v in idx]  # s + (-n2) = n3
        T13 = [(t * R.same(A, v, C, 0)).T @ R.factor(B, v) for v in idx]  # s + (-n3) = n2
        T23 = {s: (t * R.same(B, s, C, 0)).T @ As[s] for s in As}         # (-n2) + (-n3) = -s
        k = {"xxx": 0 if mu == 0 else 1, "www": 4}.get(A[0] + B[0] + C[0], 2 if mu < 5 else 3)
        T123 = (t * R.tri[:, :, k]).sum(0)
        for a, n2 in enumerate(idx):
            xb = t * R.factor(B, n2)
            kr = (xb[None, :, :, None] * Cn[:, :, None, :]).reshape(nn, -1, nb * nb)
            Aa = torch.stack([As[n2 + n3] for n3 in idx]).transpose(1, 2)
            ups[mu, a] = torch.bmm(Aa, kr).reshape(nn, nb, nb, nb)
            for b, n3 in enumerate(idx):
                ups[mu, a, b] -= (d12 * T12[b][:, None, :] + d13 * T13[a][:, :, None] +
                                  d23 * T23[n2 + n3].T[:, :, None])
            ups[mu, a] += 2.0 * d12 * d13 * T123[:, None, None]
    return ups


def _xi(R, x, w):
    return torch.stack([(x.conj()[:, None] * R.get("x", 0)).sum(0), (x[:, None] * R.get("x", -4)).sum(0),
                        (w[:, None] * R.get("w", 0)).sum(0)], 1)


def _exact_seconds(c, cen, n, per):
    return cen * n * 4e-11 + cen * per * (2 * c["nmax"] + 7) * 2.5e-10 + cen * _contraction_flops(c) / 4e11


def exact(case, seed):
    c = case
    kind = c["kind"]
    s = prepare(case, seed)
    if kind in ("map4", "real"):
        return _exact_transforms(c, s)
    pos, shear, w = s["cat"]
    if kind == "direct":
        return _exact_direct(c, s)
    x, nmax, edges = w * torch.view_as_complex(shear), c["nmax"], s["edges"]
    if kind == "batch":
        nb, nn = c["nb"], 2 * nmax + 1
        ups = torch.zeros(s["n_out"], 9, nn, nn, nb, nb, nb, dtype=torch.complex128, device=DEV)
        xi = torch.zeros(s["n_out"], nb, 3, dtype=torch.complex128, device=DEV)
        mask = s["mask"].to(DEV)
        for k in range(c["n_cat"]):
            a, b = int(s["offsets"][k]), int(s["offsets"][k + 1])
            i = a + torch.nonzero(mask[a:b]).flatten()
            R = (_tree_records if c["tree"] else _records)(pos[i], pos[a:b], shear[a:b], w[a:b], edges, nmax)
            o = 0 if c["tree"] else k
            ups[o] += _upsilon(R, x[i], w[i], nmax)
            xi[o] += _xi(R, x[i], w[i])
        return {"upsilon": torch.view_as_real(ups), "xi": torch.view_as_real(xi)}
    per = _pairs_per_centre(c)
    if kind == "measure":
        cen = c["centres"] or c["n"]
        if _exact_seconds(c, cen, c["n"], per) > 15.0:
            return None
        i = torch.nonzero(s["mask"]).flatten() if c["centres"] else torch.arange(c["n"], device=DEV)
        ups, xi = 0.0, 0.0
        for part in torch.split(i, 4096):
            R = _records(pos[part], pos, shear, w, edges, nmax)
            ups, xi = ups + _upsilon(R, x[part], w[part], nmax), xi + _xi(R, x[part], w[part])
        return {"upsilon": torch.view_as_real(ups)[None], "xi": torch.view_as_real(xi)[None]}
    if kind == "multipoles":
        i = torch.as_tensor(s["centres"], device=DEV)
        out = []
        for part in torch.split(i, 4096):
            R = _records(pos[part], pos, shear, w, edges, nmax)
            rows = [R.get("x", m) for m in range(-2 * nmax - 3, 2 * nmax)] + [R.get("w", m) for m in range(2 * nmax + 1)]
            rows += [R.get("xx", m) for m in range(-2 * nmax - 6, 2 * nmax - 1)]
            rows += [R.get("xa", m) for m in range(2 * nmax + 3)] + [R.get("ww", m) for m in range(2 * nmax + 1)]
            rows += [R.tri[:, :, k] for k in range(5)]
            out.append(torch.cat(rows, 1))
        return {"records": torch.view_as_real(torch.cat(out))}
    if c["n"] * per * (2 * nmax + 7) * 2.5e-10 + c["n"] ** 2 * 4e-11 > 15.0:
        return None
    ups3 = torch.zeros(5, 2 * nmax + 1, c["nb"], c["nb"], dtype=torch.complex128, device=DEV)
    for part in torch.split(torch.arange(c["n"], device=DEV), 4096):
        R = _records(pos[part], pos, shear, w, edges, nmax)
        centre = {"x": x[part], "c": x[part].conj(), "w": w[part].to(x.dtype)}
        for k, (t, F1, F2) in enumerate(_FACTORS3):
            t = centre[t][:, None]
            for a, n in enumerate(range(-nmax, nmax + 1)):
                v = (t * R.factor(F1, n)).T @ R.factor(F2, n)
                v -= torch.diag((t * R.same(F1, n, F2, n)).sum(0))
                ups3[k, a] += v if k == 4 else -v
    return {"upsilon3": torch.view_as_real(ups3)}


def _exact_direct(c, s):
    pos, shear, w = s["cat"]
    order = torch.argsort(pos[:, 1])
    pos, g, w = pos[order], shear[order], w[order]
    records, moments = [], []
    for th, cen in zip(s["thetas"].tolist(), s["centres"]):
        R2, rec = (4.0 * th) * (4.0 * th), torch.zeros(cen.shape[0], 8, dtype=torch.float64, device=DEV)
        done = 0
        if cen.shape[0]:
            ys, counts = torch.unique(cen[:, 1], return_counts=True)  # lattice rows, in order
            byrow = torch.argsort(cen[:, 1], stable=True)
            for y, m in zip(ys.tolist(), counts.tolist()):
                rows = byrow[done:done + m]
                done += m
                lim = torch.tensor([y - 4.0 * th - 1e-6, y + 4.0 * th + 1e-6], dtype=torch.float64, device=DEV)
                a, b = torch.searchsorted(pos[:, 1].contiguous(), lim).tolist()
                for part in torch.split(rows, max(1, int(3e7 // max(b - a, 1)))):
                    dx = pos[None, a:b, 0] - cen[part, None, 0]
                    dy = pos[None, a:b, 1] - cen[part, None, 1]
                    r2 = dx * dx + dy * dy
                    inside = (r2 < R2).to(torch.float64)
                    t = -(g[None, a:b, 0] * (dx * dx - dy * dy) + 2.0 * g[None, a:b, 1] * dx * dy)
                    q = inside * w[None, a:b]
                    v = q * t * torch.exp(r2 * (-0.5 / (th * th))) / (4.0 * math.pi * th ** 4)
                    for col, z in ((0, v), (3, q)):
                        z2 = z * z
                        p1, p2, p3, p4 = z.sum(1), z2.sum(1), (z2 * z).sum(1), (z2 * z2).sum(1)
                        e2 = 0.5 * (p1 * p1 - p2)
                        e3 = (e2 * p1 - p1 * p2 + p3) / 3.0
                        rec[part, col] = p1
                        rec[part, col + 1] = e2
                        rec[part, col + 2] = 0.25 * (e3 * p1 - e2 * p2 + p1 * p3 - p4)
                    rec[part, 6] = inside.sum(1)
        for col in (1, 4):
            rec[:, col] *= rec[:, 6] >= 2
            rec[:, col + 1] *= rec[:, 6] >= 4
        records.append(rec)
        m = [rec[:, k].sum().item() for k in (2, 5, 1, 4)]
        area = math.pi * R2
        m4 = area ** 4 * m[0] / m[1] if m[1] > 0 else 0.0
        m2 = area ** 2 * m[2] / m[3] if m[3] > 0 else 0.0
        moments.append(m + [float(cen.shape[0]), m4, m2, m4 - 3.0 * m2 * m2])
    return {"moments": torch.tensor(moments, dtype=torch.float64, device=DEV), "records": torch.cat(records)}


_CONJ = [(), (0,), (1,), (2,), (3,), (0, 1), (0, 2), (0, 3)]  # conjugated apertures per component
_LABELS = ["tttt", "xttt", "txtt", "ttxt", "tttx", "ttxx", "txtx", "txxt", "xttx", "xtxt", "xxtt", "txxx", "xtxx",
           "xxtx", "xxxt", "xxxx"]


def _eb(pattern):
    """E/B moments [n_ap][16] from the 16 conjugation patterns {(0/1, ...): [n_ap] complex}."""
    out = []
    for lab in _LABELS:
        v = 0.0
        for beta, val in pattern.items():
            f = 1.0
            for a in range(4):
                f = f * (0.5 if lab[a] == "t" else (0.5j if beta[a] else -0.5j))
            v = v + f * val
        out.append(v.real)
    return torch.stack(out, 1)


def _exact_transforms(c, s):
    nb, N, ph = c["nb"], c["nmax"], c["nphi"]
    nn, tri = 2 * N + 1, nb ** 3
    U = torch.view_as_complex(s["ups"]).reshape(9, nn, nn, tri).permute(3, 0, 1, 2)
    n = torch.arange(-N, N + 1, device=DEV, dtype=torch.float64)
    ang = torch.arange(ph + 1, device=DEV, dtype=torch.float64) * (2.0 * math.pi / ph)
    turn = torch.exp(1j * n[:, None] * ang[None, :])
    E = (turn[:, 1:] - turn[:, :-1]) / (1j * n[:, None] + (n[:, None] == 0)) / (2.0 * math.pi)
    E[N] = 1.0 / ph
    dphi = 2.0 * math.pi / ph
    mid = (torch.arange(ph, device=DEV, dtype=torch.float64) + 0.5) * dphi
    turn1 = torch.exp(1j * mid)
    real = c["kind"] == "real"
    gam = torch.zeros(8, tri, ph, ph, dtype=torch.complex128, device=DEV) if real else None
    norm = torch.zeros(tri, ph, ph, dtype=torch.float64, device=DEV) if real else None
    if not real:
        e = torch.as_tensor(s["edges"], device=DEV)
        lo, hi = e[:-1], e[1:]
        tb = 2.0 / 3.0 * (hi ** 3 - lo ** 3) / (hi ** 2 - lo ** 2)
        area = 0.5 * (hi ** 2 - lo ** 2)
        th = torch.as_tensor(s["radii"], device=DEV)
        h = 0.5 * th ** 2
        m4 = torch.zeros(th.numel(), 8, dtype=torch.complex128, device=DEV)
    for a in range(0, tri, 40):
        b = min(tri, a + 40)
        D = E.T @ (U[a:b] @ E)
        nv = D[:, 8].real
        G = torch.where((nv != 0.0)[:, None], D[:, :8] / nv[:, None], torch.zeros((), dtype=D.dtype, device=DEV))
        if real:
            gam[:, a:b], norm[a:b] = G.transpose(0, 1), nv
            continue
        k = torch.arange(a, b, device=DEV)
        k1, k2, k3 = k // (nb * nb), (k // nb) % nb, k % nb
        one = torch.ones(ph, dtype=torch.complex128, device=DEV)
        v1 = tb[k1][:, None, None] * one[None, :, None] * one[None, None, :]
        v2 = tb[k2][:, None, None] * turn1[None, :, None] * one[None, None, :]
        v3 = tb[k3][:, None, None] * one[None, :, None] * turn1[None, None, :]
        mean = 0.25 * (v1 + v2 + v3)
        d = [-mean, v1 - mean, v2 - mean, v3 - mean]
        sd2 = sum((q * q.conj()).real for q in d).reshape(b - a, -1)
        ex = torch.exp(-sd2[:, :, None] / (2.0 * th * th))
        vol = (2.0 * math.pi * dphi * dphi * area[k1] * area[k2] * area[k3])[:, None, None]
        for mu, cj in enumerate(_CONJ):
            P, Q = [torch.ones_like(mean)], [torch.ones_like(mean)]
            phase = torch.ones_like(mean)
            for q, z in enumerate((None, one[:, None], turn1[:, None], turn1[None, :])):
                poly, root = (Q, d[q]) if q in cj else (P, d[q].conj())
                for _ in range(2):
                    lift = [torch.zeros_like(mean)] + poly
                    poly[:] = [root * low + up for low, up in zip(poly + [torch.zeros_like(mean)], lift)]
                z2 = turn1[None, :] if q == 0 else z * z  # e^{2 i zeta}, zeta_0 = phi_13 / 2
                phase = phase * (z2.conj() if q in cj else z2)
            base = G[:, mu] * phase * vol
            for t in range(min(len(P), len(Q))):
                m = (base * P[t] * Q[t]).reshape(b - a, 1, -1)
                part = torch.complex(torch.bmm(m.real, ex), torch.bmm(m.imag, ex))[:, 0].sum(0)
                m4[:, mu] += part * math.pi * math.factorial(t) * h ** (t + 1)
    if real:
        full = torch.view_as_real(gam).reshape(8, nb, nb, nb, ph, ph, 2)
        return {"gamma": full, "norm": norm.reshape(nb, nb, nb, ph, ph)}
    m4 = m4 / ((4.0 * math.pi * th ** 4) ** 4)[:, None]
    pat = {}
    for mu, cj in enumerate(_CONJ):
        beta = tuple(int(q in cj) for q in range(4))
        pat[beta], pat[tuple(1 - v for v in beta)] = m4[:, mu], m4[:, mu].conj()
    xi = torch.view_as_complex(s["xi"])
    xq = (tb[:, None] / th[None, :]) ** 2
    g = torch.exp(-0.25 * xq) * area[:, None] / th ** 2 / 128.0
    den = xi[:, 2].real
    plus = ((xi[:, 0].real / den)[:, None] * (xq * xq - 16.0 * xq + 32.0) * g).sum(0).to(torch.complex128)
    minus = ((xi[:, 1] / den)[:, None] * xq * xq * g).sum(0)
    wick = {}
    for code in range(16):
        be = tuple((code >> (3 - a)) & 1 for a in range(4))

        def two(p, q):
            return plus if be[p] != be[q] else (minus.conj() if be[p] else minus)

        wick[be] = two(0, 1) * two(2, 3) + two(0, 2) * two(1, 3) + two(0, 3) * two(1, 2)
    return {"m4": m4.cpu().numpy(), "eb": _eb(pat).cpu().numpy(), "disc": _eb(wick).cpu().numpy()}
