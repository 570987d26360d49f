"""The map of the independent sums, as the kernels compile it (csrc/basis.cuh, here by the host compiler),
against the factors generated from beta: at every (n2, n3) the family, its column and the two row
factors that a component is read from are the component's centre factor and three multipoles."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include "basis.cuh"
#include <cstdio>
int main() {
  using namespace ext4pcf;
  for (int mu = 0; mu < 9; ++mu)
    for (int n2 = -5; n2 <= 5; ++n2)
      for (int n3 = -5; n3 <= 5; ++n3) {
        const BasisTerm t = basis_term(mu, n2, n3);
        printf("%d %d %d %d %d %d %d %d %d %d %d %d %d\n", mu, n2, n3, t.q, t.place, t.sg, t.k[0], t.k[1], t.k[2],
               (int)t.flip, t.q < 4 ? basis_col_index(t.q, t.sg) : 0, (int)(t.q < 4 && basis_col_conj(t.q)),
               t.q < 4 ? (int)basis_centre_conj(t.q) : 2);
      }
}
"""


@pytest.fixture(scope="module")
def terms(tmp_path_factory):
    d = tmp_path_factory.mktemp("basis")
    (d / "terms.cpp").write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    r = subprocess.run(["g++", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"), "-I",
                        os.path.join(ROOT, "paper_2509_07974_gb300", "csrc"), str(d / "terms.cpp"), "-o",
                        str(d / "terms")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(d / "terms")], capture_output=True, text=True).stdout
    return np.array([[int(v) for v in line.split()] for line in out.splitlines()])


def test_every_component_is_read_from_its_own_factors(terms):
    from paper_2509_07974_gb300 import build, ext4pcf
    build.build()
    assert len(terms) == 9 * 11 * 11
    for mu, n2, n3, q, place, sg, k0, k1, k2, flip, col, conj, centre in terms:
        table = ext4pcf.ext4pcf_nth_order_factors(4, mu if mu < 8 else -1)
        want = [(arr, cj, a2 * n2 + a3 * n3 + b) for arr, cj, a2, a3, b in table[2:].reshape(3, 5)]
        k = [k0, k1, k2]
        assert table[0] == 1 and table[1] == centre, (mu, n2, n3)
        if mu == 8:  # W_{-m} = W_m^*: a conjugated sum has every index of the other sign
            assert q == 4 and k0 >= 0, (n2, n3)
            assert want == [(1, 0, -m if flip else m) for m in k], (n2, n3)
            continue
        got = [(0, conj, col) if l == place else (0, 0, k[l]) for l in range(3)]
        assert got == want, (mu, n2, n3)
        rows = [k[l] for l in range(3) if l != place]
        assert sum(rows) == sg and not flip, (mu, n2, n3)
        if q < 2:  # any factor in the column's place: the same index from the other sums
            assert sum(k) == (-4 if q else -8), (mu, n2, n3)
