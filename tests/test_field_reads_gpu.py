"""Field reads of domains that take several staging chunks and a result array
whose pages are brought in by threads: the moments are those of the populations,
value for value, on both sides of the sizes where that begins."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# cells: below and above one chunk (2^21), an odd number above, 32 MB of results
SIZES = [(1 << 11, 1 << 10), ((1 << 11) + 1, (1 << 10) + 1), (1024, 1024), (1023, 1024)]


@pytest.mark.parametrize("prec", ["fp64", "fp16"])
@pytest.mark.parametrize("n", SIZES)
def test_macros_are_the_moments_of_the_populations(n, prec):
    from paper_1407_4524_gb300 import lbm
    c, _, _ = lbm.lbm_lattice_table(9)
    dom = lbm.Domain(dict(lattice="D2Q9", n=n, tau=0.7, precision=prec, u0=(0.03, -0.02)), device=0)
    rng = np.random.default_rng(3)
    dom.set_populations(dom.populations() * (1.0 + 0.05 * rng.standard_normal((9, 1, n[1], n[0]))))
    dom.step(2)
    f, got = dom.populations(), dom.macros()
    want = np.zeros_like(got)
    for i in range(9):
        want[0] += f[i]
        for a in range(2):
            if c[i, a]:
                want[1 + a] += c[i, a] * f[i]
    assert np.array_equal(got, want)
