"""Field reads that go through both halves of the staging buffer several times
(three and five chunks of 2^21 cells, the last one ragged): every value is that
of the populations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(2049, 2051), (2903, 2899)])
def test_macros_of_many_chunks(n):
    from paper_1407_4524_gb300 import lbm
    c, _, _ = lbm.lbm_lattice_table(9)
    dom = lbm.Domain(dict(lattice="D2Q9", n=n, tau=0.7, precision="fp16", u0=(0.03, -0.02)), device=0)
    rng = np.random.default_rng(5)
    dom.set_populations(dom.populations() * (1.0 + 0.05 * rng.standard_normal((9, 1, n[1], n[0]))))
    dom.step(1)
    f, got = dom.populations(), dom.macros()
    want = np.zeros_like(got)
    for i in range(9):
        want[0] += f[i]
        for a in range(2):
            if c[i, a]:
                want[1 + a] += c[i, a] * f[i]
    assert np.array_equal(got, want)
    assert np.array_equal(dom.macros(), got)  # and again, into other pages
    dom.close()
