"""FP64 moments and relaxation, which leave out the operations that cannot
change the result (products with 0 and 1, what a pair of opposite directions
shares), against the oracle's written-out formulas: the same bits for both
equilibria, a reference density of 1 and another one, with and without a body
force, from random states -- and from states that hold an infinity, a NaN or
values whose squares overflow, where a left-out product would show."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BAD = {"random": None, "inf": np.inf, "minus_inf": -np.inf, "nan": np.nan, "huge": 1e200}


@pytest.mark.parametrize("state", sorted(BAD))
@pytest.mark.parametrize("force", [None, (1e-4, -2e-4, 3e-4)])
@pytest.mark.parametrize("eq,rho0", [("incomp", 1.0), ("incomp", 1.3), ("standard", 1.0)])
@pytest.mark.parametrize("lattice,n", [("D2Q9", (9, 7)), ("D3Q19", (6, 5, 7))])
def test_fp64_step_same_bits(oracle_mod, lattice, n, eq, rho0, force, state):
    from paper_1407_4524_gb300 import lbm
    spec = dict(lattice=lattice, n=n, tau=0.7, eq=eq, rho0=rho0, precision="fp64", u0=(0.02, -0.01))
    if force is not None:
        spec["force"] = force[:len(n)]
    ref = oracle_mod.Oracle(spec)
    f = ref.f() * (1.0 + 0.05 * np.random.default_rng(7).standard_normal(ref.f().shape))
    if BAD[state] is not None:
        flat = f.reshape(f.shape[0], -1)
        for i, cell in ((1, 3), (f.shape[0] - 1, 17), (0, 40)):
            flat[i, cell] = BAD[state]
    ref.set_f(f)
    dom = lbm.Domain(spec, device=0)
    dom.set_populations(f)
    assert np.array_equal(dom.populations(), ref.fhat(), equal_nan=True)
    dom.step(3)
    ref.step(3)
    assert np.array_equal(dom.populations(), ref.fhat(), equal_nan=True)
