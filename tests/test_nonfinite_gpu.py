"""Populations that are not finite (a solve that blew up, FP16 storage that
overflowed) give the moments and the wall nodes that the written-out formulas
give: operations that a kernel leaves out because they cannot change a finite
result must not hide an infinity or a NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _written_out(f, c, eq, rho0):
    rho = np.zeros(f.shape[1:])
    j = np.zeros((3,) + f.shape[1:])
    with np.errstate(all="ignore"):
        for i in range(f.shape[0]):
            rho += f[i]
            for a in range(3):
                j[a] += float(c[i, a]) * f[i]
        j /= rho0 if eq == "incomp" else rho
    return np.concatenate([rho[None], j])


@pytest.mark.parametrize("eq", ["incomp", "standard"])
@pytest.mark.parametrize("lattice,n", [("D2Q9", (9, 7)), ("D3Q19", (6, 5, 7))])
def test_macros_of_overflowed_populations(lattice, n, eq):
    from paper_1407_4524_gb300 import lbm
    c = np.zeros((9 if lattice == "D2Q9" else 19, 3), dtype=int)
    table = lbm.lbm_lattice_table(len(c))[0]
    c[:, :table.shape[1]] = table
    # a relaxation so slow that one population beyond FP16's range stays the only one
    dom = lbm.Domain(dict(lattice=lattice, n=n, tau=1e7, eq=eq, rho0=1.0, precision="fp16"), device=0)
    f = dom.populations()
    flat = f.reshape(f.shape[0], -1)
    for i, cell in ((1, 3), (4, 17), (f.shape[0] - 1, 29), (0, 40)):
        flat[i, cell] = 1e5
    dom.set_populations(f)
    got_f = dom.populations()
    bad = ~np.isfinite(got_f).reshape(len(c), -1)
    assert bad[:, [3, 17, 29, 40]].sum(0).tolist() == [1, 1, 1, 1] and bad.sum() == 4
    got = dom.macros()
    assert np.array_equal(got, _written_out(got_f, c, eq, 1.0), equal_nan=True)
    assert np.isposinf(got[1].ravel()[3]) == (eq == "incomp") and np.isnan(got[2].ravel()[3])


@pytest.mark.parametrize("edges", [{"y": ("wall", "wall")}, {"x": ("wall", "wall")}, {"x": ("wall", "outlet")}])
@pytest.mark.parametrize("lattice,n", [("D2Q9", (9, 7)), ("D3Q19", (6, 5, 7))])
def test_resting_wall_of_an_overflowed_node(lattice, n, edges):
    """Standard model: a wall link at rest adds 6 w_i rho (c_i . u_B) with u_B =
    0 and the node's own density, so a node whose density overflowed has no
    finite population after the step."""
    from paper_1407_4524_gb300 import lbm
    dom = lbm.Domain(dict(lattice=lattice, n=n, tau=1e7, eq="standard", precision="fp16", edges=edges), device=0)
    f = dom.populations()
    # a node of the y-low (x-low) wall row; its large population leaves along +x (+y)
    i, at, to, away = (1, 3, 4, 2) if "y" in edges else (2 if lattice == "D2Q9" else 3, n[0], 2 * n[0], 0)
    f.reshape(f.shape[0], -1)[i, at] = 1e5
    dom.set_populations(f)
    before = dom.populations().reshape(f.shape[0], -1)
    assert np.isposinf(before[i, at]) and np.isfinite(np.delete(before, i, 0)).all()
    dom.step(1)
    after = dom.populations().reshape(f.shape[0], -1)
    assert np.isnan(after[:, at]).all()
    assert not np.isfinite(after[:, to]).any() and np.isfinite(after[:, away]).all()
