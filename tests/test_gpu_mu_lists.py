"""css_solve_mu on Ritz lists around the length at which a list is cut into pieces (4096 values)."""
import numpy as np
import pytest

from tests.test_gpu_concurrency import _mu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(4096,), (4097, 0, 1), (8192, 5, 4095), (100_000, 3)])
def test_long_lists(sizes):
    import paper_2605_20918_gb300 as css
    rng = np.random.default_rng(sum(sizes))
    lists = [(rng.standard_normal(n) * 5.0, rng.random(n)) for n in sizes]
    lam, w = (np.concatenate([l[i] for l in lists]) for i in (0, 1))
    with css.Context(0) as ctx:
        mu = ctx.solve_mu(lists, kT=0.05, n_elec=float(w.sum()))
        assert mu == ctx.solve_mu(lists, kT=0.05, n_elec=float(w.sum()))
    assert abs(mu - _mu(lam, w, 0.05, float(w.sum()))) < 1e-9
