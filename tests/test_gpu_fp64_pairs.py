"""CSS_FP64_SPLIT in FP32 pairs (k_spmm_df): the kernel of systems whose digits of H exceed their bound or the
memory, selected here by a fixed launch variant (CSS_SPMM_VARIANT at css_create), which turns the digits off."""
import numpy as np
import pytest

import oracle
from paper_2605_20918_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return pytest.importorskip("torch")


@pytest.fixture
def ctx(monkeypatch):
    import paper_2605_20918_gb300 as css
    monkeypatch.setenv("CSS_SPMM_VARIANT", "0")
    c = css.Context(0)
    monkeypatch.delenv("CSS_SPMM_VARIANT")
    yield c
    c.close()


def _system(n, kind, r_col):
    g = synth.water_box(n)
    H = synth.hamiltonian(g, kind)
    col, nc = oracle.color(g.pos, g.box, r_col, 1004)
    return H, col, oracle.probes(col, H.b, 1005), nc


# both block widths, a second pass that regenerates the basis, one column tile and several
@pytest.mark.parametrize("n,kind,r_col,m,flags", [(64, "minimal", 8.0, 10, 1), (125, "minimal", 10.0, 12, 0),
                                                  (64, "minimal", 8.0, 10, 3), (27, "dzp", 6.0, 6, 1),
                                                  (64, "dzp", 8.0, 8, 3)])
def test_pairs_match_the_oracle(torch, ctx, n, kind, r_col, m, flags):
    import paper_2605_20918_gb300 as css
    from tests.test_gpu_parity import FP64_TOL, gpu_density
    H, col, s, nc = _system(n, kind, r_col)
    ne = synth.n_electrons(n)
    ref = oracle.density(H, col, s, nc, kT=0.05, n_elec=ne, solve_mu=True, m=m, flags=flags & ~2)
    got = gpu_density(torch, css, ctx, H, col, s, nc, kT=0.05, n_elec=ne, solve_mu=True, m=m, flags=flags,
                      precision=css.CSS_FP64_SPLIT)
    assert float(np.abs(got["P"] - ref["P"]).max()) < FP64_TOL
    assert abs(got["trP"] - ref["trP"]) < 1e-8


def test_batch_in_pairs_equals_single(torch, ctx):
    """The split copy of V is one per context, so a batch's passes run in turn."""
    import paper_2605_20918_gb300 as css
    from tests.test_gpu_parity import gpu_density
    systems = [_system(n, "minimal", 8.0) for n in (64, 27, 40)]
    ne = [synth.n_electrons(n) for n in (64, 27, 40)]
    one = [gpu_density(torch, css, ctx, *x, kT=0.05, n_elec=e, m=6, precision=css.CSS_FP64_SPLIT)["P"] for x, e in zip(systems, ne)]
    Hs = [css.DeviceBSR.from_host(H) for H, *_ in systems]
    Ps = [torch.empty_like(H.val) for H in Hs]
    ctx.density_batch(Hs, [torch.as_tensor(c, device="cuda") for _, c, _, _ in systems],
                      [torch.as_tensor(s, device="cuda") for _, _, s, _ in systems], [nc for *_, nc in systems], Ps,
                      [dict(kT=0.05, n_elec=e) for e in ne], m=6, precision=css.CSS_FP64_SPLIT)
    for a, P in zip(one, Ps):
        assert np.abs(a - P.cpu().numpy()).max() < 1e-12
