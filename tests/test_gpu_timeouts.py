"""Bounded waits that run out return CSS_ERR_TIMEOUT and leave the device usable; the waits are held by test
hooks read at css_create, nothing faults."""
import numpy as np
import pytest

import oracle
from paper_2605_20918_gb300 import synth

pytestmark = pytest.mark.gpu


def _times_out_then_works(monkeypatch, hook, n, kind, m, precision):
    torch = pytest.importorskip("torch")
    import paper_2605_20918_gb300 as css
    g = synth.water_box(n)
    H = synth.hamiltonian(g, kind)
    col, nc = oracle.color(g.pos, g.box, 6.0, 1004)
    sign = oracle.probes(col, H.b, 1005)
    args = (css.DeviceBSR.from_host(H), torch.as_tensor(col, device="cuda"), torch.as_tensor(sign, device="cuda"), nc)
    P = torch.empty((H.nnzb, H.b, H.b), dtype=torch.float64, device="cuda")
    kw = dict(kT=0.05, mu=-4.0, solve_mu=False, m=m, precision=getattr(css, precision))
    monkeypatch.setenv(hook, "1")
    bad = css.Context(0)
    monkeypatch.delenv(hook)
    with bad, pytest.raises(css.CSSError) as e:
        bad.density(*args, P, **kw)
    assert e.value.status == css.CSS_ERR_TIMEOUT
    torch.cuda.synchronize()  # no sticky CUDA error
    with css.Context(0) as ctx:
        ctx.density(*args, P, **kw)
    ref = oracle.density(H, col, sign, nc, kT=0.05, mu=-4.0, solve_mu=False, m=m)
    assert float(np.abs(P.cpu().numpy() - ref["P"]).max()) < (1e-10 if precision == "CSS_FP64" else 1e-6)


# the sweeps of the band reduction: band in shared memory, and in L2 with several CTAs a colour
@pytest.mark.parametrize("n,kind,m", [(64, "minimal", 10), (40, "dzp", 26)])
def test_band_reduction_sweeps(monkeypatch, n, kind, m):
    _times_out_then_works(monkeypatch, "CSS_TEST_BAND_HOLD", n, kind, m, "CSS_FP64")


# the colouring, with a few vertices on many warps and with several per warp: vertex 0 is never coloured, so its own
# warp, its dependants' and theirs have to give up
@pytest.mark.parametrize("n", [40, 20_000])
def test_colouring(monkeypatch, n):
    torch = pytest.importorskip("torch")
    import paper_2605_20918_gb300 as css
    g = synth.water_box(n)
    xyz = torch.as_tensor(g.pos, device="cuda")
    col = torch.empty(n, dtype=torch.int32, device="cuda")
    monkeypatch.setenv("CSS_TEST_COLOUR_HOLD", "1")
    bad = css.Context(0)
    monkeypatch.delenv("CSS_TEST_COLOUR_HOLD")
    with bad, pytest.raises(css.CSSError) as e:
        bad.color(xyz, g.box, 6.0, 1004, col)
    assert e.value.status == css.CSS_ERR_TIMEOUT
    torch.cuda.synchronize()  # no sticky CUDA error
    with css.Context(0) as ctx:
        nc = ctx.color(xyz, g.box, 6.0, 1004, col)
    ref, nref = oracle.color(g.pos, g.box, 6.0, 1004)
    assert nc == nref and np.array_equal(col.cpu().numpy(), ref)


# the FP32 row passes' rings of tiles: one tile per chunk of rows (only the stores wait), and in one chunk more tiles
# than stages (loads and products wait too)
@pytest.mark.parametrize("n,kind,m", [(64, "minimal", 6), (40, "dzp", 4), (6000, "minimal", 2), (3000, "dzp", 2)])
def test_row_passes(monkeypatch, n, kind, m):
    if n < 1000:
        return _times_out_then_works(monkeypatch, "CSS_TEST_ROWS_HOLD", n, kind, m, "CSS_MIXED_FP32")
    torch = pytest.importorskip("torch")
    import paper_2605_20918_gb300 as css
    g = synth.water_box(n)
    H = css.DeviceBSR.from_host(synth.hamiltonian(g, kind))
    col = torch.arange(n, dtype=torch.int32, device="cuda") % 60
    sign = torch.ones(n * H.b, dtype=torch.int8, device="cuda")
    P = torch.empty_like(H.val)
    monkeypatch.setenv("CSS_TEST_ROWS_HOLD", "1")
    bad = css.Context(0)
    monkeypatch.delenv("CSS_TEST_ROWS_HOLD")
    with bad, pytest.raises(css.CSSError) as e:
        bad.density(H, col, sign, 60, P, mu=-4.0, solve_mu=False, m=m, precision=css.CSS_MIXED_FP32)
    assert e.value.status == css.CSS_ERR_TIMEOUT
    torch.cuda.synchronize()  # no sticky CUDA error
