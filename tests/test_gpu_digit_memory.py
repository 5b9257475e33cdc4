"""Memory of the digits of the FP64 H*V: the digits of V in turns, and a device with too little left for the
digits of H, at the block width whose digits are largest against its blocks (b = 1)."""
import numpy as np
import pytest

from paper_2605_20918_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.fixture(scope="module")
def css(torch):
    import paper_2605_20918_gb300 as m
    return m


def _ring(torch, css, n, reach, nc):
    """n sites of one orbital on a ring, coupled up to `reach` sites apart; colours in turn."""
    rng = np.random.default_rng(n)
    off = np.arange(-reach, reach + 1)
    col = (np.arange(n)[:, None] + off[None, :]) % n
    t = np.concatenate([[rng.uniform(-3.0, 3.0, n)], 0.5 * rng.standard_normal((reach, n)) / np.arange(1, reach + 1)[:, None]])
    i = np.arange(n)[:, None] + np.zeros_like(off)[None, :]
    val = t[np.abs(off)[None, :], np.where(off[None, :] >= 0, i, col)]
    order = np.argsort(col, axis=1)
    H = synth.BSR(n, 1, (np.arange(n + 1) * len(off)).astype(np.int32),
                  np.take_along_axis(col, order, 1).reshape(-1).astype(np.int32),
                  np.ascontiguousarray(np.take_along_axis(val, order, 1)).reshape(-1, 1, 1))
    colour = (np.arange(n) % nc).astype(np.int32)
    sign = np.where(rng.random(n) < 0.5, -1, 1).astype(np.int8)
    return css.DeviceBSR.from_host(H), torch.as_tensor(colour, device="cuda"), torch.as_tensor(sign, device="cuda"), nc


KW = dict(mu=0.2, kT=0.3, m=5)


def test_digits_of_v_in_turns(torch, css):
    """300 colours of 20,000 sites are 19 tiles of 82 MB, of which 13 fit the buffer: the second turn has six, the last
    with 12 of 16 columns.  The sums are exact, so the columns of P are those of calls that fit in one turn."""
    H, col, sign, nc = _ring(torch, css, 20_000, 14, 300)
    P = torch.empty_like(H.val)
    with css.Context(0) as ctx:
        ctx.density(H, col, sign, nc, P, flags=0, solve_mu=False, **KW)
        total = torch.zeros_like(P)
        for part in (range(0, 150), range(150, 300)):
            owned, Pr = np.zeros(nc, np.uint8), torch.empty_like(P)
            owned[list(part)] = 1
            ctx.density_colours(H, col, sign, nc, owned, Pr, **KW)
            total += Pr
    assert torch.equal(P, total)


def test_short_memory_takes_the_dfma_kernel(torch, css, monkeypatch):
    """580,000 blocks have 1.2 GB of digits and 0.3 GB of padded blocks: with 1 GB left the call runs as it did before
    there were digits, bitwise, and a repeated call allocates nothing."""
    H, col, sign, nc = _ring(torch, css, 20_000, 14, 30)
    P, ref, digits = (torch.empty_like(H.val) for _ in range(3))
    with css.Context(0) as ctx:
        ctx.density(H, col, sign, nc, digits, solve_mu=False, **KW)
    monkeypatch.setenv("CSS_SPMM_VARIANT", "0")
    with css.Context(0) as ctx:
        ctx.density(H, col, sign, nc, ref, solve_mu=False, **KW)
    monkeypatch.delenv("CSS_SPMM_VARIANT")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    with css.Context(0) as ctx:
        ballast = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")
        ctx.density(H, col, sign, nc, P, solve_mu=False, **KW)
        held = ctx.info()["workspace_bytes"]
        ctx.density(H, col, sign, nc, P, solve_mu=False, **KW)
        assert ctx.info()["workspace_bytes"] == held
        del ballast
    torch.cuda.empty_cache()
    assert torch.equal(P, ref)
    assert float((P - digits).abs().max()) < 1e-12 and not torch.equal(ref, digits)
