"""Edges of the GPU kernels' work splits: sizes at which a warp, tile or chunk is partly filled,
exactly filled or exceeded, each against the CPU oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return pytest.importorskip("torch")


@pytest.fixture(scope="module")
def css():
    import paper_2605_20918_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(css):
    c = css.Context(0)
    yield c
    c.close()


def _complete(n):
    adj = np.array([j for i in range(n) for j in range(n) if j != i], np.int32)
    return np.arange(n + 1, dtype=np.int32) * (n - 1), adj


def _ring(n):
    i = np.arange(n)
    adj = np.stack([(i - 1) % n, (i + 1) % n], axis=1).reshape(-1).astype(np.int32)
    return np.arange(n + 1, dtype=np.int32) * 2, adj


# complete graphs: as many colours as vertices, around the 256 colours of one search and the 32
# parents of one look; rings: one vertex per warp, several, and more than the 32 a warp watches at once
@pytest.mark.parametrize("graph,n", [(_complete, 33), (_complete, 256), (_complete, 300), (_ring, 20_001),
                                     (_ring, 400_000)])
def test_colour_graph_splits(torch, ctx, graph, n):
    ptr, adj = graph(n)
    col = torch.empty(n, dtype=torch.int32, device="cuda")
    nc = ctx.color_graph(torch.as_tensor(ptr, device="cuda"), torch.as_tensor(adj, device="cuda"), 1004, col)
    ref, nref = oracle.color_graph(ptr, adj, 1004)
    assert nc == nref and np.array_equal(col.cpu().numpy(), ref)


# 8, 16 or 32 lanes per sweep (b = 8 / 9, 16 / 17), the band in shared memory or in L2 (m), and in L2
# with four, two or one CTA per colour (38, 39 and 77 colours); tolerances of the eigen-stage tests
@pytest.mark.parametrize("b,m,n_col", [(2, 2, 3), (8, 23, 7), (8, 200, 2), (9, 20, 7), (16, 70, 3), (17, 12, 5),
                                       (32, 16, 38), (32, 16, 39), (32, 16, 77)])
def test_band_reduction_splits(torch, ctx, b, m, n_col):
    from tests.test_gpu_eigen import check, random_blocks
    rng = np.random.default_rng(1000 * b + m)
    A, B = random_blocks(rng, n_col, m, b)
    nblk = np.full(n_col, m)
    nblk[-1] = 1
    check(torch, ctx, A, B, nblk, rng.integers(1, 50, n_col), mu=0.3, kT=0.5)


# FP32 row passes: rows that leave part of a tile (n b mod 64), one, an odd number and more than one
# group of colours (b = 23: groups of four, whose columns start at four offsets within 16 bytes), and a Krylov space that is exhausted before depth m (nearly dependent blocks, then
# breakdown); fixed mid-gap mu, the mixed-precision tolerance of the parity tests
@pytest.mark.parametrize("kind,n,nc,m", [("minimal", 33, 1, 5), ("minimal", 33, 11, 5), ("minimal", 64, 21, 5),
                                         ("minimal", 75, 75, 4), ("minimal", 9, 9, 12), ("dzp", 9, 1, 5),
                                         ("dzp", 14, 5, 5), ("dzp", 20, 20, 4), ("dzp", 6, 6, 8)])
def test_fp32_row_pass_splits(torch, css, ctx, kind, n, nc, m):
    from paper_2605_20918_gb300 import synth
    from tests.test_gpu_parity import MIXED_P_TOL, gpu_density
    g = synth.water_box(n)
    H = synth.hamiltonian(g, kind)
    col = (np.arange(n) % nc).astype(np.int32)
    s = oracle.probes(col, H.b, 1005)
    kw = dict(kT=0.05, n_elec=synth.n_electrons(n), m=m, mu=-4.0, solve_mu=False)
    ref = oracle.density(H, col, s, nc, **kw)
    got = gpu_density(torch, css, ctx, H, col, s, nc, precision=css.CSS_MIXED_FP32, **kw)
    scale = max(1.0, float(np.abs(ref["P"]).max()))
    assert float(np.abs(got["P"] - ref["P"]).max()) < MIXED_P_TOL * scale


def _dense_bsr(n, b, scale, seed):
    """Symmetric matrix with every block present; row and column i scaled by scale[i]."""
    from paper_2605_20918_gb300 import synth
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((n * b, n * b)) / np.sqrt(n * b)
    A = (A + A.T) * np.sqrt(scale)[:, None] * np.sqrt(scale)[None, :]
    A[np.arange(n * b), np.arange(n * b)] += rng.uniform(-20.0, 20.0, n * b) * scale
    val = np.ascontiguousarray(A.reshape(n, b, n, b).transpose(0, 2, 1, 3)).reshape(n * n, b, b)
    ptr = (np.arange(n + 1) * n).astype(np.int32)
    return synth.BSR(n, b, ptr, np.tile(np.arange(n, dtype=np.int32), n), val)


# FP64 H*V from exact digit products: block widths at the edges of the 8-row and 16-column tiles and past
# the rule's last (b = 25), one to nine tiles of 16 columns (a partly filled last one, a second CTA), rows
# with fewer, as many and more blocks than one exact sum takes (146 / b), rows graded over eight decades.  A fixed mu; the
# tolerance of the FP64 parity tests
@pytest.mark.parametrize("n,b,nc,m,grade", [(1, 1, 1, 1, 0), (150, 1, 9, 6, 0), (37, 6, 24, 5, 0), (24, 6, 3, 5, 8),
                                            (19, 8, 2, 4, 0), (18, 9, 5, 4, 0), (9, 16, 9, 3, 8), (9, 17, 1, 4, 0),
                                            (13, 23, 4, 5, 0), (7, 24, 3, 3, 0), (7, 25, 3, 3, 0)])
def test_fp64_digit_products(torch, css, monkeypatch, n, b, nc, m, grade):
    from tests.test_gpu_parity import FP64_TOL, gpu_density
    scale = 10.0 ** np.linspace(0.0, -grade, n * b)
    H = _dense_bsr(n, b, scale, 100 * n + b)
    col = (np.arange(n) % nc).astype(np.int32)
    s = oracle.probes(col, b, 1005)
    kw = dict(kT=0.5, n_elec=float(n * b), m=m, mu=0.1, solve_mu=False)
    ref = oracle.density(H, col, s, nc, **kw)
    for variant in (None, "0"):  # the default and the general (DFMA) kernel
        if variant is not None:
            monkeypatch.setenv("CSS_SPMM_VARIANT", variant)
        c = css.Context(0)
        try:
            got = gpu_density(torch, css, c, H, col, s, nc, precision=css.CSS_FP64, **kw)
        finally:
            c.close()
        assert float(np.abs(got["P"] - ref["P"]).max()) < FP64_TOL, variant
        assert abs(got["trP"] - ref["trP"]) < 1e-8


# FP64 row passes: one row tile partly filled, exactly filled and exceeded, one colour and many, chunks of
# two tiles with a partly filled last chunk (450 molecules), and a Krylov space that is exhausted before
# depth m (third CholeskyQR pass, then breakdown); the tolerance of the FP64 parity tests
@pytest.mark.parametrize("kind,n,nc,m", [("minimal", 1, 1, 1), ("minimal", 16, 1, 5), ("minimal", 33, 11, 5),
                                         ("minimal", 450, 3, 4), ("minimal", 9, 9, 12), ("dzp", 9, 1, 5),
                                         ("dzp", 32, 5, 4), ("dzp", 20, 20, 4), ("dzp", 6, 6, 8)])
def test_fp64_row_pass_splits(torch, css, ctx, kind, n, nc, m):
    from paper_2605_20918_gb300 import synth
    from tests.test_gpu_parity import FP64_TOL, gpu_density
    g = synth.water_box(n)
    H = synth.hamiltonian(g, kind)
    col = (np.arange(n) % nc).astype(np.int32)
    s = oracle.probes(col, H.b, 1005)
    kw = dict(kT=0.05, n_elec=synth.n_electrons(n), m=m, mu=-4.0, solve_mu=False)
    ref = oracle.density(H, col, s, nc, **kw)
    got = gpu_density(torch, css, ctx, H, col, s, nc, precision=css.CSS_FP64, **kw)
    assert float(np.abs(got["P"] - ref["P"]).max()) < FP64_TOL


# FP32 H*V at b = 6, rows side by side: one column tile of few columns, half a tile (the last that packs rows
# into a warp), one colour more, full tiles with such tails, and rows that do not fill a CTA; every variant
# bitwise equal to the ring kernel
@pytest.mark.parametrize("n,nc", [(1, 1), (33, 1), (75, 10), (75, 11), (75, 22), (130, 32), (130, 33), (130, 64)])
def test_hv6_rows_equal_the_ring_kernel_bitwise(torch, css, monkeypatch, n, nc):
    from paper_2605_20918_gb300 import synth
    from tests.test_gpu_parity import gpu_density
    g = synth.water_box(n)
    H = synth.hamiltonian(g, "minimal")
    col = (np.arange(n) % nc).astype(np.int32)
    s = oracle.probes(col, H.b, 1005)
    P = []
    for v in "3012":
        monkeypatch.setenv("CSS_SPMM_DUP_VARIANT", v)
        c = css.Context(0)
        try:
            P.append(gpu_density(torch, css, c, H, col, s, nc, kT=0.05, n_elec=synth.n_electrons(n), m=min(n, 4), mu=-4.0,
                                 solve_mu=False, precision=css.CSS_MIXED_FP32)["P"])
        finally:
            c.close()
    for v in range(1, 4):
        assert np.array_equal(P[0], P[v]), v


# CholeskyQR's two ways to end a colour, a pivot that is not positive and a diagonal below the breakdown limit, at
# the block widths whose factor kernel has the most warps: Krylov spaces that are exhausted before depth m; the
# status and P of the oracle, and the same bits in repeated calls
@pytest.mark.parametrize("n,b,nc,m", [(3, 32, 3, 6), (4, 32, 2, 9), (5, 24, 5, 7), (4, 16, 1, 8)])
def test_breakdown_of_wide_blocks(torch, css, ctx, n, b, nc, m):
    from tests.test_gpu_parity import FP64_TOL, gpu_density
    H = _dense_bsr(n, b, np.ones(n * b), 10 * n + b)
    col = (np.arange(n) % nc).astype(np.int32)
    s = oracle.probes(col, b, 1005)
    kw = dict(kT=0.5, n_elec=float(n * b), m=m, mu=0.1, solve_mu=False)
    ref = oracle.density(H, col, s, nc, **kw)
    runs = [gpu_density(torch, css, ctx, H, col, s, nc, precision=css.CSS_FP64, **kw) for _ in range(8)]
    assert float(np.abs(runs[0]["P"] - ref["P"]).max()) < FP64_TOL
    assert (runs[0]["status"] == css.CSS_WARN_BREAKDOWN) == (ref["n_breakdown"] > 0)
    for r in runs[1:]:
        assert r["status"] == runs[0]["status"] and np.array_equal(r["P"], runs[0]["P"])


# Sums of the Gram partials at narrow blocks, where many threads could share an entry: as many partials as threads and
# fewer (1 to 40 chunks of rows).  P of the oracle, and a step at b = 1 takes no longer than one at b = 4 (1.21 times
# as long when idle threads' zeros were added too; the least of many calls)
@pytest.mark.parametrize("n", [3, 70, 300])
def test_gram_sums_of_narrow_blocks(torch, css, monkeypatch, n):
    from tests.test_gpu_parity import FP64_TOL, gpu_density
    monkeypatch.setenv("CSS_TIMING", "1")
    step = {}
    with css.Context(0) as c:
        for b in (1, 2, 4):
            H = _dense_bsr(n, b, np.ones(n * b), 10 * n + b)
            col = (np.arange(n) % 3).astype(np.int32)
            s = oracle.probes(col, b, 1005)
            kw = dict(kT=0.5, n_elec=float(n * b), m=1 if n == 3 else 6, mu=0.1, solve_mu=False)
            ref = oracle.density(H, col, s, 3, **kw)
            times = []
            for _ in range(30 if n == 70 else 1):
                got = gpu_density(torch, css, c, H, col, s, 3, precision=css.CSS_FP64, **kw)
                times.append(c.info()["ms_rows"])
            assert float(np.abs(got["P"] - ref["P"]).max()) < FP64_TOL
            step[b] = min(times)
    if n == 70:
        assert step[1] < 1.15 * step[4], step
