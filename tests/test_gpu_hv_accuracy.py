"""Accuracy of the FP64 H*V where large terms cancel: weakly coupled molecules, whose on-site terms (tens
of eV) drop out of the first residual H Q_0 - Q_0 A_0 and leave couplings of 1e-3 eV and less."""
import numpy as np
import pytest

import oracle
from paper_2605_20918_gb300 import synth

pytestmark = pytest.mark.gpu


def weakly_coupled(n, b, coupling, seed):
    rng = np.random.default_rng(seed)
    val = np.empty((n, n, b, b))
    for i in range(n):
        u = np.linalg.qr(rng.standard_normal((b, b)))[0]
        val[i, i] = (u * rng.uniform(-30.0, 30.0, b)) @ u.T
        val[i, i] = 0.5 * (val[i, i] + val[i, i].T)
        for j in range(i):
            val[i, j] = coupling / np.sqrt(b) * rng.standard_normal((b, b))
            val[j, i] = val[i, j].T
    ptr = (np.arange(n + 1) * n).astype(np.int32)
    return synth.BSR(n, b, ptr, np.tile(np.arange(n, dtype=np.int32), n), np.ascontiguousarray(val.reshape(n * n, b, b)))


def bounds(H, B0):
    """Largest errors of A_1 and B_0.  An FP64 result is off by N rounding errors of |H| and of |B_0|; on top
    of that each entry of H Q_0 may be off by 2^-63 of its row's power of two (rounding of the entries of H;
    those of Q_0 are +-1), which B_0 takes as a Frobenius norm over the N b entries, Q_1 over the least singular
    value of B_0, and A_1 = Q_1^T H Q_1 twice."""
    N, norm = H.n_brow * H.b, 30.0 + 1.0
    entry = 2.0 ** -63 * 2.0 ** np.ceil(np.log2(np.abs(H.val).max()))
    F = np.sqrt(N * H.b) * entry
    eps = 2.0 ** -52
    return 2.0 * norm * F / np.linalg.svd(B0)[1].min() + N * eps * norm, F + N * eps * np.linalg.norm(B0)


@pytest.mark.parametrize("n,b,coupling", [(12, 6, 1e-3), (8, 13, 1e-3), (8, 16, 1e-4), (6, 23, 1e-3), (6, 24, 1e-4)])
def test_projected_blocks_of_weakly_coupled_molecules(n, b, coupling):
    torch = pytest.importorskip("torch")
    import paper_2605_20918_gb300 as css
    H = weakly_coupled(n, b, coupling, 7 * n + b)
    col = np.arange(n, dtype=np.int32)
    s = oracle.probes(col, b, 1005)
    Hd = css.DeviceBSR.from_host(H)
    P = torch.empty((H.nnzb, b, b), dtype=torch.float64, device="cuda")
    with css.Context(0) as ctx:
        ctx.density(Hd, torch.as_tensor(col, device="cuda"), torch.as_tensor(s, device="cuda"), n, P, mu=0.1, kT=0.5,
                    solve_mu=False, m=3, precision=css.CSS_FP64)
        A, B, _ = ctx.projected()
    for c in range(n):
        T = oracle.lanczos(H, col, s, c, 2)
        A1, B0 = T[b:, b:], T[b:, :b]
        tol_a, tol_b = bounds(H, B0)
        assert np.abs(np.asarray(A[c, 1]) - A1).max() < tol_a, c
        assert np.abs(np.asarray(B[c, 0]) - B0).max() < tol_b, c
