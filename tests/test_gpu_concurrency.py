"""Results that must not depend on what else runs: the chemical potentials of many systems while another
stream keeps the GPU busy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.fixture(scope="module")
def css():
    import paper_2605_20918_gb300 as m
    return m


def _mu(lam, w, kT, n_elec):
    """Midpoint of {mu : |N(mu) - n_elec/2| <= 1e-4 max(1, n_elec/2)}, each end by bisection."""
    half = 0.5 * n_elec
    ends = []
    for tol in (-1e-4 * max(1.0, half), 1e-4 * max(1.0, half)):
        lo, hi = lam.min() - 1.0, lam.max() + 1.0
        for _ in range(100):
            mid = 0.5 * (lo + hi)
            if (0.5 * (1.0 - np.tanh((lam - mid) / (2.0 * kT))) * w).sum() - half - tol < 0.0:
                lo = mid
            else:
                hi = mid
        ends.append(0.5 * (lo + hi))
    return 0.5 * sum(ends)


# The search for mu runs all systems in one cooperative launch whose CTAs and warps have to leave it in the
# same round.  More systems than threads, spectra and temperatures over four decades so that they end in
# different rounds; the brackets are 1e-13 wide, the tolerance is that of the batch tests
def test_mu_of_many_systems_beside_a_busy_stream(torch, css):
    from paper_2605_20918_gb300 import synth
    rng = np.random.default_rng(3)
    n_sys = 300
    ptr, idx = np.array([0, 2, 4], np.int32), np.array([0, 1, 0, 1], np.int32)
    Hs, fermis = [], []
    for s in range(n_sys):
        A = rng.standard_normal((4, 4)) * 10.0 ** (4.0 * s / n_sys - 2.0)
        A = (A + A.T).reshape(2, 2, 2, 2).transpose(0, 2, 1, 3).reshape(4, 2, 2)
        Hs.append(css.DeviceBSR.from_host(synth.BSR(2, 2, ptr, idx, np.ascontiguousarray(A))))
        fermis.append({"kT": 10.0 ** rng.uniform(-3.0, 1.0), "n_elec": float(rng.uniform(1.0, 7.0)), "solve_mu": True})
    colour = torch.tensor([0, 1], dtype=torch.int32, device="cuda")
    sign = torch.ones(4, dtype=torch.int8, device="cuda")
    P = [torch.empty((4, 2, 2), dtype=torch.float64, device="cuda") for _ in range(n_sys)]
    busy, x = torch.cuda.Stream(), torch.ones(1 << 22, device="cuda")
    torch.cuda.synchronize()
    first = None
    with css.Context(0) as ctx:
        for rep in range(16):
            if rep % 2:
                with torch.cuda.stream(busy):
                    for _ in range(300):
                        x.mul_(1.0)
            mu = np.asarray(ctx.density_batch(Hs, [colour] * n_sys, [sign] * n_sys, [2] * n_sys, P, fermis, m=2)["mu"])
            if first is None:
                first = mu
                lists = ctx.ritz()
                for s, f in enumerate(fermis):
                    lam, w = (np.concatenate([np.asarray(l[i]) for l in lists[2 * s:2 * s + 2]]) for i in (0, 1))
                    assert abs(mu[s] - _mu(lam, w, f["kT"], f["n_elec"])) < 1e-9 * max(1.0, abs(mu[s])), s
            assert np.array_equal(mu, first), rep
    torch.cuda.synchronize()


# Two threads with a context each, systems of different sizes: a kernel's limit of dynamic shared memory belongs to
# the process, so one thread's small launch must not lower it under the other's large one.  Repeated calls
# are bitwise equal
@pytest.mark.parametrize("precision", ["CSS_FP64", "CSS_MIXED_FP32"])
def test_two_threads_with_systems_of_different_sizes(torch, css, precision):
    import threading
    from paper_2605_20918_gb300 import synth
    import oracle
    jobs = []
    for n, r_col, m in ((64, 8.0, 30), (8, 4.0, 4)):
        g = synth.water_box(n)
        H = synth.hamiltonian(g, "minimal")
        col, nc = oracle.color(g.pos, g.box, r_col, 1004)
        jobs.append((css.DeviceBSR.from_host(H), torch.as_tensor(col, device="cuda"),
                     torch.as_tensor(oracle.probes(col, H.b, 1005), device="cuda"), nc, synth.n_electrons(n), m))
    torch.cuda.synchronize()
    failed = []

    def work(Hd, col, sign, nc, ne, m):
        try:
            stream = torch.cuda.Stream()
            P = torch.empty_like(Hd.val)
            first = None
            with torch.cuda.stream(stream), css.Context(0) as ctx:
                for _ in range(150):
                    ctx.density(Hd, col, sign, nc, P, kT=0.05, n_elec=ne, m=m, precision=getattr(css, precision))
                    stream.synchronize()
                    first = P.clone() if first is None else first
                    if not torch.equal(P, first):
                        raise AssertionError("results differ between repeats")
        except Exception as e:
            failed.append(repr(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
