"""GPU tests of the ways out: waits that give up, devices smaller than a kernel wants,
state after a failed allocation."""
import numpy as np
import pytest

import oracle
import workloads
from workloads import DIRICHLET as D, PERIODIC as P, UNSCREENED as U, SCREENED as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kx():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2406_16998_gb300 import build
    build.build()
    import paper_2406_16998_gb300 as k
    return k


def rand(*shape, seed=1, cplx=False):
    g = np.random.default_rng(seed)
    x = g.standard_normal(shape)
    return torch.from_numpy(x + 1j * g.standard_normal(shape) if cplx else x).cuda()


@pytest.mark.parametrize("call", ["ace_apply", "kpoints"])
def test_bulk_copy_ring_given_up(kx, call, monkeypatch):
    """A kernel whose bulk copies run ahead of it gives up its first wait (KX_FAULT=wait): it
    waits for the copies in flight, reports the timeout and returns; the next call is right."""
    n = (24, 16, 24)
    plan = kx.Plan(n, (0.4, 0.45, 0.5), (P, P, P), S, precision=1)
    if call == "ace_apply":  # three steps of eight vectors per tile of points
        xi, phi = rand(20, plan.N), rand(70, plan.N, seed=2)
        run = lambda: (kx.kx_ace_apply(plan, xi, phi),)
    else:  # twelve vectors through a ring of two
        psi, theta, wk = rand(2, 12, plan.N, cplx=True), [[0.0, 0.0, 0.0], [1.0, 0.5, -0.7]], [0.5, 0.5]
        run = lambda: kx.kx_vx_kpoints(plan, theta, wk, psi)
    want = [t.clone() for t in run()]
    assert plan.status() == kx.KX_OK
    monkeypatch.setenv("KX_FAULT", "wait")
    run()
    assert plan.status() == kx.KX_ERR_TIMEOUT
    monkeypatch.delenv("KX_FAULT")
    got = run()
    assert plan.status() == kx.KX_OK
    for a, b in zip(got, want):
        assert torch.equal(a, b)
