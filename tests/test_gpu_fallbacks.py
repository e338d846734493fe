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


@pytest.mark.parametrize("prec", [0, 1])
def test_pair_list_after_a_failed_allocation(kx, prec, monkeypatch):
    """The tables of a longer pair list cannot be allocated: the call reports it, and the plan
    still answers for the list it had."""
    plan = kx.Plan((16, 24, 16), (0.4, 0.45, 0.5), (D, P, D), U, precision=prec)
    psi = rand(40, plan.N)
    small = psi[:5].contiguous()
    want, ex = (t.clone() for t in kx.kx_vx_apply(plan, small))
    monkeypatch.setenv("KX_FAULT", "alloc")
    with pytest.raises(kx.KxError) as ei:
        kx.kx_vx_apply(plan, psi)
    assert ei.value.code == kx.KX_ERR_NOMEM
    monkeypatch.delenv("KX_FAULT")
    got, ex2 = kx.kx_vx_apply(plan, small)
    assert torch.equal(got, want) and torch.equal(ex2, ex)
    big = kx.kx_vx_apply(plan, psi)[0]
    fresh = kx.Plan((16, 24, 16), (0.4, 0.45, 0.5), (D, P, D), U, precision=prec)
    assert torch.equal(big, kx.kx_vx_apply(fresh, psi)[0])


@pytest.mark.parametrize("prec", [0, 1])
def test_pair_lists_in_turn_on_a_side_stream(kx, prec):
    """Calls with two orbital counts back to back on a stream that does not synchronise with
    the default one: each runs with its own pair list."""
    n = (48, 48, 48) if prec else (16, 16, 16)
    plan = kx.Plan(n, (0.4, 0.45, 0.5), (P, P, P), S, precision=prec)
    psi = rand(30, plan.N)
    sizes = (30, 7, 18, 3)
    want = [[t.clone() for t in kx.kx_vx_apply(plan, psi[:k].contiguous())] for k in sizes]
    parts = [psi[:k].contiguous() for k in sizes]
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        got = [[t.clone() for t in kx.kx_vx_apply(plan, p)] for _ in range(5) for p in parts]
    side.synchronize()
    assert plan.status() == kx.KX_OK
    for i, (vx, ex) in enumerate(got):
        assert torch.equal(vx, want[i % 4][0]) and torch.equal(ex, want[i % 4][1])
