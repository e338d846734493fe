"""GPU tests of the ways out: waits that give up, devices smaller than a kernel wants,
state after a failed allocation."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

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


@pytest.fixture(scope="module")
def hooks(kx, tmp_path_factory):
    """plan_hooks.cu, compiled against the library."""
    from paper_2406_16998_gb300 import build
    here = os.path.dirname(os.path.abspath(__file__))
    out = str(tmp_path_factory.mktemp("hooks") / "plan_hooks.so")
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", os.path.join(here, "plan_hooks.cu"),
           build.LIB, "-lcudart", "-o", out, "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(build.LIB)]
    subprocess.run(cmd, check=True, capture_output=True, text=True)
    return ctypes.CDLL(out)


def rand(*shape, seed=1, cplx=False):
    g = np.random.default_rng(seed)
    x = g.standard_normal(shape)
    return torch.from_numpy(x + 1j * g.standard_normal(shape) if cplx else x).cuda()


@pytest.mark.parametrize("call", ["ace_apply", "kpoints"])
def test_bulk_copy_ring_given_up(kx, hooks, call, monkeypatch):
    """A kernel whose bulk copies run ahead of it gives up its first wait (KX_FAULT=wait): it
    waits for the copies in flight, reports the timeout and returns; the next call is right."""
    n = (24, 16, 24)
    plan = kx.Plan(n, (0.4, 0.45, 0.5), (P, P, P), S, precision=1)
    hooks.hook_num_sms(plan.handle, 1)  # few SMs: the forms for many points per SM
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
def test_pair_list_without_host_memory(kx, prec, monkeypatch):
    """A host allocation that throws while a pair list is made becomes an error code at the C
    boundary; the list before it, and the plain one after a call with explicit blocks, hold."""
    plan = kx.Plan((16, 24, 16), (0.4, 0.45, 0.5), (D, P, D), U, precision=prec)
    psi = rand(12, plan.N)
    want, ex = (t.clone() for t in kx.kx_vx_apply(plan, psi))
    monkeypatch.setenv("KX_FAULT", "host")
    for call in (lambda: kx.kx_vx_apply(plan, psi[:7].contiguous()),
                 lambda: kx.kx_vx_apply_block_pairs(plan, psi, [(0, 1), (2, 2)])):
        with pytest.raises(kx.KxError) as ei:
            call()
        assert ei.value.code == kx.KX_ERR_NOMEM
    monkeypatch.delenv("KX_FAULT")
    got, ex2 = kx.kx_vx_apply(plan, psi)
    assert torch.equal(got, want) and torch.equal(ex2, ex)


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


# bands, third axis, boundaries and k-points of a plane of 64 x 64 points, where two
# products run per kernel
FUSED = [(3, 64, (P, P, D), U, 3, None), (4, 32, (P, D, P), U, 2, "5"), (3, 64, (P, P, P), S, 2, "7"),
         (1, 32, (D, P, P), S, 2, None)]


def fused_case(kx, n_orb, n3, bc, kind, nk):
    plan = kx.Plan((64, 64, n3), (0.3, 0.35, 0.4), bc, kind, precision=1)
    theta = np.random.default_rng(n3).uniform(-3, 3, (nk, 3))
    # bands of very different sizes: the splits' scales span many octaves
    psi = rand(nk, n_orb, plan.N, seed=n3, cplx=True) * torch.logspace(-4, 3, n_orb, device="cuda")[:, None]
    wk = [1.0 / nk] * nk

    def run():
        vx, ex = kx.kx_vx_kpoints(plan, theta, wk, psi)
        one = kx.kx_vx_apply_kpoint(plan, theta, wk, psi, nk - 1, psi[0].contiguous())
        e_only = kx.kx_energy_kpoints(plan, theta, wk, psi)
        launches = plan.profile_read()["bloch"][1]
        assert plan.status() == kx.KX_OK
        return [vx, one, ex, e_only], launches

    plan.profile(False)
    return plan, run


@pytest.mark.parametrize("n_orb,n3,bc,kind,nk,chunk", FUSED)
def test_fused_kpoint_products_bit_for_bit(kx, n_orb, n3, bc, kind, nk, chunk, monkeypatch):
    """The kernels with two products and the single products (KX_BLOCH_FUSED=0) give the same bits."""
    if chunk:
        monkeypatch.setenv("KX_CHUNK_PAIRS", chunk)
    plan, run = fused_case(kx, n_orb, n3, bc, kind, nk)
    two, n_two = run()
    monkeypatch.setenv("KX_BLOCH_FUSED", "0")
    one, n_one = run()
    assert n_one - n_two > n_two  # other kernels: twice as many launches and more
    for a, b in zip(two, one):
        assert torch.equal(a, b)


@pytest.mark.parametrize("sms", [16, 31, 4096])
@pytest.mark.parametrize("n_orb,n3,bc,kind,nk,chunk", FUSED[:3])
def test_fused_kpoint_products_on_another_share_of_the_device(kx, hooks, sms, n_orb, n3, bc, kind, nk, chunk,
                                                              monkeypatch):
    """With fewer SMs than an item has tiles (a CTA would wait for its own next tile), and with
    more CTAs than the device holds at once (the launch is refused), the calls take the
    single products and give the same bits; E_x differs by the grouping of its partial sums."""
    if chunk:
        monkeypatch.setenv("KX_CHUNK_PAIRS", chunk)
    plan, run = fused_case(kx, n_orb, n3, bc, kind, nk)
    want, _ = run()
    old = hooks.hook_num_sms(plan.handle, sms)
    try:
        got, _ = run()
    finally:
        hooks.hook_num_sms(plan.handle, old)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    for a, b in zip(got[2:], want[2:]):
        assert abs(a.item() - b.item()) < 1e-6 * abs(b.item())


# Three kinds of k-point products (two per kernel, single ones, CUDA cores with up to 200 KB
# of shared memory) and the widest sums, before and after a reset of the device: what was
# set for the kernels in the first context is gone in the second.
RESET = """
import ctypes, sys
import numpy as np
import paper_2406_16998_gb300 as kx
L = kx.lib()
rt = ctypes.CDLL("libcudart.so.13")  # the one the library is linked to
dp = ctypes.POINTER(ctypes.c_double)

def buf(a):
    p = ctypes.c_void_p()
    assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(a.nbytes)) == 0
    assert rt.cudaMemcpy(p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes), 1) == 0
    return p

def run(n, n_orb):
    plan = kx.Plan(n, (0.4, 0.45, 0.5), (1, 1, 1), 1, precision=1)
    psi = np.random.default_rng(n_orb).standard_normal((2, n_orb, plan.N, 2))
    theta, wk = np.array([[0.0, 0.0, 0.0], [1.0, 0.5, -0.7]]), np.array([0.5, 0.5])
    d_psi, d_vx = buf(psi), buf(np.zeros_like(psi))
    host = lambda a: a.ctypes.data_as(L.kx_vx_kpoints.argtypes[2])
    rc = L.kx_vx_kpoints(plan.handle, 2, host(theta), host(wk), n_orb, d_psi, None, d_vx, None, None)
    detail = ctypes.create_string_buffer(256)
    L.kx_last_error_detail(detail, 256)
    assert rc == 0, (n, rc, detail.value)
    out = np.empty_like(psi)
    assert rt.cudaMemcpy(out.ctypes.data_as(ctypes.c_void_p), d_vx, ctypes.c_size_t(out.nbytes), 2) == 0
    plan.close()
    assert np.isfinite(out).all() and np.abs(out).max() > 0
    return out.tobytes()

calls = [((64, 64, 32), 5), ((64, 32, 32), 2), ((48, 40, 56), 2), ((16, 16, 16), 20)]
first = [run(*c) for c in calls]
assert rt.cudaDeviceReset() == 0
assert [run(*c) for c in calls] == first
print("same")
"""


def test_kpoints_in_a_second_context(kx):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RESET], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stdout + r.stderr


@pytest.mark.parametrize("prec,big,small", [(2, (96, 96, 4), (8, 9, 5)), (1, (96, 96, 8), (16, 8, 8))])
def test_two_threads_with_kernels_of_different_size(kx, hooks, prec, big, small):
    """Two host threads, each with its own plan and stream, launch the same kernels with much and
    with little shared memory: neither takes the other's limit away."""
    plans = [kx.Plan(n, (0.5,) * 3, (P, P, P), S, precision=prec) for n in (big, small)]
    b = [rand(1, p.N) for p in plans]
    want = [kx.kx_apply_fL(p, x).clone() for p, x in zip(plans, b)]
    got = [torch.zeros_like(x) for x in b]
    torch.cuda.synchronize()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    assert hooks.hook_two_threads(plans[0].handle, ptr(b[0]), ptr(got[0]), plans[1].handle, ptr(b[1]), ptr(got[1]),
                                  5000) == 0
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("n,axis,n_rhs", [
    ((12, 9, 16), 0, 3), ((9, 13, 8), 1, 2), ((8, 16, 70), 2, 2),
    ((128, 32, 40), 0, 64), ((8, 128, 8), 1, 3), ((40, 32, 101), 2, 64),  # the widest forms, many and few pencils
])
@pytest.mark.parametrize("angle", [1e-7, 0.6])
def test_float64_eigenvectors_without_parity(kx, hooks, n, axis, n_rhs, angle):
    """Eigenvectors of a Dirichlet axis that are neither even nor odd, by a little or altogether,
    take the dense form, which drops nothing of them."""
    bc = [P, P, P]
    bc[axis] = D
    plan = kx.Plan(n, (0.4, 0.45, 0.5), bc, S, precision=0)
    assert hooks.hook_mix_eigenvectors(plan.handle, axis, 1, ctypes.c_double(angle)) == 0
    V = [torch.from_numpy(np.asarray(plan.eig(a)[1])).cuda() for a in range(3)]
    f = torch.from_numpy(np.asarray(plan.ftable()).reshape(n[2], n[1], n[0])).cuda()

    def solve(b):
        t = b.view(-1, n[2], n[1], n[0])
        t = torch.einsum("rzyx,zk,yj,xi->rkji", t, V[2], V[1], V[0]) * f
        return torch.einsum("rkji,zk,yj,xi->rzyx", t, V[2], V[1], V[0]).reshape(b.shape)

    b = rand(n_rhs, plan.N)
    ref, x = solve(b), kx.kx_apply_fL(plan, b)
    assert (x - ref).abs().max() < 1e-11 * ref.abs().max()
    psi = b[:2].contiguous()
    rho = torch.stack([psi[0] * psi[0], psi[0] * psi[1], psi[1] * psi[1]])
    phi = solve(rho)
    vx_ref = -torch.stack([psi[0] * phi[0] + psi[1] * phi[1], psi[0] * phi[1] + psi[1] * phi[2]])
    dV = 0.4 * 0.45 * 0.5
    ex_ref = -0.5 * dV * ((rho * phi).sum(1) * torch.tensor([1.0, 2.0, 1.0], device="cuda", dtype=torch.float64)).sum()
    vx, ex = kx.kx_vx_apply(plan, psi)
    assert (vx - vx_ref).abs().max() < 1e-11 * vx_ref.abs().max()
    for e in (ex.item(), kx.kx_energy(plan, psi).item()):
        assert abs(e - ex_ref.item()) < 1e-11 * abs(ex_ref.item())


@pytest.mark.parametrize("n,n_orb,n_vec,chunk", [
    ((16, 8, 8), 1, 9, None), ((16, 16, 8), 4, 6, "7"), ((8, 16, 16), 5, 8, "11"), ((16, 8, 16), 9, 3, "20"),
    ((16, 16, 16), 17, 5, "50"), ((16, 8, 16), 24, 2, None), ((12, 10, 9), 6, 7, "11"),
])
def test_kpoint_sums_of_few_and_of_many_points(kx, hooks, n, n_orb, n_vec, chunk, monkeypatch):
    """The one-pass sums (many points per SM) and the kernels that spread a chunk's vectors over
    the SMs (few) give the same bits, forward alone and both ways, over the band counts a
    thread holds and chunks that split a vector's bands."""
    if chunk:
        monkeypatch.setenv("KX_CHUNK_PAIRS", chunk)
    plan = kx.Plan(n, (0.4, 0.45, 0.5), (P, P, P), S, precision=1 if all(m % 8 == 0 for m in n) else 2)
    psi, phi = rand(3, n_orb, plan.N, cplx=True), rand(n_vec, plan.N, seed=2, cplx=True)
    occ = torch.linspace(0.2, 1.0, 3 * n_orb, dtype=torch.float64, device="cuda").view(3, n_orb)
    theta, wk = np.random.default_rng(n_orb).uniform(-3, 3, (3, 3)), [0.5, 0.3, 0.2]
    run = lambda: [kx.kx_vx_kpoints(plan, theta, wk, psi, occ)[0],
                   kx.kx_vx_apply_kpoint(plan, theta, wk, psi, 1, phi, occ)]
    few = run()  # the device's SMs: at most 36 blocks of points
    sms = hooks.hook_num_sms(plan.handle, 1)
    many = run()
    hooks.hook_num_sms(plan.handle, sms)
    assert plan.status() == kx.KX_OK
    for a, b in zip(few, many):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n,n_xi,n_vec", [
    ((16, 8, 8), 1, 1), ((24, 40, 16), 7, 33), ((24, 40, 16), 64, 64), ((32, 16, 40), 65, 130), ((16, 8, 8), 200, 3),
])
def test_combinations_of_few_and_of_many_points(kx, hooks, n, n_xi, n_vec):
    """The combination of grid vectors by bulk copies (many points per SM) and by 8-byte copies (few)
    against the products in float64: the projections are rounded alike, 2e-6 as elsewhere."""
    plan = kx.Plan(n, (0.4, 0.45, 0.5), (D, P, D), U, precision=1)
    xi, phi = rand(n_xi, plan.N) * 0.3, rand(n_vec, plan.N, seed=2)
    ref = -(0.4 * 0.45 * 0.5) * (phi @ xi.T) @ xi
    for sms in (1, None):
        old = hooks.hook_num_sms(plan.handle, sms) if sms else None
        out = kx.kx_ace_apply(plan, xi, phi)
        if sms:
            hooks.hook_num_sms(plan.handle, old)
        assert plan.status() == kx.KX_OK
        assert (out - ref).abs().max() < 2e-6 * ref.abs().max()


def test_fused_kpoint_products_refused_then_captured(kx, hooks):
    """A launch that is refused inside a capture would invalidate it: a plan that has met a
    refusal captures the single products, with the same bits."""
    plan = kx.Plan((64, 64, 64), (0.3, 0.35, 0.4), (P, P, D), U, precision=1)
    psi = rand(2, 4, plan.N, cplx=True)
    theta, wk = [[0.0, 0.0, 0.0], [0.5, 0.2, 0.1]], [0.5, 0.5]
    want = kx.kx_vx_kpoints(plan, theta, wk, psi)[0].clone()
    vx, ex = torch.empty_like(psi), torch.empty(1, dtype=torch.float64, device="cuda")
    old = hooks.hook_num_sms(plan.handle, 4096)
    try:
        kx.kx_vx_kpoints(plan, theta, wk, psi, out=vx, e_x=ex)  # refused; sizes the workspace
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            kx.kx_vx_kpoints(plan, theta, wk, psi, out=vx, e_x=ex)
    finally:
        hooks.hook_num_sms(plan.handle, old)
    vx.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert plan.status() == kx.KX_OK
    assert torch.equal(vx, want)
