"""Edges of the two-float window of the J/K build: exponents on both sides of
the limits that keep the seeds pref (-2 alpha)^m F_m of a class pair inside the
FP32 exponent range, density elements far below the largest one, and handles
in and out of the range in one batch.

Tolerance of a default FP64 build: a primitive quartet in the window is below
line = 2^-13 max(G_ab)^2 max|D| and held to 2^-40 of itself (2^-44 with four bits
for the cancellation in the recursion), at most n^2 of them add up in an
element; everything else is FP64 and held to 2^-44 of the largest element."""
import numpy as np
import pytest

import molgen
import oracle

pytestmark = pytest.mark.gpu

TOL_MIXED = 1e-7


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required")
    import paper_2407_21445_gb300 as fk
    return torch, fk


def _build(env, bas, D, tau, **kw):
    torch, fk = env
    b = fk.JKBuilder(bas, tau, fk.make_opts(**kw))
    J, K = b.build(torch.tensor(D, device="cuda"))
    torch.cuda.synchronize()
    assert fk.fock_stream_status() == 0
    b.close()
    return J.cpu().numpy(), K.cpu().numpy()


def _tolerance(bas, D, Jo, Ko):
    gmax = float(np.max(oracle.schwarz(bas)[0]))
    line = 2.0 ** -13 * gmax ** 2 * np.abs(D).max()
    return len(D) ** 2 * line * 2.0 ** -40 + 2.0 ** -44 * max(np.abs(Jo).max(), np.abs(Ko).max())


def _one_exponent(ls, a, small, spread=1.0):
    """An s shell of exponent 1 with D = 1 and shells `ls` of exponent `a` within
    `spread` of their radius with D = `small` times random numbers: their quartets
    among themselves lie in the two-float window."""
    rng = np.random.Generator(np.random.PCG64(720))
    shells = [(0, np.zeros(3), [1.0], [1.0])]
    shells += [(l, spread / np.sqrt(a) * rng.uniform(-1, 1, 3), [a], [1.0]) for l in ls]
    bas = molgen.single_shell_basis(shells)
    n = oracle.nbf(bas)
    D = small * rng.uniform(-1, 1, (n, n))
    D = 0.5 * (D + D.T)
    D[0, 0] = 1.0
    return bas, D


# With one exponent a on every shell the limits 2^120 and 2^-100 of the seeds lie
# at 690 and 1.7e-3 for (ff|ff), at 3200 and 5e-4 for (fd|fd); (dd|dd) ends at
# 1e4 by the limit of the exponents themselves.
RANGE = [([3, 3], a) for a in (2e-4, 1.5e-3, 3e-3, 600.0, 900.0, 2000.0, 5000.0)]
RANGE += [([3, 2], a) for a in (4e-4, 1e-3, 1500.0, 2500.0, 9000.0)]
RANGE += [([2, 2], a) for a in (2e-4, 9e3, 1.1e4)]


@pytest.mark.parametrize("spread", [0.0, 1.0])
@pytest.mark.parametrize("ls,a", RANGE)
def test_exponents_at_the_edges(env, ls, a, spread):
    bas, D = _one_exponent(ls, a, 1e-4, spread)
    Jo, Ko = oracle.jk(bas, D, 1e-10)
    J, K = _build(env, bas, D, 1e-10)
    tol = _tolerance(bas, D, Jo, Ko)
    assert np.abs(J - Jo).max() <= tol and np.abs(K - Ko).max() <= tol


@pytest.mark.parametrize("group", [0, 8])
@pytest.mark.parametrize("exps", [(1e-3, 1e3), (2e-3, 3.0), (1.0, 5e3)])
def test_exponents_of_several_sizes(env, exps, group):
    """Contracted f, d and p shells that hold tight and diffuse primitives."""
    rng = np.random.Generator(np.random.PCG64(721))
    shells = [(0, np.zeros(3), [1.0], [1.0])]
    shells += [(l, 0.3 * rng.uniform(-1, 1, 3), list(exps), [0.6, 0.4]) for l in (3, 2, 1, 3)]
    bas = molgen.single_shell_basis(shells)
    n = oracle.nbf(bas)
    D = 1e-4 * rng.uniform(-1, 1, (n, n))
    D = 0.5 * (D + D.T)
    D[0, 0] = 1.0
    Jo, Ko = oracle.jk(bas, D, 1e-10)
    J, K = _build(env, bas, D, 1e-10, group_override=group)
    tol = _tolerance(bas, D, Jo, Ko)
    assert np.abs(J - Jo).max() <= tol and np.abs(K - Ko).max() <= tol


def test_batch_with_one_handle_out_of_range(env):
    """A batch whose handles lie inside, partly outside (f pairs only) and wholly
    outside the two-float range gives what each handle gives."""
    torch, fk = env
    mols = [_one_exponent([3, 2], 5.0, 1e-4), _one_exponent([3, 3], 5e3, 1e-4), _one_exponent([1, 2], 1e8, 1e-4)]
    for pick in ([0, 1], [0, 1, 2]):
        bs = [fk.JKBuilder(mols[i][0], 1e-10) for i in pick]
        D = [torch.tensor(mols[i][1], device="cuda") for i in pick]
        J, K = [torch.full_like(d, float("nan")) for d in D], [torch.full_like(d, float("nan")) for d in D]
        fk.fock_build_jk_batched([b.handle for b in bs], D, 1e-10, J, K)
        torch.cuda.synchronize()
        assert fk.fock_stream_status() == 0
        for i, j, k in zip(pick, J, K):
            bas, Dn = mols[i]
            Jo, Ko = oracle.jk(bas, Dn, 1e-10)
            tol = _tolerance(bas, Dn, Jo, Ko)
            assert np.abs(j.cpu().numpy() - Jo).max() <= tol and np.abs(k.cpu().numpy() - Ko).max() <= tol
        for b in bs:
            b.close()


@pytest.mark.parametrize("log2_scale", [-24, -39, -41, -59])
def test_small_elements_of_a_small_density(env, log2_scale):
    """Densities whose elements spread over 2^-36 of the largest, on both sides of
    the smallest max|D| that the window takes (2^-40): every element counts."""
    rng = np.random.Generator(np.random.PCG64(722))
    bas = molgen.random_shells(rng, [0, 1, 2, 0, 1, 3], spread=4.0, kmax=4)
    n = oracle.nbf(bas)
    sizes = [oracle.ncart(int(l)) for l in bas["l"]]
    w = np.repeat(2.0 ** -np.array([0.0, 4.0, 8.0, 12.0, 16.0, 18.0]), sizes)
    D = rng.uniform(-1, 1, (n, n)) * w[:, None] * w[None]
    D = 0.5 * (D + D.T)
    D[0, 0] = 1.0
    D *= 2.0 ** log2_scale
    tau = 1e-22 * 2.0 ** log2_scale
    Jo, Ko = oracle.jk(bas, D, tau)
    J, K = _build(env, bas, D, tau)
    tol = 1e-10 * 2.0 ** log2_scale
    assert np.abs(J - Jo).max() <= tol and np.abs(K - Ko).max() <= tol


def test_large_density_element_far_away(env):
    """One element of D is 2^30 times the others, on a shell too far away to
    exchange with them: every contribution to the near shells' K lies in the
    window (2^-40 of itself), or, with the window turned off, is FP64."""
    torch, fk = env
    rng = np.random.Generator(np.random.PCG64(724))
    bas = molgen.random_shells(rng, [0, 0, 1, 2, 3, 1], spread=2.0, kmax=4)
    bas["center"][0] = [0.0, 0.0, 90.0]
    n = oracle.nbf(bas)
    D = rng.uniform(-1, 1, (n, n))
    D = 0.5 * (D + D.T)
    D[0, :] = D[:, 0] = 0.0
    D[0, 0] = 2.0 ** 30
    Jo, Ko = oracle.jk(bas, D, 1e-12)
    g2 = float(np.max(oracle.schwarz(bas)[0][1:, 1:])) ** 2
    for two_float, rel in ((True, 2.0 ** -40), (False, 2.0 ** -46)):
        J, K = _build(env, bas, D, 1e-12, two_float=two_float)
        assert np.abs(J - Jo).max() <= 2.0 ** -44 * np.abs(Jo).max()
        assert np.abs(K - Ko)[1:, 1:].max() <= n * n * g2 * rel


def test_window_turned_off(env):
    """FOCK_NO_TWO_FLOAT: no launch of its own for two floats, and the same J and K."""
    torch, fk = env
    p = molgen.problem(0)
    b = [fk.JKBuilder(p.basis, p.tau, fk.make_opts(two_float=t)) for t in (True, False)]
    assert fk.fock_kernels_per_build(b[1].handle) < fk.fock_kernels_per_build(b[0].handle)
    D = torch.tensor(p.D, device="cuda")
    (J0, K0), (J1, K1) = (x.build(D) for x in b)
    assert float((J0 - J1).abs().max()) <= 1e-10 and float((K0 - K1).abs().max()) <= 1e-10
    with pytest.raises(fk.FockError):  # one choice per batch
        fk.fock_build_jk_batched([x.handle for x in b], [D, D], p.tau, [J0, J1], [K0, K1])
    for v in (2, 0x102, 0x200, -1):
        with pytest.raises(fk.FockError):
            fk.JKBuilder(p.basis, p.tau, fk.make_opts(precision=v))
    for x in b:
        x.close()


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("group", [0, 4])
@pytest.mark.parametrize("ls,a", [([3, 3], 2e-4), ([3, 3], 600.0), ([3, 2], 2000.0), ([3, 3], 5000.0), ([2, 2], 5e4)])
def test_mixed_exponents_at_the_edges(env, ls, a, group, batched):
    """Mixed builds whose f and d quartets lie below the FP32 cutoff: where the
    seeds would leave the FP32 exponent range the class pair runs in FP64."""
    torch, fk = env
    bas, D = _one_exponent(ls, a, 1e-8)
    Jo, Ko = oracle.jk(bas, D, 1e-13)
    opts = dict(precision=fk.FOCK_MIXED, group_override=group)
    if batched:
        b = fk.JKBuilder(bas, 1e-13, fk.make_opts(**opts))
        Dt = torch.tensor(D, device="cuda")
        J, K = torch.empty_like(Dt), torch.empty_like(Dt)
        fk.fock_build_jk_batched([b.handle], [Dt], 1e-13, [J], [K])
        torch.cuda.synchronize()
        J, K = J.cpu().numpy(), K.cpu().numpy()
        b.close()
    else:
        J, K = _build(env, bas, D, 1e-13, **opts)
    assert np.abs(J - Jo).max() <= TOL_MIXED and np.abs(K - Ko).max() <= TOL_MIXED


def test_mixed_stats_out_of_range(env):
    """No FP32 quartet is counted for a class pair that runs in FP64."""
    torch, fk = env
    bas, D = _one_exponent([3], 5000.0, 1e-8)
    b = fk.JKBuilder(bas, 1e-13, fk.make_opts(precision=fk.FOCK_MIXED))
    st = b.stats(D)
    c = fk.JKBuilder(_one_exponent([3], 500.0, 1e-8)[0], 1e-13, fk.make_opts(precision=fk.FOCK_MIXED)).stats(D)
    b.close()
    assert st["quartets_evaluated"] == c["quartets_evaluated"]
    assert st["quartets_fp32"] < c["quartets_fp32"]


def test_fp32_overflow_shows(env):
    """FP32 quartets whose digested value passes the largest FP32 number: the
    element is infinite or NaN, never a finite wrong number."""
    torch, fk = env
    rng = np.random.Generator(np.random.PCG64(723))
    bas = molgen.random_shells(rng, [0, 1, 2, 3], spread=0.5, kmax=2)
    D = np.full((oracle.nbf(bas),) * 2, 3e38)
    Jo, Ko = oracle.jk(bas, D, 1e-10)
    J, K = _build(env, bas, D, 1e-10, precision=fk.FOCK_MIXED, fp32_cutoff=1e300)
    assert not (np.isfinite(J).all() and np.isfinite(K).all())
    for x, xo in ((J, Jo), (K, Ko)):
        ok = np.isfinite(x)
        assert np.abs(x - xo)[ok].max(initial=0.0) <= 1e-4 * np.abs(xo).max()
