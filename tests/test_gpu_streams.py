"""Builds of several streams at once and beside graph captures: the pool of
internal streams is shared by every caller, and what it does must not show."""
import threading

import pytest

import molgen

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required")
    import paper_2407_21445_gb300 as fk
    return torch, fk


def _diff(a, b):
    return max(float((x - y).abs().max()) for x, y in zip(a, b))


@pytest.mark.parametrize("entry", ["fock_build_jk_noalloc", "fock_build_jk"])
def test_build_beside_a_global_capture(env, entry):
    """While a global-mode capture (torch's default) is open on one stream, builds
    of its thread and of another one on streams that own no set of the pool leave
    it intact."""
    torch, fk = env
    build = getattr(fk.fock, entry)
    p = molgen.problem(1, carbons=3)
    b = fk.JKBuilder(p.basis, p.tau)
    D = torch.tensor(p.D, device="cuda")
    ref = b.build(D)
    streams = [torch.cuda.Stream() for _ in range(5)]
    out = [tuple(torch.full_like(D, float("nan")) for _ in range(2)) for _ in range(3)]
    torch.cuda.synchronize()
    for s in streams[:3]:  # the sets of the pool have had owners
        build(b.handle, D, p.tau, *out[0], stream=s)
    torch.cuda.synchronize()
    for J, K in out:
        J.fill_(float("nan"))
        K.fill_(float("nan"))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=streams[3]):
        fk.fock.fock_build_jk(b.handle, D, p.tau, *out[0], stream=streams[3])
        build(b.handle, D, p.tau, *out[1], stream=streams[4])  # not captured
        t = threading.Thread(target=lambda: build(b.handle, D, p.tau, *out[2], stream=streams[4]))
        t.start()
        t.join()
    torch.cuda.synchronize()
    assert _diff(out[1], ref) <= TOL and _diff(out[2], ref) <= TOL
    g.replay()
    torch.cuda.synchronize()
    assert _diff(out[0], ref) <= TOL
    b.close()


def test_more_streams_than_sets(env):
    """Builds of four streams in flight together, more than the pool has sets: the
    others run on the caller's stream alone and give the same."""
    torch, fk = env
    p = molgen.problem(1, carbons=10)
    b = fk.JKBuilder(p.basis, p.tau)
    scale = (1.0, 0.5, -2.0, 3.0)
    D = [torch.tensor(s * p.D, device="cuda") for s in scale]
    ref = [b.build(d) for d in D]  # each its own: the screening weighs the density
    out = [tuple(torch.full_like(D[0], float("nan")) for _ in range(2)) for _ in D]
    streams = [torch.cuda.Stream() for _ in D]
    torch.cuda.synchronize()
    for _ in range(3):
        for d, o, s in zip(D, out, streams):
            b.build(d, *o, stream=s)
    torch.cuda.synchronize()
    for o, r in zip(out, ref):
        assert _diff(o, r) <= TOL
    b.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_captured_build_writes_both_matrices(env, precision):
    """J and K are both rewritten by every replay, from the density it finds."""
    torch, fk = env
    p = molgen.problem(1, carbons=4)
    b = fk.JKBuilder(p.basis, p.tau, fk.make_opts(precision=precision))
    D = torch.tensor(p.D, device="cuda")
    J, K = torch.empty_like(D), torch.empty_like(D)
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        b.build(D, J, K, stream=s)
    for scale in (1.0, 0.25):
        D.copy_(torch.tensor(scale * p.D))
        ref = b.build(D)
        J.fill_(float("nan"))
        K.fill_(float("nan"))
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert _diff((J, K), ref) <= (TOL if precision == 0 else 1e-7)
    b.close()
