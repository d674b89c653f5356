"""fock_window_stats: quartets and modelled operations by the arithmetic that
evaluates them, against the rules of the kernels restated here in numpy, and in
the cases where one arithmetic takes everything."""
import numpy as np
import pytest

import molgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required")
    import paper_2407_21445_gb300 as fk
    return torch, fk


def _builder(fk, bas, tau, **kw):
    return fk.JKBuilder(bas, tau, fk.make_opts(**kw))


def test_one_arithmetic_takes_everything(env):
    """Window off: all FP64, the operations of fock_work_stats.  A cutoff of more
    than 2^-24 of the largest bound: nothing is left to FP64."""
    torch, fk = env
    p = molgen.problem(1, carbons=3)
    b = _builder(fk, p.basis, p.tau, two_float=False)
    st, w = b.stats(p.D), b.window_stats(p.D)
    assert w["flops_two_float"] == w["flops_fp32"] == w["quartets_two_float"] == w["quartets_fp32"] == 0.0
    assert w["flops_fp64"] == st["flops_model"] and w["quartets_fp64"] == st["quartets_evaluated"]
    b.close()
    b = _builder(fk, p.basis, p.tau, precision=fk.FOCK_MIXED, fp32_cutoff=1e-5)
    st, w = b.stats(p.D), b.window_stats(p.D)
    assert w["quartets_fp64"] == 0.0 and w["flops_fp64"] == 0.0
    assert w["quartets_fp32"] == st["quartets_fp32"] > 0
    assert w["quartets_two_float"] == st["quartets_evaluated"] - st["quartets_fp32"] > 0
    b.close()


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -20, 2.0 ** -50])
@pytest.mark.parametrize("cutoff", [0.0, 1e-9])
def test_quartets_against_the_rules(env, scale, cutoff):
    """Uncontracted shells (one primitive quartet each): the edge is 2^-13 of
    max(G)^2 max|D| in FP32 arithmetic, nothing for max|D| below 2^-40."""
    torch, fk = env
    rng = np.random.Generator(np.random.PCG64(730))
    bas = molgen.random_shells(rng, [0, 1, 2, 3, 0, 1, 0], spread=5.0, kmax=1)
    n, ns = oracle.nbf(bas), len(bas["l"])
    D = rng.uniform(-1, 1, (n, n)) * 10.0 ** rng.uniform(-4, 0, (n, 1))
    D = scale * 0.5 * (D + D.T)
    tau, cutoff = 1e-12 * scale, cutoff * scale
    b = _builder(fk, bas, tau, precision=fk.FOCK_MIXED if cutoff else fk.FOCK_FP64, fp32_cutoff=cutoff)
    w = b.window_stats(D)
    b.close()
    G = oracle.schwarz(bas)[0]
    off = np.concatenate([[0], np.cumsum([oracle.ncart(int(l)) for l in bas["l"]])])
    Ds = np.array([[np.abs(D[off[i]:off[i + 1], off[j]:off[j + 1]]).max() for j in range(ns)] for i in range(ns)])
    dmax, g2 = np.abs(D).max(), G.max() ** 2
    pairs = [(i, j) for i in range(ns) for j in range(i + 1)]
    count = {"quartets_fp64": 0, "quartets_two_float": 0, "quartets_fp32": 0}
    close = 0  # quartets too near a line for a recount in other roundings
    for x, (i, j) in enumerate(pairs):
        for k, l in pairs[:x + 1]:
            g = G[i, j] * G[k, l]
            d = max(Ds[i, j], Ds[k, l], Ds[i, k], Ds[i, l], Ds[j, k], Ds[j, l])
            if g < tau or g * d < tau:
                continue
            if cutoff and g * d < cutoff:
                name, line = "quartets_fp32", cutoff
            elif dmax <= 2.0 ** -40 or (not (cutoff and cutoff >= 2.0 ** -24 * g2 * dmax)
                                        and g * d >= 2.0 ** -13 * g2 * dmax):
                name, line = "quartets_fp64", 2.0 ** -13 * g2 * dmax
            else:
                name, line = "quartets_two_float", 2.0 ** -13 * g2 * dmax
            count[name] += 1
            close += min(abs(g * d / y - 1) for y in (line, tau)) < 1e-5
    for name in count:
        assert abs(w[name] - count[name]) <= close, (w, count)
    assert sum(count.values()) > 100
