"""When FP64 products of 4-function atoms go in quads of four: the lists that too few triples fill are not kept, and
both kinds of product agree with the CUDA cores on either side of their lines."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1404_5776_gb300 as m
    m.build()
    return m


def _radii(r):
    return {k: r for k in ("r_Sinv", "r_T", "r_U", "r_K", "r_M")}


def _system(cell=3):
    return synth.diamond_system(cell, "sp4", 6.0, 6.0, seed=0)


# 3.0, 4.5, 5.9 and 9.7 triples to a product of quads on P_U
@pytest.mark.parametrize("radius,quads", [(6.0, False), (7.0, False), (7.5, True), (8.0, True)])
@pytest.mark.parametrize("prop", ["em", "cn", "m4"])
def test_lists_of_quads_are_kept_where_they_are_taken(rt, prop, radius, quads):
    s = _system()
    lists = []
    for precision in ("fp32", "fp64"):
        ctx = rt.RT(s, prop=prop, dt=0.05, precision=precision, **_radii(radius))
        lists.append([ctx.debug_check()])
        ctx.inverse()
        ctx.propagator(0.0)
        ctx.unitarity(0)  # takes none
        lists[-1].append(ctx.debug_check())
        ctx.close()
    mixed, fp64 = lists  # the mixed modes have no quads
    assert (fp64[0] > mixed[0]) == quads
    assert fp64[1] - fp64[0] == mixed[1] - mixed[0]


# n atoms that all reach one another: n triples to a block
@pytest.mark.parametrize("n,quads", [(2, False), (7, False), (8, True), (20, True)])
def test_smallest_systems_take_no_quads(rt, n, quads):
    from test_gpu_x64_range import _chain
    H = np.random.default_rng(n).normal(size=(4 * n, 4 * n))
    s, _ = _chain(H + H.T, 4, 0.1)
    lists = []
    for precision in ("fp32", "fp64"):
        ctx = rt.RT(s, prop="em", dt=0.05, precision=precision, **_radii(6.0))
        lists.append(ctx.debug_check())
        ctx.close()
    assert (lists[1] > lists[0]) == quads


@pytest.mark.parametrize("cell,radius", [(3, 7.5), (3, 8.0), (4, 7.0), (4, 7.5), (0, 9), (0, 21)])
# cell 0: 9 or 21 atoms that all reach one another
@pytest.mark.parametrize("prop", ["em", "cn"])
def test_quads_agree_with_the_cuda_cores(rt, monkeypatch, prop, cell, radius):
    from test_gpu_memory import Limited
    from test_gpu_x64_range import _chain
    if cell:
        s = _system(cell)
    else:
        H = np.random.default_rng(0).normal(size=(4 * radius, 4 * radius))
        s, _ = _chain(H + H.T, 4, 0.1)
    rng = np.random.default_rng(1)

    def trajectory(refused):
        mem = Limited(rt)
        get = lambda n, stream, user: None if n == refused else mem.hooks[0](n, stream, user)
        hooks = rt.ALLOC_FN(get), mem.hooks[1]
        monkeypatch.setattr(rt, "_torch_allocator", lambda: hooks)
        ctx = rt.RT(s, prop=prop, dt=0.01, **_radii(max(radius, 6.0) if cell else 6.0))
        ctx.inverse()
        rowptr, col = ctx.pattern(0, rt.RT_PAT_U)
        K0 = rng.normal(size=16 * len(col)) + 1j * rng.normal(size=16 * len(col))
        ctx.set_density(0, 0, K0 if refused is None else out["K0"])
        ctx.step(2)
        got = [ctx.matrix(0, m) for m in (rt.RT_MAT_SINV, rt.RT_MAT_U, rt.RT_MAT_K)]
        ctx.close()
        rows = np.repeat(np.arange(s.n_atoms), np.diff(rowptr))
        blocks = len(set(zip((rows // 4).tolist(), (col // 4).tolist())))
        out.setdefault("K0", K0)
        return got, mem, (8192 * blocks + 16 + 255) // 256 * 256  # the digits of one split operand

    out = {}
    with_quads, mem, digits = trajectory(None)
    assert digits in mem.sizes
    without, mem, _ = trajectory(digits)
    assert digits not in mem.sizes
    for a, b in zip(with_quads, without):  # either route rounds a product to 2^-53 of a few hundred terms
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
