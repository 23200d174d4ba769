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


@pytest.mark.parametrize("cell,radius", [(3, 7.5), (3, 8.0), (4, 7.0), (4, 7.5)])
@pytest.mark.parametrize("prop", ["em", "cn"])
def test_quads_agree_with_the_cuda_cores(rt, monkeypatch, prop, cell, radius):
    from test_gpu_memory import Limited
    s = _system(cell)
    rng = np.random.default_rng(1)

    def trajectory(limit):
        mem = Limited(rt, limit)
        monkeypatch.setattr(rt, "_torch_allocator", lambda: mem.hooks)
        ctx = rt.RT(s, prop=prop, dt=0.05, **_radii(radius))
        ctx.inverse()
        ctx.set_density(0, 0, K0)
        ctx.step(2)
        out = [ctx.matrix(0, m) for m in (rt.RT_MAT_SINV, rt.RT_MAT_U, rt.RT_MAT_K)]
        ctx.close()
        return out, mem

    probe = rt.RT(s, prop=prop, dt=0.05, **_radii(radius))
    n = 16 * len(probe.pattern(0, rt.RT_PAT_K)[1])
    probe.close()
    K0 = rng.normal(size=n) + 1j * rng.normal(size=n)
    with_quads, mem = trajectory(None)
    without, _ = trajectory(mem.peak - sum(sorted(mem.sizes)[-2:]))
    for a, b in zip(with_quads, without):  # either route rounds a product to 2^-53 of a few hundred terms
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
