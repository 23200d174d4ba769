"""Densities, matrices and states of more than 8 MB in pageable memory: they come back as they went in, also where the
device has no memory to spare, and a copy takes about the time of one plain copy of that size."""
import time

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


def _cluster(target):
    pos, species = synth.si_h_cluster(target=target)
    return synth.build_system(pos, None, species, 6.0, 6.0)


def _values(rt, ctx, s, rng):
    rowptr, col = ctx.pattern(0, rt.RT_PAT_K)
    rows = np.repeat(np.arange(s.n_atoms), np.diff(rowptr))
    n = int((s.bsize[rows] * s.bsize[col]).sum())
    return rng.normal(size=n) + 1j * rng.normal(size=n)


# 13 functions (no padding); 1 and 4 functions (padded to 4)
@pytest.mark.parametrize("system", ["diamond", "cluster"])
def test_large_matrices_and_states_round_trip(rt, system):
    s = synth.diamond_system(2, "spd13", 7.0, 7.0, seed=0) if system == "diamond" else _cluster(500)
    rng = np.random.default_rng(0)
    ctx, other = (rt.RT(s, prop="em", dt=0.05, **_radii(8.0 if system == "diamond" else 14.0)) for _ in range(2))
    for _ in range(2):
        K = _values(rt, ctx, s, rng)
        assert K.nbytes > 8 << 20
        ctx.set_density(0, 0, K)
        assert np.array_equal(ctx.matrix(0, rt.RT_MAT_K), K)
    other.set_state(ctx.get_state())
    assert np.array_equal(other.matrix(0, rt.RT_MAT_K), K)
    ctx.close()
    other.close()


def test_a_pageable_density_is_set_at_the_rate_of_a_plain_copy(rt):
    import torch
    s = synth.diamond_system(4, "spd13", 7.0, 7.0, seed=0)
    ctx = rt.RT(s, prop="em", dt=0.05, precision="fp32", **_radii(8.0))
    K = _values(rt, ctx, s, np.random.default_rng(0))
    plain = torch.empty(K.size, dtype=torch.complex128, device="cuda")

    def best(f):
        t = []
        for _ in range(9):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            f()
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t)

    copy = best(lambda: plain.copy_(torch.from_numpy(K)))
    assert best(lambda: ctx.set_density(0, 0, K)) <= 2.0 * copy
    ctx.close()


# 13 functions (real matrices packed), 1 and 4 functions (all packed)
@pytest.mark.parametrize("system,precision", [("diamond", "fp64"), ("diamond", "fp32"), ("cluster", "fp64")])
def test_matrices_are_read_and_set_without_device_memory_to_spare(rt, monkeypatch, system, precision):
    from test_gpu_memory import Limited
    s = synth.diamond_system(2, "spd13", 6.0, 6.0, seed=0) if system == "diamond" else _cluster(150)
    mem = Limited(rt)
    monkeypatch.setattr(rt, "_torch_allocator", lambda: mem.hooks)
    ctx = rt.RT(s, prop="em", dt=0.05, precision=precision, **_radii(8.0))
    ctx.inverse()
    K = _values(rt, ctx, s, np.random.default_rng(0))
    ctx.set_density(0, 0, K)
    read = lambda: [ctx.matrix(0, m) for m in (rt.RT_MAT_SINV, rt.RT_MAT_T, rt.RT_MAT_K)]
    ctx.step(1)
    before, held = read(), dict(mem.held)
    mem.limit = mem.now
    for got, want in zip(read(), before):
        assert np.array_equal(got, want)
    ctx.set_density(0, 0, K)
    assert np.array_equal(ctx.matrix(0, rt.RT_MAT_K), K)
    ctx.step(1)
    mem.limit = None
    assert np.array_equal(ctx.matrix(0, rt.RT_MAT_K), before[2])
    assert mem.held == held  # the split operands among it
    ctx.close()
