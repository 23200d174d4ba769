"""Densities, matrices and states of more than 8 MB in pageable memory: they come back as they went in, and a copy takes
about the time of one plain copy of that size."""
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
