"""Contexts whose device memory is refused: what fits without the split operands of the FP64 products has to run
(on the CUDA cores), whether they are refused themselves or hold what a later request needs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1404_5776_gb300 as m
    m.build()
    return m


class Limited:
    """The library's allocator with a limit on the bytes handed out; remembers the peak and the largest requests."""

    def __init__(self, rt, limit=None):
        import torch
        self.limit, self.now, self.peak, self.sizes, self.held = limit, 0, 0, [], {}
        dev = torch.cuda.current_device()

        def get(nbytes, stream, user):
            if self.limit is not None and self.now + nbytes > self.limit:
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), dev, stream or 0)
            self.held[p] = nbytes
            self.sizes.append(nbytes)
            self.now += nbytes
            self.peak = max(self.peak, self.now)
            return p

        def put(p, stream, user):
            self.now -= self.held.pop(p)
            torch.cuda.caching_allocator_delete(int(p))

        self.hooks = rt.ALLOC_FN(get), rt.FREE_FN(put)


def _system(basis, cell):
    import synth
    return synth.diamond_system(cell, basis, 6.0, 6.0, seed=0)


RADII = {k: 8.0 for k in ("r_Sinv", "r_T", "r_U", "r_K", "r_M")}


@pytest.mark.parametrize("basis,prop", [("spd13", "em"), ("spd13", "cn"), ("sp4", "em"), ("sp4", "cn")])
def test_fp64_context_without_room_for_split_operands(rt, monkeypatch, basis, prop):
    s = _system(basis, 2 if basis == "spd13" else 3)
    rng = np.random.default_rng(3)
    K0 = rng.normal(size=(s.n, s.n))
    K0 = (K0 + K0.T).astype(complex)

    def trajectory(limit):
        mem = Limited(rt, limit)
        monkeypatch.setattr(rt, "_torch_allocator", lambda: mem.hooks)
        ctx = rt.RT(s, prop=prop, dt=0.05, **RADII)
        split = sorted(mem.sizes)[-2:]  # the digits of the two operands (a later, larger product may ask for more)
        ctx.inverse()
        ctx.set_density_dense(0, 0, K0)
        ctx.step(2)
        ctx.kick(0, 0, 0, 1e-3)
        ctx.step(1)
        unit = ctx.unitarity(0)
        ctx.step(1)
        out = ctx.observables(0, 0, 4), ctx.matrix(0, rt.RT_MAT_K), np.asarray(unit)
        ctx.close()
        assert not mem.held
        return out, mem.peak, split

    (obs, K, unit), peak, split = trajectory(None)
    for less in (1, split[0], sum(split)):
        (obs2, K2, unit2), _, _ = trajectory(peak - less)
        # both routes round products to 2^-53 of a few hundred terms
        assert np.abs(K2 - K).max() <= 1e-12 * np.abs(K).max()
        live = np.abs(obs[:, 1:9]).max()
        assert np.abs(obs2[:, 1:9] - obs[:, 1:9]).max() <= 1e-12 * live
        assert np.abs(unit2 - unit).max() <= 1e-12
