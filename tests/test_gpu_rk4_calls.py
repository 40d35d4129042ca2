"""Time stepping cut into calls: n steps in one call are n calls of one step, bit for bit."""
import numpy as np
import pytest

import oracle
import synth

from test_gpu_parity import T, nrel, pb  # noqa: F401 - pb is a fixture

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hole", [0.0, 1e-3, 1e-8], ids=["hot", "full-1e-3", "full-1e-8"])
@pytest.mark.parametrize("n,kw", [(16, {}), (16, dict(tile_sweep=2)), (17, dict(variant="c32")), (30, {})],
                         ids=["chained", "whole-tiles", "c32", "ring"])
def test_steps_in_one_call_and_in_many(pb, n, kw, hole):  # noqa: F811
    """The stages' input and a call's own are the same function of f, also in nearly full states, where
    1 - f has few of the bits that f is stored to.  (30^3: 272 tiles, the ring.)"""
    m = synth.make_window4(n)
    o = oracle.Oracle(m) if n < 20 else None
    ch = pb.Channels.from_model(m)
    dev = pb.Device(ch, **kw)
    rng = np.random.default_rng(83)
    f = 1.0 - hole * rng.uniform(0, 1, ch.nstate) if hole else rng.uniform(0, 1, ch.nstate)
    a, b = T(f), T(f)
    dev.rk4(a, 0.5, 5)
    for _ in range(5):
        dev.rk4(b, 0.5, 1)
    assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
    if o is not None and not kw:
        # df/dt of nearly full states is of the order of the holes: its own norm is the measure
        assert nrel(dev.collision(T(f)).cpu().numpy(), o.collision(f)) <= 1e-12
    dev.check()


@pytest.mark.parametrize("hole", [0.0, 1e-8])
@pytest.mark.parametrize("precision", ["ff", "c32", "fp32"])
def test_batch_steps_in_one_call_and_in_many(pb, precision, hole):  # noqa: F811
    b = pb.Batch([pb.Channels.from_model(synth.make_window4(n)) for n in (12, 17)], precision=precision)
    rng = np.random.default_rng(89)
    f = 1.0 - hole * rng.uniform(0, 1, b.nstate) if hole else rng.uniform(0, 1, b.nstate)
    x, y = T(f), T(f)
    b.rk4(x, 0.5, 4)
    for _ in range(4):
        b.rk4(y, 0.5, 1)
    assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
