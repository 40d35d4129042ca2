"""The energy-ordered tiles: only the block pairs within reach of a phonon are stored, and the sums
are those of the whole pair matrix (the rows of the same list, and the oracle)."""
import numpy as np
import pytest

import oracle
import synth

from test_gpu_parity import C32_TOL, MUTUAL, TOL, T, check_I, nrel, pb  # noqa: F401 - pb is a fixture

pytestmark = pytest.mark.gpu

# name: (model, whether fewer tiles than the whole triangle are stored)
CASES = {
    "narrow": (lambda: synth.make_window4(16, sigma=4e-4), True),   # reach 0.066 eV: a thin band
    "default": (lambda: synth.make_window4(17), True),              # ragged last block
    "full": (lambda: synth.make_window4(12, sigma=0.3), False),     # reach beyond the spectrum
    "flat": (lambda: synth.make_flat_einstein(5), False),           # one energy: 125 states, 2 blocks
    "cold": (lambda: synth.make_tiny(6).with_(T=20.0), True),       # many Bose factors near zero
}


@pytest.mark.parametrize("variant", ["ff", "c32"])
@pytest.mark.parametrize("name", list(CASES))
def test_energy_ordered_tiles_hold_every_nonzero_pair(pb, name, variant):  # noqa: F811
    make, fewer = CASES[name]
    m = make()
    o = oracle.Oracle(m)
    ch = pb.Channels.from_model(m)
    dev = pb.Device(ch, variant=variant)
    nb = (ch.nstate + 63) // 64
    tiles = dev.bytes_per_channel * ch.nchannels / (4096 * (16 if variant == "ff" else 8))
    assert (tiles < nb * (nb + 1) // 2 - 0.5) == (fewer and variant == "ff")  # c32: state order, all tiles
    f = np.random.default_rng(41).uniform(0, 1, o.nstate)
    ref, ab = o.collision(f, with_abs=True)
    I = dev.collision(T(f)).cpu().numpy()
    if variant == "ff":
        check_I(I, ref, ab)
        rows = pb.Device(ch, dense_rows=2)
        assert np.abs(I - rows.collision(T(f)).cpu().numpy()).max() <= MUTUAL * ab.max()
    else:
        assert np.abs(I - ref).max() <= C32_TOL * ab.max()
    tol = TOL if variant == "ff" else C32_TOL
    assert nrel(dev.rates(T(f)).cpu().numpy(), o.rates(f)) <= tol
    f0 = o.window_values(m.f_hot())
    ft = T(f0)
    dev.rk4(ft, 1.0, 2)
    assert nrel(ft.cpu().numpy(), o.rk4(f0, 1.0, 2)) <= tol
    dev.check()
    # after set_g2 the rows replace the tiles (and read f in state order again)
    if variant == "ff":
        dev.set_g2(T(ch.export()["g2"]))
        assert np.abs(dev.collision(T(f)).cpu().numpy() - I).max() <= MUTUAL * ab.max()


@pytest.mark.parametrize("name", list(CASES))
def test_transport_over_tiles(pb, name):  # noqa: F811
    """The automatic transport shape on the tiles: one map against the oracle and the row sweep, the
    residual numbers, the weights that stay in use after set_g2 until the next setup, and the row
    form after it."""
    m = CASES[name][0]()
    o = oracle.Oracle(m)
    ch = pb.Channels.from_model(m)
    dev, rows = pb.Device(ch, transport=True), pb.Device(ch, transport=True, dense_rows=2)
    rng = np.random.default_rng(43)
    f0, v = o.window_values(m.f_fermi(m.emin() - 0.2)), o.window_values(m.vel)
    F = rng.normal(size=(o.nstate, 3))
    ref, _ = o.transport_map(f0, v, F)
    got = dev.transport_map(T(f0), T(v), T(F)).cpu().numpy()
    assert nrel(got, ref) <= TOL
    assert nrel(rows.transport_map(T(f0), T(v), T(F)).cpu().numpy(), got) <= TOL
    res = T(np.zeros(3))
    dev.transport_iterate(T(v), T(F), resid=res)
    d, top = np.abs(got - F).max(), np.abs(got).max()
    assert np.abs(res.cpu().numpy() - np.array([d / top, d, top])).max() <= 1e-14 * max(d, top)
    dev.set_g2(T(2.0 * ch.export()["g2"]))
    assert np.array_equal(dev.transport_iterate(T(v), T(F)).cpu().numpy(), got)
    dev.transport_setup(T(f0))
    twice = dev.transport_iterate(T(v), T(F)).cpu().numpy()  # tau halves, tau W stays
    assert np.abs(twice - (got - 0.5 * v / o.rates(f0)[:, None])).max() <= TOL * np.abs(got).max()
    dev.check()


def test_transport_segments_of_many_tiles(pb):  # noqa: F811
    """A CTA's run of one block row longer than the 16 tiles that one lazily renormalised sum may
    take (92 blocks of states at one energy): sampled rows against the oracle."""
    m = synth.make_flat_einstein(18)
    o = oracle.Oracle(m)
    dev = pb.Device(pb.Channels.from_model(m), transport=True)
    rng = np.random.default_rng(47)
    f0, v, F = rng.uniform(0, 1, o.nstate), rng.normal(size=(o.nstate, 3)), rng.normal(size=(o.nstate, 3))
    rows = np.concatenate([np.arange(3), rng.integers(0, o.nstate, 20), [o.nstate - 1]]).astype(np.int32)
    ref, _ = o.transport_map(f0, v, F, rows=rows)
    got = dev.transport_map(T(f0), T(v), T(F)).cpu().numpy()
    assert np.abs(got[rows] - ref).max() <= TOL * np.abs(got).max()
    dev.check()


@pytest.mark.parametrize("name", list(CASES))
def test_dense_mixed_sweep_skips_pairs_out_of_reach(pb, name):  # noqa: F811
    """The dense FP32 |g|^2 sweep over the pairs in reach, alone and in the batch, and its adjoint
    against the channel-list form of the same device type, which sweeps every channel: both evaluate
    the same FP32 Gaussians (whose own error against FP64 is about 2^-24 of the exponent: beyond
    1e-6 where a narrow delta function leaves only far tails), so they agree to FP32 rounding of the
    terms."""
    m = CASES[name][0]()
    o = oracle.Oracle(m)
    ch = pb.Channels.from_model(m)
    dev, lanes = pb.Device(ch, variant="g32", channel_per_lane=5), pb.Device(ch, variant="g32", channel_per_lane=4)
    b = pb.Batch([ch, ch])
    rng = np.random.default_rng(53)
    f, lam = rng.uniform(0, 1, o.nstate), rng.normal(size=o.nstate)
    ab = o.collision(f, with_abs=True)[1]
    ref = lanes.collision(T(f)).cpu().numpy()
    assert np.abs(dev.collision(T(f)).cpu().numpy() - ref).max() <= 1e-6 * ab.max()
    both = b.collision(T(np.concatenate([f, f]))).cpu().numpy()
    assert np.array_equal(both[:o.nstate], both[o.nstate:])
    assert np.abs(both[:o.nstate] - ref).max() <= 1e-6 * ab.max()
    assert nrel(dev.rates(T(f)).cpu().numpy(), lanes.rates(T(f)).cpu().numpy()) <= 1e-6
    f0 = o.window_values(m.f_hot())
    ft, fb, want = T(f0), T(np.concatenate([f0, f0])), T(f0)
    dev.rk4(ft, 1.0, 2)
    b.rk4(fb, 1.0, 2)
    lanes.rk4(want, 1.0, 2)
    want = want.cpu().numpy()
    assert nrel(ft.cpu().numpy(), want) <= 1e-6 and nrel(fb.cpu().numpy()[o.nstate:], want) <= 1e-6
    g = [d.collision_vjp(T(f), T(lam), grad_g2=T(np.zeros(ch.nchannels))).cpu().numpy() for d in (dev, lanes)]
    assert np.abs(g[0] - g[1]).max() <= 1e-6 * np.abs(o.rates(f)).max() * np.abs(lam).max()


@pytest.mark.parametrize("ctas", [0, 2])
@pytest.mark.parametrize("n", [3, 4, 10, 11])
def test_half_tile_sweep_of_small_and_larger_lists(pb, n, ctas):  # noqa: F811
    """Whole triangles around the lines of the half-tile sweep: 27 and 64 states (one diagonal tile,
    ragged and full), 1000 states (136 tiles: a CTA per half-tile, chained; twice that in the batch, which
    takes the ring) and 1331 (231 tiles, the ring), against the oracle; the batch also with itself."""
    m = synth.make_flat_einstein(n)
    o = oracle.Oracle(m)
    ch = pb.Channels.from_model(m)
    dev = pb.Device(ch, dense_rows=3, ctas_per_sm=ctas)
    rng = np.random.default_rng(59)
    f = rng.uniform(0, 1, o.nstate)
    ref, ab = o.collision(f, with_abs=True)
    check_I(dev.collision(T(f)).cpu().numpy(), ref, ab)
    assert nrel(dev.rates(T(f)).cpu().numpy(), o.rates(f)) <= TOL
    ft = T(f)
    dev.rk4(ft, 1.0, 3)
    assert nrel(ft.cpu().numpy(), o.rk4(f, 1.0, 3)) <= TOL
    dev.check()
    b = pb.Batch([ch, ch], precision="ff", layout=2)
    both = b.collision(T(np.concatenate([f, f]))).cpu().numpy()
    assert np.array_equal(both[:o.nstate], both[o.nstate:])
    check_I(both[:o.nstate], ref, ab)
    fb = T(np.concatenate([f, f]))
    b.rk4(fb, 1.0, 3)
    assert nrel(fb.cpu().numpy()[o.nstate:], o.rk4(f, 1.0, 3)) <= TOL


@pytest.mark.parametrize("opts", [{}, dict(tile_sweep=1)])
@pytest.mark.parametrize("name", list(CASES) + ["ring"])
def test_adjoint_over_tiles(pb, name, opts):  # noqa: F811
    """The FF adjoint over the tiles (a CTA per half-tile; "ring", 231 tiles, and tile_sweep 1 a CTA per
    tile) against the oracle and, for the |g|^2 gradient, the row form, which takes the same table."""
    m = synth.make_flat_einstein(11) if name == "ring" else CASES[name][0]()
    o = oracle.Oracle(m)
    ch = pb.Channels.from_model(m)
    dev, rows = pb.Device(ch, dense_rows=3, **opts), pb.Device(ch, dense_rows=2)
    rng = np.random.default_rng(61)
    f, lam = rng.uniform(0, 1, o.nstate), rng.normal(size=o.nstate)
    gg = [T(np.zeros(ch.nchannels)) for _ in range(2)]
    got, ref = [d.collision_vjp(T(f), T(lam), grad_g2=q).cpu().numpy() for d, q in zip((dev, rows), gg)]
    assert nrel(got, o.collision_vjp(f, lam)) <= 1e-11
    assert nrel(got, ref) <= 1e-11
    assert np.array_equal(gg[0].cpu().numpy(), gg[1].cpu().numpy())
    f0 = o.window_values(m.f_hot())
    l1 = T(lam)
    for _ in range(2):  # twice: the replayed sequence too
        l1.copy_(T(lam))
        dev.rk4_vjp(T(f0), l1, 1.0)
        assert nrel(l1.cpu().numpy(), o.rk4_vjp(f0, 1.0, 1, lam)) <= 1e-11
    # after set_g2 the rows replace the tiles
    dev.set_g2(T(ch.export()["g2"]))
    assert nrel(dev.collision_vjp(T(f), T(lam)).cpu().numpy(), got) <= 1e-11
    dev.check()
