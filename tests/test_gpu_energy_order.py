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
    assert (tiles < nb * (nb + 1) // 2 - 0.5) == fewer
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
