"""1/tau of the transport setup where the rate R - B cancels: occupied states."""
import numpy as np
import pytest

import oracle
import synth

from test_gpu_parity import T, nrel, pb  # noqa: F401 - pb is a fixture

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sigma,T_K,mus", [(16, 4e-4, 100.0, (0.15, 0.6, 3.0)), (17, 1e-3, 100.0, (0.3, 3.0)),
                                             (12, 8e-3, 300.0, (-0.2, 0.3, 3.0))])
def test_tau_with_occupied_states(pb, n, sigma, T_K, mus):  # noqa: F811
    """tau from one pass with F = 0 and v = 1 (tau (v + W F) = tau), state by state against the
    oracle's positive sum, mu from below the band to above its top.  Each weight is within 2^-45 (two
    products of values stored to 2^-49, their sum), the oracle and the device each within
    3 2^-53 z^2 / 2 of a Gaussian at z widths, z^2 / 2 up to 30 where the narrow delta function
    leaves tails: 5e-14 together.  (R - B alone is 8e-14 to 1.6e-13 off in the first model.)"""
    m = synth.make_window4(n, sigma=sigma).with_(T=T_K)
    o = oracle.Oracle(m)
    ch = pb.Channels.from_model(m)
    dev, big = pb.Device(ch, transport=True), pb.Device(ch, transport=True, tile_sweep=2)
    one, zero = np.ones((o.nstate, 3)), np.zeros((o.nstate, 3))
    for mu in mus:
        f0 = o.window_values(m.f_fermi(m.emin() + mu))
        rate = o.rates(f0)
        tau = dev.transport_map(T(f0), T(one), T(zero)).cpu().numpy()
        assert np.abs(tau * rate[:, None] - 1.0).max() <= 5e-14
        # one column slot per tile instead of two: the same sums in another order
        other = big.transport_map(T(f0), T(one), T(zero)).cpu().numpy()
        assert np.abs(tau / other - 1.0).max() <= 5e-14


def test_tau_of_signed_and_single_block_inputs(pb):  # noqa: F811
    """27 states (one ragged diagonal tile) with f0 outside [0, 1], where the weights change sign, and
    1000 at one energy, uniform f0: against the oracle."""
    for m, f in ((synth.make_flat_einstein(3), lambda r, n: r.uniform(-0.5, 0.4, n)),
                 (synth.make_flat_einstein(10), lambda r, n: r.uniform(0, 1, n))):
        o = oracle.Oracle(m)
        dev = pb.Device(pb.Channels.from_model(m), transport=True)
        f0 = f(np.random.default_rng(71), o.nstate)
        v = np.random.default_rng(72).normal(size=(o.nstate, 3))
        got = dev.transport_map(T(f0), T(v), T(np.zeros_like(v))).cpu().numpy()
        assert nrel(got, v / o.rates(f0)[:, None]) <= 1e-12
