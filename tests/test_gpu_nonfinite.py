"""Inputs that are not finite: what a NaN or an infinity in one state's numbers reaches."""
import numpy as np
import pytest

import oracle
import synth

from test_gpu_parity import T, pb  # noqa: F401 - pb is a fixture

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [{}, dict(dense_rows=2), dict(variant="f64")], ids=["tiles", "rows", "f64"])
@pytest.mark.parametrize("bad", ["f0", "vel"])
def test_transport_of_numbers_that_are_not_finite_does_not_converge(pb, opts, bad):  # noqa: F811
    """One NaN in f0, one infinite velocity: the solve ends unconverged with an infinite residual at once
    (every maximum that drops a NaN would call it converged), a pass reports residual numbers that are
    not finite, and the handle's next solve is not touched by it."""
    m = synth.make_window4(16)
    o = oracle.Oracle(m)
    dev = pb.Device(pb.Channels.from_model(m), transport=True, **opts)
    f0, v = o.window_values(m.f_fermi(m.emin() - 0.2)), o.window_values(m.vel)
    F, it, res, ok = dev.transport(T(f0), T(v), tol=1e-10, maxit=200)
    assert ok and it > 1 and res <= 1e-10
    fb, vb = f0.copy(), v.copy()
    if bad == "f0":
        fb[o.nstate // 3] = np.nan
    else:
        vb[o.nstate // 3, 1] = np.inf
    Fb, itb, resb, okb = dev.transport(T(fb), T(vb), tol=1e-10, maxit=200)
    assert not okb and itb == 1 and resb == np.inf
    assert not np.isfinite(Fb.cpu().numpy()).all()
    r3 = T(np.zeros(3))
    dev.transport_iterate(T(vb), Fb, resid=r3)
    assert not np.isfinite(r3.cpu().numpy()).any()
    F2, it2, _, ok2 = dev.transport(T(f0), T(v), tol=1e-10, maxit=200)
    assert ok2 and it2 == it and np.array_equal(F2.cpu().numpy(), F.cpu().numpy())


FORMS = {"tiles": {}, "whole-tiles": dict(tile_sweep=2), "rows": dict(dense_rows=2), "f64": dict(variant="f64"),
         "c32": dict(variant="c32"), "g32": dict(variant="g32", channel_per_lane=5),
         "g32-lanes": dict(variant="g32", channel_per_lane=4), "h16": dict(variant="h16", channel_per_lane=5),
         "batch-ff": "ff", "batch-c32": "c32", "batch-fp32": "fp32"}
IN_REACH_ONLY = ("g32", "h16", "batch-fp32")  # the dense forms hold no pair out of reach


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_state_that_is_not_finite_spoils_the_states_it_is_coupled_to(pb, form, bad):  # noqa: F811
    """Every state within 60 meV + 8 sigma of the bad one (some branch within 8 widths: a nonzero
    coefficient in FP32 too) becomes not finite, in each form; in the dense forms no state beyond
    the reach of the FP32 Gaussian (13.3 widths) does, whichever state it is: the last one too,
    which padding lanes would read."""
    m = synth.make_window4(16)
    o = oracle.Oracle(m)
    ch = pb.Channels.from_model(m)
    kw = FORMS[form]
    dev = pb.Batch([ch], precision=kw) if isinstance(kw, str) else pb.Device(ch, **kw)
    e = m.eps.reshape(-1)[o.ids]
    f = np.random.default_rng(97).uniform(0, 1, o.nstate)
    for k in (o.nstate - 1, 0, o.nstate // 2):
        fb = f.copy()
        fb[k] = bad
        I = dev.collision(T(fb)).cpu().numpy()
        de = np.abs(e - e[k])
        assert not np.isfinite(I[de <= 0.06 + 8 * m.sigma]).any()
        if form in IN_REACH_ONLY:
            assert np.isfinite(I[de > 0.06 + 13.5 * m.sigma]).all()
        assert np.isfinite(dev.collision(T(f)).cpu().numpy()).all()
