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
