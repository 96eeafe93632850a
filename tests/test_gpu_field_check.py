"""GPU: what a multi-step run whose grid barrier gave up leaves behind.  The barriers give up by
host-side injection (LF2_FAULT=timeout): the run ends by itself and nothing faults."""
import numpy as np
import pytest

from paper_1508_05610_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPE = (16, 12, 10)
KW = dict(dx=1.0, dt=0.1, lam=1.0, eta=1.0, m2=0.0)


@pytest.fixture(scope="module")
def lf2():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1508_05610_gb300 import build, lf2 as binding
    build.build()
    binding.load()
    return binding


def timed_out(lf2, f):
    try:
        lf2.lf2_field_check(f)
    except lf2.LF2Error as e:
        assert e.status == lf2.LF2_ERR_TIMEOUT
        return True
    return False


@pytest.mark.parametrize("later", ["leapfrog", "leapfrog_energy"])
def test_a_timeout_is_kept_until_it_is_reported(lf2, monkeypatch, later):
    """A later run on the field neither clears the report nor stops for it; a check with no run
    behind it (scratch just allocated) reports nothing."""
    import torch
    monkeypatch.setenv("LF2_TUNE", "off")
    p = lf2.params(**KW)
    phi0 = inputs.gaussian_field(*SHAPE, 1, sigma=0.1, seed=941)
    rec = torch.zeros((4, 16), dtype=torch.float64, device="cuda")
    with lf2.System(SHAPE, 1, "f64") as s, lf2.System(SHAPE, 1, "f64") as t:
        for q in (s, t):
            q.upload(phi0, np.zeros_like(phi0))
            lf2.lf2_leapfrog_init(q.phi, q.pi, p)
        assert not timed_out(lf2, s.phi)
        monkeypatch.setenv("LF2_FAULT", "timeout")
        lf2.lf2_leapfrog_energy(s.phi, s.pi, p, 4, rec.data_ptr())
        monkeypatch.delenv("LF2_FAULT")
        s.upload(phi0, np.zeros_like(phi0))
        lf2.lf2_leapfrog_init(s.phi, s.pi, p)
        if later == "leapfrog":
            lf2.lf2_leapfrog(s.phi, s.pi, p, 4)
        else:
            lf2.lf2_leapfrog_energy(s.phi, s.pi, p, 4, rec.data_ptr())
            assert torch.isfinite(rec).all()
        lf2.lf2_leapfrog_ex(t.phi, t.pi, p, 4, kernel=lf2.LF2_KERNEL_SITE)
        got, ref = s.download(), t.download()
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
        assert timed_out(lf2, s.phi)
        assert not timed_out(lf2, s.phi)  # once


@pytest.mark.parametrize("prec", ["f64", "f32k"])
def test_injected_timeout_reaches_lf2_leapfrog(lf2, monkeypatch, prec):
    """LF2_FAULT=timeout makes the barriers of lf2_leapfrog's one-launch runs give up as well: the
    check reports it, and a run of freshly uploaded fields steps as the site kernel does."""
    monkeypatch.setenv("LF2_TUNE", "off")
    p = lf2.params(**KW)
    phi0 = inputs.gaussian_field(*SHAPE, 1, sigma=0.1, seed=942)
    with lf2.System(SHAPE, 1, prec) as s, lf2.System(SHAPE, 1, prec) as t:
        for q in (s, t):
            q.upload(phi0, np.zeros_like(phi0))
            lf2.lf2_leapfrog_init(q.phi, q.pi, p)
        monkeypatch.setenv("LF2_FAULT", "timeout")
        lf2.lf2_leapfrog(s.phi, s.pi, p, 4)
        monkeypatch.delenv("LF2_FAULT")
        assert timed_out(lf2, s.phi)
        s.upload(phi0, np.zeros_like(phi0))
        lf2.lf2_leapfrog_init(s.phi, s.pi, p)
        lf2.lf2_leapfrog(s.phi, s.pi, p, 4)
        assert not timed_out(lf2, s.phi)
        lf2.lf2_leapfrog_ex(t.phi, t.pi, p, 4, kernel=lf2.LF2_KERNEL_SITE)
        got, ref = s.download(), t.download()
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
