"""GPU: lattices with more rows or planes than a launch has blocks along y or z (65535), which the
default step takes with taller or longer tiles or with the kernels for any shape; bitwise the
one-thread-per-site kernel.  Two steps, so that the buffers change places."""
import numpy as np
import pytest

from paper_1508_05610_gb300 import inputs

pytestmark = pytest.mark.gpu
KW = dict(dx=0.9, dt=0.07, lam=1.3, eta=0.8, m2=0.1)


@pytest.fixture(scope="module")
def lf2():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1508_05610_gb300 import build, lf2 as binding
    build.build()
    binding.load()
    return binding


def same_as_site(lf2, shape, ncomp, prec, step):
    nx, ny, nz = shape
    phi0 = inputs.gaussian_field(nx, ny, nz, ncomp, sigma=0.4, seed=951)
    pi0 = inputs.gaussian_field(nx, ny, nz, ncomp, sigma=0.2, seed=952)
    p = lf2.params(**KW)
    with lf2.System(shape, ncomp, prec) as a, lf2.System(shape, ncomp, prec) as b:
        for s in (a, b):
            s.upload(phi0, pi0)
        step(a, p)
        lf2.lf2_leapfrog_ex(b.phi, b.pi, p, 2, kernel=lf2.LF2_KERNEL_SITE)
        got, ref = a.download(), b.download()
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])


@pytest.mark.parametrize("prec", ["f64", "f32k", "f32"])
@pytest.mark.parametrize("shape,ncomp", [((4, 131072, 1), 1),   # 65536 pairs of rows
                                         ((4, 131074, 2), 1),   # pairs, but no fours
                                         ((4, 131076, 1), 3),
                                         ((2, 262140, 1), 2),   # the most rows in fours
                                         ((4, 2, 196612), 1),   # more than 65535 chunks of three planes
                                         ((4, 4, 262148), 1)])  # of four
def test_default_step_of_long_lattices(lf2, monkeypatch, shape, ncomp, prec):
    monkeypatch.setenv("LF2_TUNE", "off")
    same_as_site(lf2, shape, ncomp, prec, lambda s, p: lf2.lf2_leapfrog(s.phi, s.pi, p, 2))


@pytest.mark.parametrize("shape", [(4, 131072, 1), (4, 4, 262148)])
def test_streaming_without_a_tile_on_long_lattices(lf2, shape):
    same_as_site(lf2, shape, 1, "f32k",
                 lambda s, p: lf2.lf2_leapfrog_ex(s.phi, s.pi, p, 2, kernel=lf2.LF2_KERNEL_STREAM))


def test_streaming_tiles_that_do_not_fit_are_refused(lf2):
    shape = (4, 131072, 1)
    with lf2.System(shape, 1, "f32") as s:
        with pytest.raises(lf2.LF2Error) as e:
            lf2.lf2_leapfrog_ex(s.phi, s.pi, lf2.params(**KW), 1, kernel=lf2.LF2_KERNEL_STREAM, tile_y=2)
    assert e.value.status == lf2.LF2_ERR_UNSUPPORTED


def test_one_step_plan_of_a_lattice_that_only_tall_tiles_fit(lf2):
    shape = (4, 262152, 1)
    with lf2.System(shape, 1, "f32") as s:
        plan = lf2.lf2_tune(s.phi, s.pi, lf2.params(**KW), flags=lf2.LF2_TUNE_FORCE | lf2.LF2_TUNE_ONE_STEP)
    assert plan["kernel"] == lf2.LF2_KERNEL_STREAM and plan["tile_y"] == 8
    same_as_site(lf2, shape, 1, "f32", lambda s, p: lf2.lf2_leapfrog(s.phi, s.pi, p, 2))


@pytest.mark.parametrize("nz", [131080, 262144, 524288])
def test_one_step_plan_launches_on_more_planes_than_the_tuner_times(lf2, nz):
    """The tuner times 256 planes; chunks of two or four planes that win there are more than 65535 chunks
    here."""
    shape = (16, 4, nz)
    with lf2.System(shape, 1, "f32k") as s:
        plan = lf2.lf2_tune(s.phi, s.pi, lf2.params(**KW), flags=lf2.LF2_TUNE_FORCE | lf2.LF2_TUNE_ONE_STEP)
    assert plan["kernel"] == lf2.LF2_KERNEL_STREAM and plan["zchunk"] * 65535 >= nz
    same_as_site(lf2, shape, 1, "f32k", lambda s, p: lf2.lf2_leapfrog(s.phi, s.pi, p, 2))
