"""GPU: the step that lattices take whose rows are no whole vectors, against the one-thread-per-site
kernel (bitwise) and the FP64 oracle: every component count and precision, sides of 1, 2 and 3,
planes smaller and larger than a block, z-chunks of one plane and with a remainder."""
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


@pytest.mark.parametrize("prec", ["f64", "f32k", "f32"])
@pytest.mark.parametrize("shape,ncomp", [((1, 1, 1), 1), ((2, 1, 3), 1), ((3, 2, 1), 2), ((1, 5, 67), 1),
                                         ((513, 1, 9), 1), ((33, 31, 19), 1), ((257, 21, 10), 1), ((33, 5, 7), 2),
                                         ((17, 9, 5), 3), ((9, 7, 5), 4), ((19, 6, 5), 5), ((7, 9, 5), 6)])
def test_default_step_equals_site_kernel_and_oracle(lf2, ora, monkeypatch, shape, ncomp, prec):
    monkeypatch.setenv("LF2_TUNE", "off")
    nx, ny, nz = shape
    phi0 = inputs.gaussian_field(nx, ny, nz, ncomp, sigma=0.4, seed=901)
    pi0 = inputs.gaussian_field(nx, ny, nz, ncomp, sigma=0.2, seed=902)
    p = lf2.params(**KW)
    with lf2.System(shape, ncomp, prec) as a, lf2.System(shape, ncomp, prec) as b:
        for s in (a, b):
            s.upload(phi0, pi0)
        lf2.lf2_leapfrog(a.phi, a.pi, p, 5)
        lf2.lf2_leapfrog_ex(b.phi, b.pi, p, 5, kernel=lf2.LF2_KERNEL_SITE)
        got, ref = a.download(), b.download()
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    ophi, opi = ora.evolve(phi0, pi0, 5, **KW)
    tol = 1e-12 if prec == "f64" else 1e-5  # as in test_gpu_parity.py, there for 10 steps
    assert np.max(np.abs(got[0] - ophi)) <= tol * np.max(np.abs(ophi))
    assert np.max(np.abs(got[1] - opi)) <= tol * np.max(np.abs(opi))


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("ncomp", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 1), (7, 5, 3), (4, 3, 2), (12, 7, 5), (132, 3, 4), (260, 5, 2),
                                   (1028, 3, 2), (515, 2, 3)])
def test_derivative_of_every_row_length(lf2, shape, ncomp, prec):
    """(phi(x+i) - phi(x-i)) * (1 / (2 dx)) in the storage type, exactly: rows shorter than a vector,
    of whole vectors and not, within one block and over several, an odd number of rows."""
    nx, ny, nz = shape
    dtype = np.float64 if prec == "f64" else np.float32
    v = inputs.gaussian_field(nx, ny, nz, ncomp, sigma=1.0, seed=903).astype(dtype)
    inv = dtype(0.5 / 0.7)
    with lf2.System(shape, ncomp, prec) as s:
        lf2.lf2_field_upload(s.phi, v.astype(np.float64))
        for dim in range(3):
            lf2.lf2_field_derivative(s.phi, s.pi, dim, 0.7)
            want = (np.roll(v, -1, 2 - dim) - np.roll(v, 1, 2 - dim)) * inv
            got = lf2.lf2_field_download(s.pi, s.host_shape)
            assert np.array_equal(got, want.astype(np.float64)), dim


@pytest.mark.parametrize("prec", ["f64", "f32k", "f32"])
@pytest.mark.parametrize("shape,ncomp", [((1, 1, 1), 1), ((5, 3, 2), 2), ((16, 16, 16), 1), ((31, 9, 8), 3),
                                         ((48, 40, 36), 1), ((20, 18, 14), 4), ((13, 11, 9), 5), ((16, 12, 10), 6),
                                         ((60, 60, 60), 1), ((61, 61, 61), 1), ((64, 64, 64), 1), ((64, 64, 40), 2)])
def test_many_steps_of_small_lattices_equal_single_steps(lf2, monkeypatch, shape, ncomp, prec):
    """Runs of 2, 7 and 1 steps (one cooperative launch where every site has a resident thread, else a
    launch per step), even and odd, bitwise as many single calls of the site kernel; the runs reuse
    the scratch and continue from each other's state."""
    monkeypatch.setenv("LF2_TUNE", "off")
    nx, ny, nz = shape
    phi0 = inputs.gaussian_field(nx, ny, nz, ncomp, sigma=0.4, seed=911)
    pi0 = inputs.gaussian_field(nx, ny, nz, ncomp, sigma=0.2, seed=912)
    p = lf2.params(**KW)
    with lf2.System(shape, ncomp, prec) as a, lf2.System(shape, ncomp, prec) as b:
        for s in (a, b):
            s.upload(phi0, pi0)
            lf2.lf2_leapfrog_init(s.phi, s.pi, p)
        for n in (2, 7, 1):
            lf2.lf2_leapfrog(a.phi, a.pi, p, n)
            for _ in range(n):
                lf2.lf2_leapfrog_ex(b.phi, b.pi, p, 1, kernel=lf2.LF2_KERNEL_SITE)
            got, ref = a.download(), b.download()
            assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), n
        lf2.lf2_field_check(a.phi)


@pytest.mark.parametrize("prec,ncomp,depth,cx,tile", [("f32k", 1, 4, 4, (56, 24)), ("f32", 2, 4, 2, (24, 24)),
                                                      ("f32k", 1, 6, 2, (20, 12)), ("f32", 1, 8, 1, (8, 4)),
                                                      ("f32k", 4, 4, 1, (8, 24)), ("f32k", 3, 3, 1, (10, 8)),
                                                      ("f32k", 6, 2, 1, (12, 12)), ("f64", 1, 4, 2, (24, 8)),
                                                      ("f32k", 1, 3, 4, (56, 26))])
def test_steps_left_over_by_temporal_blocking(lf2, prec, ncomp, depth, cx, tile):
    """Every remainder of a run by the depth (shallower passes of the same region, then single steps)
    gives bitwise the site kernel's state, on a lattice of ragged tiles and as an ensemble of two."""
    shape = (72, 30, 12)
    nx, ny, nz = shape
    phi0 = inputs.gaussian_field(nx, ny, nz, ncomp, sigma=0.4, seed=921)
    pi0 = inputs.gaussian_field(nx, ny, nz, ncomp, sigma=0.2, seed=922)
    p = lf2.params(**KW)
    cfg = dict(depth=depth, cx=cx, tile_x=tile[0], tile_y=tile[1])
    with lf2.System(shape, ncomp, prec) as a, lf2.System(shape, ncomp, prec) as b, \
            lf2.System(shape, ncomp, prec) as c, lf2.System(shape, ncomp, prec) as d:
        for s in (a, b, c, d):
            s.upload(phi0, pi0)
        e = lf2.lf2_ensemble_create([c.phi, d.phi], [c.pi, d.pi], [p, p])
        try:
            lf2.lf2_ensemble_set_config(e, **cfg)
            for rest in range(depth):
                lf2.lf2_leapfrog_ex(a.phi, a.pi, p, depth + rest, kernel=lf2.LF2_KERNEL_TBLOCK, **cfg)
                lf2.lf2_leapfrog_ex(b.phi, b.pi, p, depth + rest, kernel=lf2.LF2_KERNEL_SITE)
                lf2.lf2_ensemble_run(e, depth + rest)
                ref = b.download()
                for s in (a, c, d):
                    got = s.download()
                    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), rest
        finally:
            lf2.lf2_ensemble_destroy(e)


@pytest.mark.parametrize("prec", ["f32k", "f32"])
@pytest.mark.parametrize("shape", [(131, 121, 61), (133, 121, 111), (133, 121, 112), (257, 193, 67), (1, 515, 1201)])
def test_column_walk_over_chunks_of_several_planes(lf2, monkeypatch, shape, prec):
    """Chunks of 2, 4 and 8 planes, whole and with 1 or 3 planes left in the last one, bitwise the
    site kernel; three steps, so that the buffers change places."""
    monkeypatch.setenv("LF2_TUNE", "off")
    nx, ny, nz = shape
    phi0 = inputs.gaussian_field(nx, ny, nz, 1, sigma=0.4, seed=931)
    pi0 = inputs.gaussian_field(nx, ny, nz, 1, sigma=0.2, seed=932)
    p = lf2.params(**KW)
    with lf2.System(shape, 1, prec) as a, lf2.System(shape, 1, prec) as b:
        for s in (a, b):
            s.upload(phi0, pi0)
        lf2.lf2_leapfrog(a.phi, a.pi, p, 3)
        lf2.lf2_leapfrog_ex(b.phi, b.pi, p, 3, kernel=lf2.LF2_KERNEL_SITE)
        got, ref = a.download(), b.download()
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])


@pytest.mark.parametrize("shape,ncomp,prec", [((16, 16, 16), 1, "f64"), ((20, 18, 14), 2, "f32k")])
def test_small_lattice_run_captured_into_a_graph(lf2, monkeypatch, shape, ncomp, prec):
    """A run of several steps in one launch, captured (an even number of steps, so that the buffers are
    where they were) and replayed three times, bitwise as many steps of the site kernel."""
    import torch
    monkeypatch.setenv("LF2_TUNE", "off")
    phi0 = inputs.gaussian_field(*shape, ncomp, sigma=0.4, seed=941)
    pi0 = inputs.gaussian_field(*shape, ncomp, sigma=0.2, seed=942)
    p = lf2.params(**KW)
    with lf2.System(shape, ncomp, prec) as a, lf2.System(shape, ncomp, prec) as b:
        for s in (a, b):
            s.upload(phi0, pi0)
            lf2.lf2_leapfrog_init(s.phi, s.pi, p)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            lf2.lf2_leapfrog(a.phi, a.pi, p, 6, torch.cuda.current_stream())
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        lf2.lf2_leapfrog_ex(b.phi, b.pi, p, 18, kernel=lf2.LF2_KERNEL_SITE)
        got, ref = a.download(), b.download()
        lf2.lf2_field_check(a.phi)
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
