"""The adjoint's chunks and view slices at the sizes where they change: volumes lower than a chunk,
whole chunks, chunks that overlap by one voxel and by all but one, fewer views than slices, and
rows that no ray of the volume uses.

Bars: the operators' relative L2 of 1e-4 against the FP64 oracle (FP32 ray parameters on volumes
of ~30 mm against 1 mm voxels: ~1e-6 expected). Rows whose rays miss the volume have weight 0 in
every voxel: whatever they hold, the result is bit for bit the same."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cb():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1008_2042_gb300 import build
    build.build()
    import paper_1008_2042_gb300 as m
    m.load_library()
    return m


def geom(nz, views, nx=37, ny=21, nv=60):
    return synth.Geometry(nx=nx, ny=ny, nz=nz, dx=1.0, dy=1.1, dz=1.2, nu=33, nv=nv, du=1.7, dv=1.3, u_off=0.6, v_off=-0.35,
                          n_views=views, angles=tuple(0.17 + 2 * np.pi * np.arange(views) / views))


def dev(x):
    return torch.tensor(x, dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("nz", [1, 2, 7, 8, 9, 11, 15, 16, 17, 18, 19, 23, 33])
@pytest.mark.parametrize("views", [1, 3, 8, 17])
def test_backproject_parity_at_chunk_edges(cb, nz, views):
    g = geom(nz, views)
    y = synth.random_projections(g, 77)
    with cb.Geometry(g) as h:
        b = cb.backproject(h, dev(y)).cpu().numpy()
    ref = oracle.backproject(g, y)
    assert np.linalg.norm(b - ref) <= 1e-4 * np.linalg.norm(ref)


# imager rows at v = 0 +- 0.0005 pitches, and away from it, against chunks that begin and end at z = 0
@pytest.mark.parametrize("v_off", [0.65 - 0.00065, 0.65 + 0.00065, 0.1])
@pytest.mark.parametrize("nz", [16, 24, 28, 32, 36, 64])
def test_chunks_that_meet_at_the_orbit_plane(cb, nz, v_off):
    g = synth.Geometry(nx=37, ny=21, nz=nz, dx=1.0, dy=1.1, dz=1.2, nu=33, nv=120, du=1.7, dv=1.3, u_off=0.6, v_off=v_off,
                       n_views=5, angles=tuple(0.17 + 2 * np.pi * np.arange(5) / 5))
    y = synth.random_projections(g, 80)
    with cb.Geometry(g) as h:
        b = cb.backproject(h, dev(y)).cpu().numpy()
    ref = oracle.backproject(g, y)
    assert np.linalg.norm(b - ref) <= 1e-4 * np.linalg.norm(ref)


def test_wide_grid_of_whole_chunks(cb):
    """Enough columns for one slice per patch, 70 = 5 x 14 voxels, sampled voxels in the oracle."""
    g = synth.Geometry(nx=640, ny=600, nz=70, dx=0.4, dy=0.4, dz=1.0, nu=40, nv=60, du=9.7, dv=2.1, u_off=0.6, v_off=-0.35,
                       n_views=2, angles=(0.4, 2.1))
    y = synth.random_projections(g, 78)
    with cb.Geometry(g) as h:
        b = cb.backproject(h, dev(y)).cpu().numpy()
    ref = oracle.backproject(g, y)
    assert np.linalg.norm(b - ref) <= 1e-4 * np.linalg.norm(ref)


def test_rows_that_miss_the_volume_do_not_matter(cb):
    g = geom(9, 4)
    y = synth.random_projections(g, 79)
    hit = oracle.project(g, np.ones(g.vol_shape)).max(axis=(0, 2)) > 0
    above = np.arange(g.nv) > np.nonzero(hit)[0].max()
    assert above.sum() >= 3
    a, b = y.copy(), y.copy()
    a[:, above, :] = 0.0
    b[:, above, :] = np.nan
    with cb.Geometry(g) as h:
        fa, fb = cb.backproject(h, dev(a)), cb.backproject(h, dev(b))
        assert bool(torch.isfinite(fb).all())
        assert torch.equal(fa, fb)
