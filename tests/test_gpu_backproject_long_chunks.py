"""The adjoint's chunks of 12, 14, 16 and 18 voxels, on grids with enough columns for them: one whole
chunk, chunks that meet and chunks that overlap by little and by all but one voxel, and chunks that begin, end
or lie across z = 0, whose middle plane rounds to 0 (dz = 1.25) or not (dz = 1.7); one and several view
slices; rows below the volume that hold other values.

Bars: the operators' relative L2 of 1e-4 against the FP64 oracle (FP32 ray parameters on volumes of ~70 mm
against voxels of 0.5 mm: ~1e-6 expected). A row below the volume is part of every prefix above it, so that another
value there moves a voxel by roundings of the prefixes: two per visit of at most 2^-24 of the largest prefix, times the
weight of a visit (the ray's length in a voxel column)."""
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
    import paper_1008_2042_gb300 as m
    m.load_library()
    return m


def geom(nz, dz=1.25, views=3, v_off=0.1, nv=None):
    nv = nv or int(1.2 * nz * dz / 0.9) + 4
    return synth.Geometry(nx=136, ny=84, nz=nz, dx=0.5, dy=0.55, dz=dz, nu=61, nv=nv, du=1.9, dv=1.3, u_off=0.6, v_off=v_off,
                          n_views=views, angles=tuple(0.17 + 2 * np.pi * np.arange(views) / views))


def run(cb, g, y):
    with cb.Geometry(g) as h:
        return cb.backproject(h, torch.tensor(y, dtype=torch.float32, device="cuda")).cpu().numpy()


def check(cb, g, seed=81):
    y = synth.random_projections(g, seed)
    b, ref = run(cb, g, y), oracle.backproject(g, y)
    assert np.linalg.norm(b - ref) <= 1e-4 * np.linalg.norm(ref)


@pytest.mark.parametrize("nz", [7, 9, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20, 21, 22, 24, 25, 28, 29, 31, 33, 35, 36, 42, 51])
def test_chunks_of_every_length(cb, nz):
    check(cb, geom(nz))


# imager rows at v = 0 +- 0.0005 pitches, and away from it
@pytest.mark.parametrize("v_off", [0.65 - 0.00065, 0.65 + 0.00065, 0.1])
@pytest.mark.parametrize("dz", [1.25, 1.7])
@pytest.mark.parametrize("nz", [16, 24, 28, 32, 36, 48])
def test_long_chunks_at_the_orbit_plane(cb, nz, dz, v_off):
    check(cb, geom(nz, dz=dz, v_off=v_off, nv=2 * (int(0.6 * nz * dz) + 2)))


@pytest.mark.parametrize("views", [1, 2, 8])
@pytest.mark.parametrize("nz", [12, 28, 36])
def test_long_chunks_in_view_slices(cb, nz, views):
    check(cb, geom(nz, views=views))


def test_rows_below_the_volume_move_roundings_only(cb):
    g = geom(28, views=4, nv=80)
    a = synth.random_projections(g, 82)
    rows = oracle.project(g, np.ones(g.vol_shape)).max(axis=(0, 2)) > 0
    below = np.arange(g.nv) < np.nonzero(rows)[0].min()
    assert below.sum() >= 3
    b = a.copy()
    b[:, below, :] = 1.0 - a[:, below, :]
    fa, fb = run(cb, g, a), run(cb, g, b)
    top = np.hypot(g.sdd, 100.0) * max(x.sum(axis=1).max() for x in (a, b))  # above every prefix of |D - S| g
    # a voxel sees at most 3 imager columns a view, each over a chord of at most its diagonal, as a part of the ray
    weight = np.hypot(g.dx, g.dy) / g.sdd
    assert np.abs(fa - fb).max() <= g.n_views * 3 * 2 * 2 * 2.0**-24 * top * weight
