"""The projector's table build and line fills at the sizes where they change: padded z-lines of
every remainder, one or two imager rows per thread and more rows than a block, volumes taller
than a TMA box, traces that end inside, at and just after a table, and the packed z-lines of the
allocation-free entry point.

Bars: the operators' relative L2 of 1e-4 against the FP64 oracle (FP32 ray parameters on volumes
of at most ~60 mm against voxels of 0.4 mm or more: ~1e-6 expected); the two entry points run the
same sums in the same order and are equal."""
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


def geom(nx, ny, nz, nu, nv, dz=1.0, du=2.1, dv=1.3, views=3):
    return synth.Geometry(nx=nx, ny=ny, nz=nz, dx=1.0, dy=1.1, dz=dz, nu=nu, nv=nv, du=du, dv=dv, u_off=0.6, v_off=-0.35,
                          n_views=views, angles=tuple(0.17 + 2 * np.pi * np.arange(views) / views))


CASES = {
    **{f"nz{nz}": geom(33, 29, nz, 21, 30) for nz in (1, 2, 3, 4, 5, 6, 7, 8, 63, 64, 65)},
    "rows192": geom(30, 30, 20, 9, 192, dv=0.2), "rows193": geom(30, 30, 20, 9, 193, dv=0.2),
    "rows385": geom(30, 30, 20, 9, 385, dv=0.1),
    "box256": geom(20, 18, 256, 9, 60, dz=0.4, dv=2.7), "box257": geom(20, 18, 257, 9, 60, dz=0.4, dv=2.7),
    # traces of about 80, 112 and 160 segments along the axes (views near 0 and 90 degrees)
    **{f"trace{n}": synth.Geometry(nx=n, ny=6, nz=9, dx=0.5, dy=0.5, dz=1.0, nu=9, nv=14, du=0.31, dv=1.0, u_off=0.1,
                                   v_off=0.2, n_views=2, angles=(0.003, np.pi)) for n in (79, 80, 81, 111, 112, 113, 160)},
}


@pytest.mark.parametrize("name", list(CASES))
def test_project_parity_at_table_edges(cb, name):
    g = CASES[name]
    f = synth.random_volume(g, 911)
    with cb.Geometry(g) as h:
        ft = torch.tensor(f, dtype=torch.float32, device="cuda")
        p = cb.project(h, ft).cpu().numpy()
        q = torch.full(g.proj_shape, float("nan"), dtype=torch.float32, device="cuda")
        cb.project_static(h, ft, q)
    ref = oracle.project(g, f)
    assert np.linalg.norm(p - ref) <= 1e-4 * np.linalg.norm(ref)
    assert np.array_equal(p, q.cpu().numpy())


def test_static_projection_of_packed_lines_equals_project(cb):
    """A volume that fits the fixed scratch only without the padding of its z-lines."""
    g = synth.Geometry(nx=1100, ny=1200, nz=3, dx=0.2, dy=0.2, dz=1.0, nu=24, nv=10, du=8.0, dv=0.7, u_off=0.3, n_views=2,
                       angles=(0.2, 1.9))
    assert g.nx * g.ny * g.nz <= 4194304 < g.nx * g.ny * 4
    f = torch.rand(g.vol_shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5))
    with cb.Geometry(g) as h:
        p = cb.project(h, f)
        q = torch.full(g.proj_shape, float("nan"), dtype=torch.float32, device="cuda")
        cb.project_static(h, f, q)
        assert torch.equal(p, q)
