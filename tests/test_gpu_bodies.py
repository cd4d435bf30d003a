"""Bodies at the limits of what a lattice takes."""
import ctypes

import numpy as np
import pytest

from paper_2110_00967_gb300 import vplbm as V
from paper_2110_00967_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def lattice(w, **over):
    lat = V.Lattice(V.config_of(w, **over))
    lat.set_body(V.body_of(w))
    return lat


@pytest.mark.parametrize("field", ["x_c", "y_c", "angle"])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_a_body_at_no_finite_place_is_refused(field, value):
    """Placed, or in a snapshot's header: EINVAL, and the lattice goes on as it was."""
    w = W.naca(5.0, dtype="f32", nx=512, ny=256)
    lat, twin = lattice(w), lattice(w)
    lat.step(3)
    bad = V.body_of(w)
    setattr(bad, field, value)
    with pytest.raises(V.VplbmError) as e:
        V.vplbm_set_body(lat.ctx, bad)
    assert e.value.status == V.EINVAL
    snap = lat.save_state()
    at = 16 + ctypes.sizeof(V.vplbm_config) + getattr(V.vplbm_body, field).offset
    assert snap[at:at + 8].view(np.float64)[0] == getattr(V.body_of(w), field)
    snap[at:at + 8].view(np.float64)[0] = value
    with pytest.raises(V.VplbmError) as e:
        lat.load_state(snap)
    assert e.value.status == V.EINVAL
    lat.step(4)
    twin.step(7)
    np.testing.assert_array_equal(lat.get_f(), twin.get_f())
    np.testing.assert_array_equal(lat.history(V.MEM, 7), twin.history(V.MEM, 7))


@pytest.mark.parametrize("field,value", [("x_c", 5.0), ("y_c", 1e9), ("length", 1e9), ("length", 600.0)])
def test_a_snapshot_of_a_body_beyond_the_lattice_is_refused(field, value):
    """No such body can have been placed: EINVAL, and the lattice goes on as it was."""
    w = W.naca(5.0, dtype="f32", nx=512, ny=256)
    lat, twin = lattice(w), lattice(w)
    lat.step(3)
    snap = lat.save_state()
    at = 16 + ctypes.sizeof(V.vplbm_config) + getattr(V.vplbm_body, field).offset
    snap[at:at + 8].view(np.float64)[0] = value
    with pytest.raises(V.VplbmError) as e:
        lat.load_state(snap)
    assert e.value.status == V.EINVAL
    lat.step(4)
    twin.step(7)
    np.testing.assert_array_equal(lat.get_f(), twin.get_f())


@pytest.mark.parametrize("dtype", ["f64", "f32", "f16"])
@pytest.mark.parametrize("length", [0.0, 20.0])
def test_an_empty_lattice_has_nothing_to_move(dtype, length):
    """kind NONE with the moving flag set (a length, a density ratio and gravity beside
    it): the flow of an empty lattice, no mask, no force, no instability."""
    w = W.Workload(name="none", nx=401, ny=263, dtype=dtype, collision="trt", tau_plus=0.6, u_in=(0.04, 0.01),
                   bc=("inlet", "outlet", "symmetry", "symmetry"), body=W.Body("none"), steps=1)
    odd = V.body_of(w)
    odd.moving, odd.length, odd.x_c, odd.y_c, odd.density_ratio = 1, length, 200.0, 130.0, 1.5
    odd.gravity[1] = -1e-4
    lat, twin = V.Lattice(V.config_of(w)), lattice(w)
    lat.set_body(odd)
    f = W.random_field(5, (9, w.ny, w.nx), lo=0.10, hi=0.12)
    for x in (lat, twin):
        x.set_state(f, f, post_collision=False)
        x.step(1)
        x.step(6)
        x.check()
    np.testing.assert_array_equal(lat.get_f(), twin.get_f())
    assert not lat.get_mask().any()
    assert not lat.history(V.MEM, 7).any()


def test_a_large_disk_moving_onto_one_more_column_of_tiles():
    """A disk whose box covers 16 columns of tiles where it is placed and 17 a step later
    (16,388 tiles): every node of the box is updated.  The same steps are taken by a
    lattice set to each level's populations before its step, which updates every tile
    of the lattice."""
    body = W.Body("disk", length=1918.0, x_c=1084.0, y_c=980.0, moving=True, density_ratio=50.0, n_sim_points=1000)
    w = W.Workload(name="wide", nx=2112, ny=1960, dtype="f32", collision="trt", tau_plus=0.7, u_in=(0.0, 0.0),
                   bc=("noslip",) * 4, body=body, steps=1)
    b = V.body_of(w)
    b.u[0] = 0.2
    runs, whole = V.Lattice(V.config_of(w)), V.Lattice(V.config_of(w))
    f = W.random_field(5, (9, w.ny, w.nx), lo=0.10, hi=0.12)
    for lat in (runs, whole):
        lat.set_body(b)
        lat.set_state(f, f, post_collision=False)
    for _ in range(5):
        runs.step(1)
        whole.step(1)
        f = runs.get_f()
        # offsets of up to 0.4 read back and set again: one unit of FP32 at most
        np.testing.assert_allclose(f, whole.get_f(), rtol=0, atol=2.0 ** -22)
        np.testing.assert_allclose(runs.get_body(), whole.get_body(), rtol=1e-9, atol=1e-9)
        whole.set_state(f, f, post_collision=False)
    assert runs.get_body()[0] > 1084.5
    runs.check()
