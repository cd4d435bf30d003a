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
