"""Two steps per launch (fixed bodies on larger lattices): runs replayed from step
graphs, which take their steps in pairs, end bit-identical -- populations, force
histories, running sums -- to the same lattice stepped one step per call, over the
storage forms, side conditions, body kinds, SIM orders, launch forms and the ragged
sizes at which strips, row runs and tiles end."""
import numpy as np
import pytest

from paper_2110_00967_gb300 import vplbm as V
from paper_2110_00967_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the GPU tests need a CUDA device"
    V.lib()
    yield


def run_both(w, lengths, variant=None, start=None, **over):
    """The workload stepped in runs of the given lengths and one step per call."""
    lats = []
    for _ in range(2):
        lat = V.Lattice(V.config_of(w, **over))
        lat.set_body(V.body_of(w))
        if variant is not None:
            lat.bulk_variant = variant
        if start is not None:
            lat.set_state(start, start, post_collision=True)
        lats.append(lat)
    runs, single = lats
    launches = []
    for n in lengths:
        l0 = runs.launches
        runs.step(n)
        launches.append(runs.launches - l0)
    total = sum(lengths)
    for _ in range(total):
        single.step(1)
    np.testing.assert_array_equal(runs.get_f(), single.get_f())
    for est in (V.MEM, V.SIM, V.ANGOT):
        np.testing.assert_array_equal(runs.history(est, total), single.history(est, total))
    for a, b in zip(runs.sums(), single.sums()):
        np.testing.assert_array_equal(a, b)
    assert runs.steps == single.steps == total
    runs.check()
    return launches


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16", "f16sr", "bf16sr"])
@pytest.mark.parametrize("force", [False, True])
def test_airfoil_runs_equal_single_steps(dtype, force):
    w = W.naca(9.0, dtype=dtype, nx=517, ny=263)
    w = w.with_(body_force=(1e-6, -2e-6) if force else (0.0, 0.0))
    launches = run_both(w, (1, 2, 7, 32, 5))
    # 32 steps are 16 launches and one that finalizes the forces
    assert launches[3] == 16 + 1


# strips of 60 nodes between the two outermost columns on either side: widths one
# below, at and one above their multiples, a narrow and a low lattice
SIZES = [(4 * 60 + 4, 2 * 62 + 4 + 300), (4 * 60 + 5, 433), (8 * 60 + 3, 16 * 14 + 4), (62 * 8, 16 * 14 + 5),
         (62 * 8 + 1, 16 * 14 + 3), (2 * 480 + 4, 128), (1500, 70), (67, 1571)]


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("shape", SIZES)
def test_ragged_sizes(dtype, shape):
    nx, ny = shape
    body = W.Body("disk", length=15.0, x_c=min(0.4 * nx, 70.3), y_c=0.5 * ny + 0.2)
    w = W.Workload(name="ragged", nx=nx, ny=ny, dtype=dtype, collision="trt", tau_plus=0.6, u_in=(0.04, 0.0),
                   bc=("inlet", "outlet", "symmetry", "symmetry"), body=body, steps=1, u_ref=(0.04, 0.0))
    run_both(w, (1, 4, 3))


# rows per warp 5, 6 and 8 (by the lattice's size): a last run of one row, of a full
# run and of all but one row, and 0, 2 and 3 warps in the last block of four
RUNS = [(514, 5 * 41 + 5), (490, 5 * 43 + 4), (424, 5 * 48 + 8), (724, 6 * 93 + 5), (904, 8 * 97 + 5)]


@pytest.mark.parametrize("dtype", ["f32", "f16sr"])
@pytest.mark.parametrize("shape", RUNS)
def test_last_runs_and_warps(dtype, shape):
    nx, ny = shape
    body = W.Body("disk", length=17.0, x_c=80.4, y_c=0.5 * ny - 0.3)
    w = W.Workload(name="runs", nx=nx, ny=ny, dtype=dtype, collision="trt", tau_plus=0.6, u_in=(0.04, 0.0),
                   bc=("inlet", "outlet", "symmetry", "symmetry"), body=body, steps=1, u_ref=(0.04, 0.0))
    run_both(w, (1, 4, 2))


BCS = [("periodic", "periodic", "periodic", "periodic"), ("periodic", "periodic", "noslip", "noslip"),
       ("inlet", "outlet_free", "noslip", "noslip"), ("noslip", "noslip", "periodic", "periodic"),
       ("inlet", "noslip", "symmetry", "noslip"), ("inlet", "outlet", "periodic", "periodic")]


@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("kind", ["none", "disk"])
def test_side_conditions_from_a_random_state(bc, kind):
    """From random populations, so that every edge carries a signal."""
    nx, ny = 401, 259
    body = W.Body("none") if kind == "none" else W.Body("disk", length=21.0, x_c=200.0, y_c=129.0)
    w = W.Workload(name="sides", nx=nx, ny=ny, dtype="f32", collision="trt", tau_plus=0.7, u_in=(0.03, 0.01),
                   bc=bc, body=body, steps=1, u_ref=(0.02, 0.01))
    start = W.random_field(5, (9, ny, nx), lo=0.10, hi=0.12)
    run_both(w, (2, 6, 1, 4), start=start)


@pytest.mark.parametrize("over", [{"sim_order": 1}, {"sim_every": 0}])
def test_sim_options(over):
    run_both(W.naca(4.0, dtype="f32", nx=512, ny=256), (1, 9, 4), **over)


@pytest.mark.parametrize("variant", [0, 1, 2])
@pytest.mark.parametrize("dtype", ["f32", "f16sr"])
def test_launch_forms(variant, dtype):
    run_both(W.naca(12.0, dtype=dtype, nx=700, ny=301), (1, 8, 3), variant=variant)


@pytest.mark.parametrize("x,y", [(20.0, 130.0), (250.0, 21.0), (24.0, 24.0), (480.5, 239.0)])
def test_bodies_next_to_the_edges(x, y):
    """A body near the edges: within the clearance of the pair kernels the box comes
    close to the frame; nearer, the lattice is stepped singly."""
    body = W.Body("disk", length=17.0, x_c=x, y_c=y)
    w = W.Workload(name="near", nx=517, ny=263, dtype="f32", collision="trt", tau_plus=0.6, u_in=(0.04, 0.0),
                   bc=("inlet", "outlet", "noslip", "noslip"), body=body, steps=1, u_ref=(0.04, 0.0))
    run_both(w, (1, 6, 3))


def test_snapshot_between_pairs():
    """A snapshot taken in the middle of a run and restored into another lattice
    continues bit for bit, in pairs."""
    w = W.naca(6.0, dtype="f32", nx=512, ny=256)
    a = V.Lattice(V.config_of(w))
    a.set_body(V.body_of(w))
    a.step(13)
    snap = a.save_state()
    b = V.Lattice(V.config_of(w))
    b.load_state(snap)
    for lat in (a, b):
        lat.step(21)
    np.testing.assert_array_equal(a.get_f(), b.get_f())
    np.testing.assert_array_equal(a.history(V.SIM, 34), b.history(V.SIM, 34))


def test_batch_of_lattices_stepped_in_pairs_and_singly():
    """A prepared batch call of 10 steps moves a lattice stepped in pairs to its other
    buffer and one stepped singly not: repeated calls still equal lone lattices."""
    works = [W.naca(7.0, dtype="f32", nx=512, ny=256), W.naca(7.0, dtype="f32", nx=256, ny=128)]

    def make():
        out = []
        for w in works:
            lat = V.Lattice(V.config_of(w))
            lat.set_body(V.body_of(w))
            out.append(lat)
        return out

    members, alone = make(), make()
    batch = V.Batch(members)
    batch.step(1)
    batch.prepare(10)
    for n in (10, 10, 3, 10, 10):
        batch.step(n)
    batch.close()
    for a, m in zip(alone, members):
        a.step(44)
        np.testing.assert_array_equal(a.get_f(), m.get_f())
        np.testing.assert_array_equal(a.history(V.MEM, 44), m.history(V.MEM, 44))


@pytest.mark.parametrize("count, per_lattice", [(7, 4 + 1), (8, 2 * 8 + 1)])
def test_sixteen_bit_batches_pair_up_to_their_nodes_and_lattices(count, per_lattice):
    """16-bit lattices of 448 x 256 nodes: seven together step in pairs, eight do not
    (each lattice weighs its nodes and a constant); the results are the same."""
    works = [W.naca(2.0 * k, dtype="f16", nx=448, ny=256) for k in range(count)]
    lats = [V.Lattice(V.config_of(w)) for w in works]
    for lat, w in zip(lats, works):
        lat.set_body(V.body_of(w))
    batch = V.Batch(lats)
    batch.step(1)
    before = [lat.launches for lat in lats]
    batch.step(8)
    assert [lat.launches - b for lat, b in zip(lats, before)] == [per_lattice] * count
    for lat, w in list(zip(lats, works))[:2]:
        alone = V.Lattice(V.config_of(w))
        alone.set_body(V.body_of(w))
        for _ in range(9):
            alone.step(1)
        np.testing.assert_array_equal(lat.get_f(), alone.get_f())
        for est in (V.MEM, V.SIM):
            np.testing.assert_array_equal(lat.history(est, 9), alone.history(est, 9))
    batch.close()


@pytest.mark.parametrize("history_len", [1, 2, 3])
def test_short_force_histories(history_len):
    """A history of one row, of a pair's two, and of three: after every run the last
    steps' forces are those of a lattice stepped one step per call."""
    w = W.naca(9.0, dtype="f32", nx=517, ny=263)
    runs, single = (V.Lattice(V.config_of(w, history_len=history_len)) for _ in range(2))
    for lat in (runs, single):
        lat.set_body(V.body_of(w))
    for n in (1, 2, 6, 5, 32):
        runs.step(n)
        for _ in range(n):
            single.step(1)
        keep = min(history_len, runs.steps)
        for est in (V.MEM, V.SIM, V.ANGOT):
            np.testing.assert_array_equal(runs.history(est, keep), single.history(est, keep))
        np.testing.assert_array_equal(runs.force_mem(), single.force_mem())
        np.testing.assert_array_equal(runs.force_sim(), single.force_sim())
        np.testing.assert_array_equal(runs.force_angot(), single.force_angot())
        for a, b in zip(runs.sums(), single.sums()):
            np.testing.assert_array_equal(a, b)


# rows per warp 20, as batches of more than four million FP32 nodes take them: a last
# run of 20, one and 19 rows, and two, three and one warps in the last block of four
LARGE = [(2044, 20 * 51 + 4), (1500, 20 * 50 + 5), (2084, 20 * 38 + 23)]


def test_large_batches_equal_single_steps():
    works = [W.naca(4.0 + 5 * k, dtype="f32", nx=nx, ny=ny) for k, (nx, ny) in enumerate(LARGE)]
    members, alone = ([V.Lattice(V.config_of(w)) for w in works] for _ in range(2))
    for lats in (members, alone):
        for lat, w in zip(lats, works):
            lat.set_body(V.body_of(w))
    batch = V.Batch(members)
    batch.step(1)
    batch.prepare(8)
    before = [m.launches for m in members]
    for n in (8, 3, 8):
        batch.step(n)
    # four launches and one that finalizes for 8 steps; one pair, one step and their
    # finalizing launches for 3
    assert [m.launches - b for m, b in zip(members, before)] == [5 + 2 + 3 + 5] * len(LARGE)
    batch.close()
    for a, m in zip(alone, members):
        for _ in range(20):
            a.step(1)
        np.testing.assert_array_equal(a.get_f(), m.get_f())
        for est in (V.MEM, V.SIM, V.ANGOT):
            np.testing.assert_array_equal(a.history(est, 20), m.history(est, 20))
        for p, q in zip(a.sums(), m.sums()):
            np.testing.assert_array_equal(p, q)


# frame tiles of 30 nodes along the rows and along the columns between them: sizes at,
# one above and one below their multiples
FRAMES = [(30 * 14, 30 * 10 + 4), (30 * 14 + 1, 30 * 10 + 5), (30 * 14 + 29, 30 * 10 + 33)]


@pytest.mark.parametrize("length", range(15, 29))
def test_ends_of_frame_and_box_tiles(length):
    """Box tiles of 14 x 6 nodes around disks of fourteen sizes, so that the last tile
    of either direction is of every size; frame tiles in turn."""
    nx, ny = FRAMES[length % 3]
    body = W.Body("disk", length=float(length), x_c=90.3, y_c=0.5 * ny + 0.2)
    w = W.Workload(name="tiles", nx=nx, ny=ny, dtype="f32" if length % 2 else "f16sr", collision="trt",
                   tau_plus=0.6, u_in=(0.04, 0.0), bc=("inlet", "outlet", "symmetry", "noslip"), body=body,
                   steps=1, u_ref=(0.04, 0.0))
    start = W.random_field(length, (9, ny, nx), lo=0.10, hi=0.12)
    run_both(w, (1, 4, 3), start=start)
