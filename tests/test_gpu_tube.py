"""Sec. V tube flow: a neutral squirmer (R = 9) in a round tube of diameter
D = 20R/3 and length 3 pi R, periodic along the axis (workloads.tube_oscillation).

The boundary-element trajectories the paper compares with are not in its
text, so the run is checked by parity with the FP64 oracle over its first
steps, at full size, and by the mirror symmetry of a start on the axis."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle.oracle import OracleSim  # noqa: E402
from paper_1903_04799_gb300 import Lattice  # noqa: E402
from paper_1903_04799_gb300 import workloads as W  # noqa: E402


def _rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def _gpu(t, storage="f64"):
    b = t.body
    g = Lattice(t.shape, collision="trt", storage=storage)
    tube = g.add_round_tube(t.axis[0], t.axis[1], t.radius)
    gi = g.add_squirmer(b.pos, b.e, b.R, b.B1, b.beta, mobile=True)
    g.set_contact(*t.contact)
    return g, gi, tube


def test_tube_run_first_steps_match_oracle():
    """The paper's configuration at full size (64 x 64 x 85), started at
    y0 = -R: 120 steps in FP64 against the oracle.  Owners bit-exact; fields
    and the squirmer's state within 1e-12."""
    t = W.tube_oscillation(y0_over_R=-1.0)
    b = t.body
    g, gi, _ = _gpu(t)
    o = OracleSim(*t.shape, lambda_e=1.0, collision="trt")
    o.add_tube(t.axis[0], t.axis[1], t.radius)
    oi = o.add_sphere(b.pos, b.e, b.R, b.B1, b.beta, mobile=True)
    o.set_contact(*t.contact)
    for _ in range(3):
        g.step(40)
        o.step(40)
        assert (g.owner() == o.owner()).all()
        _, ug = g.fields()
        _, uo = o.fields()
        assert _rel(ug, uo) < 1e-12
        for a, c in zip(g.state(gi), o.state(oi)):
            assert np.abs(a - c).max() < 1e-12
    g.close()


def test_tube_centred_start_stays_on_the_axis():
    """A squirmer started on the axis, parallel to it: the lattice, the tube
    and the sphere are mirror-symmetric about the planes x = c and y = c
    (c = 31.5, between two nodes), so it must swim along the axis without
    drifting or turning, and its flow must keep the symmetry: after 3000
    FP64 steps the centre stays within 1e-10 of the axis, e within 1e-12 of
    +z, and u_x, u_y odd under the mirror to 1e-12 of max|u|."""
    t = W.tube_oscillation(y0_over_R=0.0)
    g, gi, _ = _gpu(t)
    g.step(3000)
    p, v, e, w = g.state(gi)
    c = np.array(t.axis)
    assert np.abs(p[:2] - c).max() < 1e-10, p
    assert np.abs(e - np.array([0.0, 0.0, 1.0])).max() < 1e-12, e
    assert v[2] > 0.5 * (2 * t.body.B1 / 3)  # it does swim
    _, u = g.fields()
    nx, ny, nz = t.shape
    ux, uy = u[0].reshape(nz, ny, nx), u[1].reshape(nz, ny, nx)
    scale = np.abs(u).max()
    assert np.abs(ux + ux[:, :, ::-1]).max() < 1e-12 * scale
    assert np.abs(uy + uy[:, ::-1, :]).max() < 1e-12 * scale
    assert np.abs(ux - ux[:, ::-1, :]).max() < 1e-12 * scale
    g.close()


@pytest.mark.parametrize("shape,axis,radius", [((23, 21, 5), (11.0, 10.0), 9.3), ((30, 31, 3), (14.6, 15.2), 13.0),
                                               ((12, 12, 4), (5.5, 5.5), 1.4), ((40, 17, 3), (30.2, 8.1), 7.7)])
def test_tube_links_brute_force(shape, axis, radius):
    """The tube's link list, built from the nodes near its wall only, against
    every fluid node with a wall neighbour: wide and narrow tubes (radius below
    the margin: every node is looked at) and an axis off the box's centre."""
    from paper_1903_04799_gb300 import Lattice

    nx, ny, nz = shape
    with Lattice(shape, storage="f32") as g:
        tube = g.add_round_tube(*axis, radius)
        links = set(g.links(tube).tolist())
        wall = (g.owner() == tube).reshape(nz, ny, nx)
    c = np.array([[0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0],
                  [0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1],
                  [0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1]])
    want = set()
    for i in range(1, 19):
        near = np.roll(wall, (-c[2, i], -c[1, i], -c[0, i]), (0, 1, 2))
        want |= {32 * int(n) + i for n in np.flatnonzero((~wall & near).reshape(-1))}
    assert links == want and len(links) > 0


@pytest.mark.parametrize("shape,axis,radius", [((32, 32, 4), (4.0, 16.0), 10.0), ((32, 32, 4), (0.0, 16.0), 10.0),
                                               ((64, 64, 4), (34.0, 32.0), 33.0), ((20, 26, 3), (19.0, 25.0), 8.5)])
def test_tube_links_across_the_periodic_edge(shape, axis, radius):
    """Tubes whose cross-section the box's periodic edge cuts: a fluid node at
    the edge has the nodes across it as neighbours, and those may be wall
    however near the axis the first lies.  The link list against every fluid
    node with a wall neighbour, in cell and direction order."""
    from paper_1903_04799_gb300 import Lattice

    nx, ny, nz = shape
    with Lattice(shape, storage="f32") as g:
        tube = g.add_round_tube(*axis, radius)
        links = g.links(tube).tolist()
        wall = (g.owner() == tube).reshape(nz, ny, nx)
    c = np.array([[0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0],
                  [0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1],
                  [0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1]])
    edge = ~wall & (np.hypot(np.arange(nx)[None, None, :] - axis[0], np.arange(ny)[None, :, None] - axis[1])
                    < radius - 1.5)
    want, crossing = [], 0
    for i in range(1, 19):
        near = ~wall & np.roll(wall, (-c[2, i], -c[1, i], -c[0, i]), (0, 1, 2))
        want += [32 * int(n) + i for n in np.flatnonzero(near.reshape(-1))]
        crossing += int((near & edge).sum())
    assert links == sorted(want) and crossing > 0


@pytest.mark.parametrize("axis,r,pos,e", [((4.0, 16.0), 10.0, (3.4, 15.7, 12.2), (-1.0, 0.1, 0.2)),
                                          ((15.0, 27.0), 10.0, (15.2, 27.6, 11.8), (0.1, 1.0, -0.2)),
                                          ((0.0, 16.0), 20.0, (3.4, 15.7, 12.2), (-1.0, 0.1, 0.2))])
def test_swimmer_at_the_cut_edge_of_a_tube_matches_oracle(axis, r, pos, e):
    """A squirmer that swims at the periodic edge cutting its tube and covers
    nodes whose neighbours across the edge are wall (30 steps, FP64): owners
    and link lists as the oracle's, populations and states within 1e-12."""
    shape, R = (32, 32, 24), 3.0
    g = Lattice(shape, collision="trt")
    o = OracleSim(*shape, lambda_e=1.0, collision="trt")
    g.add_round_tube(*axis, r)
    o.add_tube(*axis, r)
    gi = g.add_squirmer(pos, e, R, 0.05, 0.0, mobile=True)
    oi = o.add_sphere(pos, e, R, 0.05, 0.0, mobile=True)
    first = g.owner()
    edge = np.zeros((24, 32, 32), bool)
    edge[:, :, 0] = edge[:, 31, :] = True
    covered = False
    for _ in range(6):
        g.step(5)
        o.step(5)
        own = g.owner()
        assert (own == o.owner()).all()
        covered |= bool(((own != first) & edge.reshape(-1)).any())
        fluid = own == 0  # solid cells hold nothing in the oracle
        assert _rel(g.populations()[:, fluid], o.populations()[:, fluid]) < 1e-12
        for a, c in zip(g.state(gi), o.state(oi)):
            assert np.abs(a - c).max() < 1e-12
    assert covered  # nodes of the edge changed hands
    g.close()
