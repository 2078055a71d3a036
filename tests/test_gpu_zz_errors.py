"""Failure detection on the GPU without a GPU fault: a state the scheme cannot
carry (NaN populations, injected from the host) is caught by the body update
on the device, reported at the next synchronising call as LB_ERR_DIVERGED,
and the context then refuses to step (LB_ERR_STATE).  The diverged body is
held in place, so no kernel indexes from a runaway position."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_04799_gb300 import Lattice  # noqa: E402
from paper_1903_04799_gb300.lbsq import LB_ERR_DIVERGED, LB_ERR_STATE, LBError  # noqa: E402


@pytest.mark.parametrize("shape,pos,R", [((28, 26, 30), (13.3, 12.7, 14.1), 4.5),
                                         ((128, 96, 96), (64.3, 40.7, 50.1), 6.0)])
def test_nan_state_is_reported_as_divergence(shape, pos, R):
    """The second lattice splits its steps (near window, pending body step)."""
    g = Lattice(shape, collision="trt", storage="f64")
    gi = g.add_squirmer(pos, (0.3, -0.4, 1.0), R, 0.03, -2.0, mobile=True)
    g.step(5)
    f = g.populations()
    f[:] = np.nan
    g.set_populations(f)
    g.step(3)
    with pytest.raises(LBError) as ei:
        g.state(gi)
    assert ei.value.status == LB_ERR_DIVERGED
    with pytest.raises(LBError) as ei:
        g.step(1)
    assert ei.value.status == LB_ERR_STATE
    g.close()


def test_force_that_the_links_hold_back_is_no_divergence():
    """Two light spheres pushed apart so hard that in some steps the contact
    and conversion forces alone would take them past |v| = 1/2, where the
    drag of the links keeps them below (on the oracle: at most 0.43, and 0.51
    without the links' force).  The fused kernel runs its update on scratch
    without the links' force, which must not report divergence.  States as the
    oracle's to 1e-9 (8 steps at |v| of order 1)."""
    from oracle.oracle import OracleSim

    shape, R, gap = (24, 24, 72), 3.2, 10.0
    put = [((14.2, 13.8, 36.0 - R - gap / 2), (0.0, 0.0, -1.0)), ((14.3, 13.9, 36.1 + R + gap / 2), (0.0, 0.0, 1.0))]
    g = Lattice(shape, collision="trt", storage="f64")
    o = OracleSim(*shape, lambda_e=1.0, collision="trt")
    gi = [g.add_squirmer(p, e, R, 0.0, 0.0, mobile=True) for p, e in put]
    oi = [o.add_sphere(p, e, R, 0.0, 0.0, mobile=True) for p, e in put]
    g.set_contact(12.0, 1.9)
    o.set_contact(12.0, 1.9)
    mass, most = 4.0 / 3.0 * np.pi * R ** 3, 0.0
    for _ in range(8):
        booked = [o.pending_conversion(i)[0] for i in oi]
        g.step(1)
        o.step(1)
        for a, b, f0 in zip(gi, oi, booked):
            for x, y in zip(g.state(a), o.state(b)):
                assert np.abs(x - y).max() < 1e-9
            most = max(most, np.linalg.norm(o.state(b)[1] - (o.force_torque(b)[0] - f0) / mass))
    assert most > 0.505  # the scratch update does leave the scheme
    g.close()
