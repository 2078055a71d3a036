"""Density, velocity and total mass / momentum read-outs against exactly rounded host sums.

The kernels sum deviations in 64-bit fixed point (unit 2^-60 of rho0) and take FP64 sums where a
deviation leaves the fixed-point range; both are compared with math.fsum over the populations the
library exports, on lattices with edges 1 and odd edges, on both parities, for every storage.

Tolerances: an exported population carries one rounding (2^-53 of itself), FP64 sums of 19 terms at
most 19 roundings of the gross sum, so |rho - fsum f| and |j - fsum f c| stay below
2^-53 (2 * 19) sum |f| < 2^-47 sum |f|; u = j / rho adds four roundings of u.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1903_04799_gb300 import Lattice  # noqa: E402

C = np.array([[0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0],
              [0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1],
              [0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1]], dtype=np.float64)
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _check(g, rho0, inc):
    f = g.populations()
    rho, u = g.fields()
    mass, mom = g.mass()
    fluid = g.owner() == 0
    gross = np.abs(f).sum(0)
    r = np.array([math.fsum(c) for c in f.T])
    j = np.array([[math.fsum(C[a] * c) for c in f.T] for a in range(3)])
    den = rho0 if inc else r
    tol = 2.0 ** -47 * gross
    assert (np.abs(rho - r)[fluid] <= tol[fluid]).all()
    assert (np.abs(u - j / den)[:, fluid] <= (tol / np.abs(den) + 2.0 ** -51 * np.abs(j / den))[:, fluid]).all()
    assert (rho[~fluid] == 0).all() and (u[:, ~fluid] == 0).all()
    total = 2.0 ** -47 * gross[fluid].sum()
    assert abs(mass - math.fsum(r[fluid])) <= total
    for a in range(3):
        assert abs(mom[a] - math.fsum(j[a][fluid])) <= total


@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("shape,rho0,inc,spread", [
    ((1, 1, 1), 1.0, False, 0.1),
    ((3, 1, 2), 1.0, False, 0.1),
    ((17, 5, 3), 1.0, True, 0.1),
    ((17, 16, 9), 1.9, False, 0.3),
    ((33, 7, 11), 0.03, False, 0.05),
    ((19, 8, 6), 1.0, False, 3.0),  # some cells outside the fixed-point range
])
def test_fields_and_totals(storage, shape, rho0, inc, spread):
    n = math.prod(shape)
    rng = np.random.default_rng(n)
    f = rho0 * W[:, None] * (1.0 + spread * rng.uniform(-0.3, 1.0, (19, n)))
    with Lattice(shape, collision="trt", storage=storage, rho0=rho0,
                 equilibrium="incompressible" if inc else "compressible") as g:
        if min(shape) >= 3:
            g.add_plane_wall(2, 1)  # solid cells read as zero
        g.set_populations(f)
        _check(g, rho0, inc)  # even parity
        g.step(1)
        _check(g, rho0, inc)  # odd parity


@pytest.mark.parametrize("offset", [0, 8, 72])
def test_large_read_out_into_fresh_and_existing_pages(offset):
    """A read-out of 23 MB (five blocks and a part, no whole number of pages) into
    a buffer whose pages do not exist yet, at several alignments, against one
    into a buffer that has been written: the same bytes, and none outside."""
    import mmap

    from paper_1903_04799_gb300 import lbsq

    shape = (61, 47, 53)
    n = math.prod(shape)
    f = W[:, None] * (1.0 + 0.05 * np.random.default_rng(3).uniform(-1, 1, (19, n)))
    with Lattice(shape, storage="f64") as g:
        g.set_populations(f)
        lib = lbsq.load()
        warm = np.ones(19 * n)
        lbsq._check(g.ctx, lib.lb_get_populations(g.ctx, lbsq._dp(warm)), "lb_get_populations")
        m = mmap.mmap(-1, 19 * n * 8 + (1 << 20))
        fresh = np.frombuffer(m, dtype=np.float64, count=19 * n, offset=offset)
        lbsq._check(g.ctx, lib.lb_get_populations(g.ctx, lbsq._dp(fresh)), "lb_get_populations")
        assert np.array_equal(fresh, warm)
        rest = np.frombuffer(m, dtype=np.uint8)
        assert not rest[:offset].any() and not rest[offset + 19 * n * 8:].any()
        assert np.abs(warm.reshape(19, n) - f).max() < 1e-16  # two roundings of at most 2^-54
