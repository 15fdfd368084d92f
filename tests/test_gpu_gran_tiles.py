"""The tiled granulation kernels at the edges of their range, against the
oracle: the widest disk they take (16 pixels) and the next one (plain
kernels), a plane one tile wide, disks of unequal extent in x and y, ties
that take many batches of rounds."""
import numpy as np
import pytest

import inputs
from oracle.granulation import GranParams, Granulation as OracleGran

pytestmark = pytest.mark.gpu

BASE = dict(v0=1.0, vmin_frac=0.78, lifetime=300.0, lifetime_spread=0.10, amp_spread=0.15, f_rot=5.0)


# FP64 on both sides in different orders: 1e-12 of the field's maximum, as in
# the driver's other tests; radii half a pixel off the lattice keep every disk
# decision away from rounding
@pytest.mark.parametrize("nx,ny,dx,dy,ri,rg,rl", [
    (64, 64, 1.0, 1.0, 2.55, 9.3, 16.45), (64, 64, 1.0, 1.0, 2.55, 9.3, 17.45),
    (32, 8, 1.0, 1.0, 1.35, 2.2, 3.45), (32, 128, 1.0, 0.25, 2.05, 2.6, 3.45), (16, 64, 1.0, 1.0, 1.35, 2.2, 3.45),
    (128, 16, 0.5, 1.0, 0.3, 0.8, 2.3)])
def test_tiles_match_the_oracle(nx, ny, dx, dy, ri, rg, rl):
    from paper_1908_08557_gb300 import Granulation
    gp = dict(BASE, r_inner=ri, r_granule=rg, r_lane=rl)
    gen, ref = Granulation(nx, ny, dx, dy, gp), OracleGran(nx, ny, dx, dy, GranParams(**gp))
    for u, t in enumerate((0.0, 150.0, 290.0, 420.0)):
        d = inputs.granulation_draws(nx, ny, seed=21, update=u)
        gen.update(t, *d)
        ref.update(t, *d)
        occ, par = gen.granules()
        o_occ, o_par = ref.maps()
        assert np.array_equal(occ.cpu().numpy(), o_occ)
        np.testing.assert_allclose(par.cpu().numpy(), o_par, rtol=1e-14, atol=0)
    v = gen.velocity(430.0, precision=64).cpu().numpy()
    w = np.stack(ref.velocity(430.0))
    assert np.abs(v - w).max() <= 1e-12 * np.abs(w).max()


def test_ties_take_many_rounds():
    from paper_1908_08557_gb300 import Granulation
    gp = dict(BASE, r_inner=1.6, r_granule=2.0, r_lane=3.45)
    gen, ref = Granulation(64, 32, 1.0, 1.0, gp), OracleGran(64, 32, 1.0, 1.0, GranParams(**gp))
    keys = np.full((32, 64), 7, np.uint32)
    _, cl, ca = inputs.granulation_draws(64, 32, seed=2)
    rounds = gen.update(0.0, keys, cl, ca)
    ref.update(0.0, keys, cl, ca)
    assert rounds > 8
    assert np.array_equal(gen.granules()[0].cpu().numpy(), ref.maps()[0])
