"""The mixed SRD kernel at the edges of its tiling (GPU, bit-exact against the
oracle).  A warp owns 4 to 32 cells by the size of the box and takes them in
sub-tiles of 1 to 32 cells by the density, with at most 192 members: densities
on both sides of every change of the sub-tile, rows of 188 and 192 records (the
longest it takes) and of 196 (the warp-spread kernel), ragged boxes whose last
warp and block are partly or wholly beyond the grid, and a box large enough for
32 cells a warp.  Beads in sub-tiles of two cells, and a body force."""
import numpy as np
import pytest

import oracle
from paper_1801_10187_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1801_10187_gb300 as pkg  # noqa: E402

CASES = [((5, 3, 2), 1), ((7, 5, 3), 5), ((23, 17, 9), 6), ((9, 4, 5), 10), ((9, 4, 5), 13),
         ((6, 5, 4), 21), ((6, 5, 4), 36), ((4, 4, 3), 79), ((3, 3, 2), 90), ((3, 2, 2), 118),
         ((3, 2, 2), 121), ((3, 2, 2), 122), ((40, 40, 50), 3), ((41, 39, 53), 5)]


@pytest.mark.parametrize("thermostat", [False, True])
@pytest.mark.parametrize("n,rho", CASES)
def test_sub_tiles_match_the_oracle(n, rho, thermostat):
    s = inputs.solvent(n, rho, seed=rho + 3, mixed=True)
    kw = dict(n=n, seed=rho + 3, thermostat=thermostat)
    box = pkg.Box(precision="mixed", body_force=(0.01, -0.02, 0.03), **kw)
    box.set_state(s.pos, s.vel, step=7)
    box.step(3)
    pos, vel, _, _, step = box.get_state()
    cells, counts = box.last_cells()
    box.close()
    ref = oracle.State(s.pos.copy(), s.vel.copy(), step=7)
    rc, rk = oracle.step(oracle.Params(precision=oracle.MIXED, g=(0.01, -0.02, 0.03), **kw), ref, 3,
                         want_cells=True)
    assert step == ref.step
    np.testing.assert_array_equal(cells, rc)
    np.testing.assert_array_equal(counts, rk)
    np.testing.assert_array_equal(pos, ref.pos)
    np.testing.assert_array_equal(vel, ref.vel)


def test_beads_in_narrow_sub_tiles():
    n, rho = (5, 4, 4), 70
    s = inputs.solvent(n, rho, seed=9, mixed=True)
    sp, sv = inputs.chains(n, 12, 10, 0.5, bead_mass=5.0, seed=10)
    kw = dict(n=n, seed=9, thermostat=True, chain_len=10, md_substeps=4, solute_mass=5.0, bond_k=300.0,
              bond_r0=0.5)
    box = pkg.Box(precision="mixed", **kw)
    box.set_state(s.pos, s.vel, sp, sv)
    box.step(2)
    got = box.get_state()
    box.close()
    ref = oracle.State(s.pos.copy(), s.vel.copy(), sp.copy(), sv.copy())
    oracle.step(oracle.Params(precision=oracle.MIXED, **kw), ref, 2)
    np.testing.assert_array_equal(got[0], ref.pos)
    np.testing.assert_array_equal(got[1], ref.vel)
    np.testing.assert_allclose(got[2], ref.spos, rtol=0, atol=1e-10)
    np.testing.assert_allclose(got[3], ref.svel, rtol=0, atol=1e-10 * max(1.0, np.abs(ref.svel).max()))
