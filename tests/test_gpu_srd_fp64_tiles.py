"""The FP64 SRD kernel with integer members (GPU, against the oracle) where its
tiling and its number format can go wrong: every width of the sub-tile, the
longest row it takes (112 records) and one beyond, ragged boxes and a box large
enough for 32 cells a warp; velocities of very different and very large or small
size within a cell (the shared exponent), a cell at rest, and the double path
(exponents beyond the integers' range, overflowing rows).

Tolerance: velocities |dv| / max(|v|, scale) <= 1e-12 with scale the largest
speed of the box, as the shared exponent resolves it to 2^-59 and each step
rounds a handful of times at 2^-53; cells exact."""
import numpy as np
import pytest

import oracle
from paper_1801_10187_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1801_10187_gb300 as pkg  # noqa: E402


def compare(n, pos, vel, steps, kT=1.0, **kw):
    box = pkg.Box(n=n, precision="fp64", kT=kT, **kw)
    box.set_state(pos, vel, step=5)
    box.step(steps)
    p, v, _, _, st = box.get_state()
    cells, counts = box.last_cells()
    box.close()
    g = kw.pop("body_force", (0.0, 0.0, 0.0))
    ref = oracle.State(pos.copy(), vel.copy(), step=5)
    rc, rk = oracle.step(oracle.Params(n=n, precision=oracle.FP64, kT=kT, g=g, **kw), ref, steps,
                         want_cells=True)
    assert st == ref.step
    np.testing.assert_array_equal(cells, rc)
    np.testing.assert_array_equal(counts, rk)
    scale = np.abs(ref.vel).max(initial=0.0)
    assert np.abs(v - ref.vel).max(initial=0.0) <= 1e-12 * scale
    d = np.abs(p - ref.pos)
    assert np.minimum(d, np.array(n, dtype=float) - d).max(initial=0.0) <= 1e-12 * max(max(n), scale)


CASES = [((5, 3, 2), 1), ((7, 5, 3), 3), ((23, 17, 9), 5), ((9, 4, 5), 10), ((9, 4, 5), 11),
         ((6, 5, 4), 21), ((6, 5, 4), 40), ((4, 3, 3), 58), ((4, 3, 3), 60), ((40, 40, 50), 3)]


@pytest.mark.parametrize("thermostat", [False, True])
@pytest.mark.parametrize("n,rho", CASES)
def test_sub_tiles_match_the_oracle(n, rho, thermostat):
    s = inputs.solvent(n, rho, seed=rho + 3)
    compare(n, s.pos, s.vel, 3, seed=rho + 3, thermostat=thermostat, body_force=(0.01, -0.02, 0.03))


@pytest.mark.parametrize("thermostat", [False, True])
@pytest.mark.parametrize("scale", [1e-200, 1e-9, 1.0, 3e5])
def test_velocity_scales(scale, thermostat):
    n = (6, 5, 4)
    s = inputs.solvent(n, 6, seed=4)
    compare(n, s.pos, s.vel * scale, 1, seed=4, thermostat=thermostat, kT=max(scale * scale, 1e-300))


def test_mixed_scales_and_rest():
    n = (6, 5, 4)
    s = inputs.solvent(n, 6, seed=8)
    rng = np.random.default_rng(1)
    vel = s.vel * 10.0 ** rng.uniform(-12, 2, (len(s.vel), 1))
    vel[s.pos[:, 0] < 2.0] = 0.0
    compare(n, s.pos, vel, 2, seed=8)
    compare(n, s.pos, np.zeros_like(vel), 2, seed=8)


def test_exponents_beyond_the_integers_and_overflowing_rows():
    n = (4, 4, 4)
    s = inputs.solvent(n, 6, seed=9)
    compare(n, s.pos, s.vel * 1e-290, 1, seed=9)  # below 2^-900
    pos = s.pos.copy()
    pos[:200] = 1.3 + 0.4 * np.random.default_rng(2).random((200, 3))  # one cell, a full row and more
    compare(n, pos, s.vel, 1, seed=9, thermostat=True)


@pytest.mark.parametrize("thermostat", [False, True])
@pytest.mark.parametrize("n,rho", [((8, 6, 5), 6), ((23, 17, 9), 2), ((4, 3, 3), 58)])
@pytest.mark.parametrize("fast", [1e6, 1e9, 1e12, 1e18])
def test_a_fast_particle_costs_no_other_cell_precision(fast, n, rho, thermostat):
    """One particle `fast` times faster than the rest, in one cell: every particle within the
    parity bound of its own cell, 1e-12 of the largest speed that the cell's members had or got
    (a collision rounds a handful of times at 2^-53 of that), and a particle alone in its
    cell keeps its velocity to the bit, small components beside large ones included."""
    s = inputs.solvent(n, rho, seed=21)
    vel = s.vel.copy()
    vel[::5, 1] *= 1e-14
    vel[0] *= fast / np.linalg.norm(vel[0])
    box = pkg.Box(n=n, seed=21, precision="fp64", thermostat=thermostat)
    box.set_state(s.pos, vel, step=5)
    box.step(1)
    p, v, _, _, _ = box.get_state()
    cells, counts = box.last_cells()
    box.close()
    ref = oracle.State(s.pos.copy(), vel.copy(), step=5)
    rc, rk = oracle.step(oracle.Params(n=n, seed=21, precision=oracle.FP64, thermostat=thermostat), ref, 1,
                         want_cells=True)
    np.testing.assert_array_equal(cells, rc)
    np.testing.assert_array_equal(counts, rk)
    np.testing.assert_array_equal(p, ref.pos)
    speed = np.maximum(np.linalg.norm(vel, axis=1), np.linalg.norm(ref.vel, axis=1))
    largest = np.zeros(len(rk))
    np.maximum.at(largest, rc, speed)
    assert (np.linalg.norm(v - ref.vel, axis=1) / largest[rc]).max() <= 1e-12
    lone = rk[rc] == 1
    assert lone.any() or rho > 10
    np.testing.assert_array_equal(v[lone], vel[lone])


@pytest.mark.parametrize("thermostat", [False, True])
@pytest.mark.parametrize("rho", [7, 12, 18, 36, 58])
def test_sub_tiles_that_may_not_fit(rho, thermostat):
    """Sub-tiles of 32 cells a warp that take up to 16, 8, 4 or 2 cells (mean 96 to 146 of 112 members):
    what does not fit waits for the next, which starts at any cell."""
    n = (31, 32, 31)
    s = inputs.solvent(n, rho, seed=rho)
    compare(n, s.pos, s.vel, 2, seed=rho, thermostat=thermostat)
