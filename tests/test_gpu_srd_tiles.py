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


RULES = [dict(collision="at"), dict(angular=True), dict(angular=True, thermostat=True)]


@pytest.mark.parametrize("rule", RULES)
@pytest.mark.parametrize("n,rho", [((5, 3, 2), 1), ((23, 17, 9), 6), ((9, 4, 5), 13), ((6, 5, 4), 36),
                                   ((3, 2, 2), 121), ((3, 2, 2), 122), ((40, 40, 50), 3)])
def test_other_rules_match_the_oracle(n, rho, rule):
    s = inputs.solvent(n, rho, seed=rho + 5, mixed=True)
    box = pkg.Box(n=n, seed=rho + 5, precision="mixed", body_force=(0.01, -0.02, 0.03), **rule)
    box.set_state(s.pos, s.vel, step=7)
    box.step(3)
    pos, vel, _, _, step = box.get_state()
    box.close()
    kw = dict(rule)
    if kw.get("collision") == "at":
        kw["collision"] = oracle.AT
    ref = oracle.State(s.pos.copy(), s.vel.copy(), step=7)
    oracle.step(oracle.Params(n=n, seed=rho + 5, precision=oracle.MIXED, g=(0.01, -0.02, 0.03), **kw), ref, 3)
    assert step == ref.step
    np.testing.assert_array_equal(pos, ref.pos)
    np.testing.assert_array_equal(vel, ref.vel)


@pytest.mark.parametrize("rule", RULES)
def test_other_rules_with_large_velocities_and_a_full_row(rule):
    """The exact sums (|v|, dv or a term of the correction beyond 1024) and the overflow list."""
    n = (4, 4, 4)
    s = inputs.solvent(n, 6, seed=3, mixed=True)
    rng = np.random.default_rng(4)
    pos, vel = s.pos.copy(), s.vel.copy()
    pos[:120] = (1.3 + 0.4 * rng.random((120, 3))).astype(np.float32)
    vel[::9] = rng.uniform(1024.0, 1500.0, vel[::9].shape).astype(np.float32)
    kT = 4e6 if rule.get("collision") == "at" else 1.0
    box = pkg.Box(n=n, seed=3, precision="mixed", kT=kT, **rule)
    box.set_state(pos, vel)
    box.step(1)
    p, v, *_ = box.get_state()
    box.close()
    kw = dict(rule)
    if kw.get("collision") == "at":
        kw["collision"] = oracle.AT
    ref = oracle.State(pos.copy(), vel.copy())
    oracle.step(oracle.Params(n=n, seed=3, precision=oracle.MIXED, kT=kT, **kw), ref, 1)
    np.testing.assert_array_equal(p, ref.pos)
    np.testing.assert_array_equal(v, ref.vel)


@pytest.mark.parametrize("n,rho,density", [((5, 4, 1), 10, 10.0), ((7, 5, 2), 3, 0.0), ((9, 7, 3), 30, 45.5),
                                           ((40, 40, 8), 5, 5.0)])
def test_walls_match_the_oracle(n, rho, density):
    """Channel walls, from one layer of cells on: cells exact; velocities to the rounding
    that double log and cospi of the virtual particles leave in float (2e-6 a step, as the
    other wall tests state)."""
    s = inputs.solvent(n, rho, seed=5, mixed=True)
    kw = dict(n=n, seed=5, thermostat=True, walls_z=True, virt_density=density)
    box = pkg.Box(precision="mixed", body_force=(0.01, 0.02, 0.0), **kw)
    box.set_state(s.pos, s.vel)
    box.step(4)
    pos, vel, *_ = box.get_state()
    cells, counts = box.last_cells()
    box.close()
    ref = oracle.State(s.pos.copy(), s.vel.copy())
    kw["virt_density"] = density or float(rho)  # (0: the library's default, N / V)
    rc, rk = oracle.step(oracle.Params(precision=oracle.MIXED, g=(0.01, 0.02, 0.0), **kw), ref, 4,
                         want_cells=True)
    np.testing.assert_array_equal(cells, rc)
    np.testing.assert_array_equal(counts, rk)
    scale = np.maximum(np.linalg.norm(ref.vel, axis=1), 1.0)
    assert (np.linalg.norm(vel - ref.vel, axis=1) / scale).max() <= 8e-6
    assert np.all((pos[:, 2] >= 0) & (pos[:, 2] < n[2]))


@pytest.mark.parametrize("precision,rho", [("mixed", 6), ("mixed", 700), ("fp64", 6)])
def test_read_out_of_large_and_small_states(precision, rho):
    """The state comes back in input order through buckets of 4096 (FP64: 2048)
    tags, the last one partly filled, as through the direct scatter; overflowing
    rows and cell numbers included."""
    n = (61, 43, 47) if rho == 6 else (11, 10, 10)
    s = inputs.solvent(n, rho, seed=2, mixed=precision == "mixed")
    pos = s.pos.copy()
    pos[:500] = pos[0]  # one cell beyond its row
    box = pkg.Box(n=n, seed=2, precision=precision)
    box.set_state(pos, s.vel)
    p, v, *_ = box.get_state()
    np.testing.assert_array_equal(p, pos)
    np.testing.assert_array_equal(v, s.vel)
    box.step(1)
    p, v, *_ = box.get_state()
    cells, counts = box.last_cells()
    box.close()
    assert np.array_equal(np.bincount(cells, minlength=len(counts)), counts)
    d = np.abs(p - (pos + 0.1 * s.vel))
    L = np.array(n, dtype=float)
    assert np.minimum(d, np.abs(d - L)).max() < 1e-4


def test_many_steps_in_one_call_equal_single_steps():
    """Runs long enough for the graph of many steps, beads and all, against steps
    one at a time."""
    n = (6, 6, 6)
    s = inputs.solvent(n, 5, seed=12, mixed=True)
    sp, sv = inputs.chains(n, 4, 8, 0.5, bead_mass=5.0, seed=13)
    got = []
    for split in ([1] * 75, [75], [3, 33, 39]):
        box = pkg.Box(n=n, seed=12, precision="mixed", thermostat=True, chain_len=8, md_substeps=5,
                      solute_mass=5.0, bond_k=300.0, bond_r0=0.5)
        box.set_state(s.pos, s.vel, sp, sv)
        for k in split:
            box.step(k)
        got.append(box.get_state())
        box.close()
    for g in got[1:]:
        assert g[4] == got[0][4] == 75
        for a, b in zip(g[:4], got[0][:4]):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("mass", [1.0, 0.3, 1e-3, 4096.0, 5000.0])
def test_observables_of_any_mass(mass):
    """Mixed observables, summed from velocities and multiplied by the mass at the end, against
    plain NumPy: the totals to the rounding of a double sum; the cells' temperatures to their
    fixed point: 2^-32 m' a particle and component (m <= m' < 2 m, m' |v| < 2 max(m |v|)), over
    M (n - 1) >= 2 m, times the centre's speed.  Speeds that leave the split range included."""
    n = (9, 7, 5)
    s = inputs.solvent(n, 6, seed=9, mixed=True)
    vel = (s.vel / np.sqrt(mass)).astype(np.float32)
    vel[:40] *= 3000.0
    box = pkg.Box(n=n, seed=9, precision="mixed", mass=mass)
    box.set_state(s.pos, vel.astype(np.float64))
    ob = box.observables()
    box.close()
    v = vel.astype(np.float64)
    np.testing.assert_allclose(ob["P"], mass * v.sum(axis=0), atol=1e-13 * mass * np.abs(v).sum(), rtol=0)
    np.testing.assert_allclose(ob["KE"], 0.5 * mass * (v * v).sum(), rtol=1e-13)
    c = np.minimum(np.floor(s.pos), np.array(n) - 1).astype(int)
    c = c[:, 0] + n[0] * (c[:, 1] + n[1] * c[:, 2])
    cnt = np.bincount(c, minlength=np.prod(n))
    ok = cnt >= 2
    u = np.stack([np.bincount(c, v[:, k], cnt.size) for k in range(3)], 1)[ok] / cnt[ok, None]
    full = np.zeros((cnt.size, 3))
    full[ok] = u
    T = np.bincount(c, mass * ((v - full[c]) ** 2).sum(1), cnt.size)[ok] / (3.0 * (cnt[ok] - 1))
    err = 2.0 * cnt[ok] * 2.0 ** -32 * (1.0 + np.linalg.norm(u, axis=1) * 2) / (3.0 * (cnt[ok] - 1))
    kk = np.bincount(c, mass * (v * v).sum(1), cnt.size)[ok] / (3.0 * (cnt[ok] - 1))
    assert abs(ob["T_cell_mean"] - T.mean()) <= err.mean() + 1e-13 * kk.mean()
    assert ob["occupied_cells"] == int((cnt > 0).sum())


@pytest.mark.parametrize("beads", [False, True])
def test_narrow_warps_on_long_rows_keep_results(beads):
    """Rows beyond 192 records under the tuner's candidates of 16 and 8 cells a warp (idle lanes, a
    ragged last part, a bead group shared by warps): real steps, bit for bit those of 32."""
    n, rho, kw, sp, sv = (6, 5, 4), 130, {}, None, None
    s = inputs.solvent(n, rho, seed=31, mixed=True)
    if beads:
        kw = dict(chain_len=10, md_substeps=4, solute_mass=5.0, bond_k=300.0, bond_r0=0.5)
        sp, sv = inputs.chains(n, 12, 10, 0.5, bead_mass=5.0, seed=32)
    got = []
    for tuned in (True, False):
        box = pkg.Box(n=n, seed=31, precision="mixed", thermostat=True, body_force=(0.01, 0.0, -0.02), **kw)
        box.set_state(s.pos, s.vel, sp, sv)
        if tuned:
            taken = box.tune(1)[2]
        else:
            box.step(taken)
        box.step(2)
        got.append(box.get_state())
        box.close()
    assert got[0][4] == got[1][4] == taken + 2
    for a, b in zip(got[0][:4], got[1][:4]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("n,rho", [((41, 39, 53), 11), ((43, 41, 45), 14), ((53, 40, 37), 30), ((45, 43, 41), 45),
                                   ((44, 42, 43), 90)])
def test_sub_tiles_that_may_not_fit(n, rho):
    """With the thermostat and 32 cells a warp a sub-tile takes up to 16, 8, 4 or 2 cells whose members
    fill the staging area (mean 176 to 240 of 192): the cells that do not fit wait for the next,
    and a sub-tile starts at any cell."""
    s = inputs.solvent(n, rho, seed=rho, mixed=True)
    kw = dict(n=n, seed=rho, thermostat=True)
    box = pkg.Box(precision="mixed", **kw)
    box.set_state(s.pos, s.vel, step=7)
    box.step(2)
    pos, vel, *_ = box.get_state()
    box.close()
    ref = oracle.State(s.pos.copy(), s.vel.copy(), step=7)
    oracle.step(oracle.Params(precision=oracle.MIXED, **kw), ref, 2)
    np.testing.assert_array_equal(pos, ref.pos)
    np.testing.assert_array_equal(vel, ref.vel)


@pytest.mark.parametrize("n,rho,nch,thermostat", [((100, 80, 76), 1, 300, True), ((100, 80, 76), 5, 3000, True),
                                                  ((64, 63, 58), 18, 300, False), ((64, 63, 58), 45, 2000, False)])
def test_beads_of_large_boxes(n, rho, nch, thermostat):
    """Solute boxes large enough for the fused kernel's two launches, over the bead groups without
    beads and, from the list, with: sub-tiles of 32, 16, 8 and 2 cells, few beads and many."""
    s = inputs.solvent(n, rho, seed=9, mixed=True)
    sp, sv = inputs.chains(n, nch, 10, 0.5, bead_mass=5.0, seed=10)
    kw = dict(n=n, seed=9, thermostat=thermostat, chain_len=10, md_substeps=4, solute_mass=5.0, bond_k=300.0,
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
