"""The host engine (capi.cu) on a CPU: its launch rules and what it does with the errors that
a CUDA call returns, on a stand-in for the CUDA runtime and the kernels' launchers
(tests/host_engine).  Nothing is computed: a launch is a line of a log."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import paper_1801_10187_gb300 as pkg
from paper_1801_10187_gb300 import _build

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host_engine")
DEVICE, HOST = 2, 1  # cudaMemoryType
P, I64, I32, U64 = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int32, ctypes.c_uint64


@pytest.fixture(scope="module")
def engine(tmp_path_factory):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("nvcc is needed to compile the engine's host code")
    _build.build()
    out = tmp_path_factory.mktemp("engine")
    nvcc = _build._nvcc()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))

    def run(*cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr

    run("g++", "-O1", "-std=c++17", "-fPIC", "-I", os.path.join(cuda, "include"), "-c",
        os.path.join(HERE, "fake_runtime.cpp"), "-o", str(out / "runtime.o"))
    run(nvcc, *_build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-c",
        os.path.join(HERE, "fake_launchers.cu"), "-o", str(out / "launchers.o"))
    run("g++", "-shared", "-Wl,-Bsymbolic", os.path.join(_build.BUILD, "capi.o"), str(out / "runtime.o"),
        str(out / "launchers.o"), "-o", str(out / "engine.so"), "-lpthread")
    L = ctypes.CDLL(str(out / "engine.so"))
    L.fake_log.restype = ctypes.c_char_p
    L.mpcd_last_error.restype = ctypes.c_char_p
    L.fake_alloc.restype = P
    L.fake_alloc.argtypes = [ctypes.c_size_t, ctypes.c_int, ctypes.c_int]
    L.fake_cost.argtypes = [ctypes.c_int, ctypes.c_double]
    L.mpcd_get_state_device.argtypes = [P, P, P]
    L.mpcd_set_state_thermal.argtypes = [P, I64, U64, U64]
    L.mpcd_step.argtypes = [P, I64]
    L.mpcd_destroy.argtypes = [P]
    return L


class Box:
    """A box of the engine; solute: beads at random places in chains of kw's chain_len."""

    def __init__(self, L, n_solvent, n_solute=0, **kw):
        self.L, self.ctx, p = L, P(), pkg.make_params(**kw)
        assert L.mpcd_create(ctypes.byref(p), None, ctypes.byref(self.ctx)) == 0
        if n_solute:
            x = [np.random.default_rng(1).random((m, 3)) for m in (n_solvent, n_solvent, n_solute, n_solute)]
            a, b, c, d = (v.ctypes.data_as(P) for v in x)
            assert L.mpcd_set_state(self.ctx, I64(n_solvent), a, b, I64(n_solute), c, d, U64(0)) == 0
        else:
            assert L.mpcd_set_state_thermal(self.ctx, n_solvent, 1, 0) == 0
        self.log()

    def step(self, n=1):
        return self.L.mpcd_step(self.ctx, n)

    def log(self):
        return self.L.fake_log().decode().split("\n")[:-1]

    def tune(self, reps=1):
        """mpcd_tune: (blocks per SM, cells per warp)."""
        bps, cpw = I32(), I32()
        assert self.L.mpcd_tune(self.ctx, I64(reps), ctypes.byref(bps), None, None, None, ctypes.byref(cpw)) == 0
        return bps.value, cpw.value

    def close(self):
        self.L.mpcd_destroy(self.ctx)


def fused(log, mode=1):
    """(launcher, spans, grid, cells per warp) of the fused launches of a mode (1: stream after collide)."""
    out = []
    for line in log:
        name, *kv = line.split()
        kv = {k: int(v) for k, _, v in (x.partition("=") for x in kv)}
        if kv.get("mode") == mode:
            out.append((name, kv["spans"], kv["grid"], kv["cpw"]))
    return out


@pytest.mark.parametrize("precision,kernel,per_sm", [("fp64", "srdd", 4), ("mixed", "srd", 7)])
def test_a_large_launch_is_as_many_blocks_as_fit(engine, precision, kernel, per_sm):
    """Blocks per SM are those of the kernel that is launched (in the stand-in 4 and 7)."""
    box = Box(engine, 1000, n=(57, 57, 57), precision=precision)
    assert box.step(2) == 0
    (name, spans, grid, cpw), = fused(box.log())
    assert (name, spans, cpw) == (kernel, 724, 32) and grid == per_sm * 152
    box.close()


def test_the_tuner_tries_narrow_warps_on_long_rows(engine):
    """Rows of 193 to 448 records, which k_cells_warp takes: 32 cells a warp untuned, and 16 and 8
    among the tuner's candidates; the steps after it take what it chose."""
    box = Box(engine, 150000, n=(10, 10, 10), precision="mixed")
    assert box.step(2) == 0
    assert fused(box.log()) == [("warp", 4, 4, 32)]
    engine.fake_cost(8, 0.25)
    bps, cpw = box.tune()
    engine.fake_cost(8, 1.0)
    assert cpw == 8 and {x[3] for x in fused(box.log())} == {32, 16, 8}
    assert box.step(2) == 0
    assert fused(box.log()) == [("warp", 4, 16, 8)]
    box.close()


@pytest.mark.parametrize("precision,n,kernel", [("mixed", 16, "srd"), ("fp64", 10, "srdd")])
def test_the_tuner_can_keep_the_width_of_a_small_box(engine, precision, n, kernel):
    """A box that takes four cells a warp untuned takes them after the tuner, too, where they are
    the fastest; the width that the call returns has no value for them and is its smallest."""
    box = Box(engine, 10 * n ** 3, n=(n, n, n), precision=precision)
    assert box.step(2) == 0
    (name, spans, grid, cpw), = fused(box.log())
    assert (name, cpw) == (kernel, 4)
    engine.fake_cost(4, 0.25)
    assert box.tune()[1] == 8
    engine.fake_cost(4, 1.0)
    assert {x[3] for x in fused(box.log())} == {32, 16, 8, 4}
    assert box.step(2) == 0
    assert fused(box.log())[0][3] == 4
    box.close()


@pytest.mark.parametrize("n_solvent,ahead", [(200000, True), (1000, False)])
def test_cells_of_large_boxes_are_copied_behind_the_read_out(engine, n_solvent, ahead):
    """mpcd_last_cells: a large box's copies are queued while its kernels work (device errors of the
    step looked at before), a small one's after the one wait for both."""
    box = Box(engine, n_solvent, n=(20, 20, 20), precision="mixed")
    assert box.step(2) == 0
    box.log()
    cells, counts = np.empty(n_solvent, np.int32), np.empty(8000, np.int32)
    assert engine.mpcd_last_cells(box.ctx, cells.ctypes.data_as(P), counts.ctypes.data_as(P)) == 0
    log = [x for x in box.log() if x in ("extract", "wait") or x.startswith("read")]
    sized = [i for i, x in enumerate(log) if x == f"read bytes={4 * n_solvent}"]
    between = log[log.index("extract") + 1:sized[0]]
    assert ("wait" in between) != ahead
    assert ("read bytes=4" in log[:log.index("extract")]) == ahead
    box.close()


@pytest.mark.parametrize("n_solvent,ahead", [(200000, True), (1000, False)])
def test_the_host_s_threads_start_beside_a_long_read_out(engine, n_solvent, ahead):
    """mpcd_get_state: the transfer of a large state begins while its read-out runs, the step's
    errors and its counter looked at before; a small one's after the one wait for all."""
    box = Box(engine, n_solvent, n=(20, 20, 20), precision="fp64")
    assert box.step(2) == 0
    box.log()
    pos, vel, step = np.empty((n_solvent, 3)), np.empty((n_solvent, 3)), U64()
    assert engine.mpcd_get_state(box.ctx, pos.ctypes.data_as(P), vel.ctypes.data_as(P), None, None,
                                 ctypes.byref(step)) == 0
    log = [x for x in box.log() if x in ("extract", "wait") or x.startswith("read")]
    first = min(i for i, x in enumerate(log) if x.startswith("read") and int(x.split("=")[1]) > 20000)
    assert ("wait" in log[log.index("extract") + 1:first]) != ahead
    assert ("read bytes=4" in log[:log.index("extract")]) == ahead
    assert np.all(pos == 1.0) and np.all(vel == 2.0)
    box.close()


@pytest.mark.parametrize("n,chains,thermostat,split", [
    (40, 40, True, False), (64, 1000, True, False), (100, 128, True, True), (100, 1000, True, True),
    (80, 60, False, False), (100, 128, False, True), (100, 1000, False, False)])
def test_solute_boxes_take_the_faster_kernel(engine, n, chains, thermostat, split):
    """Density 5: two launches of the fused kernel on large boxes, one of the warp-spread kernel on
    small ones and, without the thermostat, on those full of beads."""
    box = Box(engine, 5 * n ** 3, 50 * chains, n=(n, n, n), precision="mixed", thermostat=thermostat,
              chain_len=50, md_substeps=4, solute_mass=5.0, bond_k=100.0, bond_r0=0.5)
    assert box.step(2) == 0
    assert [x[0] for x in fused(box.log())] == (["srd", "srd_beads"] if split else ["warp"])
    box.close()


@pytest.mark.parametrize("density,after", [(150, 0.125), (10, 0.0)])
def test_phase_times_of_the_record_updates(engine, density, after):
    """mpcd_phase_times: the kernel that ends a pass of the warp-spread kernel is a phase of its own, and
    no part of the fused step's; the fused kernel does without."""
    box = Box(engine, 1000 * density, n=(10, 10, 10), precision="mixed")
    engine.fake_cost(-1, 0.125)
    ms, n = (ctypes.c_double * 8)(), I32()
    assert engine.mpcd_phase_times(box.ctx, I64(4), ms, 8, ctypes.byref(n)) == 0
    engine.fake_cost(-1, 1.0)
    assert n.value == 3 and list(ms[:3]) == [1.0, after, 0.0]
    box.close()


def test_a_refused_launch_is_an_error_of_every_step(engine):
    """The cooperative launch of the solute's MD fails during capture: no graph without it is kept,
    so the next steps fail as well, and the first one after that takes it."""
    box = Box(engine, 500, 40, n=(5, 5, 5), precision="fp64", chain_len=10, md_substeps=5, solute_mass=5.0,
              bond_k=100.0, bond_r0=0.5, lj_epsilon=1.0, lj_sigma=0.5)
    for passes in (1, 40):
        engine.fake_fail(b"wca", 720)  # cudaErrorCooperativeLaunchTooLarge
        for _ in range(2):
            assert box.step(passes) == pkg.MPCD_ECUDA
            assert "graph" not in box.log()
        engine.fake_fail(b"wca", 0)
        assert box.step(passes) == 0
        log = box.log()
        assert "wca" in log and "graph" in log
    box.close()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_the_state_is_stored_by_a_kernel_only_into_memory_it_may_write(engine, precision):
    """mpcd_get_state_device: into this device's own memory directly; into another device's, or where
    two arrays overlap or are not aligned, through a copy; what the driver refuses, and an
    array that is too small, comes back as an error."""
    n, es = 1000, 4 if precision == "mixed" else 8
    real, bytes_ = np.float32 if es == 4 else np.float64, 3 * 1000 * es
    box = Box(engine, n, n=(5, 5, 5), precision=precision)
    box.step(1)

    def read(pos, vel):
        box.log()
        rc = engine.mpcd_get_state_device(box.ctx, pos, vel)
        return rc, [x for x in box.log() if x.startswith("copy")]

    def values(p):
        return np.frombuffer(ctypes.string_at(p, bytes_), dtype=real)

    own = [engine.fake_alloc(bytes_, DEVICE, 0) for _ in range(2)]
    other = [engine.fake_alloc(bytes_, DEVICE, 1) for _ in range(2)]
    assert read(*own) == (0, [])
    assert read(own[0], None) == (0, []) and read(None, own[1]) == (0, [])
    rc, copies = read(*other)
    assert rc == 0 and len(copies) == 2
    rc, copies = read(own[0], other[1])
    assert rc == 0 and len(copies) == 1
    for pos, vel in (own, other):
        assert np.all(values(pos) == 1) and np.all(values(vel) == 2)
    both = engine.fake_alloc(2 * bytes_, DEVICE, 0)
    assert read(both, both + bytes_) == (0, [])
    rc, copies = read(both, both + es)  # overlapping: the velocities are written last
    assert rc == 0 and len(copies) == 2 and np.all(values(both)[1:] == 2) and values(both)[0] == 1
    rc, copies = read(both + es // 2, None)  # not aligned
    assert rc == 0 and len(copies) == 1
    small = engine.fake_alloc(bytes_ - 1, DEVICE, 0)
    for bad in (small, own[0] + es, 1 << 40, engine.fake_alloc(bytes_ // 2, HOST, 0)):
        assert read(bad, own[1])[0] == pkg.MPCD_ECUDA
    assert read(*own) == (0, [])
    box.close()
