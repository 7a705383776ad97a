"""Solver states around the gathering back projection: checkpoints between a
state that gathers and one that scatters, the memory that a state needs, and a
change of the sampling mode."""
import os
import struct
import subprocess
import sys

import numpy as np
import pytest

from helpers import gpu_geom, oracle_geom, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import bsgd as OB  # noqa: E402
from oracle import projector as P  # noqa: E402
from paper_1903_11874_gb300 import binding as B  # noqa: E402
from paper_1903_11874_gb300 import synth  # noqa: E402

DEV = "cuda:0"


def solve_geometry(kN, **over):
    """The smallest size whose solver gathers; odd nv, uneven slabs (one block)."""
    M = 1 if kN == 1 else 2
    s = dict(kind="cone3d", nx=128, ny=126, nz=63 if kN == 1 else 64, dx=1.0, dy=1.0, dz=1.0, n_views=52,
             nu=110, nv=71, du=2.2, dv=2.2, dso=300.0, dsd=600.0, M=M, N=2)
    s.update(over)
    return s


def scan(og, s):
    xt = synth.ellipsoid_phantom(s["nx"], s["ny"], s["nz"], 4, seed=1).reshape(-1).astype(np.float64) * 0.01
    return P.fp(og, xt).reshape(-1).astype(np.float32)


@pytest.fixture(scope="module")
def one_block():
    s = solve_geometry(1)
    og, gg = oracle_geom(s), gpu_geom(s)
    return gg, torch.from_numpy(scan(og, s)).to(DEV)


def one_block_state(one_block, cells):
    gg, y = one_block
    prm = B.SolveParams(alpha=1.0, gamma=0.5, step_rule=B.STEP_FIXED, mu=2e-5, seed=5, cells=cells,
                        n_cells=1 if cells == B.CELLS_NONE else 4)
    return B.State(gg, prm, y)


def run_on(st, x, n):
    st.block_step(x, n)
    return x.cpu().double().numpy()


@pytest.mark.parametrize("first,second", [(B.CELLS_NONE, B.CELLS_GEOMETRIC), (B.CELLS_GEOMETRIC, B.CELLS_NONE)])
def test_checkpoint_between_sampling_modes(one_block, first, second):
    """A state created with whole views gathers, one created with detector cells
    scatters; a blob of either continues in the other.

    Bound: both runs are the same iterations in FP32, each within 1e-5 of the
    exact image (the parity bound of the solver tests): 2e-5 between them."""
    a, b = one_block_state(one_block, first), one_block_state(one_block, second)
    x = torch.zeros(one_block[0].n_cols, device=DEV)
    a.block_step(x, 4)
    blob, xb = a.save(), x.clone()
    b.restore(blob)
    assert b.query()["residual_norm"] == a.query()["residual_norm"]
    assert rel_l2(run_on(b, xb, 3), run_on(a, x, 3)) <= 2e-5


def split_blob(blob, gg, whole):
    """The blob with g moved wholly into its y-fastest part (whole = False), or
    such a blob with that part added back."""
    payload = struct.unpack_from("<q", blob, 128)[0]
    at, C = 144 + 4 * (2 * gg.compact_rows + gg.n_rows), gg.n_cols
    shape = (gg.nz, gg.ny, gg.nx)
    head, g, rest = bytearray(blob[:at]), np.frombuffer(blob, np.float32, C, at).reshape(shape), blob[at + 4 * C:]
    if whole:
        gT = np.frombuffer(rest[-4 * C:], np.float32).reshape(gg.nz, gg.nx, gg.ny)
        struct.pack_into("<q", head, 128, payload - 4 * C)
        return bytes(head) + (g + gT.transpose(0, 2, 1)).astype(np.float32).tobytes() + rest[:-4 * C]
    struct.pack_into("<q", head, 128, payload + 4 * C)
    return bytes(head) + bytes(4 * C) + rest + np.ascontiguousarray(g.transpose(0, 2, 1)).tobytes()


def test_checkpoint_with_and_without_the_y_fastest_gradient(one_block):
    """A state that gathers takes the blob of one that scatters with the same
    parameters (part of g stored y-fastest, after the trace), and the other way
    round; a blob cut short stays refused."""
    gg, _ = one_block
    a = one_block_state(one_block, B.CELLS_NONE)
    x = torch.zeros(gg.n_cols, device=DEV)
    a.block_step(x, 4)
    blob, xb = a.save(), x.clone()
    ref = run_on(a, x, 3)
    b = one_block_state(one_block, B.CELLS_NONE)
    b.restore(split_blob(blob, gg, False))
    assert np.array_equal(run_on(b, xb.clone(), 3), ref)   # the same g, and the gather is reproducible
    c = one_block_state(one_block, B.CELLS_GEOMETRIC)
    xc = torch.zeros(gg.n_cols, device=DEV)
    c.block_step(xc, 4)
    cblob, xd = c.save(), xc.clone()
    ref = run_on(c, xc, 3)
    d = one_block_state(one_block, B.CELLS_GEOMETRIC)
    d.restore(split_blob(cblob, gg, True))
    assert rel_l2(run_on(d, xd, 3), ref) <= 2e-5
    for bad in (blob[:-4], split_blob(blob, gg, False)[:-4]):
        with pytest.raises(B.BSGDError):
            b.restore(bad)


LITTLE_MEMORY = """
import torch
from helpers import gpu_geom
from paper_1903_11874_gb300 import binding as B
geo = dict(kind="cone3d", nx=128, ny=128, nz=64, dx=1.0, dy=1.0, dz=1.0, n_views=720, nu=512, nv=448,
           du=1.6, dv=1.6, dso=300.0, dsd=600.0)
gg = B.Geometry(M=1, N=2, **geo)
y = torch.ones(gg.n_rows, device="cuda:0")
prm = B.SolveParams(alpha=1.0, gamma=1.0, step_rule=B.STEP_FIXED, mu=1e-6, seed=5)
x = torch.zeros(gg.n_cols, device="cuda:0")
need = B.bsgd_request_bytes(geo, 1, 2, prm)
torch.cuda.empty_cache()
free = torch.cuda.mem_get_info()[0]
hold = torch.empty(free - need - (1 << 28), dtype=torch.uint8, device="cuda:0")
st = B.State(gg, prm, y)
st.block_step(x, 1)
torch.cuda.synchronize()
assert bool(torch.isfinite(x).all()) and float(x.abs().max()) > 0
st.close()
B.bsgd_solve(gg, B.SolveParams(alpha=1.0, gamma=1.0, step_rule=B.STEP_FIXED, mu=1e-6, seed=5, epochs=1), y, x)
print("MADE")
"""


def test_little_memory_scatters():
    """With a gigabyte more than a scattering state holds, less than the 1.7 GB of
    weights that the gather would take, the state is made and steps."""
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([here, os.path.dirname(here)]))
    res = subprocess.run([sys.executable, "-c", LITTLE_MEMORY], cwd=os.path.dirname(here), env=env,
                         capture_output=True, text=True, timeout=300)
    assert "MADE" in res.stdout, res.stderr[-2000:]


def kernels_of(f):
    """Names of the kernels that a call launches."""
    for _ in range(3):   # (a process's first profile comes back empty)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            f()
            torch.cuda.synchronize()
        names = " ".join(e.key for e in prof.key_averages())
        if "kernel" in names:
            return names
    pytest.skip("no kernel names from the profiler here")


@pytest.mark.parametrize("first", [B.CELLS_NONE, B.CELLS_UNIFORM])
def test_sampling_mode_carries_the_form(one_block, first):
    """A one-block state gathers while it draws whole views and scatters while it
    draws cells, whatever it was created with; its image after changes of the mode
    both ways is the oracle's of the same draws (the solver tests' bound)."""
    gg, y = one_block
    s = solve_geometry(1)
    og = oracle_geom(s)
    st = one_block_state(one_block, first)
    x = torch.zeros(gg.n_cols, device=DEV)
    modes = [B.CELLS_NONE, B.CELLS_UNIFORM, B.CELLS_NONE, B.CELLS_UNIFORM]
    for m in modes:
        st.set_sampling(B.PAIRS_UNIFORM, m, 1 if m == B.CELLS_NONE else 4)
        st.block_step(x, 2)
    sels = []
    for t in st.read_trace(8):
        c = t[3:3 + gg.n_views].astype(np.int64)
        sels.append(OB.Selection([(int(t[1]), int(t[2]))], [None if c[0] < 0 else c]))
    po = OB.Params(1, 2, 1.0, 0.5, 2e-5, seed=5, cells="uniform", n_cells=4)
    ost = OB.bsgd(og, y.cpu().double().numpy(), po, 8, replay=sels)
    assert rel_l2(x.cpu().double().numpy(), ost.x) <= 1e-5
    for m, gathers in ((B.CELLS_NONE, True), (B.CELLS_UNIFORM, False)):
        st.set_sampling(B.PAIRS_UNIFORM, m, 1 if m == B.CELLS_NONE else 4)
        assert ("solve_gather_kernel" in kernels_of(lambda: st.block_step(x, 2))) == gathers


def test_served_set_up_keeps_to_its_bytes():
    """The power iteration of a served request takes weights of at most an image's
    floats (the y-fastest accumulator that its bytes are counted without): one row
    block of four at a time here. Its step is the plain state's (FP32 sums in
    another order)."""
    geo = dict(kind="cone3d", nx=96, ny=96, nz=64, dx=1.0, dy=1.0, dz=1.0, n_views=96, nu=96, nv=96, du=1.7,
               dv=1.7, dso=250.0, dsd=500.0)
    prm = B.SolveParams(alpha=0.25, gamma=0.5, step_rule=B.STEP_STRIP, power_iters=3, rho=0.5, seed=5, epochs=1)
    gg = B.Geometry(M=4, N=2, **geo)
    y = np.ones(gg.n_rows, dtype=np.float32)
    srv = B.Server(budget_bytes=4 << 30, max_slots=2)
    try:
        for _ in range(3):   # (a process's first profile comes back empty)
            with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
                _x, rep = srv.wait(srv.submit(geo, 4, 2, prm, y))
                torch.cuda.synchronize()
            launches = sum(e.count for e in prof.key_averages() if "bp_gather_kernel" in e.key)
            if launches:
                break
    finally:
        srv.close()
    if not launches:
        pytest.skip("no kernel names from the profiler here")
    assert launches == 2 * 3 * 4   # blocks x iterations x passes
    st = B.State(gg, prm, torch.from_numpy(y).to(DEV))
    assert abs(rep["mu"] / st.query()["mu"] - 1.0) <= 1e-5


KINDS = {"none": B.CELLS_NONE, "geometric": B.CELLS_GEOMETRIC, "uniform": B.CELLS_UNIFORM}


@pytest.fixture(scope="module")
def two_blocks():
    s = solve_geometry(2)
    og = oracle_geom(s)
    return og, gpu_geom(s), scan(og, s)


def check_against_oracle(st, x, ost, tol):
    assert rel_l2(x.float().cpu().double().numpy(), ost.x) <= tol
    rn = ost.residual_norm()
    assert abs(st.query()["residual_norm"] - rn) <= tol * rn


@pytest.mark.parametrize("kN,cells,storage", [(1, "none", "f32"), (2, "none", "f32"), (2, "uniform", "f32"),
                                              (2, "geometric", "bf16")])
def test_separate_passes(one_block, two_blocks, kN, cells, storage):
    """FP, residual and BP apart: the weights are the residual's change on the
    block's band (zero off the drawn cell), turned row by row, and the snapshot
    follows. The solver tests' bounds."""
    if kN == 1:
        og, gg, y = oracle_geom(solve_geometry(1)), one_block[0], one_block[1].cpu().numpy()
    else:
        og, gg, y = two_blocks
    n_cells = 1 if cells == "none" else 4
    prm = B.SolveParams(alpha=1 / gg.M, gamma=kN / 2, step_rule=B.STEP_FIXED, mu=2e-5, seed=5, cells=KINDS[cells],
                        n_cells=n_cells, storage=B.F32 if storage == "f32" else B.BF16)
    st = B.State(gg, prm, torch.from_numpy(y).to(DEV))
    x = torch.zeros(gg.n_cols, device=DEV, dtype=torch.float32 if storage == "f32" else torch.bfloat16)
    st.block_step(x, 1)      # the passes alternate: both leave the same memory
    st.set_split(True)
    st.block_step(x, 3)
    ost = OB.bsgd(og, y.astype(np.float64), OB.Params(gg.M, 2, 1 / gg.M, kN / 2, 2e-5, seed=5, cells=cells,
                                                      n_cells=n_cells), 4)
    check_against_oracle(st, x, ost, 1e-5 if storage == "f32" else 1e-2)
    assert "column_change_kernel" in kernels_of(lambda: st.block_step(x, 1))


def test_replayed_pairs(two_blocks):
    """A replayed trace of several blocks takes the separate passes; it gives the
    image of the draws it replays."""
    og, gg, y = two_blocks
    yd = torch.from_numpy(y).to(DEV)
    kw = dict(alpha=0.5, gamma=1.0, step_rule=B.STEP_FIXED, mu=2e-5)
    a, b = B.State(gg, B.SolveParams(seed=5, **kw), yd), B.State(gg, B.SolveParams(seed=6, **kw), yd)
    xa, xb = torch.zeros(gg.n_cols, device=DEV), torch.zeros(gg.n_cols, device=DEV)
    a.block_step(xa, 4)
    trace = a.read_trace(4)
    b.set_replay(trace)
    b.block_step(xb, 4)
    sels = [OB.Selection([(int(t[1]), int(t[2])), (int(t[3]), int(t[4]))], [None, None]) for t in trace]
    ost = OB.bsgd(og, y.astype(np.float64), OB.Params(2, 2, 0.5, 1.0, 2e-5, seed=6), 4, replay=sels)
    check_against_oracle(b, xb, ost, 1e-5)


@pytest.mark.parametrize("cells", ["none", "uniform"])
def test_sharded_steps(two_blocks, cells):
    """One process that owns both blocks, and two that own one each (their parts of
    the sum added here), with a gathering BP."""
    og, gg, y = two_blocks
    yd = torch.from_numpy(y).to(DEV)
    n_cells = 1 if cells == "none" else 4
    prm = B.SolveParams(alpha=0.5, gamma=1.0, step_rule=B.STEP_FIXED, mu=2e-5, seed=5, cells=KINDS[cells],
                        n_cells=n_cells)
    ost = OB.bsgd(og, y.astype(np.float64), OB.Params(2, 2, 0.5, 1.0, 2e-5, seed=5, cells=cells, n_cells=n_cells), 4)
    for owners in ([[0, 1]], [[0], [1]]):
        states = [B.State(gg, prm, yd) for _ in owners]
        xs = [torch.zeros(gg.n_cols, device=DEV) for _ in owners]
        parts = [torch.zeros(st.set_shard(own), device=DEV) for st, own in zip(states, owners)]
        for _ in range(4):
            for st, x, e in zip(states, xs, parts):
                st.shard_begin(x, e)
            total = sum(parts[1:], parts[0].clone())
            for st, x in zip(states, xs):
                st.shard_end(x, total)
        check_against_oracle(states[0], sum(xs[1:], xs[0].clone()), ost, 1e-5)


@pytest.mark.parametrize("kN,cells,apart", [(2, "none", False), (3, "none", True), (4, "none", True),
                                            (3, "uniform", False), (4, "geometric", False)])
def test_blocks_that_take_separate_passes(kN, cells, apart):
    """The rule on one pass or separate ones (three and four blocks): either gives
    the oracle's image."""
    s = solve_geometry(kN, nx=96, ny=94, nz=32 * kN, n_views=20, M=2, N=kN, nu=95, nv=95, du=2.2, dv=2.2)
    og, gg = oracle_geom(s), gpu_geom(s)
    y = scan(og, s)
    n_cells = 1 if cells == "none" else 4
    prm = B.SolveParams(alpha=1.0, gamma=1.0, step_rule=B.STEP_FIXED, mu=2e-5, seed=5, cells=KINDS[cells],
                        n_cells=n_cells)
    st = B.State(gg, prm, torch.from_numpy(y).to(DEV))
    x = torch.zeros(gg.n_cols, device=DEV)
    st.profile(True)
    st.block_step(x, 3)
    prof = st.read_profile()
    assert (prof["fp"]["launches"], prof["fpbp"]["launches"]) == ((3, 0) if apart else (0, 3))
    ost = OB.bsgd(og, y.astype(np.float64), OB.Params(2, kN, 1.0, 1.0, 2e-5, seed=5, cells=cells, n_cells=n_cells), 3)
    check_against_oracle(st, x, ost, 1e-5)
    assert "solve_gather_kernel" in kernels_of(lambda: st.block_step(x, 1))
