"""The gathering back projections where their work is dealt or declined: views of
many small row blocks, and sources far away."""
import numpy as np
import pytest

from helpers import gpu_geom, oracle_geom, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import projector as P  # noqa: E402
from paper_1903_11874_gb300 import binding as B  # noqa: E402
from paper_1903_11874_gb300 import synth  # noqa: E402

DEV = "cuda:0"


def fan(n, views, nu, M, view_block):
    return dict(kind="fan2d", nx=n, ny=n, nz=1, dx=1.0, dy=1.0, dz=1.0, n_views=views, nu=nu, nv=1, du=1.7,
                dv=1.0, dso=2.0 * n, dsd=4.0 * n, M=M, N=2, view_block=np.asarray(view_block, dtype=np.int32))


@pytest.mark.parametrize("views,M,block", [(90, 45, "pairs"), (60, 60, "ones"), (300, 2, "uneven"), (90, 90, "ones")])
def test_slice_views_dealt_over_all_blocks(views, M, block):
    """Row blocks in view order: a warp takes every 8th view whichever block it is
    of, so the sums are those of one block of all views, bit for bit (blocks of
    equal size, at most 64 at a time; otherwise the views fall to other warps and
    the sums agree to FP32 rounding). Against the oracle: the bound of the plain
    gather's tests."""
    vb = {"pairs": np.arange(views) // 2, "ones": np.arange(views), "uneven": (np.arange(views) > 29) * 1}[block]
    s = fan(70, views, 97, M, vb)
    og = oracle_geom(dict(s, view_block=None))
    r = torch.from_numpy(synth.normal_array(views * 97, 3).astype(np.float32)).to(DEV)
    got, one = torch.zeros(70 * 70, device=DEV), torch.zeros(70 * 70, device=DEV)
    B.bsgd_back_project(gpu_geom(s), r, got)
    B.bsgd_back_project(gpu_geom(dict(s, M=1, view_block=None)), r, one)
    if block != "uneven" and M <= 64:
        assert torch.equal(got, one)
    ref = P.bp(og, r.cpu().double().numpy()).reshape(-1)
    assert rel_l2(got.cpu().double().numpy(), ref) <= 4e-5
    again = torch.zeros_like(got)
    B.bsgd_back_project(gpu_geom(s), r, again)
    assert torch.equal(again, got)


@pytest.mark.parametrize("views,M,pick", [(90, 45, range(0, 45, 2)), (300, 3, [2, 0]), (140, 70, range(67)),
                                          (29, 4, [1, 3])])
def test_slice_of_some_blocks(views, M, pick):
    """Blocks chosen by the caller: small ones listed, large ones one after another,
    more than a launch takes, uneven ones (the bound of the plain gather's tests)."""
    s = fan(70, views, 97, M, np.arange(views) % M)
    og, gg = oracle_geom(s), gpu_geom(s)
    r = synth.normal_array(views * 97, 3).astype(np.float32)
    x = torch.full((70 * 70,), 2.0, device=DEV)
    B.bsgd_back_project(gg, torch.from_numpy(r).to(DEV), x, row_blocks=list(pick))
    rows = np.sort(np.concatenate([P.rows_of_views(og, P.row_block_views(og, M, i)) for i in pick]))
    ref = P.bp_rows(og, r.astype(np.float64)[rows], rows, None)
    assert rel_l2(x.cpu().double().numpy(), ref.reshape(-1)) <= 4e-5


FAR = {
    "cone_3e5": dict(kind="cone3d", nx=64, ny=64, nz=40, dx=1.0, dy=1.0, dz=1.0, n_views=6, nu=70, nv=45, du=2.0,
                     dv=2.0, dso=3e5, dsd=6e5),
    "cone_1e6": dict(kind="cone3d", nx=64, ny=64, nz=40, dx=1.0, dy=1.0, dz=1.0, n_views=6, nu=70, nv=45, du=2.0,
                     dv=2.0, dso=1e6, dsd=2e6),
    "cone_1e7": dict(kind="cone3d", nx=64, ny=64, nz=40, dx=1.0, dy=1.0, dz=1.0, n_views=6, nu=70, nv=45, du=2.0,
                     dv=2.0, dso=1e7, dsd=2e7),
    "fan_1e6": dict(kind="fan2d", nx=70, ny=70, nz=1, dx=1.0, dy=1.0, dz=1.0, n_views=30, nu=300, nv=1, du=0.5,
                    dv=1.0, dso=1e6, dsd=2e6),
}


@pytest.mark.parametrize("name", list(FAR))
def test_far_sources_lose_no_ray(name):
    """The sum over the volume is that of the oracle: no voxel misses a ray.

    Bound: a ray's ends round to half an ulp of the source's distance, which moves
    its length in the volume by up to four times that, either way: five standard
    deviations of the mean over the rays, against their mean length. Rays past FP32
    (1e7) are held to a tenth. The cones here lie beyond the gather's rule."""
    s = dict(FAR[name], M=1, N=1)
    og, gg = oracle_geom(s), gpu_geom(s)
    r = synth.uniform_array(og.n_rows, 3).astype(np.float32)
    x = torch.zeros(og.n_cols, device=DEV)
    B.bsgd_back_project(gg, torch.from_numpy(r).to(DEV), x)
    chords = P.fp(og, np.ones(og.n_cols)).reshape(-1)
    n, mean = int((chords > 0).sum()), chords.sum() / (chords > 0).sum()
    ulp = float(np.spacing(np.float32(s["dso"])))
    bound = 0.1 if s["dso"] > 5e6 else 5 * 4 * 0.5 * ulp / mean / np.sqrt(n)
    ref = P.bp(og, r.astype(np.float64)).sum()
    assert abs(x.double().sum().item() / ref - 1) <= bound


def cone(n, nz, views, nu, nv, pitch, dso, mag, N):
    return dict(kind="cone3d", nx=n, ny=n, nz=nz, dx=1.0, dy=1.0, dz=1.0, n_views=views, nu=nu, nv=nv, du=pitch,
                dv=pitch, dso=dso, dsd=mag * dso, M=1, N=N)


@pytest.mark.parametrize("nz,nv", [(48, 76), (48, 77), (49, 76), (32, 61), (20, 40)])
def test_chunks_on_both_sides_of_a_near_source(nz, nv):
    """Planes below and above the source's height in one chunk of 32, with the
    source 11 voxels from the volume (rows per voxel change by up to 0.6 across a cell
    there): level rows in a face, inside a voxel, and none. The bounds are those
    of the plain gather's tests, against the oracle and the walk (thin blocks)."""
    s = cone(60, nz, 9, 70, nv, 1.8, 54.0, 2.0, nz)
    og, gg = oracle_geom(s), gpu_geom(s)
    r = synth.normal_array(og.n_rows, 3).astype(np.float32)
    rd = torch.from_numpy(r).to(DEV)
    x, thin = torch.zeros(og.n_cols, device=DEV), torch.zeros(og.n_cols, device=DEV)
    B.bsgd_back_project(gg, rd, x)
    for j in range(nz):
        B.bsgd_back_project(gg, rd, thin, col_blocks=[j])
    got = x.cpu().double().numpy()
    assert rel_l2(got, P.bp(og, r.astype(np.float64)).reshape(-1)) <= 4e-5
    assert rel_l2(got, thin.cpu().double().numpy()) <= 2e-5


def time_of(f):
    times = []
    f()
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(4):
            f()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return sorted(times)[3]


def test_near_source_chunk_costs_its_rows():
    """One chunk on both sides of the source's height takes no more than twice its
    two halves by themselves (seven times where every crossing took the rows that
    the cell nearest to the source needs)."""
    s = cone(128, 32, 60, 128, 128, 1.6, 100.0, 2.0, 2)
    gg = gpu_geom(s)
    r, x = torch.ones(gg.n_rows, device=DEV), torch.zeros(gg.n_cols, device=DEV)
    whole = time_of(lambda: B.bsgd_back_project(gg, r, x))
    halves = sum(time_of(lambda: B.bsgd_back_project(gg, r, x, col_blocks=[j])) for j in (0, 1))
    assert whole <= 2.0 * halves


def kernels_of(f):
    """Names of the kernels that a call launches."""
    f()
    torch.cuda.synchronize()
    for _ in range(3):   # (a process's first profile comes back empty)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            f()
            torch.cuda.synchronize()
        names = " ".join(e.key for e in prof.key_averages())
        if "kernel" in names:
            return names
    pytest.skip("no kernel names from the profiler here")


@pytest.mark.parametrize("dso,block,gathers", [(93.0, None, False), (96.0, None, True), (250.0, None, True),
                                               (92.0, 1, False), (100.0, 1, True)])
def test_sources_that_touch_the_volume_scatter(dso, block, gathers):
    """The rule on the padding of the weights: the back projection from a source 2.5
    voxels from the volume takes the walk, from 5.5 voxels the gather; either agrees
    with the oracle (one view: the bound of the plain gather's tests)."""
    s = cone(128, 128, 40, 128, 128, 1.6, dso, 2.0, 4)
    og, gg = oracle_geom(dict(s, n_views=1)), gpu_geom(s)
    r = np.zeros((40, 128, 128), np.float32)
    r[0] = synth.normal_array(128 * 128, 3).reshape(128, 128)
    rd, x = torch.from_numpy(r).to(DEV), torch.zeros(gg.n_cols, device=DEV)
    cb = None if block is None else [block]
    names = kernels_of(lambda: B.bsgd_back_project(gg, rd, x, col_blocks=cb))
    assert ("bp_gather_kernel" in names) == gathers and ("bp_plain_kernel" in names) != gathers
    ref = P.bp(og, r[0].reshape(-1).astype(np.float64)).reshape(128, -1)
    sl = slice(None) if block is None else slice(32 * block, 32 * block + 32)
    assert rel_l2(x.cpu().double().numpy().reshape(128, -1)[sl], ref[sl]) <= 4e-5


@pytest.mark.parametrize("M", [1, 4, 7])
def test_all_row_blocks_gather_in_view_order(M):
    """All row blocks of a geometry give the sums of one block of all views, bit for
    bit: the views are taken in order whichever blocks they are in."""
    s = cone(64, 64, 30, 70, 70, 1.8, 200.0, 2.0, 1)
    r = torch.from_numpy(synth.normal_array(30 * 70 * 70, 3).astype(np.float32)).to(DEV)
    a, b = torch.zeros(64 ** 3, device=DEV), torch.zeros(64 ** 3, device=DEV)
    B.bsgd_back_project(gpu_geom(s), r, a)
    gg = gpu_geom(dict(s, M=M))
    B.bsgd_back_project(gg, r, b)
    assert torch.equal(a, b)
    # some of the blocks, added one after another: the same sums in another order
    c = torch.zeros_like(b)
    for i in range(M):
        B.bsgd_back_project(gg, r, c, row_blocks=[i], accumulate=True)
    assert rel_l2(c.cpu().double().numpy(), a.cpu().double().numpy()) <= 1e-6


@pytest.mark.parametrize("pitch,block,gathers", [(1.2, 0, False), (1.2, 1, True), (1.6, 0, True)])
def test_slabs_that_the_detector_hardly_covers_scatter(pitch, block, gathers):
    """The rule on a slab's covered planes: the top slab of 128^3 scatters under a
    detector that covers seven of its 32 planes."""
    gg = gpu_geom(dict(cone(128, 128, 40, 128, 128, pitch, 250.0, 2.0, 4), M=2))
    r, x = torch.ones(gg.n_rows, device=DEV), torch.zeros(gg.n_cols, device=DEV)
    names = kernels_of(lambda: B.bsgd_back_project(gg, r, x, col_blocks=[block]))
    assert ("bp_gather_kernel" in names) == gathers and ("bp_plain_kernel" in names) != gathers
    names = kernels_of(lambda: B.bsgd_power_iteration(gg, block, 2))
    assert ("bp_gather_kernel" in names) == gathers and ("bp_plain_kernel" in names) != gathers


@pytest.mark.parametrize("planes,gathers", [(12, False), (16, True)])
def test_thin_slabs_of_fine_rows_scatter(planes, gathers):
    """The rule on a slab's planes holds for rows close together, too."""
    gg = gpu_geom(cone(128, planes, 40, 128, 128, 1.0, 250.0, 2.0, 1))
    r, x = torch.ones(gg.n_rows, device=DEV), torch.zeros(gg.n_cols, device=DEV)
    names = kernels_of(lambda: B.bsgd_back_project(gg, r, x))
    assert ("bp_gather_kernel" in names) == gathers and ("bp_plain_kernel" in names) != gathers


@pytest.mark.parametrize("s", [cone(64, 64, 30, 70, 70, 1.8, 200.0, 2.0, 4), fan(70, 60, 97, 2, np.arange(60) % 2)])
def test_geometry_is_one_allocation(s):
    """All tables of a geometry, the gather's lines among them, are one block of
    device memory."""
    gpu_geom(s)
    for _ in range(3):   # (a process's first profile comes back empty)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            gpu_geom(s)
            torch.cuda.synchronize()
        calls = {e.key: e.count for e in prof.key_averages()}
        if "cudaMalloc" in calls:
            assert calls["cudaMalloc"] == 1
            return
    pytest.skip("no calls from the profiler here")


def test_source_in_the_corner_scatters():
    """A source 0.0035 voxel from the corner of a tall volume, where the padding of
    the weights would not fit an int: the back projection takes the walk.

    Bound: that of the plain gather's tests at the rounding of heights up to 1500
    voxels (6.1e-5, eight times theirs), against the oracle."""
    s = cone(8, 3000, 4, 9, 4, 3.3, 8 / np.sqrt(2.0) + 0.0035, 2.0, 1)
    near = s["dso"] - 8 / np.sqrt(2.0)
    rows = s["dsd"] / (near * s["dv"])
    assert rows < 1e3 and s["dv"] / 2.0 <= 1.7 and (2 * 3000 + 32) * rows * np.sqrt(2.0) / near > 2 ** 31
    og, gg = oracle_geom(s), gpu_geom(s)
    r = synth.normal_array(og.n_rows, 3).astype(np.float32)
    rd, x = torch.from_numpy(r).to(DEV), torch.zeros(og.n_cols, device=DEV)
    names = kernels_of(lambda: B.bsgd_back_project(gg, rd, x))
    assert "bp_gather_kernel" not in names and "bp_plain_kernel" in names
    assert rel_l2(x.cpu().double().numpy(), P.bp(og, r.astype(np.float64)).reshape(-1)) <= 3.2e-4


def test_more_row_blocks_than_a_launch_takes():
    """66 row blocks of a cone (64 at a time): the second launch adds to the first's
    image. Unequal voxel sides and angles given by the caller. The bounds are those
    of the plain gather's tests."""
    s = dict(kind="cone3d", nx=64, ny=60, nz=48, dx=1.0, dy=1.2, dz=0.9, n_views=66, nu=60, nv=50, du=2.3, dv=1.7,
             dso=200.0, dsd=400.0, M=66, N=1, angles=np.sort(synth.uniform_array(66, 7)) * 6.28)
    og, gg = oracle_geom(s), gpu_geom(s)
    r = synth.normal_array(og.n_rows, 3).astype(np.float32)
    rd, x = torch.from_numpy(r).to(DEV), torch.full((og.n_cols,), 5.0, device=DEV)
    assert kernels_of(lambda: B.bsgd_back_project(gg, rd, x)).count("bp_gather_kernel") == 1
    assert rel_l2(x.cpu().double().numpy(), P.bp(og, r.astype(np.float64)).reshape(-1)) <= 4e-5
    again = torch.zeros_like(x)
    B.bsgd_back_project(gg, rd, again)
    assert torch.equal(again, x)
