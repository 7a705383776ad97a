"""The gathering back projection of the cone beam (column.cu) against the FP64
oracle, at the sizes where its pieces end: planes past a whole chunk of 32, an
odd nz (the source's height inside a voxel), a level detector row, slabs on both
sides of the source's height, detectors finer than half a voxel (more than one
pair of rows per crossing) and coarser than one, columns past a CTA's tile,
rays along the axes, 16-bit residuals, and the solver's form of it (several
column blocks, drawn detector cells)."""
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


def cone(nx, ny, nz, views, nu, nv, pitch, M=1, N=1, dso=200.0, dsd=400.0):
    return dict(kind="cone3d", nx=nx, ny=ny, nz=nz, dx=1.0, dy=1.0, dz=1.0, n_views=views, nu=nu,
                nv=nv, du=pitch, dv=pitch, dso=dso, dsd=dsd, M=M, N=N)


CASES = {
    "one_chunk_and_a_plane": cone(64, 61, 33, 8, 90, 70, 1.7),
    "odd_height_level_row": cone(67, 64, 65, 8, 81, 91, 1.9),
    "level_row_in_a_face": cone(64, 64, 64, 8, 80, 81, 2.1),
    "fine_rows": cone(64, 64, 40, 4, 200, 150, 0.7),
    "coarse_rows": cone(70, 66, 64, 16, 50, 48, 3.2),
    "nine_chunks": cone(40, 40, 260, 4, 50, 130, 2.8),
    "short_distance": cone(64, 64, 48, 8, 96, 64, 1.6, dso=80.0, dsd=200.0),
    "rise_of_most_of_a_voxel": cone(48, 48, 64, 8, 84, 84, 2.2, dso=72.0, dsd=144.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_back_projection(name):
    """Against the oracle, and against the scattering walk (thin blocks of planes
    scatter), which runs on the same FP32 rays.

    Bounds: a ray's ends are rounded to FP32 in voxels (up to 232 from the
    volume's corner: 7.6e-6), which moves a face crossing by up to ~1.5e-5 voxel;
    two crossings of a mean chord of 0.7 voxel: 4e-5 of the chord, against the
    oracle. The walks share the rays, and the gather's own crossings carry
    distances from the middle (<= 50 voxels, 1.9e-6): 2e-5 holds both."""
    s = dict(CASES[name], N=CASES[name]["nz"] // 2)
    og, gg = oracle_geom(s), gpu_geom(s)
    r = synth.normal_array(og.n_rows, 3).astype(np.float32)
    rd = torch.from_numpy(r).to(DEV)
    x = torch.full((og.n_cols,), 7.0, device=DEV)
    B.bsgd_back_project(gg, rd, x)
    got = x.cpu().double().numpy()
    assert rel_l2(got, P.bp(og, r.astype(np.float64)).reshape(-1)) <= 4e-5
    thin = torch.zeros_like(x)
    for j in range(gg.N):
        B.bsgd_back_project(gg, rd, thin, col_blocks=[j])
    assert rel_l2(got, thin.cpu().double().numpy()) <= 2e-5
    # the same sum in every run
    again = torch.zeros_like(x)
    B.bsgd_back_project(gg, rd, again)
    assert torch.equal(x, again)


SLICES = {
    "par_odd": dict(kind="par2d", nx=67, ny=66, nz=1, dx=1.0, dy=1.0, dz=1.0, n_views=37, nu=101, nv=1,
                    du=0.9, dv=1.0),
    "par_bins_in_faces": dict(kind="par2d", nx=64, ny=64, nz=1, dx=1.0, dy=1.0, dz=1.0, n_views=4, nu=67,
                              nv=1, du=1.0, dv=1.0),
    "fan_coarse": dict(kind="fan2d", nx=96, ny=64, nz=1, dx=1.0, dy=1.5, dz=1.0, n_views=30, nu=40, nv=1,
                       du=8.0, dv=1.0, dso=200.0, dsd=400.0),
    "fan_fine": dict(kind="fan2d", nx=65, ny=70, nz=1, dx=1.2, dy=1.0, dz=1.0, n_views=9, nu=600, nv=1,
                     du=0.5, dv=1.0, dso=150.0, dsd=300.0),
}


@pytest.mark.parametrize("name", list(SLICES))
def test_slice_back_projection(name):
    """2D images: the bounds of test_back_projection (ends of the rays up to 250
    voxels from the corner; single rows of pixels scatter)."""
    s = dict(SLICES[name], M=3, N=SLICES[name]["ny"])
    og, gg = oracle_geom(s), gpu_geom(s)
    r = torch.from_numpy(synth.normal_array(og.n_rows, 6)).to(DEV, torch.bfloat16)
    x = torch.full((og.n_cols,), 3.0, device=DEV)
    B.bsgd_back_project(gg, r, x)
    got, r64 = x.cpu().double().numpy(), r.double().cpu().numpy()
    assert rel_l2(got, P.bp(og, r64).reshape(-1)) <= 4e-5
    thin = torch.zeros_like(x)
    for j in range(gg.N):
        B.bsgd_back_project(gg, r, thin, col_blocks=[j])
    assert rel_l2(got, thin.cpu().double().numpy()) <= 2e-5
    # two row blocks, scaled, added onto the image
    y = x.clone()
    B.bsgd_back_project(gg, r, y, row_blocks=[2, 0], scale=-2.0, accumulate=True)
    rows = np.sort(np.concatenate([P.rows_of_views(og, P.row_block_views(og, 3, i)) for i in (0, 2)]))
    ref = got - 2.0 * P.bp_rows(og, r64[rows], rows, None)
    assert rel_l2(y.cpu().double().numpy(), ref) <= 4e-5


def test_blocks_scale_accumulate_and_storage():
    """Two separate runs of slabs (the middle one on both sides of the source's
    height), some row blocks, added onto an image, from a BF16 residual."""
    s = cone(72, 70, 160, 12, 90, 160, 1.9, M=4, N=5)
    og, gg = oracle_geom(s), gpu_geom(s)
    r = torch.from_numpy(synth.normal_array(og.n_rows, 4)).to(DEV, torch.bfloat16)
    base = synth.uniform_array(og.n_cols, 5).astype(np.float32)
    x = torch.from_numpy(base).to(DEV)
    B.bsgd_back_project(gg, r, x, row_blocks=[2, 0], col_blocks=[2, 4], scale=-0.5, accumulate=True)
    rows = np.sort(np.concatenate([P.rows_of_views(og, P.row_block_views(og, 4, i)) for i in (0, 2)]))
    r64 = r.double().cpu().numpy()
    ref = base.astype(np.float64)
    for j in (2, 4):
        ref = ref - 0.5 * P.bp_rows(og, r64[rows], rows, P.column_block(og, 5, j))
    got = x.cpu().double().numpy()
    assert rel_l2(got, ref) <= 4e-5
    untouched = np.concatenate([P.column_block_voxels(og, 5, j) for j in (0, 1, 3)])
    assert np.array_equal(got[untouched], base[untouched])


def near(mask, shape):
    """The voxels of a mask and their neighbours along the axes and diagonals."""
    m = np.pad(mask.reshape(shape), 1)
    out = np.zeros_like(m)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                out |= np.roll(m, (dz, dy, dx), (0, 1, 2))
    return out[1:-1, 1:-1, 1:-1].reshape(-1)


def test_infinite_and_nan_weights_stay_on_their_rays():
    """A NaN or infinite ray reaches the voxels it crosses, and none further off
    than a corner it grazes within rounding."""
    s = cone(64, 64, 64, 4, 80, 80, 2.1)
    og, gg = oracle_geom(s), gpu_geom(s)
    r = np.zeros((4, 80, 80), dtype=np.float32)
    r[1, 37, 40], r[2, 50, 20] = np.nan, np.inf
    x = torch.zeros(og.n_cols, device=DEV)
    B.bsgd_back_project(gg, torch.from_numpy(r.reshape(-1)).to(DEV), x)
    got = x.cpu().numpy()
    ray = np.zeros((4, 80, 80))
    ray[1, 37, 40] = 1.0
    a = P.bp(og, ray.reshape(-1)).reshape(-1)
    ray[:] = 0.0
    ray[2, 50, 20] = 1.0
    b = P.bp(og, ray.reshape(-1)).reshape(-1)
    near_a, near_b = near(a > 0, (64, 64, 64)), near(b > 0, (64, 64, 64))
    assert np.all(np.isnan(got[a > 1e-3]))
    assert np.all(np.isposinf(got[(b > 1e-3) & ~near_a]))
    assert np.all(got[~near_a & ~near_b] == 0.0)


@pytest.mark.parametrize("kN,cells,storage", [(1, "none", "f32"), (2, "none", "f32"), (2, "geometric", "f32"),
                                              (2, "uniform", "f32"), (2, "none", "bf16")])
def test_solver(kN, cells, storage):
    """BSGD at the smallest size whose solver gathers, against the oracle with the
    same draws; odd nv (a level row) and uneven slabs."""
    M = 1 if kN == 1 else 2
    s = cone(128, 126, 63 if kN == 1 else 64, 52, 110, 71, 2.2, M=M, N=2, dso=300.0, dsd=600.0)
    og, gg = oracle_geom(s), gpu_geom(s)
    xt = synth.ellipsoid_phantom(128, 126, s["nz"], 4, seed=1).reshape(-1).astype(np.float64) * 0.01
    y = P.fp(og, xt).reshape(-1).astype(np.float32)
    mu, iters = 2e-5, 4
    kinds = {"none": B.CELLS_NONE, "geometric": B.CELLS_GEOMETRIC, "uniform": B.CELLS_UNIFORM}
    n_cells = 1 if cells == "none" else 4
    prm = B.SolveParams(alpha=1 / M, gamma=kN / 2, step_rule=B.STEP_FIXED, mu=mu, seed=5, cells=kinds[cells],
                        n_cells=n_cells, storage=B.F32 if storage == "f32" else B.BF16)
    st = B.State(gg, prm, torch.from_numpy(y).to(DEV))
    x = torch.zeros(og.n_cols, device=DEV, dtype=torch.float32 if storage == "f32" else torch.bfloat16)
    st.block_step(x, iters)
    po = OB.Params(M, 2, 1 / M, kN / 2, mu, seed=5, cells=cells, n_cells=n_cells)
    ost = OB.bsgd(og, y.astype(np.float64), po, iters)
    assert rel_l2(x.cpu().double().numpy(), ost.x) <= (1e-5 if storage == "f32" else 1e-2)
    q = st.query()
    assert abs(q["residual_norm"] - ost.residual_norm()) <= (1e-5 if storage == "f32" else 1e-2) * ost.residual_norm()
    # a checkpoint carries the gathered gradient
    blob, x1 = st.save(), x.clone()
    st.block_step(x, 2)
    st2 = B.State(gg, prm, torch.from_numpy(y).to(DEV))
    st2.restore(blob)
    st2.block_step(x1, 2)
    assert torch.equal(x, x1)
