"""The gathering back projections where their work is dealt or declined: views of
many small row blocks."""
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
