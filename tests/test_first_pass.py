"""The first 1-D pass of the default order (Eq. 1 costs and their horizontal
sums): widths around its segments of 160 and 32 columns, around the two halves
of a row and the longest row of one block, ranges with their halo, partial
groups of disparities and disparities that leave the image in either view.
Maps and costs of both views against the oracle (parity rule), and bit for bit
against the same pass in short ranges."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_02300_gb300 import scenes
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_02300_gb300 import binding
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    st = binding.Stereo(0)
    yield torch, binding, st
    st.close()


@pytest.mark.parametrize("W,D,dmin,L1", [(31, 31, 0, 34), (33, 7, 20, 34), (160, 40, 0, 34), (161, 64, 3, 12),
                                         (192, 33, 0, 40), (193, 65, 0, 34), (320, 36, 100, 34), (352, 256, 0, 34),
                                         (353, 50, 0, 1), (513, 96, 0, 34), (640, 70, 0, 34), (641, 40, 0, 34),
                                         (1213, 100, 50, 34), (1300, 20, 236, 40)])
def test_rows_of_every_shape(env, W, D, dmin, L1):
    torch, binding, st = env
    H = 13
    s = scenes.plane_scene(W, H, dmin + D, 5, seed=scenes.seed_for(8, 3 * W + D), drange=(dmin, dmin + D - 1),
                           noise_sigma=2.0, texture="mixed")
    L, R = torch.from_numpy(s.left).cuda(), torch.from_numpy(s.right).cuda()
    over = dict(d_min=dmin, arm_l1=L1, arm_l2=L1 // 2)
    got = [t.cpu().numpy() for t in st.match_views(L, R, D, binding.Params.default(**over))]
    for h_chunk in (32, 100):
        for a, b in zip(got, st.match_views(L, R, D, binding.Params.default(h_chunk=h_chunk, **over))):
            assert np.array_equal(a, b.cpu().numpy()), h_chunk
    st.sync_status()
    ref = O.match(s.left, s.right, D, O.Params(**over))
    what = f"first pass {W}x{H} d in [{dmin}, {dmin + D - 1}] L1={L1}"
    parity.check_disparity(got[1], ref.disp_l, ref.best_l, ref.second_l, what + " left")
    parity.check_disparity(got[2], ref.disp_r, ref.best_r, ref.second_r, what + " right")
    parity.check_cost(got[3], ref.best_l, got[1], ref.disp_l, what + " left cost")
    parity.check_cost(got[4], ref.best_r, got[2], ref.disp_r, what + " right cost")


def test_wide_passes_give_way_to_a_budget(env):
    # the automatic pass is as wide as the slices' cap allows; a budget that
    # holds only narrow passes is met with narrow passes, by every entry point
    torch, binding, st = env
    s = scenes.plane_scene(640, 480, 128, 6, seed=scenes.seed_for(8, 9), drange=(2, 120), noise_sigma=2.0,
                           texture="mixed")
    L, R = torch.from_numpy(s.left).cuda(), torch.from_numpy(s.right).cuda()
    want = st.match(L, R, 128).cpu().numpy()
    narrow = binding.Stereo.workspace_bytes(640, 480, 128, binding.Params.default(d_chunk=32))
    assert binding.Stereo.workspace_bytes(640, 480, 128) > narrow
    with binding.Stereo(0, budget_bytes=narrow) as h:
        h.reserve(640, 480, 128)
        assert 0 < h.workspace_allocated() <= narrow
        assert np.array_equal(h.match(L, R, 128).cpu().numpy(), want)
        assert h.workspace_allocated() <= narrow
    half = binding.Stereo.workspace_bytes(320, 240, 64, binding.Params.default(d_chunk=32))
    front = 2 * (-(-3 * 320 * 240 // 256) * 256) + -(-2 * 320 * 240 // 256) * 256
    with binding.Stereo(0, budget_bytes=half + front) as h:
        got = h.depth(L, R, 64, 700.0, 0.12).cpu().numpy()
    assert np.array_equal(got, st.depth(L, R, 64, 700.0, 0.12).cpu().numpy())
