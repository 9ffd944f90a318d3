"""The second 1-D pass (Eq. 2's second sum, Eq. 3): every way its walk is dealt
out to blocks (whole strips, bands, shares that run on from strip to strip),
the edges of its steps of 32 positions and strips of 4 lines, the shortest
and longest arms, partial groups of disparities.  The maps are compared with
the oracle on row bands (parity rule) and, bit for bit, with the same pass cut
into runs of 32 positions."""
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


# W, H, D, rows checked: bands of one or several steps (first four), whole
# strips and bands (1280 wide: two rounds), whole strips and shares that run
# on (1000 x 300), one round of shares that run on (600 x 290)
SHAPES = [(66, 31, 5, None), (65, 33, 33, None), (131, 97, 40, None), (7, 65, 3, None),
          (1280, 70, 64, (30, 40)), (1000, 300, 64, (120, 126)), (600, 290, 64, (30, 36))]


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("W,H,D,rows", SHAPES)
def test_walk_equals_the_oracle_and_short_runs(env, W, H, D, rows, order):
    torch, binding, st = env
    if W < 16:
        left, right = scenes.random_pair(W, H, W + H)
    else:
        s = scenes.plane_scene(W, H, D, 4, seed=scenes.seed_for(8, W + H + D), drange=(0, D - 1), noise_sigma=2.0,
                               texture="mixed")
        left, right = s.left, s.right
    L, R = torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()
    p = binding.Params.default(agg_order=order)
    got = [t.cpu().numpy() for t in st.match_views(L, R, D, p)]
    p.v_chunk = 32
    for a, b in zip(got, st.match_views(L, R, D, p)):
        assert np.array_equal(a, b.cpu().numpy())
    ref = O.match(left, right, D, O.Params(agg_order=order), rows=rows)
    sl = slice(*rows) if rows else slice(None)
    what = f"second pass {W}x{H} D={D} order {order}"
    parity.check_disparity(got[1][sl], ref.disp_l, ref.best_l, ref.second_l, what + " left")
    parity.check_disparity(got[2][sl], ref.disp_r, ref.best_r, ref.second_r, what + " right")
    parity.check_cost(got[3][sl], ref.best_l, got[1][sl], ref.disp_l, what + " left cost")
    parity.check_cost(got[4][sl], ref.best_r, got[2][sl], ref.disp_r, what + " right cost")


@pytest.mark.parametrize("L1", [1, 3, 7, 11, 15, 16, 40])
def test_arm_limits(env, L1):
    # ring lengths: shortest, just below and above a multiple of eight rows, longest
    torch, binding, st = env
    s = scenes.plane_scene(90, 150, 37, 3, seed=scenes.seed_for(8, 40 + L1), drange=(2, 34), noise_sigma=1.0,
                           texture="mixed")
    L, R = torch.from_numpy(s.left).cuda(), torch.from_numpy(s.right).cuda()
    for order in (0, 1):
        bp = binding.Params.default(arm_l1=L1, arm_l2=L1 // 2, agg_order=order)
        out, dl, dr, cl, cr = (t.cpu().numpy() for t in st.match_views(L, R, s.D, bp))
        ref = O.match(s.left, s.right, s.D, O.Params(arm_l1=L1, arm_l2=L1 // 2, agg_order=order))
        parity.check_disparity(dl, ref.disp_l, ref.best_l, ref.second_l, f"L1={L1} order {order} left")
        parity.check_cost(cl, ref.best_l, dl, ref.disp_l, f"L1={L1} order {order} left cost")
        assert (out == O.lr_check(dl, dr, 1)).all()
