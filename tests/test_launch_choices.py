"""The choice of kernels and the deal of their blocks by the size of a launch:
maps and costs are the same whichever runs, and no size pays for the rule of
another (ratios of kernel times of the same process).
"""
import ctypes

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


def _pair(torch, W, H, D, seed=1, d_min=0):
    if W < 16:
        left, right = scenes.random_pair(W, H, W + H)
    else:
        s = scenes.plane_scene(W, H, d_min + D, 4, seed=scenes.seed_for(8, 100 + seed), noise_sigma=2.0, texture="mixed",
                               drange=(d_min, d_min + D - 1))
        left, right = s.left, s.right
    return left, right, torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()


def _us(torch, st, kernels, call, reps=9):
    """Device time of one call's launches of these kernels: the shortest of three means."""
    call()
    torch.cuda.synchronize()
    st.set_profiling(True)
    best = float("inf")
    for _ in range(3):
        st.profile_reset()
        for _ in range(reps):
            call()
        prof = st.profile()
        best = min(best, 1e3 * sum(prof[k][1] for k in kernels.split()) / reps)
    st.set_profiling(False)
    return best


def test_short_arms_are_dealt_to_the_blocks_that_are_resident(env):
    # a shorter ring must not be slower for being dealt to blocks that the
    # registers do not let in: 0.98 of the long arms' time when it was, 0.85 since
    torch, binding, st = env
    _, _, L, R = _pair(torch, 640, 480, 64)
    t = {L1: _us(torch, st, "k_vagg", lambda p=binding.Params.default(arm_l1=L1, arm_l2=L1 // 2): st.match(L, R, 64, p))
         for L1 in (8, 34)}
    assert t[8] < 0.92 * t[34], t


def test_batches_beyond_one_launch_keep_the_device_full(env):
    # pairs 65 .. 128 are a launch of their own: 1.76 times two launches of 64 when
    # the blocks were dealt over the call
    torch, binding, st = env
    _, _, L, R = _pair(torch, 320, 240, 32)
    pairs = [(L, R, 32, torch.empty((240, 320), dtype=torch.int16, device="cuda")) for _ in range(128)]
    t = {n: _us(torch, st, "k_vagg", lambda n=n: st.match_batch(pairs[:n])) for n in (64, 128)}
    assert t[128] < 2 * 1.3 * t[64], t
    for p in pairs[1:]:
        assert torch.equal(p[3], pairs[0][3])


@pytest.mark.parametrize("W,H,D,d_min", [(33, 513, 7, 0), (40, 1100, 33, 2), (513, 31, 20, 0), (600, 20, 70, 5), (7, 3, 2, 0)])
@pytest.mark.parametrize("order", [0, 1])
def test_cost_volumes_of_long_lines_and_partial_groups(env, W, H, D, d_min, order):
    torch, binding, st = env
    left, right, L, R = _pair(torch, W, H, D, W, d_min)
    ref = O.match(left, right, D, O.Params(agg_order=order, d_min=d_min), volume=True)
    for d_chunk in (0, 32):   # one pass, and passes that merge their winners
        p = binding.Params.default(agg_order=order, d_min=d_min, d_chunk=d_chunk)
        for view, want in ((0, ref.vol_l), (1, ref.vol_r)):
            parity.check_volume(st.cost_volume(L, R, D, view, p).cpu().numpy(), want,
                                f"volume {W}x{H} D={D} order {order} view {view}")


def test_a_cost_volume_takes_region_sizes_once(env):
    # 7 times the match's second pass when N(p) was summed again for every group
    torch, binding, st = env
    _, _, L, R = _pair(torch, 640, 480, 64)
    vol = _us(torch, st, "k_vagg", lambda: st.cost_volume(L, R, 64, 0))
    assert vol < 5 * _us(torch, st, "k_vagg", lambda: st.match(L, R, 64))


# sizes whose second pass runs by whole lines; h_chunk has no part in it
@pytest.mark.parametrize("W,H,D", [(96, 64, 16), (7, 65, 3), (33, 32, 32), (65, 33, 33), (131, 97, 70), (40, 511, 40),
                                   (41, 512, 31), (512, 20, 65)])
@pytest.mark.parametrize("order", [0, 1])
def test_whole_lines_equal_the_strips(env, W, H, D, order):
    torch, binding, st = env
    _, _, L, R = _pair(torch, W, H, D, H)
    for d_chunk, vote in ((0, 0), (24, 0), (0, 2)):
        over = dict(agg_order=order, d_chunk=d_chunk, vote_iters=vote, smooth_arms=vote // 2)
        lines = st.match_views(L, R, D, binding.Params.default(**over))
        strips = st.match_views(L, R, D, binding.Params.default(v_chunk=16384, **over))
        for a, b in zip(lines, strips):
            assert torch.equal(a, b), (over, W, H, D)


@pytest.mark.parametrize("W,H,D", [(333, 211, 50), (320, 240, 64)])
def test_small_launches_are_not_bound_by_one_strip(env, W, H, D):
    # strips (one block each, as v_chunk asks) against the automatic choice, which also
    # writes the costs: the same time when that was strips too
    torch, binding, st = env
    _, _, L, R = _pair(torch, W, H, D)
    p = binding.Params.default(v_chunk=16384)
    lines, strips = (_us(torch, st, "k_vagg k_end", lambda q=q: st.match_views(L, R, D, q), 25) for q in (None, p))
    assert lines < 0.95 * strips, (lines, strips)


# reference columns at the edges of the first pass's blocks (320), parts (96, 160, 352, 448)
# and segments, rows that leave disparities outside, partial groups
@pytest.mark.parametrize("W,D,d_min,L1", [(96, 16, 0, 34), (97, 20, 10, 34), (129, 40, 0, 34), (200, 50, 3, 12), (256, 33, 0, 40),
                                          (257, 64, 0, 34), (319, 36, 100, 34), (320, 70, 0, 34), (321, 40, 0, 34), (352, 50, 0, 1),
                                          (353, 96, 0, 34), (416, 33, 60, 34), (448, 40, 0, 34), (449, 64, 0, 34), (577, 40, 0, 40),
                                          (736, 40, 0, 34)])
def test_first_pass_at_the_edges_of_its_parts(env, W, D, d_min, L1):
    torch, binding, st = env
    H = 11
    left, right, L, R = _pair(torch, W, H, D, W, d_min)
    over = dict(d_min=d_min, arm_l1=L1, arm_l2=L1 // 2)
    got = st.match_views(L, R, D, binding.Params.default(**over))
    for h_chunk in (50, 300):   # ranges in blocks of eight and of sixteen warps
        for a, b in zip(got, st.match_views(L, R, D, binding.Params.default(h_chunk=h_chunk, **over))):
            assert torch.equal(a, b), h_chunk
    ref = O.match(left, right, D, O.Params(**over))
    got = [t.cpu().numpy() for t in got]
    parity.check_disparity(got[1], ref.disp_l, ref.best_l, ref.second_l, f"first pass {W} columns left")
    parity.check_disparity(got[2], ref.disp_r, ref.best_r, ref.second_r, f"first pass {W} columns right")
    parity.check_cost(got[3], ref.best_l, got[1], ref.disp_l, f"first pass {W} columns left cost")
    parity.check_cost(got[4], ref.best_r, got[2], ref.disp_r, f"first pass {W} columns right cost")


def test_short_rows_keep_the_first_pass_busy(env):
    # the same evaluations in rows of 160 and of 640 columns: 1.7 times as long in the short ones
    # while half of a block's warps had none of their columns, 1.2 since
    torch, binding, st = env

    def batch(n, W, H):
        _, _, L, R = _pair(torch, W, H, 32)
        pairs = [(L, R, 32, torch.empty((H, W), dtype=torch.int16, device="cuda")) for _ in range(n)]
        return _us(torch, st, "k_hagg", lambda: st.match_batch(pairs))
    short, long = batch(64, 160, 120), batch(4, 640, 480)
    assert short < 1.45 * long, (short, long)


def test_the_column_pass_of_tall_images_keeps_two_blocks_per_sm(env):
    # order 1 at 1280x720: 2.3 times the row pass of order 0 while its registers let one
    # block of 23 warps in, 1.8 since
    torch, binding, st = env
    _, _, L, R = _pair(torch, 1280, 720, 128)
    cols = _us(torch, st, "k_vcost", lambda p=binding.Params.default(agg_order=1): st.match(L, R, 128, p))
    rows = _us(torch, st, "k_hagg", lambda: st.match(L, R, 128))
    assert cols < 2.0 * rows, (cols, rows)


def test_one_buffer_for_the_left_view_and_the_checked_map(env):
    # dco_stereo_match_views with disp_out == disp_left: the checked map, as the
    # consistency check comes after the views, with and without costs
    torch, binding, st = env
    W, H, D = 133, 60, 24
    _, _, L, R = _pair(torch, W, H, D)
    p = lambda t: ctypes.c_void_p(t.data_ptr() if t is not None else None)   # noqa: E731
    want = st.match(L, R, D)
    assert int((want < 0).sum()) > 0
    for params in (None, binding.Params.default(v_chunk=64)):
        for cost in (None, torch.empty((H, W), dtype=torch.float32, device="cuda")):
            both = torch.full((H, W), -9, dtype=torch.int16, device="cuda")
            torch.cuda.synchronize()
            rc = binding.lib().dco_stereo_match_views(st._h, p(L), p(R), W, H, D, ctypes.byref(params) if params else None,
                                                      p(both), p(both), None, p(cost), None, None)
            st.sync_status()
            assert rc == 0 and torch.equal(both, want)


def _strips(E, F, layers, slots):
    """The deal of the strip walk: (whole rounds, strips left, bands per strip that is
    left; 0: equal shares that run on from strip to strip)."""
    units = -(-F // 4) * layers
    rounds, rest = divmod(units, slots)
    nb = slots // rest if rest else 1
    return rounds, rest, min(nb, -(-E // 32)) if nb > 1 else 1 if E <= 256 else 0


def _lines(E, F, layers, L1, nsm):
    """Whether the second pass of one pair takes whole lines."""
    warps = F * layers * -(-E // 32)
    return E <= 512 and (warps <= 110 * nsm or E <= 200 + 3 * L1 and warps <= 1000 * nsm)


def _slots(L1, nsm):
    """Resident blocks of the strip walk: by its ring in shared memory, at most four."""
    ring = (-(-(2 * L1 + 1) // 8) * 8 + 32) * 512
    return nsm * min(4, (228 << 10) // (ring + 6 * 512 + 4 * (8 * 128 + 128) + 1024))


SCHEDULES = {   # E, D, arm_l1, what the deal has to be; F is searched for
    "run-on shares after whole rounds": (310, 64, 34, lambda r, rest, b: r > 0 and rest > 0 and b == 0),
    "run-on shares alone": (500, 32, 34, lambda r, rest, b: r == 0 and b == 0),
    "whole strips after whole rounds": (240, 64, 3, lambda r, rest, b: r > 0 and rest > 0 and b == 1),
    "bands after whole rounds": (360, 64, 34, lambda r, rest, b: r > 0 and b > 1),
    "bands alone": (600, 40, 34, lambda r, rest, b: r == 0 and b > 1),
}


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("what", SCHEDULES)
def test_every_deal_of_the_strips(env, what, order):
    torch, binding, st = env
    E, D, L1, wanted = SCHEDULES[what]
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    layers = 2 * -(-D // 32)
    F = next(F for F in range(64, 1400, 20)
             if wanted(*_strips(E, F, layers, _slots(L1, nsm))) and not _lines(E, F, layers, L1, nsm))
    W, H = (F, E) if order == 0 else (E, F)
    left, right, L, R = _pair(torch, W, H, D, F)
    over = dict(agg_order=order, arm_l1=L1, arm_l2=L1 // 2)
    got = st.match_views(L, R, D, binding.Params.default(**over))
    for a, b in zip(got, st.match_views(L, R, D, binding.Params.default(v_chunk=32, **over))):
        assert torch.equal(a, b), (what, W, H)
    rows = (H // 2, H // 2 + 4)
    ref = O.match(left, right, D, O.Params(**over), rows=rows)
    got = [t.cpu().numpy()[slice(*rows)] for t in got]
    parity.check_disparity(got[1], ref.disp_l, ref.best_l, ref.second_l, f"{what}, order {order}, left")
    parity.check_cost(got[4], ref.best_r, got[2], ref.disp_r, f"{what}, order {order}, right cost")


@pytest.mark.parametrize("W,H", [(333, 251), (65, 37)])   # a thread per pixel; a thread per arm (at most two tiles per SM)
def test_both_preparations_for_every_window_and_arm_rule(env, W, H):
    torch, binding, st = env
    img, _, L, _ = _pair(torch, W, H, 16)
    tiles = -(-W // 32) * -(-H // 8)
    assert (tiles > 2 * torch.cuda.get_device_properties(0).multi_processor_count) == (W == 333)
    for cw, ch, l1, l2, t1, t2 in ((9, 7, 34, 17, 20, 6), (7, 5, 10, 4, 15, 5), (11, 5, 40, 20, 30, 8), (1, 1, 1, 0, 256, 256),
                                   (9, 7, 34, 17, 0, 6), (9, 7, 34, 2, 255, 0), (3, 3, 8, 8, 1, 1), (5, 13, 40, 0, 60, 60)):
        over = dict(census_w=cw, census_h=ch, arm_l1=l1, arm_l2=l2, tau1=t1, tau2=t2)
        p = binding.Params.default(**over)
        assert (st.census(L, p).cpu().numpy().view(np.uint64) == O.census(img, cw, ch)).all(), over
        assert (st.arms(L, p).cpu().numpy() == O.arms(img, O.Params(**over))).all(), over


def test_ragged_disparities_write_whole_sectors(env):
    # D = 10 does less than D = 16; it took 1.6 times as long while the slices of its last four
    # disparities were half sectors
    torch, binding, st = env
    _, _, L, R = _pair(torch, 1920, 1080, 16)
    few, more = (_us(torch, st, "k_hagg", lambda D=D: st.match(L, R, D)) for D in (10, 16))
    assert few < 1.15 * more, (few, more)


@pytest.mark.parametrize("W,H,order", [(1920, 100, 0), (160, 1080, 1)])
def test_short_lines_are_not_walked_in_strips(env, W, H, order):
    # strips (as v_chunk asks) against the automatic choice: the same time when that was
    # strips too, 0.68 and 0.75 of it since
    torch, binding, st = env
    _, _, L, R = _pair(torch, W, H, 64)
    auto, strips = (_us(torch, st, "k_hwta" if order else "k_vagg", lambda p=binding.Params.default(agg_order=order, v_chunk=v):
                        st.match(L, R, 64, p), 20) for v in (0, 16384))
    assert auto < 0.88 * strips, (auto, strips)


def test_a_batch_of_short_and_long_pairs(env):
    # strips and lines in one call, with and without passes and votes: each pair as alone
    torch, binding, st = env
    shapes = [(640, 480, 64), (200, 150, 40), (333, 211, 50), (96, 600, 20), (1000, 120, 33), (64, 64, 64)] * 2
    made = [_pair(torch, *s, seed=k)[2:] for k, s in enumerate(shapes)]
    outs = [torch.empty((H, W), dtype=torch.int16, device="cuda") for W, H, _ in shapes]
    for over in ({}, {"vote_iters": 2}, {"d_chunk": 32}, {"agg_order": 1}):
        p = binding.Params.default(**over)
        st.match_batch([(*m, s[2], o) for m, s, o in zip(made, shapes, outs)], p)
        for m, s, o in zip(made, shapes, outs):
            assert torch.equal(o, st.match(*m, s[2], p)), (over, s)


def test_a_vote_round_of_a_large_image(env):
    # 0.93 of the second pass of the vote with 40 registers, 0.82 since
    torch, binding, st = env
    _, _, L, R = _pair(torch, 1280, 720, 128)
    p = binding.Params.default(vote_iters=1)
    counts, sums = (_us(torch, st, k, lambda: st.match(L, R, 128, p)) for k in ("k_hvote", "k_vvote"))
    assert counts < 0.92 * sums, (counts, sums)
