"""Wide automatic passes are a choice: where the device cannot allocate their
workspace (refused here by a test flag), every entry point runs with narrow
passes, the same maps come out, and a warmed-up call allocates and synchronises
nothing (it can be captured)."""
import numpy as np
import pytest

from paper_2203_02300_gb300 import scenes

pytestmark = pytest.mark.gpu

W, H, D = 640, 480, 128   # 314 MB of slices in one pass; 79 MB in passes of 32


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_02300_gb300 import binding
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    s = scenes.plane_scene(W, H, D, 6, seed=scenes.seed_for(8, 77), drange=(2, 120), noise_sigma=2.0, texture="mixed")
    left, right = torch.from_numpy(s.left).cuda(), torch.from_numpy(s.right).cuda()
    with binding.Stereo(0) as st:
        want = st.match(left, right, D).cpu().numpy()
        assert st.workspace_allocated() == binding.Stereo.workspace_bytes(W, H, D)
    return torch, binding, left, right, want


def _narrow(binding):
    return binding.Stereo.workspace_bytes(W, H, D, binding.Params.default(d_chunk=32))


def test_a_refused_wide_workspace_is_not_asked_for_again(env):
    torch, binding, left, right, want = env
    out = torch.empty((H, W), dtype=torch.int16, device="cuda")
    with binding.Stereo(0) as st:
        st.set_test_flags(binding.DCO_TEST_REFUSE_WIDE)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            st.match(left, right, D, None, out)
        stream.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
        assert st.workspace_allocated() == _narrow(binding)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):   # an allocation or a synchronisation would end the capture
            st.match(left, right, D, None, out)
        out.fill_(-7)
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
        # the device gives again: a call that fits does not ask, a reserve does
        st.set_test_flags(0)
        assert np.array_equal(st.match(left, right, D).cpu().numpy(), want)
        assert st.workspace_allocated() == _narrow(binding)
        st.reserve(W, H, D)
        assert st.workspace_allocated() == binding.Stereo.workspace_bytes(W, H, D)


def test_reserve_and_batches_take_the_narrow_plan(env):
    torch, binding, left, right, want = env
    from paper_2203_02300_gb300.batch import BatchGraph
    with binding.Stereo(0) as st:
        st.set_test_flags(binding.DCO_TEST_REFUSE_WIDE)
        st.reserve(W, H, D)
        assert st.workspace_allocated() == _narrow(binding)
        for got in BatchGraph(st, [(W, H, D)] * 2)([left] * 2, [right] * 2):
            assert np.array_equal(got.cpu().numpy(), want)
    # groups of a budget: each as wide as the budget allows, or narrow
    budget = binding.Stereo.workspace_bytes(W, H, D) + 1000
    outs = [torch.empty((H, W), dtype=torch.int16, device="cuda") for _ in range(9)]
    for flag in (0, binding.DCO_TEST_REFUSE_WIDE):
        with binding.Stereo(0, budget_bytes=budget) as st:
            st.set_test_flags(flag)
            st.match_batch([(left, right, D, o) for o in outs])
            torch.cuda.synchronize()
            assert st.workspace_allocated() <= budget and st.batch_groups() > 1
            for o in outs:
                assert np.array_equal(o.cpu().numpy(), want)
                o.fill_(-7)


def test_a_large_batch_bounds_its_slices(env):
    # from 65 pairs on the pairs share 32 GiB of slices
    torch, binding, left, right, want = env
    w, h, n = 640, 360, 200   # alone: one pass of 256 (472 MB); among 200: passes of 64
    s = scenes.plane_scene(w, h, 256, 6, seed=scenes.seed_for(8, 78), drange=(2, 250), noise_sigma=2.0, texture="mixed")
    a, b = torch.from_numpy(s.left).cuda(), torch.from_numpy(s.right).cuda()
    outs = [torch.empty((h, w), dtype=torch.int16, device="cuda") for _ in range(n)]
    with binding.Stereo(0) as st:
        st.match_batch([(a, b, 256, o) for o in outs])
        torch.cuda.synchronize()
        assert st.workspace_allocated() < (36 << 30)
        alone = st.match(a, b, 256)
        for o in outs:
            assert torch.equal(o, alone)
