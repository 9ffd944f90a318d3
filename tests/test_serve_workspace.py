"""The serving lanes' workspace does not grow while frames are served: bursts of
the large streams' frames, which share a batch, allocate nothing."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# the small stream comes first and has most slots of a batch in stream order
SHAPES = [(320, 240, 64), (640, 480, 128), (640, 480, 128)]
TILES = [(64, 0, 0), (128, 0, 0), (128, 0, 0)]


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_02300_gb300 import binding
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    return torch, binding


def _frames(torch):
    rng = np.random.default_rng(5)
    return [[torch.from_numpy(rng.integers(0, 256, (H, W, 3), dtype=np.uint8)).pin_memory() for _ in range(2)]
            for W, H, _ in SHAPES]


def test_native_lanes_hold_the_largest_admissible_batch(env):
    torch, binding = env
    frames = _frames(torch)
    with binding.NativeServer(SHAPES, lanes=2, tiles=TILES) as srv:
        outs = [[torch.empty((H, W), dtype=torch.int16).pin_memory().numpy() for _ in range(12)] for W, H, _ in SHAPES]
        free = torch.cuda.mem_get_info()[0]
        for _ in range(4):   # the first frames occupy the lanes, the later ones share batches
            tickets = [srv.submit(s, frames[s][0].numpy(), frames[s][1].numpy(), outs[s][k])
                       for k in range(12) for s in (1, 2, 0)]
            for t in tickets:
                srv.wait(t)
        c = srv.counters()
        both = sum(binding.Stereo.workspace_bytes(*SHAPES[s], binding.Tile(*TILES[s]).apply(binding.Params.default()))
                   for s in (1, 2))
        assert both <= c["max_batch_bytes"] <= c["lane_budget"]   # two large frames did share a batch
        assert torch.cuda.mem_get_info()[0] >= free - (4 << 20)


def test_python_lanes_hold_the_largest_admissible_batch(env):
    torch, binding = env
    from paper_2203_02300_gb300.serve import Server
    frames = _frames(torch)
    srv = Server(SHAPES, lanes=2, tiles=TILES)
    try:
        held = [ln.stereo.workspace_allocated() for ln in srv.lanes]
        for f in [srv.submit(s, *frames[s]) for _ in range(12) for s in (1, 2, 0)]:
            f.result(timeout=60)
        assert [ln.stereo.workspace_allocated() for ln in srv.lanes] == held
        assert min(held) >= sum(binding.Stereo.workspace_bytes(*SHAPES[s], binding.Tile(*TILES[s]).apply(binding.Params.default()))
                                for s in (1, 2))
    finally:
        srv.close()
