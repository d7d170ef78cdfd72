"""Calls captured into a CUDA graph by the caller."""
import numpy as np
import pytest

import oracle
from paper_2510_01764_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_01764_gb300 import build

    build.build()
    oracle.build()


@pytest.mark.parametrize("n", [3, 1000])
def test_a_shape_first_used_under_capture(n):
    """A shape whose group table does not exist yet, first used inside a capture
    that allows allocations: the table is there for the graph's replays, and for
    calls outside the graph before it was ever replayed."""
    from paper_2510_01764_gb300 import octax as o

    games = W.cfg_shooter().games
    goe = (np.arange(n) % 3).astype(np.uint16)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        env = o.Env(games, n, seed=2, game_of_env=goe, stream=st)
        acts = torch.from_numpy(W.actions(2, 0, 3, n, 5)).cuda()
        a = torch.empty(n, dtype=torch.uint8, device="cuda")
        out = (torch.empty(env.obs_shape, dtype=torch.uint8, device="cuda"), torch.empty(n, device="cuda"),
               torch.empty(n, dtype=torch.uint8, device="cuda"))
    st.synchronize()
    env.set_launch(block=32, inst_per_warp=5, steps_per_launch=1, persistent=0, use_graph=0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st, capture_error_mode="relaxed"):
        env.step(a, out)
    ref = oracle.OracleEnv(games, n, seed=2, game_of_env=goe)
    for k in range(3):
        with torch.cuda.stream(st):
            a.copy_(acts[k])
            if k == 1:
                graph.replay()
            else:
                env.step(a, out)
        st.synchronize()
        o2, r2, d2 = ref.step(acts[k].cpu().numpy())
        assert np.array_equal(out[0].cpu().numpy(), o2)
        assert np.array_equal(out[1].cpu().numpy(), r2) and np.array_equal(out[2].cpu().numpy(), d2)
