"""A server whose ticks fill the device runs the instances per warp it was
configured with, also above what the spread by size ever gives."""
import numpy as np
import pytest

from paper_2510_01764_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_01764_gb300 import build

    build.build()


@pytest.mark.parametrize("variant,block,ipw,requests,n",
                         [("chip8", 128, 32, 9, 4093), ("chip8", 256, 32, 9, 4093), ("chip8", 128, 16, 9, 4093),
                          ("schip", 128, 16, 3, 2047), ("schip", 256, 16, 3, 2047)])
def test_as_plain_environments(variant, block, ipw, requests, n):
    from paper_2510_01764_gb300 import octax as o

    games = [W.random_game(70 + r) if variant == "chip8" else W.random_schip_game(70 + r) for r in range(3)]
    frame = o.frame_shape(variant)
    server = o.Server(games, memory_budget_bytes=requests * n * 5300, block=block, inst_per_warp=ipw)
    rng = np.random.default_rng(ipw)
    items = []
    for k in range(requests):
        acts = rng.integers(0, 5, size=(3, n), dtype=np.uint8)
        out = (torch.zeros((3, n, 4) + frame, dtype=torch.uint8, device="cuda"),
               torch.zeros((3, n), dtype=torch.float32, device="cuda"), torch.zeros((3, n), dtype=torch.uint8, device="cuda"))
        items.append((k % 3, acts, 11 + k, out))
    torch.cuda.synchronize()
    server.wait_batch(server.submit_batch(items))
    assert server.stats()["peak_active_envs"] == requests * n
    for game, acts, seed, out in items:
        env = o.Env([games[game]], n, seed=seed)
        want = env.step_n(torch.from_numpy(acts).cuda())
        env.sync()
        assert all(torch.equal(x, y) for x, y in zip(want, out))
    server.close()
