"""Environments that run in the launch shape chosen from their size, on both
sides of each line of that choice, against the oracle: 18 steps per call, one
launch of 16 and one of 2."""
import numpy as np
import pytest

import oracle
from paper_2510_01764_gb300 import workloads as W
from test_gpu_parity import full_compare

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_01764_gb300 import build

    build.build()
    oracle.build()


@pytest.mark.parametrize("per_sm,over", [(0, 1), (0, 5), (8, 0), (8, 1), (16, 0), (16, 1), (32, 0), (32, 1), (192, 0), (192, 1)])
def test_chip8(per_sm, over):
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over
    games = [W.replace(g, max_episode_steps=7, sticky_prob=0.25, max_noops=3) for g in W.cfg_shooter().games]
    full_compare(games, n, 18, seed=n, action_seed=n, game_of_env=(np.arange(n) % 3).astype(np.uint16), use_step_n=True)


@pytest.mark.parametrize("per_sm,over", [(0, 3), (8, 1), (16, 1), (129, 0)])
def test_schip(per_sm, over):
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over
    games = [W.replace(W.random_schip_game(41), max_episode_steps=5)]
    full_compare(games, n, 3 if n > 10000 else 18, seed=n, action_seed=n, use_step_n=True)
