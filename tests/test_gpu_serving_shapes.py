"""The server where a tick's shape and copies change: two waves of requests of
different lengths, so that the second is admitted into gaps the first left
(runs of neighbouring slots and single ones), with many, few and one instances
left per tick; every request against the oracle."""
import pytest

import oracle
from test_gpu_serving import games, make_requests, octax, run_all

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_01764_gb300 import build

    build.build()
    oracle.build()


@pytest.mark.parametrize("block,ipw,max_envs", [(128, 16, 4096), (64, 8, 700), (32, 1, 40)])
def test_two_waves(block, ipw, max_envs):
    gs = games()
    reqs = make_requests(40, block + ipw, max_envs=max_envs)
    most = max(sum(r["actions"].shape[1] for r in reqs) // 2, max(r["actions"].shape[1] for r in reqs))
    server = octax().Server(gs, memory_budget_bytes=most * 4484, block=block, inst_per_warp=ipw)
    _, _, outs = run_all(server, reqs)
    for r, (obs, rew, done) in zip(reqs, outs):
        n = r["actions"].shape[1]
        ref = oracle.OracleEnv([gs[r["game"]]], n, seed=r["seed"])
        ref.reset()
        o2, r2, d2, _ = ref.rollout(r["actions"], obs=True)
        assert (obs.numpy() == o2).all() and (rew.numpy() == r2).all() and (done.numpy() == d2).all()
    server.close()
