"""The writer-warp kernel where several lanes emulate one instance: what those
lanes share (the call stack) and where they have to meet."""
import time

import numpy as np
import pytest

import oracle
from chip8_prog import prog
from paper_2510_01764_gb300 import workloads as W
from paper_2510_01764_gb300.workloads import Clause, Term
from test_gpu_parity import full_compare, hashes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# 16, 8 and 4 lanes to an instance, one to four instances of the lanes' own per pass of a writer warp
SHAPES = [dict(block=128, inst_per_warp=2, writer_warps=1), dict(block=64, inst_per_warp=4, writer_warps=1),
          dict(block=64, inst_per_warp=8, writer_warps=2), dict(block=256, inst_per_warp=1, writer_warps=1)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_01764_gb300 import build

    build.build()
    oracle.build()


@pytest.mark.parametrize("persistent", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_returns_just_before_a_reset(shape, persistent):
    """Returns fall on every one of a step's last instructions, and the step
    after often ends the episode: the reset clears the stack those returns read.
    What follows a return decides the score and the episode's end."""
    words = [0x2208, 0x7301, 0x7A01, 0x1200,  # call; V3 and VA count the returns
             0xC103, 0x3100, 0x7401, 0x00EE]  # one to two instructions more or less before the return
    g = prog(words, instr_per_frame=7, frameskip=4, max_episode_steps=3, score=(Term("reg", 3),),
             term=(Clause(Term("reg", 4), ">=", 5), Clause(Term("reg", 10), "==", 7)))
    env, ref = full_compare([g], 517, 40, seed=6, use_step_n=True,
                            launch=dict(shape, persistent=persistent, steps_per_launch=8, use_graph=0))
    assert (ref.records()["episode_steps"] < 3).all()


@pytest.mark.parametrize("persistent", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_a_stalled_hand_over_ends_every_lane_alike(shape, persistent):
    """The writers skip their hand-over, so the emulators' waits run out, in the
    middle of programs that draw and write memory (where the lanes of an instance
    meet). The call ends within seconds, over several groups per CTA too, is
    reported once and leaves no state; the next call is exact."""
    from paper_2510_01764_gb300 import octax as o

    games = W.cfg_divergence(n_envs=64).games[:2]
    n = 24001 if persistent else 515
    goe = (np.arange(n) % 2).astype(np.uint16)
    env = o.Env(games, n, game_of_env=goe, seed=5)
    env.set_launch(**dict(shape, persistent=persistent, steps_per_launch=2, use_graph=0))
    h0 = hashes(env)
    acts = W.actions(5, 0, 2, n, 5)
    a_dev = torch.from_numpy(acts).cuda()
    env.debug_stall_writers(True)
    t0 = time.monotonic()
    env.step_n(a_dev)
    with pytest.raises(o.OctaxError) as ei:
        env.sync()
    assert ei.value.code == o.ECUDA and time.monotonic() - t0 < 20.0
    assert np.array_equal(hashes(env), h0)
    env.debug_stall_writers(False)
    obs, rew, done = env.step_n(a_dev)
    env.sync()
    ref = oracle.OracleEnv(games, n, game_of_env=goe, seed=5)
    _, r2, d2, _ = ref.rollout(acts, obs=False)
    assert np.array_equal(rew.cpu().numpy(), r2) and np.array_equal(done.cpu().numpy(), d2)
    assert np.array_equal(hashes(env), ref.hashes())
