"""Env.launch gives the shape that runs, and set_launch keeps the fields it is
not given, on both sides of each line of the choice by size."""
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


def make(per_sm, over, schip=False):
    from paper_2510_01764_gb300 import octax as o

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = W.TemplateParams(seed=1)
    return o.Env([W.schip_template_game(p) if schip else W.template_game(p)], per_sm * sms + over, seed=1)


LINES = [(0, 1, 64, 1), (8, 0, 64, 1), (8, 1, 64, 2), (16, 0, 64, 2), (16, 1, 128, 4), (32, 0, 128, 4),
         (32, 1, 128, 8), (192, 0, 128, 8), (192, 1, 128, 16)]


@pytest.mark.parametrize("per_sm,over,block,ipw", LINES)
def test_chosen_shape(per_sm, over, block, ipw):
    own = dict(block=block, inst_per_warp=ipw, steps_per_launch=16, persistent=0, use_graph=1, writer_warps=0, balance=0)
    env = make(per_sm, over)
    assert env.launch == own
    env.set_launch(use_graph=0)
    assert env.launch == dict(own, use_graph=0)
    env.set_launch(steps_per_launch=3, persistent=1)
    assert env.launch == dict(own, use_graph=0, steps_per_launch=3, persistent=1)
    env = make(per_sm, over)
    env.set_launch(**env.launch)
    assert env.launch == own


def test_chosen_shape_schip():
    assert make(192, 1, schip=True).launch["inst_per_warp"] == 8


@pytest.mark.parametrize("per_sm,over", [(0, 64), (16, 1), (192, 1)])
@pytest.mark.parametrize("kw", [dict(writer_warps=1), dict(writer_warps=2), dict(writer_warps=2, persistent=1),
                                dict(block=256, writer_warps=4), dict(block=128, writer_warps=1)])
def test_writer_warps_alone(per_sm, over, kw):
    """Accepted whatever shape was chosen, as on 64 threads x 8 instances."""
    env = make(per_sm, over)
    env.set_launch(**kw)
    got = env.launch
    assert got["writer_warps"] == kw["writer_warps"] and got["block"] == kw.get("block", got["block"])
    assert got["block"] // 32 * got["inst_per_warp"] // got["writer_warps"] in (8, 16, 32)


def test_what_is_refused_stays_refused():
    from paper_2510_01764_gb300 import octax as o

    env = make(0, 64)
    before = env.launch
    for kw in (dict(writer_warps=3), dict(block=48), dict(inst_per_warp=33), dict(steps_per_launch=0),
               dict(block=32, inst_per_warp=4, writer_warps=1), dict(block=64, inst_per_warp=1, writer_warps=1)):
        with pytest.raises(o.OctaxError):
            env.set_launch(**kw)
        assert env.launch == before
    env.set_launch(block=64, inst_per_warp=1)  # chosen by hand now
    with pytest.raises(o.OctaxError):
        env.set_launch(writer_warps=1)
    with pytest.raises(o.OctaxError):
        make(0, 64, schip=True).set_launch(writer_warps=2)


def test_a_failed_autotune_leaves_the_chosen_shape():
    from paper_2510_01764_gb300 import octax as o

    env = make(16, 1)
    before = env.launch
    with pytest.raises(o.OctaxError):
        env.autotune(0)
    assert env.launch == before


@pytest.mark.parametrize("games,each,block,ipw", [(64, 1, 32, 1), (700, 2, 64, 1), (700, 3, 64, 2), (700, 4, 128, 1),
                                                  (700, 16, 128, 4), (700, 17, 128, 8), (1200, 32, 128, 8),
                                                  (1200, 33, 128, 16)])
def test_many_games(games, each, block, ipw):
    """CTAs of one game each, cut to the instances it has where these are at most
    half of what the size alone gives a CTA; the results stay those of any shape."""
    import numpy as np

    from paper_2510_01764_gb300 import octax as o

    rng = np.random.default_rng(games + each)
    gs = [W.random_game(900 + r) for r in range(8)]
    n = games * each
    goe = rng.permutation(np.arange(n) % games).astype(np.uint16)
    env = o.Env([gs[g % 8] for g in range(games)], n, game_of_env=goe, seed=2)
    assert (env.launch["block"], env.launch["inst_per_warp"]) == (block, ipw)
    ref = o.Env(gs, n, game_of_env=goe % 8, seed=2)
    ref.set_launch(block=64, inst_per_warp=8, steps_per_launch=4)
    acts = torch.from_numpy(W.actions(4, 0, 12, n)).cuda()
    for x, y in zip(env.step_n_packed(acts), ref.step_n_packed(acts)):
        assert torch.equal(x, y)
    assert torch.equal(env.state_hash(), ref.state_hash())
