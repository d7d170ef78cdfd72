"""Forwards of more instances than one launch of the conv kernel takes, and the
device memory a policy keeps."""
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


@pytest.mark.parametrize("over", [0, 1, 3001])
def test_every_instance_as_alone(over):
    """64 batches of 8 instances per SM are one launch; what lies around the
    launches' seam and at the ends equals, bit for bit, a small forward of it."""
    from paper_2510_01764_gb300 import octax as o

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 64 * 8 * sms + over
    pol = o.Policy(W.policy_params(2, 5), max_envs=n)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(over)
    words = torch.randint(-2 ** 62, 2 ** 62, (n, 4, 32), dtype=torch.int64, device="cuda", generator=gen)
    words &= torch.randint(-2 ** 62, 2 ** 62, (n, 4, 32), dtype=torch.int64, device="cuda", generator=gen)
    frames = ((words.unsqueeze(-1) >> torch.arange(64, device="cuda")) & 1).to(torch.uint8)
    torch.cuda.synchronize()  # the policy has a stream of its own
    lg, v, _ = pol.forward(words, seed=3)
    pol.sync()
    lg8, v8, _ = pol.forward_u8(frames, seed=3)
    pol.sync()
    assert torch.equal(lg, lg8) and torch.equal(v, v8)
    step = 4096
    for a in range(0, n, step):
        x, y, _ = pol.forward(words[a:a + step].contiguous())
        pol.sync()
        assert torch.equal(x, lg[a:a + step]) and torch.equal(y, v[a:a + step]), a


def test_memory_per_instance():
    """2 KB of features and 2 KB of rollout observations per instance, and what
    one conv launch keeps, whatever the size."""
    from paper_2510_01764_gb300 import octax as o

    def taken(n):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        pol = o.Policy(W.policy_params(2, 5), max_envs=n)
        got = before - torch.cuda.mem_get_info()[0]
        del pol
        return got

    taken(1)
    assert taken(1_000_000) - taken(500_000) < 500_000 * 4096 + (16 << 20)
    assert taken(1_000_000) < 1_000_000 * 4096 + (400 << 20)
