"""The network where its launches change: one, two and three batches of 8 per
CTA of the conv kernel, one and two tiles of 128 per CTA of the heads kernel
(an odd number of tiles too), ragged ends. An instance's outputs are sums in
one order whatever the size of the call, so they equal those of small calls
bit for bit; the first and last instances are compared with the oracle within
the bounds of test_gpu_policy. Repeated calls agree (each role of the conv
kernel runs at its own pace)."""
import numpy as np
import pytest

from paper_2510_01764_gb300 import workloads as W
from test_gpu_policy import check_outputs, pack, random_frames

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_01764_gb300 import build

    build.build()


@pytest.mark.parametrize("per_sm,over,L", [(8, 0, 5), (8, 1, 5), (16, -3, 17), (17, 9, 5), (64, 0, 5), (64, 129, 1)])
def test_sizes(per_sm, over, L):
    from paper_2510_01764_gb300 import octax as o

    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over
    params = W.policy_params(n, L)
    obs = random_frames(n, 0.1, n)
    pol = o.Policy(params, max_envs=n)
    words = torch.from_numpy(pack(obs)).cuda()
    want = pol.forward(words, seed=6, step=2)
    pol.sync()
    u8 = torch.from_numpy(obs * 3).cuda()  # any nonzero byte is a lit pixel
    for _ in range(3):
        for got in (pol.forward(words, seed=6, step=2), pol.forward_u8(u8, seed=6, step=2)):
            pol.sync()
            assert all(torch.equal(x, y) for x, y in zip(want, got))
    for a in (0, max(0, n - 261)):
        lg, v, _ = pol.forward(words[a:a + 261].contiguous(), seed=6, step=2)
        pol.sync()
        assert torch.equal(lg, want[0][a:a + 261]) and torch.equal(v, want[1][a:a + 261])
    idx = np.unique(np.r_[0:9, n - 9:n])
    check_outputs(params, obs[idx], want[0][idx], want[1][idx])
