"""The micro-op table and the datapath it feeds, where they can go wrong: ROM
lengths at the ends of the table, a launch without room for the table, and
every datapath instruction from an even address (table) and from an odd one
(the general switch), under every quirk set and several lane splits, all
against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2510_01764_gb300 import workloads as W
from paper_2510_01764_gb300.workloads import GameSpec
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


def shape(ipw):
    return dict(block=64, inst_per_warp=ipw, steps_per_launch=4, persistent=0, use_graph=1)


@pytest.mark.parametrize("ipw", [1, 3, 16])
def test_rom_lengths(ipw):
    """One byte, odd lengths, and the longest ROMs: successors, skips and
    jumps that leave the table."""
    games = [W.replace(W.random_game(700 + k), rom=W.random_opcode_rom(700 + k)[:length])
             for k, length in enumerate((1, 2, 3, 4, 5, 6, 7, 63, 64, 65, 3582, 3583, 3584))]
    n = 13 * 8
    full_compare(games, n, 40, seed=6, action_seed=6, game_of_env=(np.arange(n) % 13).astype(np.uint16),
                 launch=shape(ipw), use_step_n=True)


def test_launch_without_table():
    """256 threads x 22 Super-CHIP instances per warp leave no room beside
    their records for the table of a 3,584-byte ROM."""
    games = [W.random_schip_game(3100 + r) for r in range(2)]
    n = 360
    full_compare(games, n, 24, seed=4, action_seed=4, game_of_env=(np.arange(n) % 2).astype(np.uint16),
                 launch=dict(block=256, inst_per_warp=22, steps_per_launch=6, persistent=0, use_graph=1),
                 use_step_n=True)


def straight_line(seed, start, count=400, schip=False):
    """16 random registers, then `count` datapath instructions with no jumps, from address `start`."""
    rng = np.random.default_rng(seed)
    ops = [0xC0FF | x << 8 for x in range(16)]
    for _ in range(count):
        x, y, nn = (int(v) for v in rng.integers(0, (16, 16, 256)))
        kind = int(rng.integers(0, 17 if schip else 16))
        ops.append([0x3000 | x << 8 | nn, 0x4000 | x << 8 | nn, 0x5000 | x << 8 | y << 4,
                    0x6000 | x << 8 | nn, 0x7000 | x << 8 | nn, 0x9000 | x << 8 | y << 4,
                    0xA000 | x << 8 | nn, 0xE09E | x << 8, 0xE0A1 | x << 8, 0xF007 | x << 8,
                    0xF015 | x << 8, 0xF018 | x << 8, 0xF029 | x << 8, nn, 0xF01E | x << 8,
                    0x8000 | x << 8 | y << 4 | (0, 1, 2, 3, 4, 5, 6, 7, 14)[nn % 9],
                    0xF030 | x << 8][kind])
    code = b"".join(op.to_bytes(2, "big") for op in ops)
    return (0x1000 | start).to_bytes(2, "big") + bytes(start - 0x202) + code


@pytest.mark.parametrize("quirks", [0, 0x01, 0x04, 0x20, 0x3F])
@pytest.mark.parametrize("variant", ["chip8", "schip"])
def test_datapath_from_even_and_odd_addresses(quirks, variant):
    schip = variant == "schip"
    games = [GameSpec(rom=straight_line(90 + k // 2, 0x204 + k % 2, schip=schip), instr_per_frame=7, frameskip=2,
                      stack_frames=2, action_set=(1, 2, 3, 12), variant=variant) for k in range(8)]
    n = 8 * 12
    for ipw in (4, 32):
        full_compare(games, n, 32, seed=quirks + 1, action_seed=2, quirks=quirks,
                     game_of_env=(np.arange(n) % 8).astype(np.uint16), launch=shape(ipw))
