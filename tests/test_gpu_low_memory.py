"""Programs that run in the memory below the ROM, on both sides of the ROM
length from which the micro-op table covers it, against the oracle."""
import numpy as np
import pytest

import oracle
from chip8_prog import rom
from paper_2510_01764_gb300 import workloads as W
from paper_2510_01764_gb300.workloads import Clause, GameSpec, Term
from test_gpu_parity import full_compare

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PROGRAMS = [
    [0x7A01, 0x1100],                          # through the zeros into the ROM again
    [0x7A01, 0x1000],                          # from address 0, over the font
    [0x7A01, 0x1101],                          # the same at odd addresses: a wait at the ROM's odd start
    [0x607B, 0x6105, 0xA150, 0xF155, 0x1140],  # an instruction written below the ROM, then met: VB += 5
    [0x6020, 0xB000],                          # BNNN into the zeros
    [0x7A01, 0x00EE],                          # a return from an empty stack: address 0
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_01764_gb300 import build

    build.build()
    oracle.build()


@pytest.mark.parametrize("variant", ["chip8", "schip"])
@pytest.mark.parametrize("length", [3071, 3072, 3073, 3584])
def test_programs(length, variant):
    games = [GameSpec(rom=rom(p).ljust(length, b"\0"), instr_per_frame=23, frameskip=4, action_set=(7, 9, 5, 8),
                      max_episode_steps=17, score=(Term("reg", 10), Term("reg", 11)),
                      term=(Clause(Term("reg", 11), ">=", 40),), variant=variant) for p in PROGRAMS]
    make = W.random_opcode_rom if variant == "chip8" else W.random_schip_rom
    games += [W.replace(games[0], rom=make(60 + r, n_bytes=length), instr_per_frame=10) for r in range(10)]
    n = 5 * len(games)
    env, ref = full_compare(games, n, 40, seed=length, action_seed=4, use_step_n=True,
                            game_of_env=(np.arange(n) % len(games)).astype(np.uint16))
    assert (ref.records()["env_steps"] == 40).all()
