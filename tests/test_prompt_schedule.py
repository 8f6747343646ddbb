"""The order of the prompt phase's items, replayed on the host (tests/prompt_replay.cpp compiled against csrc/mkv_schedule.h)
for prompts of equal and of different lengths."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2503_00979_b200", "csrc")


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("prompt") / "prompt_replay")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "prompt_replay.cpp"), "-o", exe], check=True)

    def run(kv_heads, layers, tiles, longest, lens=()):
        args = [kv_heads, layers, tiles, longest, *(longest - n for n in lens)]
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True)
        assert r.returncode == 0 and "ok" in r.stdout, f"{args}: {r.stdout}{r.stderr}"
        return int(r.stdout.split()[-1])

    return run


@pytest.mark.parametrize("tiles", [1, 3, 8, 14])
@pytest.mark.parametrize("lens", [
    (),                                              # equal lengths, as one number
    (3000,) * 8,                                     # equal lengths, row by row
    (3000, 900, 2400, 1200, 2900, 760, 1800, 2100),  # a quarter to the whole
    (3000, 130, 140, 180, 129, 128, 1, 127),         # one long prompt among short ones
    (1, 3000), (3000, 1024), (2999, 2945, 3000),
])
def test_runs_in_order(replay, tiles, lens):
    for kv_heads, layers in ((8, 32), (2, 5), (1, 1), (16, 3)):
        assert replay(kv_heads, layers, tiles, 3000, lens) > 0


def test_long_prompts_and_many_rows(replay):
    replay(8, 4, 8, 131072)
    replay(2, 3, 8, 40000, (40000, 300, 39999, 20000))
    for rows in (64, 511, 512, 513, 1500):
        replay(2, 3, 8, 2000, [2000 - 29 * (b % 61) for b in range(rows)])


@pytest.mark.parametrize("kv_heads,layers,P", [(8, 1, 25600), (8, 1, 12800), (2, 4, 20000), (2, 2, 40000), (1, 1, 40000), (1, 1, 200000),
                                               (8, 2, 10000), (4, 28, 1200), (2, 32, 568), (8, 16, 164), (8, 8, 2000), (8, 8, 1486),
                                               (8, 16, 1158), (8, 32, 600), (4, 28, 560), (1, 1, 100), (8, 1, 32768)])
def test_share_of_the_busiest(replay, kv_heads, layers, P):
    replay(kv_heads, layers, 0, P)
    replay(kv_heads, layers, 0, P, (P, P // 4, P // 2, P - 1))
