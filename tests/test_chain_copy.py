"""The copying warp of the one-kernel models against a model of its barriers, on the host.

A wait that gives up cannot be provoked on a GPU without hanging something, so the order of copies, waits and cluster
barriers is a plain C++ template (csrc/chain_copy.cuh) that runs here with every one of its waits failing in turn: after
that nothing may be copied (the buffer was not handed back, its barrier may be armed), what is in flight must be waited for
before the block ends, and the cluster's barriers must all be taken part in.
"""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("chain") / "model")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Wno-unknown-pragmas", "-I", os.path.join(ROOT, "paper_1901_05350_b200", "csrc"),
                    os.path.join(ROOT, "tests", "chain_copy_model.cpp"), "-o", exe], check=True)
    return lambda *args: subprocess.run([exe, *map(str, args)], capture_output=True, text=True, check=True).stdout.strip()


def random_ops(rng, n):
    """[stem, blocks ..., pool] as flat numbers: block?, units, groups, group_cols, tile_cols, Co, n_chunks."""
    flat = [0, 3, 1, 8, 8, 8, 1]
    for _ in range(n):
        tile = 8 * rng.randint(1, 8)
        cols = tile * rng.randint(1, 3)
        co = 8 * rng.randint(1, 40)
        groups = -(-co // cols)
        flat += [1, groups * rng.randint(1, 5), groups, cols, tile, co, rng.randint(1, 4)]
    return n + 2, flat + [0, 1, 1, 8, 8, 8, 1]


@pytest.mark.parametrize("seed", range(8))
def test_every_wait_of_the_copying_warp_may_give_up(model, seed):
    rng = random.Random(seed)
    n_ops, ops = random_ops(rng, rng.randint(0, 5))
    cs = rng.choice([1, 2, 4, 8, 16])
    images, rank = rng.randint(1, 3), rng.randrange(cs)
    ok, copies, waits = model(images, cs, rank, -1, n_ops, *ops).split()
    assert ok == "ok"
    for fail_at in range(min(int(waits), 60)):
        said = model(images, cs, rank, fail_at, n_ops, *ops)
        assert said.startswith("ok "), (fail_at, said)
        assert int(said.split()[1]) <= int(copies)
