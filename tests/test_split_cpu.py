"""The split of a batch over the SMs (host code of the fused path), over the prompts that a launch may hold."""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_02631_b200", "csrc")
SMS, TILE = 148, 128


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    from paper_2603_02631_b200.build import _nvcc
    exe = str(tmp_path_factory.mktemp("split") / "split_check")
    subprocess.run([_nvcc(), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    "-o", exe, os.path.join(ROOT, "tests", "split_check.cu")], check=True, capture_output=True, timeout=600)

    def run(batches, forms=False):
        text = "".join(" ".join(map(str, [*geom, *lens])) + "\n" for geom, lens in batches)
        out = subprocess.run([exe] + ["forms"] * forms, input=text, capture_output=True, text=True, check=True, timeout=300).stdout.splitlines()
        rows = [[int(x) for x in line.split()] for line in out]
        if forms:
            return rows
        return [(bool(r[0]), r[1], bool(r[2]), [tuple(r[i:i + 3]) for i in range(3, len(r), 3)]) for r in rows]

    return run


def test_one_long_prompt_and_several_of_a_few_tiles_share_a_launch(split):
    """The short ones are rounded up to a CTA each, which the long one has to give."""
    geom = (16, 8, 4, 64, 8, 2)
    batches = [(geom, [314, 111488, 378, 19]), (geom, [100000] + [20] * 15), (geom, [20] * 15 + [140000]), (geom, [1] * 16)]
    for (_, lens), (same, n, ok, _) in zip(batches, split(batches)):
        assert same and ok and n == len(lens), lens


def test_every_batch_that_is_grouped_is_split(split):
    rng = random.Random(5)
    batches = []
    for _ in range(4000):
        group, m = rng.choice([(1, 8), (2, 8), (3, 8), (4, 8), (4, 16), (8, 4), (1, 16)])
        geom = (rng.choice([1, 2, 16, 28]), rng.choice([1, 2, 8]), group, rng.choice([64, 128]), m, rng.choice([1, 2]))
        lens = [int(2 ** rng.uniform(0, rng.choice([9, 13, 17]))) for _ in range(rng.randint(2, 16))]
        batches.append((geom, lens))
    seen = 0
    for (geom, lens), (same, n, ok, prompts) in zip(batches, split(batches)):
        if not same:
            continue                                       # refused, or of both forms: not one launch
        seen += 1
        assert ok and n >= 1, (geom, lens)
        assert sum(parts * per_part for parts, per_part, _ in prompts) <= SMS
        for length, (parts, per_part, tiles) in zip(lens, prompts):
            assert 1 <= parts <= geom[0] * geom[1] and per_part * tiles >= -(-length // TILE), (geom, lens)
    assert seen > 3000


@pytest.mark.parametrize("geom,registers,kept,twice", [
    # group, d, m, bytes per key element; the most tiles an SM with the maxima in registers, with the logits kept, and the next more
    ((4, 64, 8, 2), 8, 8, 9), ((2, 64, 16, 2), 0, 6, 7), ((4, 128, 8, 2), 8, 10, 11), ((1, 64, 32, 2), 0, 5, 6),
    ((4, 64, 8, 1), 5, 5, 6), ((2, 64, 16, 1), 0, 3, 4), ((4, 128, 8, 1), 8, 8, 9), ((1, 64, 32, 1), 0, 2, 3),
    ((1, 64, 16, 2), 0, 10, 11), ((2, 64, 8, 2), 8, 12, 13), ((4, 64, 4, 2), 8, 23, 24), ((8, 64, 2, 2), 8, 25, 26),
    ((1, 64, 16, 1), 0, 10, 11), ((2, 64, 8, 1), 8, 19, 20), ((1, 128, 16, 1), 0, 14, 15), ((2, 128, 8, 1), 8, 19, 20), ((2, 128, 8, 2), 8, 19, 20),
    ((4, 64, 16, 2), 0, 0, 1)])
def test_form_by_tiles(split, geom, registers, kept, twice):
    """The edges that the tests on the GPU are placed at."""
    group, d, m, element = geom
    for tiles, form in ((registers, 2), (registers + 1, 1 if kept > registers else 0), (kept, 2 if kept == registers else 1), (twice, 0)):
        if tiles > 0:
            assert split([((3, 1, group, d, m, element), [(tiles - 1) * SMS * TILE + 1, tiles * SMS * TILE])], forms=True) == [[form, form]], tiles
