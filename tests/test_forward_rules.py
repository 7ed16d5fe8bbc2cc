"""The forward's sizing rules (host, no GPU): blocks shrink for scenes of few
units only, also where the number of units passes 2^32; the live-unit list is
bounded and its passes cover every run."""
import pytest

from tests import rules_lib


@pytest.fixture(scope="module")
def rules():
    return rules_lib.load()


def test_small_blocks_for_few_units(rules):
    # 32 x 32 scan, 1,024 points: one unit a tile, blocks of 64 pairs give 256 units
    assert rules.pairs_of_block(512, 32, 1, 512, 152) == 64
    assert rules.pairs_of_block(512, 76, 1, 1024, 152) == 512
    assert rules.pairs_of_block(512, 1, 1, 1, 152) == 64
    assert rules.pairs_of_block(256, 151, 1, 256, 152) == 128


# products of 2^32 and a little more: as 32-bit numbers they are below the number of SMs
@pytest.mark.parametrize("tiles,windows,pairs", [(1 << 16, 1 << 6, 512 << 10), (1 << 21, 1, 512 << 11),
                                                 (1431655766, 1, 3 * 512), (1 << 20, 64, (1 << 30) - 1)])
def test_many_units_keep_whole_blocks(rules, tiles, windows, pairs):
    assert (tiles * windows * -(-pairs // 512)) % (1 << 32) < 152 or pairs == (1 << 30) - 1
    assert rules.pairs_of_block(512, tiles, windows, pairs, 152) == 512


@pytest.mark.parametrize("runs,blocks", [(1, 1), (512, 1024), (4096, 1024), (4097, 1024), (2048, 16384),
                                         (7, 1 << 22), (7, (1 << 22) + 1), (3, 1 << 23), (17477, 240),
                                         ((1 << 32) - 1, 1)])
def test_list_passes(rules, runs, blocks):
    per = rules.pass_runs(runs, blocks)
    most = max(1, rules.list_entries() // blocks)
    assert 1 <= per <= most
    passes = -(-runs // per)
    assert passes == -(-runs // most)  # no more of them than the bound asks for
    assert runs * blocks > rules.list_entries() or passes == 1
