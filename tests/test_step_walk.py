"""The stages of packed weights that a group of gemm_tmw_kernel's decoding warps walks: in a model of the kernel's barriers that uses
the kernel's own index arithmetic, with loads that land in any order, no group reads a stage before it is full or after it is freed.
For the rings of either container (SPR steps per stage), four and eight stages of decoded weights, tiles of one step to many with odd
numbers and remainders among them, several tiles per pair."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("model") / "step_walk_model")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-o", exe, os.path.join(HERE, "step_walk_model.cpp")])

    def runs(spr, a_stages, kblocks, tiles, seeds, asks):
        return int(subprocess.check_output([exe] + [str(v) for v in (spr, a_stages, kblocks, tiles, seeds, asks)]))
    return runs


@pytest.mark.parametrize("spr", [2, 4])
@pytest.mark.parametrize("a_stages", [4, 8])
def test_no_stage_is_read_before_it_is_full(model, spr, a_stages):
    for kblocks in list(range(1, 14)) + [21, 33, 64]:
        for tiles in (1, 40 // kblocks + 7):
            assert model(spr, a_stages, kblocks, tiles, 60, 1) == 0, (kblocks, tiles)


@pytest.mark.parametrize("spr,a_stages,kblocks", [(2, 8, 64), (2, 8, 13), (4, 8, 5), (4, 8, 2), (4, 4, 1)])
def test_the_model_sees_groups_that_ask_too_early(model, spr, a_stages, kblocks):
    """The same walk without the two waits in front."""
    assert model(spr, a_stages, kblocks, 40 // kblocks + 7, 60, 0) > 0
