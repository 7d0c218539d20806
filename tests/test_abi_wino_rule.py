"""Which kernels F(4,3) and F(6,3) layers of a few tiles run on (host arithmetic, no GPU)."""
import ctypes

import pytest

from paper_2206_07446_b200 import binding as nb


def rule(m, C, K, tiles):
    out = (ctypes.c_int32 * 6)()
    nb._lib.nnv_internal_wino_rule(m, C, K, tiles, out)
    return dict(zip(("small", "layer", "T", "slices", "quads", "groups"), out))


@pytest.mark.parametrize("m,C,K,tiles", [(4, 512, 512, 4), (4, 64, 64, 1), (6, 256, 256, 1), (6, 64, 96, 9)])
def test_overrides_reach_layers_of_few_tiles(m, C, K, tiles):
    """An override of the GEMM's tiling is for the tensor cores' tile GEMM, in every path that a layer takes."""
    try:
        nb.nnv_tuning_set("")
        assert rule(m, C, K, tiles)["small"]
        for spec in ("gemm_tile=64,2", "gemm_ring=4", "winosmall=0"):
            nb.nnv_tuning_set(spec)
            r = rule(m, C, K, tiles)
            assert not r["small"] and not r["layer"], (spec, r)
        nb.nnv_tuning_set("winosmall=1;winolayer=0;block=0")
        assert rule(m, C, K, tiles)["small"]
        for bad in ("winosmall=2", "winolayer=on", "block=-1"):
            with pytest.raises(nb.NnvError):
                nb.nnv_tuning_set(bad)
    finally:
        nb.nnv_tuning_set(None)


@pytest.mark.parametrize("m,C,K,tiles,layer", [
    # separate kernels / one launch, us a layer in a row of them: 4.9 / 6.4, 5.2 / 6.4, 5.5 / 6.4, 5.1 / 6.0, 6.5 / 7.5, 7.1 / 8.6
    (6, 16, 192, 8, 0), (6, 32, 256, 6, 0), (6, 64, 128, 9, 0), (6, 192, 32, 4, 0), (4, 192, 192, 8, 0), (4, 256, 160, 8, 0),
    # 23.0 / 12.9, 8.6 / 6.1, 4.6 / 3.8, 23.7 / 16.1, 7.8 / 6.0, 12.7 / 6.5
    (4, 512, 512, 4, 1), (4, 256, 256, 4, 1), (4, 64, 64, 9, 1), (6, 384, 384, 4, 1), (6, 192, 192, 1, 1), (4, 96, 1024, 4, 1),
    (4, 512, 512, 5, 0), (4, 6, 64, 1, 0), (6, 64, 64, 1, 0)])         # outside what the kernel does
def test_one_launch_where_it_is_the_faster(m, C, K, tiles, layer):
    nb.nnv_tuning_set(None)
    assert rule(m, C, K, tiles)["layer"] == layer


@pytest.mark.parametrize("m,C,K,tiles,groups", [
    (4, 960, 16, 12, 1), (4, 640, 48, 9, 1), (6, 448, 32, 9, 1), (4, 1024, 256, 6, 2), (6, 1024, 96, 1, 2),     # lone warps with long sums otherwise
    (4, 96, 64, 9, 4), (4, 512, 512, 4, 4), (4, 300, 512, 8, 4), (4, 40, 800, 12, 4)])                        # summed by the one-launch layer too, or enough blocks
def test_groups_of_output_channels(m, C, K, tiles, groups):
    nb.nnv_tuning_set(None)
    assert rule(m, C, K, tiles)["small"] and rule(m, C, K, tiles)["groups"] == groups
