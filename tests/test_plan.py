"""The rules by which a layer's GEMMs are cut (a3_plan_layer), over widths and row counts.  Host only."""
from dataclasses import replace

import pytest

from paper_2511_17560_b200 import a3
from paper_2511_17560_b200 import workloads as W

SHAPE = W.ModelShape("any", 1, 128, 1, 1, 128, 128, 32000, 5e5, 1e-5)
PAIRS = 148 // 2


def one_tile_slices(rows, features, depth, part_bytes=4 * 2 * 148 * 128 * (128 + 2) * 4):
    """The slices of a residual product whose units are one token tile each: the costs in clocks that the launcher compares."""
    cdiv = lambda a, b: -(-a // b)
    blocks, tiles, kt = cdiv(features, 256), cdiv(rows, 256), depth // 64
    if blocks * tiles > PAIRS // 2:
        return 1
    n = cdiv(cdiv(rows, tiles), 16) * 16
    per_kb = max(2 * n, 256 + n)
    least, best = kt * per_kb, 1
    for s in range(2, 17):
        if s * 16 > kt or s * rows * features * 4 > part_bytes:
            break
        cost = cdiv(blocks * tiles * s, PAIRS) * (cdiv(kt // 2, s) * 2 * per_kb + 2000) + s * rows * features * 8 // 3000 + 2000
        if cost < least:
            least, best = cost, s
    return best


@pytest.mark.parametrize("rows", [1, 75, 256, 257, 272, 288, 289, 320, 352, 384, 448, 512, 513, 804])
def test_slices_do_not_depend_on_the_tiles_that_share_weights(rows):
    """Sums are the same whether a unit is one token tile or two; two only in launches of one unit per pair of CTAs, whose two
    accumulators of 256 columns fill tensor memory."""
    for d_model in range(256, 8193, 256):
        for d_ff in (1408, 4864, 8192, 10112, 10624, 13440, 14336, 18944, 28672):
            p = a3.plan_layer(replace(SHAPE, d_model=d_model, d_ff=d_ff, n_q_heads=d_model // 128), rows)
            for depth, slices, tiles in ((d_model, p["out_slices"], p["out_tiles"]), (d_ff, p["down_slices"], p["down_tiles"])):
                assert slices == one_tile_slices(rows, d_model, depth), (d_model, d_ff, depth)
                assert tiles in (1, 2)
                if tiles == 2:
                    assert 256 < rows <= 512 and slices > 1 and -(-d_model // 256) * slices <= PAIRS
                    # their weights are marked to leave L2 first: the layer is beyond its three quarters (weights_once) by far
                    assert 2 * d_model * 3 * d_ff > 2 * 126 * 2 ** 20


@pytest.mark.parametrize("rows,down", [(75, (5, 1)), (256, (5, 1)), (257, (5, 2)), (270, (5, 2)), (352, (5, 2)), (368, (2, 1)), (512, (2, 1))])
def test_down_projection_of_qwen(rows, down):
    p = a3.plan_layer(W.QWEN7B, rows)
    assert (p["down_slices"], p["down_tiles"]) == down


@pytest.mark.parametrize("d_model,d_ff,rows,tiles", [(4096, 14336, 256, 1), (4096, 14336, 257, 2), (4096, 14336, 288, 2), (4096, 14336, 289, 1),
                                                     (4096, 14336, 320, 1), (3584, 18944, 270, 2), (3584, 18944, 304, 1), (3072, 8192, 272, 2),
                                                     (2048, 16384, 257, 1), (2048, 16384, 320, 1), (2048, 8192, 272, 1), (1536, 8960, 272, 1)])
def test_token_tiles_of_the_gate_and_up_product(d_model, d_ff, rows, tiles):
    """Two on one stream of weights only where that was faster: from 257 to 288 rows, and not at the narrow widths."""
    assert a3.plan_layer(replace(SHAPE, d_model=d_model, d_ff=d_ff, n_q_heads=d_model // 128), rows)["swiglu_tiles"] == tiles


def test_bad_arguments():
    lib, desc, plan = a3._load(), a3.ModelDesc(1, 512, 4, 2, 128, 1408, 1e4, 1e-5, 0, 1), a3.LayerPlan()
    assert lib.a3_plan_layer(None, 148, 1, plan) == -1 and lib.a3_plan_layer(desc, 148, 1, None) == -1
    assert lib.a3_plan_layer(desc, 1, 1, plan) == -1 and lib.a3_plan_layer(desc, 148, -1, plan) == -1
