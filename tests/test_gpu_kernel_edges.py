"""Sizes at the edges of the kernels' tiles, chunks and dispatch rules, against the oracle."""
import pytest

import test_gpu_backward as backward
import test_gpu_parity as parity
import test_gpu_value_norm_sampling as vnorm

pytestmark = pytest.mark.gpu

FORWARD = [
    # sort: nodes of 16 chunks add up the histograms in the placement, of 17 in a launch before it; chunks of 256 and 512 rows
    parity.W("node_of_16_chunks", 1, 1, 4096, 64, "bf16", 256, 130, 7, False, 0, seed=70),
    parity.W("node_of_17_chunks", 1, 1, 4097, 64, "bf16", 256, 130, 7, False, 0, seed=71),
    parity.W("causal_nodes_of_17_chunks", 1, 1, 8704, 128, "bf16", 128, 65, 8, True, 4352, seed=72),
    parity.W("chunks_of_512_rows", 1, 20, 4000, 64, "bf16", 128, 64, 7, False, 0, seed=73),
    # query tiles paired across blocks: an odd number of tiles per block, few and as many key tiles as the ring allows
    parity.W("pairs_of_one_tile_blocks_d128", 1, 1, 1500, 128, "bf16", 128, 96, 6, False, 0, seed=74),
    parity.W("pairs_of_three_tile_blocks_d64", 1, 1, 2900, 64, "bf16", 384, 64, 6, False, 0, seed=75),
    # fp32: hash passes of 256 rows; copies beside the hash (up to 296 CTAs of 4096 entries) and in a launch of their own; query tiles halved (up to 74 tiles) and whole, second halves of one row and none
    parity.W("fp32_n257_d64", 1, 1, 257, 64, "fp32", 64, 32, 7, False, 0, seed=76),
    parity.W("fp32_n65_d128", 1, 1, 65, 128, "fp32", 32, 16, 8, False, 0, seed=77),
    parity.W("fp32_n193_d128", 1, 2, 193, 128, "fp32", 100, 16, 1, False, 0, seed=78),
    parity.W("fp32_80_tiles_d64", 1, 5, 2048, 64, "fp32", 128, 64, 7, False, 0, seed=79),
    parity.W("fp32_copies_in_a_launch_of_their_own", 1, 5, 2000, 128, "fp32", 128, 64, 7, False, 0, seed=83),
    parity.W("fp32_85_tiles_causal_d128", 1, 5, 1090, 128, "fp32", 64, 32, 6, True, 300, seed=80),
]


@pytest.mark.parametrize("w", FORWARD, ids=[w.name for w in FORWARD])
def test_forward_edges(w):
    parity.test_small_configs_every_stage(w)


BACKWARD = [
    # key tiles and query halves of 1, 2, 63 .. 66, 127 and 128 rows; chunks of query tiles that do not divide the node
    backward.W("bwd_blocks_of_64_d64", 1, 1, 1090, 64, 64, 129, 6, False, 0, seed=70),
    backward.W("bwd_blocks_of_65_d64", 1, 1, 1301, 64, 65, 1, 6, False, 0, seed=71),
    backward.W("bwd_blocks_of_130_d64", 1, 2, 1430, 64, 130, 127, 7, False, 0, seed=72),
    backward.W("bwd_blocks_of_130_d128", 1, 1, 1562, 128, 130, 128, 7, False, 0, seed=73),
    backward.W("bwd_blocks_of_383_d128", 1, 1, 1533, 128, 383, 65, 7, False, 0, seed=74),
    backward.W("bwd_one_row_blocks_d64", 1, 1, 130, 64, 1, 3, 5, False, 0, seed=75),
    # keys that several samples draw, keys that none draws, no samples
    backward.W("bwd_more_samples_than_keys_d64", 1, 2, 200, 64, 64, 500, 5, False, 0, seed=76),
    backward.W("bwd_no_samples_d128", 1, 2, 700, 128, 128, 0, 6, False, 0, seed=77),
    # leaves of one row, one tile and one row more; unsorted and sorted nodes in one call
    backward.W("bwd_leaf_of_one_row", 1, 2, 1, 64, 64, 8, 4, True, 16, seed=78),
    backward.W("bwd_leaf_of_129_rows_d64", 1, 1, 129, 64, 64, 8, 4, True, 129, seed=79),
    backward.W("bwd_leaf_of_193_rows_d128", 1, 1, 193, 128, 64, 8, 4, True, 200, seed=80),
    backward.W("bwd_sorted_over_unsorted_nodes_d64", 1, 2, 1040, 64, 200, 33, 6, True, 130, seed=81),
    backward.W("bwd_sorted_over_unsorted_nodes_d128", 1, 1, 1040, 128, 200, 33, 6, True, 130, seed=82),
]


@pytest.mark.parametrize("w", BACKWARD, ids=[w.name for w in BACKWARD])
def test_backward_edges(w):
    backward.test_backward_matches_the_oracle(w)


VALUE_NORMS = [
    # scans of 256 rows per block sum and 4096 rows per CTA; 32 lanes per draw below 16384 draws, one from there on
    vnorm.W("vnorm_n256", 1, 1, 256, 64, 64, 48, 6, False, 0, seed=70),
    vnorm.W("vnorm_n257_d128", 1, 1, 257, 128, 64, 48, 6, False, 0, seed=71),
    vnorm.W("vnorm_n4096", 1, 1, 4096, 64, 256, 64, 7, False, 0, seed=72),
    vnorm.W("vnorm_n4097_d128", 1, 2, 4097, 128, 256, 64, 7, False, 0, seed=73),
    vnorm.W("vnorm_16352_draws", 1, 32, 300, 64, 64, 511, 5, False, 0, seed=74),
    vnorm.W("vnorm_16384_draws", 1, 32, 300, 64, 64, 512, 5, False, 0, seed=75),
]


@pytest.mark.parametrize("w", VALUE_NORMS, ids=[w.name for w in VALUE_NORMS])
def test_value_norm_edges(w):
    vnorm.test_value_norm_sampling_matches_the_oracle(w)
