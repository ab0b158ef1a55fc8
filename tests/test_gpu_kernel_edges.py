"""Sizes at the edges of the kernels' tiles, chunks and dispatch rules, against the oracle."""
import ctypes as C
import math

import numpy as np
import pytest
import torch

import paper_2310_05869_b200 as ha
from paper_2310_05869_b200 import binding as B
from paper_2310_05869_b200 import workloads as WL
from oracle import hyperattn_oracle as O

import parity_util as PU
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
    # query tiles paired across blocks (an odd number of query tiles per block), few key tiles per block, ...
    parity.W("pairs_of_one_tile_blocks_d128", 1, 1, 1500, 128, "bf16", 128, 96, 6, False, 0, seed=74),
    parity.W("pairs_of_three_tile_blocks_d64", 1, 1, 2900, 64, "bf16", 384, 64, 6, False, 0, seed=75),
    # ... as many as the ring of K / V stages allows (7 at d = 64, 3 at d = 128), and one more: not paired
    parity.W("pairs_of_seven_key_tiles_d64", 1, 2, 1000, 64, "bf16", 448, 256, 6, False, 0, seed=88, n_k=4000),
    parity.W("pairs_of_seven_key_tiles_b385_d64", 1, 1, 700, 64, "bf16", 385, 40, 6, False, 0, seed=89, n_k=3000),
    parity.W("pairs_of_three_query_and_seven_key_tiles_d64", 1, 1, 2400, 64, "bf16", 448, 64, 6, False, 0, seed=90, n_k=3000),
    parity.W("eight_key_tiles_d64", 1, 1, 1000, 64, "bf16", 449, 256, 6, False, 0, seed=91, n_k=4000),
    parity.W("pairs_of_three_key_tiles_d128", 1, 2, 1300, 128, "bf16", 192, 256, 6, False, 0, seed=92, n_k=2000),
    parity.W("pairs_of_three_key_tiles_b129_d128", 1, 1, 1900, 128, "bf16", 129, 40, 6, False, 0, seed=93, n_k=2000),
    parity.W("four_key_tiles_d128", 1, 1, 1300, 128, "bf16", 193, 256, 6, False, 0, seed=94, n_k=2000),
    # blocks of three query tiles; the last nodes have fewer queries than keys, groups of two tiles, and pairs whose first tile does not exist
    parity.W("groups_of_fewer_query_tiles_than_blocks_d64", 1, 2, 4516, 64, "bf16", 264, 31, 3, True, 204, seed=101),
    # no samples: the last key tile of a pair across blocks is the second query tile's alone (d = 128: not paired)
    parity.W("no_samples_seven_key_tiles_d64", 1, 2, 1000, 64, "bf16", 448, 0, 6, False, 0, seed=98, n_k=4000),
    parity.W("no_samples_three_key_tiles_d128", 1, 2, 1300, 128, "bf16", 192, 0, 6, False, 0, seed=99, n_k=2000),
    parity.W("no_samples_two_key_tiles_causal_d128", 1, 2, 4096, 128, "bf16", 128, 0, 6, True, 512, seed=100),
    # leaves alone, two pairs of query tiles each: the last 296 (four rounds of 148 SMs) go rank by rank, the ones before leaf by leaf
    parity.W("leaves_for_more_than_four_rounds", 1, 310, 300, 64, "bf16", 64, 8, 4, True, 512, seed=102),
    # fp32: hash passes of 256 rows; copies beside the hash (up to 296 CTAs of 4096 entries) and in a launch of their own; query tiles
    # halved (up to 74 tiles) and whole, second halves of one row and none
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


# heads of a call whose pairs of query tiles are split (at most 74 of 148 SMs have one left), and of one whose pairs are not
SPLIT = [(64, 1000, 1000, 256, 64, 18, 20, {}),          # two tiles of a block; a short last block
         (128, 1100, 1100, 256, 130, 14, 16, {}),        # ... whose second tile does not exist
         (64, 1100, 1100, 100, 33, 12, 13, {}),          # pairs across blocks, an odd number of tiles
         (64, 1100, 1100, 100, 33, 12, 13, dict(precise=True)),
         (64, 1100, 1100, 100, 130, 12, 13, dict(caps=(8.0, 16.0))),
         (64, 1100, 1100, 100, 130, 12, 13, dict(value_norm_sampling=True)),
         (64, 2900, 2900, 384, 200, 6, 7, {}),           # ... of three tiles each, the last of which do not exist
         (128, 600, 1500, 128, 64, 9, 13, {}),           # ... fewer queries than keys
         (128, 600, 1500, 128, 200, 9, 13, dict(value_norm_sampling=True)),
         (64, 20000, 20000, 256, 256, 2, 3, {})]         # behind a round of whole pairs


@pytest.mark.parametrize("d,n,n_k,b,m,split,whole,option", SPLIT)
def test_split_pairs_give_the_same_results(d, n, n_k, b, m, split, whole, option):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    q, k, v = (torch.randn(1, whole, rows, d, generator=gen, device="cuda").bfloat16() for rows in (n, n_k, n_k))
    want = ha.forward(q, k, v, b, m, 6, seed=3, out_dtype=torch.float32, **option)
    got = ha.forward(q[:, :split], k[:, :split], v[:, :split], b, m, 6, seed=3, out_dtype=torch.float32, **option)
    for x, y in zip(got, want):
        assert torch.equal(x, y[:, :split])
    assert ha.last_device_status() == 0


# host buffers go through in up to sixteen groups, calls of their own: the same bits as one call of all heads, where only one of the two splits
# its pairs, and whatever else goes by the number of heads
@pytest.mark.parametrize("H,n,n_k,d,b,m,dtype,kw", [
    (32, 4096, 4096, 64, 128, 256, torch.bfloat16, {}), (16, 1100, 1100, 64, 100, 33, torch.bfloat16, {}), (16, 600, 1500, 128, 128, 64, torch.bfloat16, {}),
    (32, 4096, 4096, 64, 256, 256, torch.bfloat16, {}), (40, 1500, 1500, 64, 100, 33, torch.bfloat16, dict(causal=True, n0=400)),
    (32, 1100, 1100, 64, 100, 33, torch.float32, {}), (20, 1500, 1500, 128, 100, 33, torch.float32, dict(causal=True, n0=400))])
def test_host_buffers_in_groups_give_the_same_bits(H, n, n_k, d, b, m, dtype, kw):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(19)
    q, k, v = (torch.randn(1, H, rows, d, generator=gen, device="cuda").to(dtype) for rows in (n, n_k, n_k))
    want = ha.forward(q, k, v, b, m, 6, seed=3, **kw)
    got = [torch.empty(x.shape, dtype=x.dtype).pin_memory() for x in want]
    ha.forward_host(*(x.cpu().pin_memory() for x in (q, k, v)), *got, b, m, 6, seed=3, **kw)
    torch.cuda.synchronize()
    for x, y in zip(got, want):
        assert torch.equal(x, y.cpu())
    assert ha.last_device_status() == 0


# the permutations are stable sorts of the bucket ids: rows of a chunk, whole and short ranges of a warp, hash widths of 1 and 8 bits, and rows that
# are all equal
SORTED = [(256, "random", 1, 1000, 1000, 64, 7, False, 0), (512, "random", 20, 3999, 3999, 64, 8, False, 0),
          (512, "random", 32, 4096, 1030, 64, 1, False, 0), (768, "random", 64, 1500, 1500, 64, 7, False, 0), (1280, "random", 60, 2500, 2500, 64, 7, False, 0),
          (1024, "random", 32, 4096, 4096, 64, 7, False, 0), (768, "random", 16, 9000, 9000, 64, 7, True, 4096),
          (1536, "random", 32, 4600, 4600, 128, 7, False, 0), (1792, "random", 4, 100003, 100003, 64, 7, True, 4096),
          (1024, "random", 17, 16384, 16384, 64, 7, False, 0), (2048, "random", 40, 16384, 16384, 64, 8, False, 0), (256, "equal", 2, 5000, 5000, 128, 7, False, 0),
          (1280, "equal", 40, 9000, 9000, 64, 7, True, 2500)]


@pytest.mark.parametrize("chunk,kind,H,n,n_k,d,r,causal,n0", SORTED)
def test_permutations_are_stable_sorts_of_the_ids(chunk, kind, H, n, n_k, d, r, causal, n0):
    p, rows = B._Params(), C.c_int(0)
    B._fill(p, 1, H, n, d, 128, 32, r, causal, n0, 5, B.BF16, B.BF16, 0.0, n_k)
    assert ha.lib().hyperattn_internal_chunk_rows(C.byref(p), C.byref(rows)) == 0 and rows.value == chunk
    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)
    q, k, v = (torch.randn(1, H, rows, d, generator=gen, device="cuda").bfloat16() for rows in (n, n_k, n_k))
    if kind == "equal":
        q, k = (x[:, :, :1].expand_as(x) for x in (q, k))
    inter = ha.forward(q, k, v, 128, 32, r, causal=causal, n0=n0, seed=5, debug=True)[2]
    ids = {"q": inter["q_ids"].int(), "k": inter["k_ids"].int()}
    L = 0
    while causal and -(-n >> L) > n0:
        L += 1
    npad = -(-n >> L) << L
    for level in range(max(L, 1)):
        s = npad >> (level + 1)
        for j in range(1 << level if causal else 1):
            for side, first, end in (("q", (2 * j + 1) * s, (2 * j + 2) * s), ("k", 2 * j * s, (2 * j + 1) * s)) if causal else (("q", 0, n), ("k", 0, n_k)):
                rows = min(end, n if side == "q" else n_k) - first
                if rows <= 0:
                    continue
                want = torch.sort(ids[side][:, first:first + rows], dim=1, stable=True).indices.int()
                at = j * s if causal else 0
                assert torch.equal(inter["perm_" + side][level, :, at:at + rows], want)
                if side == "k":
                    assert torch.equal(torch.gather(inter["rank_k"][level, :, at:at + rows], 1, want.long()),
                                       torch.arange(rows, dtype=torch.int32, device="cuda").expand(H, rows))


# chunks that need a larger workspace than the share of bf16 rows asks for are left out where the caller's is smaller (more chunks: histograms and
# offsets of 1 KiB each): the same results, and one byte less is refused
@pytest.mark.parametrize("H,n,dtype,more", [(35, 8192, torch.bfloat16, 8 - 4), (20, 2349, torch.float32, 10 - 5)])
def test_chunks_by_the_workspace(H, n, dtype, more):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(23)
    q, k, v = (torch.randn(1, H, n, 64, generator=gen, device="cuda").to(dtype) for _ in range(3))
    code = B._dtype_code(dtype)
    need = ha.workspace_bytes(1, H, n, 64, 128, 64, 7, dtype=code, out_dtype=code)
    less = need - 2 * 2 * H * more * 1024
    ws = torch.full((need,), 0xff, dtype=torch.uint8, device="cuda")
    results = [ha.forward(q, k, v, 128, 64, 7, seed=2, workspace=ws[:size]) for size in (need, need - 1, less)]
    torch.cuda.synchronize()
    assert ha.last_device_status() == 0
    for other in results[1:]:
        for x, y in zip(results[0], other):
            assert torch.equal(x, y)
    with pytest.raises(ha.HyperAttnError, match="workspace too small"):
        ha.forward(q, k, v, 128, 64, 7, seed=2, workspace=ws[:less - 1])


# calls large enough for sorted nodes and everything else in launches of their own, against calls of few heads in one launch: the same bits
TWO_LAUNCHES = [(64, 64, 2048, 256, torch.bfloat16, {}), (64, 40, 128, 256, torch.bfloat16, {}), (64, 64, 2048, 256, torch.float32, dict(precise=True)),
                (128, 64, 2048, 256, torch.bfloat16, {}), (128, 64, 2048, 250, torch.float32, {}), (128, 64, 2048, 256, torch.float32, dict(precise=True)),
                (64, 64, 2048, 256, torch.bfloat16, dict(caps=(8.0, 16.0))), (128, 64, 2048, 256, torch.bfloat16, dict(caps=(8.0, 16.0))),
                (128, 64, 2048, 256, torch.float32, dict(caps=(8.0, 16.0))), (64, 64, 2048, 256, torch.bfloat16, dict(value_norm_sampling=True)),
                (128, 64, 2048, 256, torch.bfloat16, dict(value_norm_sampling=True)),
                (128, 64, 2048, 256, torch.float32, dict(value_norm_sampling=True))]


@pytest.mark.parametrize("d,H,n0,b,out_dtype,option", TWO_LAUNCHES)
def test_nodes_and_leaves_in_launches_of_their_own(d, H, n0, b, out_dtype, option):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(17)
    q, k, v = (torch.randn(1, H, 16384, d, generator=gen, device="cuda").bfloat16() for _ in range(3))
    kw = dict(causal=True, n0=n0, seed=2, out_dtype=out_dtype, **option)
    few, launches, results = 3, [], []
    for heads in (H, few):
        ha.profile_reset()
        ha.profile_enable(True)
        results.append(ha.forward(q[:, :heads], k[:, :heads], v[:, :heads], b, 128, 6, **kw))
        torch.cuda.synchronize()
        ha.profile_enable(False)
        launches.append(ha.profile_read()["launches"]["attention"])
    assert launches[0] == launches[1] + 1
    for x, y in zip(*results):
        assert torch.equal(x[:, :few], y)
    assert ha.last_device_status() == 0


# calls whose leaves go first and write dK and dV (from 192 MiB of fp32 accumulators on), against calls of few heads, which add everything; in the
# second launch sorted nodes alone, or others too, in each build (test_abi_host.py holds these shapes to the builds)
SPLIT_BACKWARD = [(64, 26, 16384, 4096, 256), (64, 26, 16800, 2100, 256), (64, 40, 10240, 700, 256), (128, 13, 16384, 4096, 256),
                  (64, 26, 16384, 512, 512), (64, 400, 1024, 512, 512), (64, 50, 8192, 512, 4096), (128, 13, 16384, 512, 512), (128, 13, 16384, 4096, 8192)]


def _backward_in_a_workspace(q, k, v, out, lse, dout, block, samples, r, grad_dtype, n0, seed):
    """The causal backward pass with every byte of its workspace and of the gradients set to 0xff (a NaN), and its launches of all kinds."""
    _, H, n, d = q.shape
    p = B._Params()
    B._fill(p, 1, H, n, d, block, samples, r, True, n0, seed, B.BF16, B.BF16, 0.0, n)
    need, code = C.c_size_t(0), B._dtype_code(grad_dtype)
    assert ha.lib().hyperattn_backward_workspace_bytes(C.byref(p), code, C.byref(need)) == 0
    ws = torch.full((need.value,), 0xff, dtype=torch.uint8, device="cuda")
    grads = [torch.full(q.shape, math.nan, dtype=grad_dtype, device="cuda") for _ in range(3)]
    p.q, p.k, p.v, p.out, p.lse = (x.data_ptr() for x in (q, k, v, out, lse))
    p.workspace, p.workspace_bytes, p.stream = ws.data_ptr(), need.value, torch.cuda.current_stream().cuda_stream
    g = B._Grads(dout.data_ptr(), *(x.data_ptr() for x in grads), code)
    ha.profile_reset()
    ha.profile_enable(True)
    rc = ha.lib().hyperattn_backward(C.byref(p), C.byref(g))
    torch.cuda.synchronize()
    ha.profile_enable(False)
    launches = ha.profile_read()["launches"]["backward"]
    ha.profile_reset()
    assert rc == 0
    return grads, launches


@pytest.mark.parametrize("d,H,n,n0,block", SPLIT_BACKWARD)
@pytest.mark.parametrize("grad_dtype", [torch.float32, torch.bfloat16])
def test_backward_with_leaves_in_a_launch_of_their_own(d, H, n, n0, block, grad_dtype):
    assert 8 * H * n * d >= 192 << 20
    gen = torch.Generator(device="cuda")
    gen.manual_seed(13)
    q, k, v, dout = (torch.randn(1, H, n, d, generator=gen, device="cuda").bfloat16() for _ in range(4))
    args = (block, 128 if block < 1024 else 8, 6)
    out, lse = ha.forward(q, k, v, *args, causal=True, n0=n0, seed=4)
    got, launches = _backward_in_a_workspace(q, k, v, out, lse, dout, *args, grad_dtype, n0, 4)
    few = 2
    part = [x[:, :few].contiguous() for x in (q, k, v, out, lse, dout)]
    want, launches_few = _backward_in_a_workspace(*part, *args, grad_dtype, n0, 4)
    assert launches == launches_few + 1
    for x, y in zip(got, want):
        # the same terms in another order: at most 200 partial sums of fp32 (2 x 200 x 2^-24 of the terms' absolute values, which add up to a few
        # times the largest entry), and bf16 results may be a step apart (2^(e - 7) for 2^e <= |y|)
        x, y = x[:, :few].float(), y.float()
        assert torch.isfinite(x).all()
        limit = 1e-4 * float(y.abs().max()) + (2.0 ** -7 * y.abs() if grad_dtype == torch.bfloat16 else 0.0)
        assert bool(((x - y).abs() <= limit).all())
    assert ha.last_device_status() == 0


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
    # leaves alone, three key tiles each: the last 198 go rank by rank
    backward.W("bwd_leaves_for_more_than_four_rounds_d64", 1, 210, 300, 64, 64, 8, 4, True, 512, seed=85),
    # more items than SMs, so that whole tiles of consecutive rows, short ones and scattered rows follow one another in a CTA, in every build
    # of the kernel (test_abi_host.py holds these shapes to the builds): without boxes ...
    backward.W("bwd_whole_short_and_scattered_tiles_d64", 1, 40, 640, 64, 64, 33, 6, True, 320, seed=83),
    backward.W("bwd_whole_short_and_scattered_tiles_d128", 1, 24, 640, 128, 64, 33, 6, True, 320, seed=84),
    # ... with boxes and eight results warps ...
    backward.W("bwd_boxes_short_and_scattered_tiles_d64", 1, 16, 1400, 64, 64, 33, 6, True, 700, seed=86),
    backward.W("bwd_boxes_short_and_scattered_tiles_d128", 1, 12, 1400, 128, 64, 33, 6, True, 700, seed=87),
    # ... and with four (d = 64)
    backward.W("bwd_four_results_warps_short_and_scattered_tiles_d64", 1, 4, 3400, 64, 64, 33, 6, True, 1700, seed=88),
]


@pytest.mark.parametrize("w", BACKWARD, ids=[w.name for w in BACKWARD])
def test_backward_edges(w):
    backward.test_backward_matches_the_oracle(w)


def _gradients(w, q, k, v, out, lse, dout, dtype):
    return ha.backward(q, k, v, out, lse, dout, w.b, w.m, w.r, causal=w.causal, n0=w.n0, seed=w.seed, grad_dtype=dtype)


def _assert_same_gradients(got, want, dtype):
    # only the order of the fp32 reductions may differ: a few hundred terms of 2^-24 each; bf16 results round once more
    for g, x in zip(got, want):
        g, x = g.double(), x.double()
        assert torch.isfinite(g).all()
        assert (g - x).abs().max() <= (2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -14) * x.abs().max()


SHORT_TILES = [
    backward.W("one_leaf_d64", 1, 2, 193, 64, 64, 8, 4, True, 256, seed=83),
    backward.W("leaves_of_130_sorted_and_unsorted_nodes_d128", 1, 2, 1040, 128, 200, 33, 6, True, 130, seed=84),
    backward.W("one_block_d128", 1, 2, 300, 128, 512, 16, 4, False, 0, seed=85),
    backward.W("blocks_of_130_d64", 1, 2, 1301, 64, 130, 65, 6, False, 0, seed=86),
]


def _forward(w, q, k, v, **kw):
    return ha.forward(q, k, v, w.b, w.m, w.r, causal=w.causal, n0=w.n0, seed=w.seed, **kw)


@pytest.mark.parametrize("bad", [math.nan, math.inf], ids=["nan", "inf"])
@pytest.mark.parametrize("w", SHORT_TILES + [
    parity.W("ragged_leaves_d128", 1, 2, 1000, 128, "bf16", 64, 40, 6, True, 130, seed=95),
    parity.W("cross_blocks_of_100_d64", 1, 2, 500, 64, "bf16", 100, 33, 6, False, 0, seed=96, n_k=1111),
], ids=lambda w: w.name)
def test_forward_of_a_head_beside_a_head_that_is_not_finite(w, bad):
    q, k, v = PU.to_device(w, WL.make_inputs(w))
    out, lse = _forward(w, q, k, v)
    for x in (q, k, v):
        x[0, 1] = bad
    got, got_lse = _forward(w, q, k, v)
    assert ha.last_device_status() == 0
    assert torch.equal(got[0, 0], out[0, 0]) and torch.equal(got_lse[0, 0], lse[0, 0])


@pytest.mark.parametrize("option", [{}, {"precise": True}, {"caps": (8.0, 16.0)}], ids=["plain", "precise", "caps"])
@pytest.mark.parametrize("d", [64, 128])
def test_forward_of_rows_that_do_not_see_a_value_that_is_not_finite(d, option):
    """Short tiles of sorted and sampled keys: a value row that is not finite reaches the queries of its block only."""
    w = parity.W("", 1, 1, 1301, d, "bf16", 130, 40, 6, False, 0, seed=97)
    q, k, v = PU.to_device(w, WL.make_inputs(w))
    out, lse, inter = _forward(w, q, k, v, debug=True, **option)
    assert not (inter["samples"][0, 0, :w.m] == 0).any()
    v[0, 0, 0] = math.nan
    got, got_lse = _forward(w, q, k, v, **option)
    assert ha.last_device_status() == 0
    beta = int(inter["rank_k"].view(-1)[0]) // w.b
    clean = torch.ones(w.n, dtype=torch.bool, device="cuda")
    clean[inter["perm_q"].view(-1)[beta * w.b:(beta + 1) * w.b].long()] = False
    assert torch.equal(got[0, 0][clean], out[0, 0][clean]) and torch.equal(got_lse, lse)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("bad", [math.nan, math.inf], ids=["nan", "inf"])
@pytest.mark.parametrize("w", SHORT_TILES, ids=[w.name for w in SHORT_TILES])
def test_backward_of_a_head_beside_a_head_that_is_not_finite(w, bad, dtype):
    """The last tile of a head or leaf is short, and what follows it in memory is the next head: nothing of that may enter."""
    q, k, v = PU.to_device(w, WL.make_inputs(w))
    out, lse = ha.forward(q, k, v, w.b, w.m, w.r, causal=w.causal, n0=w.n0, seed=w.seed)
    dout = torch.randn(q.shape, generator=torch.Generator(device="cuda").manual_seed(92), device="cuda").bfloat16()
    want = [x[0, 0] for x in _gradients(w, q, k, v, out, lse, dout, dtype)]
    tensors = [x.clone() for x in (q, k, v, dout)]
    for x in tensors:
        x[0, 1] = bad
    got = [x[0, 0] for x in _gradients(w, *tensors[:3], out, lse, tensors[3], dtype)]
    assert ha.last_device_status() == 0
    _assert_same_gradients(got, want, dtype)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("b", [130, 65])
def test_backward_of_keys_that_a_row_that_is_not_finite_does_not_see(b, d, dtype):
    """Short tiles of sorted queries: a query that is not finite reaches the keys of its own block and the sampled ones only."""
    w = backward.W("", 1, 1, 1301, d, b, 40, 6, False, 0, seed=87)
    q, k, v = PU.to_device(w, WL.make_inputs(w))
    out, lse, inter = ha.forward(q, k, v, w.b, w.m, w.r, seed=w.seed, debug=True)
    dout = torch.randn(q.shape, generator=torch.Generator(device="cuda").manual_seed(93), device="cuda").bfloat16()
    want = _gradients(w, q, k, v, out, lse, dout, dtype)
    dout[0, 0, 0] = math.nan                               # (the permutation stays: the row's Q is left alone)
    got = _gradients(w, q, k, v, out, lse, dout, dtype)
    assert ha.last_device_status() == 0
    perm_q, perm_k = (inter[x].view(-1)[:w.n].long() for x in ("perm_q", "perm_k"))
    beta = int((perm_q == 0).nonzero()) // b
    clean = torch.ones(w.n, dtype=torch.bool, device="cuda")
    clean[perm_k[beta * b:(beta + 1) * b]] = False
    clean[inter["samples"][0, 0, :w.m].long()] = False
    assert clean.sum() > w.n // 2
    _assert_same_gradients([x[0, 0][clean] for x in got[1:]], [x[0, 0][clean] for x in want[1:]], dtype)
    _assert_same_gradients([got[0][0, 0, 1:]], [want[0][0, 0, 1:]], dtype)


VALUE_NORMS = [
    # scans of 256 rows per block sum and 4096 rows per CTA; 32 lanes per draw below 16384 draws, one from there on
    vnorm.W("vnorm_n256", 1, 1, 256, 64, 64, 48, 6, False, 0, seed=70),
    vnorm.W("vnorm_n257_d128", 1, 1, 257, 128, 64, 48, 6, False, 0, seed=71),
    vnorm.W("vnorm_n4096", 1, 1, 4096, 64, 256, 64, 7, False, 0, seed=72),
    vnorm.W("vnorm_n4097_d128", 1, 2, 4097, 128, 256, 64, 7, False, 0, seed=73),
    vnorm.W("vnorm_pairs_of_seven_key_tiles", 1, 1, 1000, 64, 448, 64, 6, False, 0, seed=76, n_k=4000),
    vnorm.W("vnorm_16352_draws", 1, 32, 300, 64, 64, 511, 5, False, 0, seed=74),
    vnorm.W("vnorm_16384_draws", 1, 32, 300, 64, 64, 512, 5, False, 0, seed=75),
]


@pytest.mark.parametrize("w", VALUE_NORMS, ids=[w.name for w in VALUE_NORMS])
def test_value_norm_edges(w):
    vnorm.test_value_norm_sampling_matches_the_oracle(w)


@pytest.mark.parametrize("n,causal,value_norms", [(4097, False, True), (16385, False, False), (70001, False, True), (300000, False, False),
                                                  (300000, False, True), (65536, True, False), (65536, True, True), (40000, True, True)])
def test_sort_of_many_chunks(n, causal, value_norms):
    """Nodes of 17 to 293 chunks: the scan by one group of threads (many nodes) or by four, and what else its launch carries."""
    w = parity.W("", 1, 2 if causal else 1, n, 64, "bf16", 256, 64, 7, causal, 1024 if n == 65536 else 10000, seed=98)
    gen = torch.Generator(device="cuda").manual_seed(98)
    q, k, v = (torch.randn((w.B, w.H, n, w.d), generator=gen, device="cuda").bfloat16() for _ in range(3))
    _, _, inter = _forward(w, q, k, v, debug=True, value_norm_sampling=value_norms)
    assert ha.last_device_status() == 0
    s = n // 2 if causal else n                            # (the first level's node: the lengths are even)
    for ids, perm, first in ((inter["q_ids"], inter["perm_q"], n - s), (inter["k_ids"], inter["perm_k"], 0)):
        for g in range(w.G):
            want = torch.sort(ids[g, first:first + s].int(), stable=True).indices
            assert torch.equal(perm[0, g, :s].long(), want)
    if value_norms:
        V = v[0, 0].double().cpu().numpy()
        idx, _ = O.sample_by_value_norms(w.seed, 0, 0, w.m, O.value_norm_weights(V)[:s])
        assert (inter["samples"].cpu().numpy()[0, 0, :w.m] == idx).all()


def _check_segments(B, H, n, d, b, m, r, seed, gen_seed, per_segment=None, **kw):
    """Calls of more segments than the y and z extents of a grid: segments around 65 536 and forty others against the oracle."""
    gen = torch.Generator(device="cuda").manual_seed(gen_seed)
    q, k, v = (torch.randn((B, H, n, d), generator=gen, device="cuda").bfloat16() for _ in range(3))
    out, lse, inter = ha.forward(q, k, v, b, m, r, seed=seed, out_dtype=torch.float32, debug=True, **kw)
    torch.cuda.synchronize()
    assert ha.last_device_status() == 0
    Wd = O.directions(d, r, seed)
    rng = np.random.default_rng(5)
    for g in sorted({0, 1, 65534, 65535, 65536, B * H - 1, *rng.integers(0, B * H, 40).tolist()}):
        Q, K, V = (x.view(-1, n, d)[g].double().cpu().numpy() for x in (q, k, v))
        if per_segment:
            per_segment(g, V, inter)
        ro, rl = O.segment_forward(Q, K, V, Wd, b, m, kw.get("causal", False), kw.get("n0", 0), seed, g, scale=1.0 / math.sqrt(d),
                                   ids_q=inter["q_ids"][g].cpu().numpy(), ids_k=inter["k_ids"][g].cpu().numpy(),
                                   value_norm_sampling=kw.get("value_norm_sampling", False))
        err = np.abs(out.view(-1, n, d)[g].cpu().numpy() - ro)
        assert err.max() <= PU.OUT_MAX_ABS and err.mean() <= PU.OUT_MEAN_ABS, g
        assert (np.abs(lse.view(-1, n)[g].cpu().numpy() - rl) <= PU.LSE_REL * np.maximum(np.abs(rl), 1.0)).all(), g


@pytest.mark.parametrize("d", [64, 128])
def test_value_norms_of_more_segments_than_a_grid_has_rows(d):
    m, seed = 5, 3

    def draws(g, V, inter):
        idx, sw = O.sample_by_value_norms(seed, g, 0, m, O.value_norm_weights(V))
        assert (inter["samples"][g, 0, :m].cpu().numpy() == idx).all(), g
        np.testing.assert_allclose(inter["sample_log2w"][g, 0, :m].cpu().numpy(), np.log2(sw), atol=1e-5)

    _check_segments(16, 4100, 20, d, 8, m, 4, seed, 91, draws, value_norm_sampling=True)


@pytest.mark.parametrize("d", [64, 128])
def test_recursion_of_more_segments_than_a_grid_has_rows(d):
    _check_segments(16, 4100, 41, d, 8, 4, 4, 4, 94, causal=True, n0=12)
