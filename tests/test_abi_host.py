"""Host-side checks of the C-ABI library that need no GPU: it loads, exports every symbol the
header declares, rejects bad arguments before touching the device, and its host-side helpers
agree with the oracle."""
import ctypes as C
import os
import re

import numpy as np
import pytest

import paper_2310_05869_b200 as ha
from paper_2310_05869_b200 import binding as B
from oracle import hyperattn_oracle as O

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_exports_every_declared_symbol():
    header = open(os.path.join(ROOT, "include", "hyperattn.h")).read()
    declared = set(re.findall(r"\b(hyperattn_[a-z_]+)\s*\(", header))
    assert declared == set(B.EXPORTS)
    L = ha.lib()
    for name in declared:
        assert hasattr(L, name), name
    assert ha.version() >= 1


def test_status_strings():
    L = ha.lib()
    seen = {L.hyperattn_status_string(c).decode() for c in range(0, -7, -1)}
    assert len(seen) == 7 and "ok" in seen
    assert L.hyperattn_status_string(-99).decode() == "unknown status"


def _params(**kw):
    p = B._Params()
    base = dict(B=1, H=2, n=1024, d=64, block=128, samples=64, hash_bits=7, causal=0, n0=0, seed=0,
                dtype=B.BF16, out_dtype=B.BF16, softmax_scale=0.0)
    base.update(kw)
    for k, v in base.items():
        setattr(p, k, v)
    fake = 0x1000
    p.q, p.k, p.v, p.out, p.lse = fake, fake + 0x100000, fake + 0x200000, fake + 0x300000, fake + 0x400000
    return p


@pytest.mark.parametrize("kw,code", [
    (dict(d=96), -2), (dict(hash_bits=0), -2), (dict(hash_bits=9), -2),
    (dict(block=0), -1), (dict(samples=-1), -1), (dict(B=0), -1), (dict(dtype=5), -1),
    (dict(causal=1, n0=0), -1), (dict(causal=1, n0=100, n=1000, n_k=900), -2), (dict(n_k=-5), -1),
    (dict(n=4096, block=1024, samples=256), -2),
])
def test_bad_shapes_are_rejected_on_the_host(kw, code):
    p = _params(**kw)
    assert ha.lib().hyperattn_forward_ex(C.byref(p)) == code
    nbytes = C.c_size_t(0)
    assert ha.lib().hyperattn_workspace_bytes(C.byref(p), C.byref(nbytes)) == code


def test_bad_pointers_are_rejected_on_the_host():
    L = ha.lib()
    p = _params(); p.q = None
    assert L.hyperattn_forward_ex(C.byref(p)) == -1
    p = _params(); p.k = 0x1008
    assert L.hyperattn_forward_ex(C.byref(p)) == -3
    p = _params(); p.out = p.v
    assert L.hyperattn_forward_ex(C.byref(p)) == -3
    assert L.hyperattn_forward_ex(None) == -1
    assert L.hyperattn_forward_host(None) == -1


def test_workspace_size_grows_with_the_problem():
    small = ha.workspace_bytes(1, 2, 1024, 64, 128, 64, 7)
    big = ha.workspace_bytes(1, 2, 4096, 64, 128, 64, 7)
    causal = ha.workspace_bytes(1, 2, 4096, 64, 128, 64, 7, True, 512)
    assert 0 < small < big < causal
    assert ha.workspace_bytes(1, 1, 256, 64, 256, 0, 7) <= 4096          # single block: nothing to sort


def test_projection_matrix_matches_the_oracle_bit_for_bit():
    for d, r, seed in [(64, 7, 0), (128, 8, 2 ** 40 + 17), (64, 1, 99)]:
        w = ha.get_projections(d, r, seed)
        ref = O.directions(d, r, seed)
        assert (w.view(np.uint32) == ref.view(np.uint32)).all()


def test_cuda_tensors_are_required():
    import torch
    q = torch.zeros(1, 1, 128, 64, dtype=torch.bfloat16)
    with pytest.raises(ha.HyperAttnError):
        ha.forward(q, q, q, 64, 8, 4)


def test_binding_mirrors_the_stage_table_of_the_header():
    """The binding's stage-times structure must have the header's HYPERATTN_NUM_STAGES entries
    (hyperattn_profile_read writes that many)."""
    import re
    hdr = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include", "hyperattn.h")).read()
    n = int(re.search(r"HYPERATTN_NUM_STAGES\s*=\s*(\d+)", hdr).group(1))
    stages = re.findall(r"HYPERATTN_STAGE_(\w+)\s*=\s*(\d+)", hdr)
    from paper_2310_05869_b200 import binding as Bn
    assert Bn.NUM_STAGES == n == len(stages)
    assert [s.lower() for s, _ in sorted(stages, key=lambda t: int(t[1]))] == Bn.STAGE_NAMES


def test_backward_rejects_bad_arguments_on_the_host():
    """Nothing is launched for fp32 inputs, missing or misaligned gradient pointers, or a bad gradient type."""
    L = ha.lib()
    fake = 0x800000
    def grads(**kw):
        g = B._Grads(fake, fake + 0x100000, fake + 0x200000, fake + 0x300000, B.BF16)
        for k, v in kw.items():
            setattr(g, k, v)
        return g
    assert L.hyperattn_backward(C.byref(_params(dtype=B.FP32)), C.byref(grads())) == -2
    assert L.hyperattn_backward(C.byref(_params()), C.byref(grads(dq=0))) == -1
    assert L.hyperattn_backward(C.byref(_params()), C.byref(grads(grad_dtype=7))) == -1
    assert L.hyperattn_backward(C.byref(_params()), C.byref(grads(dk=fake + 0x100004))) == -3
    assert L.hyperattn_backward(None, C.byref(grads())) == -1
    need_f32, need_bf16, need_fwd = C.c_size_t(0), C.c_size_t(0), C.c_size_t(0)
    p = _params()
    assert L.hyperattn_backward_workspace_bytes(C.byref(p), B.FP32, C.byref(need_f32)) == 0
    assert L.hyperattn_backward_workspace_bytes(C.byref(p), B.BF16, C.byref(need_bf16)) == 0
    # bf16 gradients are accumulated in fp32 in the workspace: three tensors more than for fp32 gradients
    assert need_bf16.value - need_f32.value >= 3 * p.B * p.H * p.n * p.d * 4


def test_node_projections_match_the_oracle():
    for node in (0, 1, 7, 30):
        w = ha.get_projections(64, 7, 5, node=node)
        assert np.array_equal(w, O.directions(64, 7, 5, node=node))
    assert not np.array_equal(ha.get_projections(64, 7, 5, node=1), ha.get_projections(64, 7, 5))


# The launches of the backward kernel and their builds, by what a call's steps are: whole tiles of 128 consecutive rows, which leave as boxes; short
# tiles of consecutive rows and tiles of sorted rows, which leave row by row and want eight results warps; how often dK and dV leave (once per key
# tile); sorted nodes alone; from 192 MiB of fp32 dK and dV on, leaves that leave as boxes first.  (d = 128 always has eight warps.)
LEAVES, NODES, ALL = 1, 2, 3
OUT = ("rows", "boxes", "first", "nodes")


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("kw,out,warps", [
    (dict(n=64, causal=1, n0=64), "rows", 8), (dict(n=127, causal=1, n0=128), "rows", 8), (dict(n=128, causal=1, n0=128), "rows", 8),
    (dict(n=300, causal=1, n0=512), "rows", 8), (dict(n=127, block=128), "rows", 8), (dict(n=200, block=256), "rows", 8),
    (dict(n=512, causal=1, n0=512), "boxes", 8), (dict(n=768, causal=1, n0=768), "boxes", 8), (dict(n=300, block=512), "boxes", 8),
    (dict(n=1536, causal=1, n0=1536), "boxes", 4), (dict(n=4096, causal=1, n0=4096), "boxes", 4), (dict(n=4096, block=4096), "boxes", 4),
    (dict(n=6400, block=64, causal=1, n0=100), "rows", 8), (dict(n=1600, block=800, causal=1, n0=100), "rows", 8),
    (dict(n=32768, block=64, causal=1, n0=512), "rows", 8), (dict(n=32768, block=256, samples=256, causal=1, n0=1024), "boxes", 8),
    (dict(n=32768, block=256, samples=256, causal=1, n0=2048), "boxes", 4),
    (dict(H=1, n=131072, block=256, samples=256, causal=1, n0=4096), "boxes", 4),
    (dict(n=8192, block=4096, causal=1, n0=512), "boxes", 4),
    (dict(n=4096, block=256, samples=256), "nodes", 8), (dict(n=32768, block=64), "nodes", 8), (dict(H=32, n=131072, block=64), "nodes", 8),
    (dict(H=128, n=4096, causal=1, n0=4096), "boxes", 4),                  # (leaves alone: everything is written by one launch)
    # the shapes of test_gpu_kernel_edges.py whose items are more than the SMs: every build of a call in one launch is run there
    (dict(H=40, n=640, block=64, samples=33, causal=1, n0=320), "rows", 8), (dict(H=210, n=300, block=64, samples=8, causal=1, n0=512), "rows", 8),
    (dict(H=16, n=1400, block=64, samples=33, causal=1, n0=700), "boxes", 8),
    (dict(H=4, n=3400, block=64, samples=33, causal=1, n0=1700), "boxes", 4),
], ids=lambda x: "_".join(f"{k}{v}" for k, v in x.items()) if isinstance(x, dict) else str(x))
def test_build_of_the_backward_kernel(d, kw, out, warps):
    assert _backward_launches(d=d, **kw) == [(ALL if "causal" in kw and kw["n"] > kw["n0"] else NODES if out == "nodes" else LEAVES,
                                              out, warps if d == 64 else 8)]


# (the first of every shape is the one of test_gpu_kernel_edges.py, where every build of the second launch is run)
@pytest.mark.parametrize("d,heads,kw,first,second", [
    (64, (26, 24, 23), dict(n=16384, block=256, n0=4096), 4, ("nodes", 8)), (128, (13, 12, 11), dict(n=16384, block=256, n0=4096), 8, ("nodes", 8)),
    (64, (26, 24, 23), dict(n=16384, block=512, n0=512), 8, ("rows", 8)), (128, (13, 12, 11), dict(n=16384, block=512, n0=512), 8, ("rows", 8)),
    (64, (400, 384, 383), dict(n=1024, block=512, n0=512), 8, ("boxes", 8)), (64, (50, 48, 47), dict(n=8192, block=4096, n0=512), 8, ("boxes", 4)),
    (128, (13, 12, 11), dict(n=16384, block=8192, n0=4096), 8, ("boxes", 8)),
], ids=lambda x: "_".join(f"{k}{v}" for k, v in x.items()) if isinstance(x, dict) else None)
def test_builds_of_the_backward_kernel_in_two_launches(d, heads, kw, first, second):
    for H in heads[:2]:
        assert _backward_launches(d=d, H=H, causal=1, samples=8, **kw) == [(LEAVES, "first", first), (NODES, *second)]
    assert [x[0] for x in _backward_launches(d=d, H=heads[2], causal=1, samples=8, **kw)] == [ALL]


# Rows per chunk: evened out over the unit; halved where the busiest SM gets less to do, and at d = 64 from 2048 rows also where it gets as much and
# the sort keeps to one launch (nodes of up to 16 chunks); fp32 inputs, whose hash works in passes of 256 rows, by the passes, to as many launches
# and nodes of up to 64 chunks
@pytest.mark.parametrize("kw,d64,d128", [
    (dict(H=1, n=1000), 256, 256), (dict(H=32, n=4096), 1024, 1024), (dict(H=40, n=16384), 2048, 2048),
    (dict(H=35, n=8192), 1024, 2048), (dict(H=64, n=4096), 1024, 2048), (dict(H=17, n=16384), 1024, 2048), (dict(H=30, n=7687, causal=1, n0=4096), 1024, 2048),
    (dict(H=9, n=30000), 2048, 2048), (dict(H=8, n=32800), 2048, 2048),         # ... nodes of more than 16 chunks
    (dict(H=60, n=2500), 1280, 1280),                                            # ... more rows for the busiest SM
    (dict(H=37, n=8192), 2048, 2048),                                            # ... two CTAs for an SM
])
def test_rows_per_chunk(kw, d64, d128):
    assert (_chunk_rows(d=64, **kw), _chunk_rows(d=128, **kw)) == (d64, d128)


@pytest.mark.parametrize("kw,d64,d128", [
    (dict(H=1, n=1024), 256, 256), (dict(H=4, n=4096), 256, 256), (dict(H=20, n=2349), 256, 256), (dict(H=10, n=4000), 256, 256),
    (dict(H=50, n=700), 256, 256), (dict(H=15, n=2500, causal=1, n0=700), 256, 256), (dict(H=4, n=10000), 256, 256),
    (dict(H=20, n=3000, causal=1, n0=1024), 768, 512), (dict(H=20, n=2247, causal=1, n0=1024), 768, 512),    # as many passes, more CTAs
    (dict(H=5, n=8000), 512, 512), (dict(H=12, n=5000), 512, 512),               # ... a launch more
    (dict(H=2, n=20000), 512, 512),                                              # ... nodes of 79 chunks
    (dict(H=40, n=16384), 2048, 2048),
])
def test_rows_per_chunk_of_fp32_inputs(kw, d64, d128):
    assert (_chunk_rows(d=64, dtype=B.FP32, **kw), _chunk_rows(d=128, dtype=B.FP32, **kw)) == (d64, d128)


def _chunk_rows(**kw):
    rows = C.c_int(0)
    assert ha.lib().hyperattn_internal_chunk_rows(C.byref(_params(**kw)), C.byref(rows)) == 0
    return rows.value


def _backward_launches(**kw):
    got = (C.c_int * 7)()
    assert ha.lib().hyperattn_internal_backward_launches(C.byref(_params(**kw)), got) == 0
    return [(got[1 + 3 * i], OUT[got[2 + 3 * i]], got[3 + 3 * i]) for i in range(got[0])]
