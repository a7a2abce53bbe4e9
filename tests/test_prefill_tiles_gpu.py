"""Prefill attention at the edges of its tiles, against the fp64 oracle: head
counts and group sizes that leave a lone head in a tile, ranks at both ends of
what the call takes (one 16-wide k-step, and past four 64-wide stages), value
ranks that end inside a stage, sequences cut at the 256-row tiles, caches
packed and pooled (the same launches for the same sequences), a long context,
one sequence with nearly all of the batch's new tokens, and the output written
over the queries.

The bound is the decode one, max|o - o_ref| / ||o_ref||_inf <= 2e-2: keys,
values and probabilities are rounded to bf16 (2^-9 each) before products that
accumulate in fp32.
"""

import numpy as np
import pytest
import torch

import oracle
from paper_2607_24331_gb300 import dck, device
from paper_2607_24331_gb300 import synth as S
from gpu_util import assert_parity

pytestmark = pytest.mark.gpu


def _layer(hq, groups, ranks, rv, theta=1e4):
    hkv = sum(len(g) for g in groups)
    return S.LayerSpec(256, hq, hkv, 128, groups, ranks, rv, "bf16", theta)


LAYERS = {
    "lone-heads": _layer(3, ((2,), (0, 1)), (16, 272), 48),
    "one-head-gqa": _layer(8, ((0,),), (112,), 80, 1e6),
    "five-heads-gqa2": _layer(10, ((4, 1, 0), (3, 2)), (64, 144), 128),
    "gqa4": _layer(8, ((1, 0),), (32,), 16),
}
SHAPES = [
    ((1, 255, 256, 257), (1, 255, 10, 257)),
    ((600, 0, 513), (599, 0, 1)),
    ((20000,), (3,)),
    ((40, 1100, 300, 1, 700), (1, 1100, 2, 1, 0)),
]


@pytest.mark.parametrize("pool", [1, 5])
@pytest.mark.parametrize("shape", SHAPES, ids=["edges", "chunk", "long", "one-long"])
@pytest.mark.parametrize("name", list(LAYERS))
def test_prefill_tiles(name, shape, pool):
    spec = LAYERS[name]
    lens, q_lens = shape
    B, q_max = len(lens), max(q_lens) + 2
    rows = [pool * n for n in lens]
    di = S.make_decode_inputs(spec, rows, seed=11)
    q = S.make_prefill_q(spec, B, q_max, seed=12)
    buf = device.DecodeBuffers(spec, rows).load_host(di)
    qd = torch.from_numpy(q).to("cuda", torch.bfloat16)
    out = qd  # the results replace the queries
    ql = torch.tensor(q_lens, dtype=torch.int32, device="cuda")
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    n = dck.dck_prefill_workspace_size(buf.layer, buf.n_rows)
    ws = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")  # NaN bit patterns where nothing is rebuilt
    dck.check(dck.dck_prefill_attention(buf.layer, qd, ql, q_max, buf.kcache, buf.vcache, buf.n_rows, buf.B_k,
                                        buf.B_v, buf.seq_start, sl, B, max(lens), spec.rope_theta, out, ws, n),
              "dck_prefill_attention")
    assert dck.dck_last_launch_count() == 2  # by the sequences, not by the size of the caller's cache
    torch.cuda.synchronize()
    assert dck.dck_last_device_error() == dck.DCK_OK
    got = out.float().cpu().numpy().astype(np.float64)
    live = [b for b in range(B) if q_lens[b]]
    ref = oracle.prefill_attention(spec, q[live], [q_lens[b] for b in live], di.kcache, di.vcache, di.B_k, di.B_v,
                                   di.seq_start[live], np.asarray(lens)[live])
    for i, b in enumerate(live):
        Q = q_lens[b]
        assert_parity(got[b, :Q], ref[i, :Q], "bf16", f"{name} sequence {b}")
    for b in range(B):
        assert (got[b, q_lens[b]:] == q[b, q_lens[b]:]).all(), "rows past Q_b keep their contents"
