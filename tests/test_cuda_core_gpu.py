"""The CUDA-core decode kernel and the few-token append at the edges of their
tiles, against the fp64 oracle: sequences cut at 32 tokens, more sequences than
a block has threads, both head dims, one and several query heads per KV head,
the smallest and the largest group rank, value ranks past one column per
thread, hidden widths that no lane count divides.

Decode bound: max|o - o_ref| / ||o_ref||_inf <= 1e-5 (fp32) or 2e-2 (bf16
outputs).  Append bound per element: u |c| + K 2^-23 sum_k |x_k a_k|.
"""

import numpy as np
import pytest
import torch

import oracle
from paper_2607_24331_gb300 import dck, device
from paper_2607_24331_gb300 import synth as S
from gpu_util import assert_parity, gpu_decode, oracle_decode
from test_step_gpu import _step

pytestmark = pytest.mark.gpu


def _layer(hq, groups, ranks, rv, d, dtype="f32", hidden=200):
    hkv = sum(len(g) for g in groups)
    return S.LayerSpec(hidden, hq, hkv, d, groups, ranks, rv, dtype, 1e4)


LAYERS = {
    "mha64": _layer(3, ((2,), (0, 1)), (16, 96), 160, 64),
    "mha128": _layer(2, ((1,), (0,)), (256, 48), 272, 128),
    "gqa4-64": _layer(8, ((1, 0),), (32,), 528, 64),
    "gqa8-128": _layer(8, ((0,),), (256,), 48, 128),
    "mha128-bf16": _layer(2, ((1, 0),), (112,), 272, 128, "bf16"),
    "gqa2-64-bf16": _layer(4, ((1,), (0,)), (16, 48), 32, 64, "bf16"),
}


@pytest.mark.parametrize("name", list(LAYERS))
@pytest.mark.parametrize("lens", [(1, 31, 32, 33, 0, 65, 500), (3000,)], ids=["edges", "long"])
def test_decode_tiles(name, lens):
    spec = LAYERS[name]
    got, di = gpu_decode(spec, lens, seed=4, kernel=1)
    live = [b for b, n in enumerate(lens) if n]  # the oracle takes no empty sequence: its output is zero
    ref = oracle_decode(di, batch_ids=live)
    assert_parity(got[live], ref[live], spec.dtype, f"{name} {lens}")
    assert all((got[b] == 0).all() for b, n in enumerate(lens) if not n)


def test_many_sequences():
    spec = LAYERS["mha64"]
    lens = tuple(1 + (7 * i) % 70 for i in range(300))
    got, di = gpu_decode(spec, lens, seed=5, kernel=1)
    assert_parity(got, oracle_decode(di), "f32", "300 sequences")


@pytest.mark.parametrize("lens", [(1,), (33, 400, 64), tuple(range(1, 70))], ids=["one", "three", "many"])
def test_step_fp32(lens):
    _step(S.workload(0).layer, lens, seed=6)


@pytest.mark.parametrize("hidden,rv,n", [(200, 32, 5), (130, 32, 5), (256, 64, 300), (256, 32, 300), (36, 2048, 40)],
                         ids=["cluster", "few", "pairs", "tiles", "core-tiles"])
@pytest.mark.parametrize("qpg", [1, 2])
def test_step_bf16_behind_each_append(hidden, rv, n, qpg):
    """The decode kernel starts early behind the step's own append: bf16 layers of head dim 64 behind each kernel that
    appends for them, the last tokens (all of a one-token sequence) being this step's own."""
    lens = (1, 31, 33, 400, 1) if n == 5 else tuple(1 + (13 * i) % 40 for i in range(n))
    _step(S.LayerSpec(hidden, 2 * qpg, 2, 64, ((1,), (0,)), (16, 48), rv, "bf16", 1e4), lens, seed=hidden + rv)


@pytest.mark.parametrize("hidden", [1, 8, 127, 128, 130, 200, 512, 1100])
@pytest.mark.parametrize("n_tok", [1, 8, 9, 129, 256, 512, 513])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_append_few(dtype, n_tok, hidden):
    # (bf16 layers whose hidden width is a multiple of 8 take the tensor-core cluster: here with output widths
    # below its 64 columns and with fewer 64-wide K blocks than CTAs; the other bf16 layers go the fp32 way)
    spec = _layer(2, ((1,), (0,)), (16, 32), 16, 64, dtype, hidden)
    x, A_k, A_v = S.make_append_inputs(spec, n_tok, seed=hidden)
    rows = np.random.default_rng(n_tok).choice(n_tok + 5, size=n_tok, replace=False)
    buf = device.AppendBuffers(spec, n_tok, n_tok + 5).load_host(x, A_k, A_v, rows)
    dck.check(buf.run(), "dck_latent_append")
    torch.cuda.synchronize()
    assert dck.dck_last_device_error() == dck.DCK_OK
    u = 2.0 ** -8 if dtype == "bf16" else 2.0 ** -23
    for got, ref, A in zip((buf.kcache, buf.vcache), oracle.latent_append(x, A_k, A_v), (A_k, A_v)):
        got = got.float().cpu().numpy().astype(np.float64)
        bound = u * np.abs(ref) + hidden * 2.0 ** -23 * (np.abs(x.astype(np.float64)) @ np.abs(A.astype(np.float64)))
        assert (np.abs(got[rows] - ref) <= bound).all()
        assert (got[np.setdiff1d(np.arange(n_tok + 5), rows)] == 0).all()


def _wide(dtype, hidden, width):
    return S.LayerSpec(hidden, 2, 2, 64, ((1,), (0,)), (width // 4, width // 4), width // 2, dtype, 1e4)


@pytest.mark.parametrize("dtype,hidden", [("f32", 200), ("bf16", 196)])
@pytest.mark.parametrize("width,side", [(2048, 0), (2048, 1), (512, 0), (512, 1)])
def test_append_few_or_tiles(dtype, hidden, width, side):
    """Either side of the line between the few-token and the tile kernel: n_tok (R_k + r_v) (D + 256) = 400000 D."""
    n_tok = 400000 * hidden // ((hidden + 256) * width) + side
    spec = _wide(dtype, hidden, width)
    x, A_k, A_v = S.make_append_inputs(spec, n_tok, seed=width)
    rows = np.random.default_rng(n_tok).choice(n_tok + 5, size=n_tok, replace=False)
    buf = device.AppendBuffers(spec, n_tok, n_tok + 5).load_host(x, A_k, A_v, rows)
    dck.check(buf.run(), "dck_latent_append")
    torch.cuda.synchronize()
    assert dck.dck_last_device_error() == dck.DCK_OK
    u = 2.0 ** -8 if dtype == "bf16" else 2.0 ** -23
    for got, ref, A in zip((buf.kcache, buf.vcache), oracle.latent_append(x, A_k, A_v), (A_k, A_v)):
        got = got.float().cpu().numpy().astype(np.float64)
        bound = u * np.abs(ref) + hidden * 2.0 ** -23 * (np.abs(x.astype(np.float64)) @ np.abs(A.astype(np.float64)))
        assert (np.abs(got[rows] - ref) <= bound).all()


@pytest.mark.parametrize("hidden,width", [(512, 4096), (64, 4096), (512, 1024)])
def test_wide_append_takes_no_longer_than_one_token_more(hidden, width):
    """512 tokens against 513 (the tile kernel): 5.5, 11 and 1.5 times as long while every call of up to 512 tokens
    went to the few-token kernel."""
    spec = _wide("f32", hidden, width)
    us = {}
    for n_tok in (512, 513):
        x, A_k, A_v = S.make_append_inputs(spec, n_tok)
        buf = device.AppendBuffers(spec, n_tok, n_tok).load_host(x, A_k, A_v, np.arange(n_tok))
        times = []
        for _ in range(15):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            dck.check(buf.run(), "dck_latent_append")
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        us[n_tok] = sorted(times)[7]
    assert us[512] <= 1.3 * us[513], us


def test_current_stream():
    """A call without a stream goes to the current one."""
    torch.cuda.init()
    side = torch.cuda.Stream()
    assert dck._stream(None) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert dck._stream(None) == side.cuda_stream != torch.cuda.default_stream().cuda_stream
    assert dck._stream(side) == side.cuda_stream
