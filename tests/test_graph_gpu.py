"""Calls captured into a CUDA graph: their launches depend on one another by
programmatic edges there too.  Each graph is replayed on two sets of inputs and
must give the bits of the eager calls."""

import numpy as np
import pytest
import torch

from paper_2607_24331_gb300 import dck, device
from paper_2607_24331_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _inputs(spec, lens, q_max, seed):
    """One set of the tensors that a replay reads or writes."""
    di = S.make_decode_inputs(spec, lens, seed=seed)
    x, A_k, A_v = S.make_append_inputs(spec, len(lens), seed=seed + 1)
    q = S.make_prefill_q(spec, len(lens), q_max, seed=seed + 2)
    up = lambda a: device.upload(a, spec.dtype)  # noqa: E731
    return [up(t) for t in (di.kcache, di.vcache, di.B_k, di.B_v, di.q, q, x, A_k, A_v)]


@pytest.mark.parametrize("kind,cfg", [("step", 0), ("step", 1), ("step", 2), ("append", 1), ("prefill", 1),
                                      ("prefill", 2)])
def test_replays_match_eager_calls(kind, cfg):
    spec = S.workload(cfg).layer
    lens, q_lens = (257, 1, 700), (200, 1, 130)
    B = len(lens)
    layer = dck.Layer.from_spec(spec)
    starts = S.seq_starts(np.asarray(lens))
    n_rows = sum(lens)
    i64 = lambda a: torch.from_numpy(np.asarray(a, dtype=np.int64)).cuda()  # noqa: E731
    i32 = lambda a: torch.from_numpy(np.asarray(a, dtype=np.int32)).cuda()  # noqa: E731
    seq_start, seq_len, q_len, rows = i64(starts), i32(lens), i32(q_lens), i64(starts + np.asarray(lens) - 1)
    sets = [_inputs(spec, lens, max(q_lens), seed) for seed in (3, 50)]
    live = [torch.zeros_like(t) for t in sets[0]]
    kc, vc, bk, bv, q, qp, x, ak, av = live
    out = torch.zeros_like(qp if kind == "prefill" else q)
    size = max(dck.dck_decode_step_workspace_size(layer, B, n_rows), dck.dck_prefill_workspace_size(layer, n_rows),
               dck.dck_latent_append_workspace_size(layer, B))
    ws = torch.empty(max(size, 256), dtype=torch.uint8, device="cuda")

    def call():
        if kind == "step":
            return dck.dck_decode_step(layer, x, ak, av, rows, q, kc, vc, n_rows, bk, bv, seq_start, seq_len, B,
                                       spec.rope_theta, out, ws, size)
        if kind == "append":
            return dck.dck_latent_append(layer, x, B, ak, av, rows, kc, vc, n_rows, ws, size)
        return dck.dck_prefill_attention(layer, qp, q_len, max(q_lens), kc, vc, n_rows, bk, bv, seq_start, seq_len,
                                         B, max(lens), spec.rope_theta, out, ws, size)

    def results(run):
        got = []
        for s in sets:
            for a, b in zip(live, s):
                a.copy_(b)
            out.zero_()
            run()
            torch.cuda.synchronize()
            got.append([t.clone() for t in (kc, vc, out)])
        return got

    eager = results(lambda: dck.check(call(), kind))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        dck.check(call(), kind)
    replayed = results(g.replay)
    assert dck.dck_last_device_error() == dck.DCK_OK
    for e, r in zip(eager, replayed):
        assert all(torch.equal(a, b) for a, b in zip(e, r))
    assert any(not torch.equal(a, b) for a, b in zip(*eager))  # the two sets differ
