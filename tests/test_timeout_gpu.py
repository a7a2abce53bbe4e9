"""Failure detection on the GPU without a fault: a bounded wait on a barrier
that nothing arrives at gives up by its own limit, the kernel reports the
timeout through the device error word, and the context keeps working."""

import time

import numpy as np
import pytest
import torch

from gpu_util import assert_parity, gpu_decode, oracle_decode
from paper_2607_24331_gb300 import dck, device
from paper_2607_24331_gb300 import synth as S

pytestmark = pytest.mark.gpu


def test_bounded_wait_gives_up_and_the_context_stays_usable():
    assert dck.dck_last_device_error() == dck.DCK_OK  # start from a clear error word
    t0 = time.perf_counter()
    dck.check(dck.dck_selftest_bounded_wait(2_000_000), "dck_selftest_bounded_wait")  # about 1 ms of SM clock
    assert dck.dck_last_device_error() == dck.DCK_ERR_TIMEOUT
    assert time.perf_counter() - t0 < 10.0
    assert dck.dck_last_device_error() == dck.DCK_OK  # reading the word cleared it
    # a regular call on the same context afterwards
    spec = S.workload(1).layer
    got, di = gpu_decode(spec, (129, 7), seed=4)
    assert_parity(got, oracle_decode(di), "bf16", "after the timeout")


@pytest.mark.parametrize("n_tok,hidden", [(1, 64), (100, 512), (200, 4096), (300, 512)])
def test_append_whose_operands_do_not_arrive(n_tok, hidden):
    """The cluster append (up to 256 tokens; one K block in all, a few per CTA, more than its ring holds) and the
    tile append (300 tokens, widths off 64): a block of operands that is never loaded ends the call by the wait's
    own limit, no cache row holds a sum that is not whole, and the same append afterwards is right."""
    spec = S.LayerSpec(hidden, 2, 2, 128, ((1,), (0,)), (80, 112), 176, "bf16", 1e4)
    x, A_k, A_v = S.make_append_inputs(spec, n_tok, seed=hidden)
    rows = np.arange(n_tok) + 3
    buf = device.AppendBuffers(spec, n_tok, n_tok + 5).load_host(x, A_k, A_v, rows)
    assert dck.dck_last_device_error() == dck.DCK_OK
    t0 = time.perf_counter()
    dck.check(dck.dck_selftest_append_timeout(buf.layer, buf.x, n_tok, buf.A_k, buf.A_v, buf.rows, buf.kcache,
                                              buf.vcache, buf.n_rows, 2_000_000), "dck_selftest_append_timeout")
    assert dck.dck_last_device_error() == dck.DCK_ERR_TIMEOUT
    assert time.perf_counter() - t0 < 1.0  # the other CTAs of a cluster are told, and do not wait for their 2 s
    assert not buf.kcache.any() and not buf.vcache.any()
    dck.check(buf.run(), "dck_latent_append")
    torch.cuda.synchronize()
    assert dck.dck_last_device_error() == dck.DCK_OK
    for got, ref in zip((buf.kcache, buf.vcache), (x @ A_k, x @ A_v)):
        assert np.abs(got.float().cpu().numpy()[rows] - ref).max() <= 2.0 ** -7 * np.abs(ref).max()
