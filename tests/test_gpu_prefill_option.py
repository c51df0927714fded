"""MTP_OPT_PREFILL_TC: prefill attention never in tensor-core tiles, always, or by the pass's rows."""
import pytest

import synth
from oracle.mtp import MTPOracle

from gpu_util import assert_logits_close, decoder, lib_module

pytestmark = pytest.mark.gpu

WIDE = synth.ModelConfig(layers=2, d_model=1024, n_attn_heads=16, d_ffn=1024, phone_vocab=128)


def test_values():
    mtp = lib_module()
    dec, _ = decoder(synth.TINY_BF16, max_ctx=64)
    try:
        assert mtp.mtp_get_option(dec.ctx, 10) == 2
        for value, kept in ((0, 0), (1, 1), (2, 2), (0, 0), (-1, 1), (7, 1)):
            mtp.mtp_set_option(dec.ctx, 10, value)
            assert mtp.mtp_get_option(dec.ctx, 10) == kept
    finally:
        dec.close()


@pytest.mark.parametrize("value", [0, 1, 2])
def test_long_prompt(value):
    mtp = lib_module()
    dec, w = decoder(synth.TINY_BF16, max_ctx=1700)
    ph, ac = synth.make_prompt(77, 400, 1237, synth.TINY_BF16.phone_vocab)
    try:
        mtp.mtp_set_option(dec.ctx, 10, value)
        dec.prefill(0, ph, ac, 8)
        dec.decode_step(4, 4)
        o = MTPOracle(synth.TINY_BF16, w)
        o.prefill(ph, ac, 8)
        assert_logits_close(dec.logits(4)[0][0], o.step(4, 4).logits, f"value {value}")
    finally:
        dec.close()


def test_never_means_never():
    """2000 rows of 16 heads take about half as long again in groups of 8 rows as in tiles."""
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    dec, _ = decoder(WIDE, max_ctx=2048)
    ph, ac = synth.make_prompt(78, 500, 1500, WIDE.phone_vocab)
    took = {}
    try:
        for value in (0, 1, 2):
            mtp.mtp_set_option(dec.ctx, 10, value)
            times = []
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                mtp.mtp_prefill(dec.ctx, 0, ph, ac, 8)
                b.record()
                torch.cuda.synchronize()
                mtp.mtp_release(dec.ctx, 0)
                times.append(a.elapsed_time(b))
            took[value] = min(times)
    finally:
        dec.close()
    assert took[0] >= 1.15 * took[1] and took[2] <= 1.1 * took[1], took
