"""Prefill attention on both sides of the line between groups of 8 rows and tiles of 128 (4 heads on
152 SMs: 1216 rows of long prompts, 2432 of prompts shorter than a tile), against the oracle."""
import copy

import pytest

import synth
from oracle.mtp import MTPOracle

from gpu_util import assert_logits_close, decoder, lib_module

pytestmark = pytest.mark.gpu

MODEL = synth.TINY_BF16


@pytest.mark.parametrize("lengths", [[1216], [1217], [600, 616], [600, 617], [100] * 20, [100] * 24, [121] * 20])
def test_both_sides(lengths):
    mtp = lib_module()
    prompts = [synth.make_prompt(500 + b, t // 4, t - t // 4, MODEL.phone_vocab) for b, t in enumerate(lengths)]
    dec, w = decoder(MODEL, max_batch=len(lengths), max_ctx=max(lengths) + 32)
    try:
        for b, (ph, ac) in enumerate(prompts):
            dec.admit(b, ph, ac, 8)
        assert mtp.mtp_prefill_pending(dec.ctx) == 1
        dec.decode_step(4, 4)
        lg = dec.logits(4)[0]
        first = MTPOracle(MODEL, w)
        for b in sorted({0, 1, len(lengths) // 2, len(lengths) - 1} & set(range(len(lengths)))):
            o = copy.copy(first)
            o.prefill(*prompts[b], 8)
            assert_logits_close(lg[b], o.step(4, 4).logits, f"slot {b}")
    finally:
        dec.close()
