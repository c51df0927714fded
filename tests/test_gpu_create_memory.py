"""A context fits beside a KV pool that leaves little of the GPU's memory: the buffers of long
prefill passes shrink to what is left, and prompts run in shorter passes."""
import pytest

import synth
from oracle.mtp import MTPOracle

from gpu_util import assert_logits_close, decoder, lib_module

pytestmark = pytest.mark.gpu

MODEL = synth.TINY_BF16


def test_little_memory_left():
    torch = pytest.importorskip("torch")
    lib_module()
    decoder(MODEL, max_ctx=64)[0].close()          # the library's code and weights generator are loaded
    torch.cuda.empty_cache()
    page_bytes = MODEL.layers * 2 * MODEL.n_attn_heads * 64 * 64 * 2
    pages = (torch.cuda.mem_get_info()[0] - (72 << 20)) // page_bytes
    # whole passes would be 14592 rows of 7168 bytes: 105 MB
    dec, w = decoder(MODEL, max_batch=16, max_ctx=1024, n_pages=int(pages))
    try:
        prompts = [synth.make_prompt(600 + b, 100, 900, MODEL.phone_vocab) for b in range(4)]
        for b, (ph, ac) in enumerate(prompts):
            dec.admit(b, ph, ac, 8)
        assert lib_module().mtp_prefill_pending(dec.ctx) >= 2
        dec.decode_step(4, 4)
        lg = dec.logits(4)[0]
        for b in (0, 3):
            o = MTPOracle(MODEL, w)
            o.prefill(*prompts[b], 8)
            assert_logits_close(lg[b], o.step(4, 4).logits, f"slot {b}")
    finally:
        dec.close()
