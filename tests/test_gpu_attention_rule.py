"""mtp_attention on both sides of the lines at which a call takes a CTA per group and head, or shares
its batches out over a wave of CTAs: contexts of two batches and one key more, of 640 keys and one
more, groups that are just three quarters of the SMs, just a wave, and one more."""
import pytest

from test_gpu_attention_stream import H, _check, _inputs

from gpu_util import lib_module

pytestmark = pytest.mark.gpu

THREE_QUARTERS, WAVE = -(-3 * 152 // (4 * H)), 4 * 152 // H   # groups, on 152 SMs


@pytest.mark.parametrize("groups,longest,rows,page", [
    (1, 33, 1, 64), (2, 128, 3, 16), (2, 129, 3, 16), (1, 257, 8, 128),
    (THREE_QUARTERS - 1, 640, 2, 64), (THREE_QUARTERS, 640, 2, 64), (THREE_QUARTERS, 641, 2, 64),
    (WAVE, 200, 1, 32), (WAVE + 1, 200, 1, 32), (3, 1024, 4, 64), (3, 1025, 4, 64),
])
def test_both_sides(groups, longest, rows, page):
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    ctx = [longest] + [max(rows, longest - 1 - (53 * g) % longest) for g in range(1, groups)]
    pool, table, q, seq, pos = _inputs(torch, ctx, rows, page, 0, False)
    out = torch.full((len(seq), H * q.shape[-1]), -7.0, device="cuda")
    row_seq, row_pos = (torch.tensor(x, dtype=torch.int32, device="cuda") for x in (seq, pos))
    args = mtp.attention_args(rows=len(seq), rows_per_group=rows, n_heads=H, page_size=page, layers=1, layer=0,
                              bt_stride=table.shape[1], max_keys=longest, q=q.view(len(seq), -1), kv_pool=pool,
                              block_table=table, row_seq=row_seq, row_pos=row_pos, out=out)
    nbytes = mtp.mtp_attention_workspace_bytes(args)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        out.fill_(-7.0)
        mtp.mtp_attention(args, ws, nbytes, torch.cuda.current_stream())
    torch.cuda.synchronize()
    _check(torch, out, pool, table, q, seq, pos)
