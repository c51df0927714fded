"""How far the attention operators are from 64 bits where a sum over many keys could drift or an
exact input could lose bits."""
import pytest

from gpu_util import lib_module

pytestmark = pytest.mark.gpu

HD, P = 64, 64


def _error(tc, heads, keys, rows, value_mean, query_bits):
    """Relative error (2-norms) of one slot's last `rows` rows over `keys` cached keys."""
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    gen = torch.Generator(device="cuda").manual_seed(keys + rows)
    pages = -(-keys // P)
    kv = torch.randn(pages, 2, heads, P, HD, device="cuda", generator=gen)
    kv[:, 1] += value_mean
    kv = kv.bfloat16()
    pool = kv
    if tc:  # the cache's row layout: chunk c of row t at chunk c ^ (t mod 8)
        t, c = torch.arange(P, device="cuda")[:, None], torch.arange(8, device="cuda")[None, :]
        pool = kv.view(pages, 2, heads, P, 8, 8)[..., t, c ^ (t & 7), :].flatten(-2).contiguous()
    q = torch.randn(rows, heads, HD, device="cuda", generator=gen)
    if query_bits == 8:
        q = q.bfloat16().float()
    ints = lambda x: torch.tensor(x, dtype=torch.int32, device="cuda")  # noqa: E731
    table, seq, pos = ints([list(range(pages))]), ints([0] * rows), ints(list(range(keys - rows, keys)))
    out = torch.zeros(rows, heads * HD, device="cuda")
    args = mtp.attention_args(rows=rows, rows_per_group=min(8, rows), n_heads=heads, page_size=P, layers=1, layer=0,
                              bt_stride=pages, max_keys=keys, q=q.view(rows, heads * HD), kv_pool=pool,
                              block_table=table, row_seq=seq, row_pos=pos, out=out)
    nbytes = (mtp.mtp_attention_tc_workspace_bytes if tc else mtp.mtp_attention_workspace_bytes)(args)
    ws = torch.zeros(max(16, nbytes), dtype=torch.uint8, device="cuda")
    (mtp.mtp_attention_tc if tc else mtp.mtp_attention)(args, ws, nbytes, torch.cuda.current_stream())
    k, v = kv.double().permute(1, 2, 0, 3, 4).flatten(2, 3)[:, :, :keys]
    a = torch.einsum("rhd,hkd->hrk", q.double(), k) / 8.0
    a = a.masked_fill(torch.arange(keys, device="cuda")[None, :] > pos.double()[:, None], float("-inf"))
    ref = torch.einsum("hrk,hkd->rhd", torch.softmax(a, -1), v).flatten(1)
    return ((out.double() - ref).norm() / ref.norm()).item()


def test_prompt_sums_do_not_drift():
    """Values of mean 1: an accumulation only grows, and the tensor core truncates it at every MMA, by less than
    2^-23.  64 keys are eight MMAs; what lies behind them is added in fp32."""
    assert _error(True, 4, 2000, 1900, 1.0, 8) <= 8 * 2.0 ** -23


@pytest.mark.parametrize("tc", [False, True])
@pytest.mark.parametrize("keys,rows", [(100, 100), (1100, 64)])
@pytest.mark.parametrize("queries", ["zero", "cancelling"])
def test_equal_weights_give_the_rounded_mean(tc, keys, rows, queries):
    """Where every score is zero the weights are equal, and whole values make the sums exact: what is left is one
    division, which is rounded once.  Queries (3, 5) against keys (5 t, -3 t) are zero only if the scaled queries
    are exact, as bf16-valued ones are when scaled by 1/8."""
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    heads, pages = 2, -(-keys // P)
    gen = torch.Generator(device="cuda").manual_seed(keys)
    kv = torch.randn(pages, 2, heads, P, HD, device="cuda", generator=gen).bfloat16()
    kv[:, 1] = torch.randint(-128, 129, (pages, heads, P, HD), device="cuda", generator=gen).bfloat16()
    q = torch.zeros(rows, heads * HD, device="cuda")
    if queries == "cancelling":
        q[:, 0::2], q[:, 1::2] = 3.0, 5.0
        t = torch.randint(-25, 26, (pages, heads, P, HD // 2), device="cuda", generator=gen)
        kv[:, 0, ..., 0::2], kv[:, 0, ..., 1::2] = (5 * t).bfloat16(), (-3 * t).bfloat16()
    pool = kv
    if tc:  # the cache's row layout: chunk c of row t at chunk c ^ (t mod 8)
        t, c = torch.arange(P, device="cuda")[:, None], torch.arange(8, device="cuda")[None, :]
        pool = kv.view(pages, 2, heads, P, 8, 8)[..., t, c ^ (t & 7), :].flatten(-2).contiguous()
    ints = lambda x: torch.tensor(x, dtype=torch.int32, device="cuda")  # noqa: E731
    table, seq, pos = ints([list(range(pages))]), ints([0] * rows), ints(list(range(keys - rows, keys)))
    out = torch.zeros(rows, heads * HD, device="cuda")
    args = mtp.attention_args(rows=rows, rows_per_group=min(8, rows), n_heads=heads, page_size=P, layers=1, layer=0,
                              bt_stride=pages, max_keys=keys, q=q, kv_pool=pool, block_table=table, row_seq=seq,
                              row_pos=pos, out=out)
    nbytes = (mtp.mtp_attention_tc_workspace_bytes if tc else mtp.mtp_attention_workspace_bytes)(args)
    ws = torch.zeros(max(16, nbytes), dtype=torch.uint8, device="cuda")
    (mtp.mtp_attention_tc if tc else mtp.mtp_attention)(args, ws, nbytes, torch.cuda.current_stream())
    sums = kv[:, 1].double().permute(1, 0, 2, 3).flatten(1, 2).cumsum(1)[:, keys - rows:keys]
    want = (sums / (pos.double() + 1)[None, :, None]).float().transpose(0, 1).flatten(1)
    assert torch.equal(out, want)
