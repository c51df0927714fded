"""mtp_attention's stream of key batches shared out over CTAs, against a float64 softmax, where
the sharing can go wrong: fewer batches than CTAs, groups cut by CTA ranges at every place,
more groups than one scan takes (128), groups without active rows, a row count that is no
multiple of the group, every page size, scores that move the softmax reference, and a
workspace smaller than the call asks for (fewer CTAs per head)."""
import pytest

from gpu_util import lib_module

pytestmark = pytest.mark.gpu

H, HD = 4, 64

CASES = [  # contexts (0: a group without active rows), rows per group, page size
    ([1], 1, 64),
    ([64, 65, 63], 3, 64),
    ([1500], 8, 16),
    ([300, 0, 77, 0, 0, 513], 4, 32),
    ([33 + 7 * g for g in range(40)], 2, 128),
    ([1 + (37 * g) % 190 for g in range(300)], 1, 64),     # groups past the first scan
    ([0] * 130 + [200, 0, 900], 5, 64),                    # the stream starts past the first scan
    ([2000, 10, 10, 1990, 64, 128], 4, 64),
    ([1 + (29 * g) % 128 for g in range(50)] + [0, 128], 1, 64),  # short contexts: a CTA per group
]


def _inputs(torch, ctx, rpg, page, drop, sharp):
    gen = torch.Generator(device="cuda").manual_seed(len(ctx) * 1000 + rpg * 10 + page)
    per = max(1, -(-max(ctx) // page))
    pool = torch.randn(len(ctx) * per, 1, 2, H, page, HD, device="cuda", generator=gen)
    if sharp:  # scores up to about 8 * 30: the reference moves from batch to batch
        pool[:, :, 0] *= 1.0 + 29.0 * torch.rand(len(ctx) * per, 1, 1, 1, 1, device="cuda", generator=gen)
    pool = pool.bfloat16()
    table = torch.randperm(len(ctx) * per, device="cuda", generator=gen).to(torch.int32).view(len(ctx), per)
    rows = len(ctx) * rpg - drop
    q = torch.randn(rows, H, HD, device="cuda", generator=gen)
    seq = [g if c > 0 else -1 for g, c in enumerate(ctx) for _ in range(rpg)][:rows]
    pos = [max(0, c - rpg + j) for c in ctx for j in range(rpg)][:rows]
    return pool, table, q, seq, pos


def _check(torch, out, pool, table, q, seq, pos):
    got = out.view(len(seq), H, HD).double()
    for r, (s, p) in enumerate(zip(seq, pos)):
        if s < 0:
            assert (got[r] == -7.0).all(), f"row {r} of no sequence was written"
            continue
        kv = pool[table[s].long(), 0].permute(1, 2, 0, 3, 4).flatten(2, 3)[:, :, :p + 1].double()
        a = torch.einsum("hd,hkd->hk", q[r].double(), kv[0]) / 8.0
        ref = torch.einsum("hk,hkd->hd", torch.softmax(a, -1), kv[1])
        # Q and P keep 16 bits: a weight is off by 2^-17 of the score's terms, |q||k| / 8 in all
        bound = 1e-5 + 2 ** -16 * (q[r].double().norm() * kv[0].norm(dim=-1).max() / 8.0).item()
        assert (got[r] - ref).abs().max() <= bound * max(1.0, ref.abs().max().item()), f"row {r}"


@pytest.mark.parametrize("ctx,rpg,page", CASES)
@pytest.mark.parametrize("sharp", [False, True])
@pytest.mark.parametrize("room", ["asked", "least"])
def test_stream(ctx, rpg, page, sharp, room):
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    drop = rpg // 2 if ctx[-1] else 0
    pool, table, q, seq, pos = _inputs(torch, ctx, rpg, page, drop, sharp)
    out = torch.full((len(seq), H * HD), -7.0, device="cuda")
    row_seq, row_pos = (torch.tensor(x, dtype=torch.int32, device="cuda") for x in (seq, pos))
    args = mtp.attention_args(rows=len(seq), rows_per_group=rpg, n_heads=H, page_size=page, layers=1, layer=0,
                              bt_stride=table.shape[1], max_keys=max(ctx), q=q.view(len(seq), H * HD),
                              kv_pool=pool, block_table=table, row_seq=row_seq, row_pos=row_pos, out=out)
    nbytes = mtp.mtp_attention_workspace_bytes(args)
    if room == "least":   # the counters and one part of every group, what the smallest calls ask for
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        parts = max(1, min(sms // (len(ctx) * H), -(-max(ctx) // page), 32))
        up = lambda x: -(-x // 256) * 256  # noqa: E731
        nbytes = min(nbytes, up(len(ctx) * H * parts * 8 * 66 * 4) + up(len(ctx) * H * 4))
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    for _ in range(2):    # the counters come back to zero
        out.fill_(-7.0)
        mtp.mtp_attention(args, ws, nbytes, torch.cuda.current_stream())
    torch.cuda.synchronize()
    _check(torch, out, pool, table, q, seq, pos)
    with pytest.raises(mtp.MTPError):
        mtp.mtp_attention(args, ws, 16, torch.cuda.current_stream())
