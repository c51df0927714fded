"""mtp_attention_tc (Sec. III-A prompt attention) where its row runs and its running
softmax reference can go wrong, against a float64 softmax: rows of one slot in several
runs of a tile, runs of one row, tiles without rows, and scores whose maximum jumps
from item to item (the reference moves and the accumulated output is rescaled) or is
far below zero."""
import pytest

from gpu_util import lib_module

pytestmark = pytest.mark.gpu

H, HD, P = 2, 64, 64


def _spec(kind):
    """(slot, position) per row; slot -1: no sequence."""
    if kind == "interleaved":      # two slots alternate row by row: 128 runs of one row
        return [(r & 1, 40 + r) for r in range(128)]
    if kind == "split run":        # slot 0 before and after slot 1 within a tile
        return [(0, r) for r in range(50)] + [(1, 200 + r) for r in range(30)] + [(0, 300 + r) for r in range(60)]
    if kind == "empty tile":       # a tile of padding rows between two prompts
        return [(0, r) for r in range(100)] + [(-1, 0)] * 156 + [(1, r) for r in range(9)]
    return [(0, r) for r in range(500)]   # "one prompt": four tiles, up to four items


@pytest.mark.parametrize("kind", ["interleaved", "split run", "empty tile", "one prompt"])
@pytest.mark.parametrize("scores", ["plain", "rising", "low"])
def test_rows_and_scores(kind, scores):
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    spec, slots, pages = _spec(kind), 2, 8
    gen = torch.Generator(device="cuda").manual_seed(len(spec) + 7 * len(scores))
    kv = torch.randn(slots, 2, H, pages * P, HD, device="cuda", generator=gen)
    q = torch.randn(len(spec), H, HD, device="cuda", generator=gen)
    if scores == "rising":   # keys of later items point along the queries: the maximum grows by about 25 per item
        q = q * 0.1 + 1.0
        kv[:, 0] = kv[:, 0] * 0.1 + 3.0 * (torch.arange(pages * P, device="cuda") // 128)[:, None]
    elif scores == "low":    # every score about -200: weights relative to the row's own maximum
        q = q * 0.1 + 5.0
        kv[:, 0] = kv[:, 0] * 0.5 - 5.0
    kv = kv.bfloat16()
    # one page per 64 keys, rows swizzled as the cache stores them
    pool = kv.view(slots, 2, H, pages, P, 8, 8).permute(0, 3, 1, 2, 4, 5, 6)
    t, c = torch.arange(P, device="cuda")[:, None], torch.arange(8, device="cuda")[None, :]
    pool = pool[..., t, c ^ (t & 7), :].contiguous()
    table = torch.arange(slots * pages, device="cuda", dtype=torch.int32).view(slots, pages)
    seq = torch.tensor([s for s, _ in spec], dtype=torch.int32, device="cuda")
    pos = torch.tensor([p for _, p in spec], dtype=torch.int32, device="cuda")
    out = torch.full((len(spec), H * HD), -7.0, device="cuda")
    args = mtp.attention_args(rows=len(spec), rows_per_group=8, n_heads=H, page_size=P, layers=1, layer=0,
                              bt_stride=pages, max_keys=pages * P, q=q.view(len(spec), H * HD).contiguous(),
                              kv_pool=pool, block_table=table, row_seq=seq, row_pos=pos, out=out)
    nbytes = mtp.mtp_attention_tc_workspace_bytes(args)
    ws = torch.zeros(max(16, nbytes), dtype=torch.uint8, device="cuda")
    mtp.mtp_attention_tc(args, ws, nbytes, torch.cuda.current_stream())
    torch.cuda.synchronize()
    got = out.view(len(spec), H, HD).double()
    for r, (s, p) in enumerate(spec):
        if s < 0:
            assert (got[r] == -7.0).all()
            continue
        k, v = kv[s].double()
        a = torch.einsum("hd,hkd->hk", q[r].double(), k[:, :p + 1]) / 8.0
        ref = torch.einsum("hk,hkd->hd", torch.softmax(a, -1), v[:, :p + 1])
        # Q and P keep 16 bits: a weight is off by 2^-17 of the score's terms, |q||k| / 8 in all
        bound = 1e-5 + 2 ** -16 * (q[r].double().norm() * k[:, :p + 1].norm(dim=-1).max() / 8.0).item()
        assert (got[r] - ref).abs().max() <= bound * max(1.0, ref.abs().max().item()), f"row {r}"
