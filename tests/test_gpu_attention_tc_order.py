"""mtp_attention_tc takes a tile's rows in any order: rows of one slot that lie in several runs are one
segment, in the result (against a float64 softmax) and in the time."""
import random

import pytest

from gpu_util import lib_module

pytestmark = pytest.mark.gpu

H, HD, P = 2, 64, 64


def _call(torch, mtp, spec, slots, pages):
    gen = torch.Generator(device="cuda").manual_seed(len(spec) + slots)
    kv = torch.randn(slots, 2, H, pages * P, HD, device="cuda", generator=gen).bfloat16()
    # one page per 64 keys, rows swizzled as the cache stores them
    pool = kv.view(slots, 2, H, pages, P, 8, 8).permute(0, 3, 1, 2, 4, 5, 6)
    t, c = torch.arange(P, device="cuda")[:, None], torch.arange(8, device="cuda")[None, :]
    pool = pool[..., t, c ^ (t & 7), :].contiguous()
    q = torch.randn(len(spec), H, HD, device="cuda", generator=gen)
    table = torch.arange(slots * pages, device="cuda", dtype=torch.int32).view(slots, pages)
    seq, pos = (torch.tensor([x[i] for x in spec], dtype=torch.int32, device="cuda") for i in (0, 1))
    out = torch.full((len(spec), H * HD), -7.0, device="cuda")
    args = mtp.attention_args(rows=len(spec), rows_per_group=8, n_heads=H, page_size=P, layers=1, layer=0,
                              bt_stride=pages, max_keys=pages * P, q=q.view(len(spec), H * HD), kv_pool=pool,
                              block_table=table, row_seq=seq, row_pos=pos, out=out)
    nbytes = mtp.mtp_attention_tc_workspace_bytes(args)
    ws = torch.zeros(max(16, nbytes), dtype=torch.uint8, device="cuda")
    keep = (pool, table, seq, pos)
    return lambda: (mtp.mtp_attention_tc(args, ws, nbytes, torch.cuda.current_stream()), keep), q, kv, out


def _spec(kind):
    if kind == "descending":          # each slot one run, the last slot first
        return [(3 - r // 40, 100 + r % 40) for r in range(150)], 4
    if kind == "round robin":         # three slots and rows of none in turn
        return [(-1, 0) if r % 4 == 3 else (r % 4, 5 + r) for r in range(300)], 3
    if kind == "shuffled":            # every slot many short runs
        rows = [(s, p) for s in range(7) for p in range(60 + 40 * s)]
        random.Random(3).shuffle(rows)
        return rows, 7
    if kind == "a slot a row":        # 128 segments, not in order
        return [((37 * r) % 128, 3 * r) for r in range(128)], 128
    return [(r % 64, 300 - r) for r in range(128)], 64   # "twice": every slot twice, half a tile apart


@pytest.mark.parametrize("kind", ["descending", "round robin", "shuffled", "a slot a row", "twice"])
def test_any_order(kind):
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    spec, slots = _spec(kind)
    run, q, kv, out = _call(torch, mtp, spec, slots, 6)
    run()
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


def test_alternating_rows_share_their_keys():
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    took = []
    for spec in ([(s, p) for s in (0, 1) for p in range(300)], [(s, p) for p in range(300) for s in (0, 1)]):
        run = _call(torch, mtp, spec, 2, 5)[0]
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                run()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        took.append(min(times))
    # a tile's rows see both slots' keys up to its last position: up to twice the items of a tile in order.  With a
    # segment for every run, 64 times as many for each slot.
    assert took[1] <= 5 * took[0], f"{took[1] / took[0]:.1f} times as long as in order"
