"""One workspace, zeroed once, serves calls of mtp_attention and mtp_attention_tc of any sizes one
after the other: the partials of a call never lie where another call's merge counters are.
Against a float64 softmax, with the buffer's whole size given or each call's own, and with the
smallest size that a call accepts."""
import pytest

from gpu_util import lib_module

pytestmark = pytest.mark.gpu

H, HD, P = 16, 64, 64


class _Call:
    def __init__(self, torch, mtp, contexts, rows, tc):
        gen = torch.Generator(device="cuda").manual_seed(len(contexts) * 7 + rows)
        self.torch, self.contexts, self.rows, per = torch, contexts, rows, -(-max(contexts) // P)
        self.kv = torch.randn(len(contexts), per, 2, H, P, HD, device="cuda", generator=gen).bfloat16()
        pool = self.kv
        if tc:  # the cache's row layout: chunk c of row t at chunk c ^ (t mod 8)
            t, c = torch.arange(P, device="cuda")[:, None], torch.arange(8, device="cuda")[None, :]
            pool = pool.view(*pool.shape[:-1], 8, 8)[..., t, c ^ (t & 7), :].flatten(-2).contiguous()
        n = len(contexts)
        table = torch.arange(n * per, dtype=torch.int32, device="cuda").view(n, per)
        seq = torch.arange(n, dtype=torch.int32, device="cuda").repeat_interleave(rows)
        pos = torch.tensor([c - rows + j for c in contexts for j in range(rows)], dtype=torch.int32, device="cuda")
        self.q = torch.randn(n * rows, H, HD, device="cuda", generator=gen)
        self.out = torch.empty(n * rows, H * HD, device="cuda")
        self.args = mtp.attention_args(rows=n * rows, rows_per_group=min(rows, 8), n_heads=H, page_size=P, layers=1,
                                       layer=0, bt_stride=per, max_keys=max(contexts), q=self.q.view(n * rows, H * HD),
                                       kv_pool=pool, block_table=table, row_seq=seq, row_pos=pos, out=self.out)
        self.keep = (pool, table, seq, pos)
        self.call = mtp.mtp_attention_tc if tc else mtp.mtp_attention
        self.size = (mtp.mtp_attention_tc_workspace_bytes if tc else mtp.mtp_attention_workspace_bytes)(self.args)

    def run(self, ws, nbytes):
        self.out.fill_(-7.0)
        self.call(self.args, ws, nbytes, self.torch.cuda.current_stream())

    def check(self, what):
        torch = self.torch
        for s, c in enumerate(self.contexts):
            k, v = self.kv[s].double().permute(1, 2, 0, 3, 4).flatten(2, 3)[:, :, :c]
            q = self.q[s * self.rows:(s + 1) * self.rows].double().transpose(0, 1)
            a = q @ k.transpose(1, 2) / 8.0
            pos = torch.arange(c - self.rows, c, device="cuda")[:, None]
            a = a.masked_fill(torch.arange(c, device="cuda")[None, :] > pos, float("-inf"))
            ref = (torch.softmax(a, -1) @ v).transpose(0, 1).flatten(1)
            got = self.out[s * self.rows:(s + 1) * self.rows].double()
            # Q and P keep 16 bits: a weight is off by 2^-17 of the score's terms, |q||k| / 8 in all
            bound = 1e-5 + 2 ** -16 * (q.norm(dim=-1).max() * k.norm(dim=-1).max() / 8.0).item()
            assert (got - ref).abs().max() <= bound * max(1.0, ref.abs().max().item()), f"{what}, slot {s}"


@pytest.mark.parametrize("given", ["whole buffer", "own size"])
def test_one_buffer(given):
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    make = lambda n, lo, step, rows, tc: _Call(  # noqa: E731
        torch, mtp, [lo + (step * i) % 301 for i in range(n)], rows, tc)
    calls = {"32": make(32, 300, 37, 4, False), "96": make(96, 200, 53, 1, False), "8": make(8, 500, 41, 8, False),
             "130": make(130, 140, 29, 1, False), "1": make(1, 1999, 0, 2, False),
             "tc 1": make(1, 2000, 0, 100, True), "tc 3": make(3, 1300, 70, 40, True)}
    assert calls["tc 1"].size > 0
    ws = torch.zeros(max(c.size for c in calls.values()), dtype=torch.uint8, device="cuda")
    order = ["32", "96", "8", "130", "96", "32", "1", "130"] + ["tc 1", "96", "tc 3", "32", "tc 1", "8", "tc 3", "130"]
    for i, name in enumerate(order):
        c = calls[name]
        c.run(ws, ws.numel() if given == "whole buffer" else c.size)
        torch.cuda.synchronize()
        c.check(f"call {i} ({name})")


def test_smallest_accepted_size():
    """Sizes as the operators have always asked for them: partials of their splits, a counter per group and head."""
    torch = pytest.importorskip("torch")
    mtp = lib_module()
    up = lambda x: -(-x // 256) * 256  # noqa: E731
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n, ctx, rows, tc in ((1, 30, 1, False), (3, 1500, 4, False), (40, 400, 2, False), (1, 2000, 100, True),
                             (2, 1100, 20, True)):
        c = _Call(torch, mtp, [ctx] * n, rows, tc)
        if tc:
            tiles = -(-n * rows // 128)
            splits = max(1, min(sms // (tiles * H), -(-ctx // 128) // 4))
            least = up(tiles * H * splits * 128 * 68 * 4) + up(tiles * H * 4)
        else:
            parts = max(1, min(sms // (n * H), -(-ctx // P), 32))
            least = up(n * H * parts * 8 * 66 * 4) + up(n * H * 4)
        ws = torch.zeros(least, dtype=torch.uint8, device="cuda")
        for _ in range(2):
            c.run(ws, least)
            torch.cuda.synchronize()
            c.check(f"{n} slots of {ctx}, tc={tc}")
        with pytest.raises(mtp.MTPError):
            c.run(ws, least - 1)
