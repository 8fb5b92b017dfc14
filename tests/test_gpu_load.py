"""Packets from host memory at the edges of the load kernel's 4 KB pieces and 48-packet launches, pinned and not pinned:
the materialised cache holds exactly the bytes that device-registered packets give."""
import pytest
import torch

from paper_2604_13226_b200 import binding as kvp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,n_kv,lens", [
    ("bf16", 128, 8, [1, 15, 16, 17, 33, 512]),          # runs below, at and above one piece and several
    ("bf16", 64, 2, [1, 32, 33, 700]),
    ("f32", 64, 1, [1, 7, 300]),
    ("f32", 128, 2, [9, 8]),
    ("bf16", 128, 1, [3 + i % 40 for i in range(101)]),  # three launches a layer
])
@pytest.mark.parametrize("pinned", [True, False])
def test_host_packets_arrive_whole(dtype, d, n_kv, lens, pinned):
    L, dt = 2, torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator().manual_seed(len(lens))
    caches = []
    host = [tuple(torch.randn((L, n_kv, n, d), generator=g).to(dt) for _ in range(2)) for n in lens]
    if pinned:
        host = [(k.pin_memory(), v.pin_memory()) for k, v in host]
    for from_host in (True, False):
        ctx = kvp.Context(L, 2 * n_kv, n_kv, d, dtype, pool_tokens=sum(lens) + 8, max_packets=len(lens), max_adapters=0,
                          max_slots=len(lens), max_prefix_tokens=sum(lens), max_query_tokens=8, max_ws_rows=sum(lens) + 16)
        for (k, v), n in zip(host, lens):
            if from_host:
                ctx.register_packet_host(k, v, n, 0)
            else:
                ctx.register_packet(k.permute(0, 2, 1, 3).contiguous().cuda(), v.permute(0, 2, 1, 3).contiguous().cuda(), n, 0)
        aid, plen = ctx.assemble([[(i, -1) for i in range(len(lens))]], kvp.MATERIALIZE)
        assert plen == [sum(lens)]
        caches.append([ctx.export_cache(aid, l, 0, plen[0], 0) for l in range(L)])
        assert ctx.status_word() == 0
        ctx.close()
    for a, b in zip(*caches):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
