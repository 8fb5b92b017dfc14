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


@pytest.mark.parametrize("pinned", ["whole", "unpinned later", "ends only", "pinned later"])
def test_buffers_pinned_in_part_or_for_a_time(pinned):
    # what is pinned when a packet is copied in decides who copies it, whatever it was at registration; a buffer that is
    # pinned in part is no kernel's to read, and the driver refuses its copy with an error code
    import mmap
    L, hkv, d, n, page = 2, 2, 128, 3000, mmap.PAGESIZE
    rt = torch.cuda.cudart()
    ctx = kvp.Context(L, 4, hkv, d, "bf16", pool_tokens=n, max_packets=1, max_slots=1, max_prefix_tokens=n, max_query_tokens=1,
                      max_ws_rows=n + 8)
    maps = [mmap.mmap(-1, (L * hkv * n * d * 2 + page - 1) // page * page) for _ in range(2)]
    buf = [torch.frombuffer(m, dtype=torch.bfloat16)[:L * hkv * n * d].view(L, hkv, n, d) for m in maps]
    g = torch.Generator()
    g.manual_seed(5)
    ranges = []
    for b, m in zip(buf, maps):
        b.copy_(torch.randn(b.shape, generator=g))
        at = b.data_ptr()
        ranges += [(at, page), (at + len(m) - page, page)] if pinned == "ends only" else [(at, len(m))]

    def pin():
        for at, size in ranges:
            assert int(rt.cudaHostRegister(at, size, 0)) == 0

    def unpin():
        for at, _ in ranges:
            assert int(rt.cudaHostUnregister(at)) == 0

    def check():
        aid, _ = ctx.assemble([[(0, -1)]], 0)
        for l in range(L):
            k, v = ctx.export_cache(aid, l, 0, n, 0)
            torch.cuda.synchronize()
            assert torch.equal(k.cpu(), buf[0][l].transpose(0, 1)) and torch.equal(v.cpu(), buf[1][l].transpose(0, 1))
        assert ctx.status_word() == 0

    if pinned != "pinned later":
        pin()
    ctx.register_packet_host(buf[0], buf[1], n, 0)
    if pinned == "unpinned later":
        unpin()
    if pinned == "ends only":
        with pytest.raises(kvp.KvpError) as e:
            ctx.assemble([[(0, -1)]], 0)
        assert e.value.code == 6
        unpin()
        ctx.evict_packet(0)
    check()
    for b in buf:
        b.mul_(2)
    if pinned == "pinned later":
        pin()
    ctx.evict_packet(0)
    check()
    if pinned in ("whole", "pinned later"):
        unpin()
    ctx.close()
