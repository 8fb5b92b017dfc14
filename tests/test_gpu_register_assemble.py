"""An assemble right behind the registrations it reads, without anything in between: the composed cache that the gather
copies (values byte for byte, keys re-based) is that of the same assembly made after a synchronisation."""
import pytest
import torch

from paper_2604_13226_b200 import binding as kvp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("materialize", [True, False])
@pytest.mark.parametrize("side_stream", [False, True])
def test_assemble_right_behind_registration(dtype, materialize, side_stream):
    L, hq, hkv, d, n, f = 2, 8, 4, 128, 700, 24
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    flags = kvp.REBASE | (kvp.MATERIALIZE if materialize else 0)
    for trial in range(8):
        ctx = kvp.Context(L, hq, hkv, d, dtype, pool_tokens=4 * (n + 2 * f), max_packets=2, max_adapters=2, max_slots=2,
                          max_prefix_tokens=2 * (n + 2 * f), max_query_tokens=1, max_ws_rows=2 * (n + 2 * f) + 8, max_assemblies=2)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(trial)
        x = [torch.randn(L, m, hkv, d, generator=gen, device="cuda", dtype=dt) for m in (n, n, f, f, f, f)]
        torch.cuda.synchronize()
        with torch.cuda.stream(torch.cuda.Stream() if side_stream else torch.cuda.current_stream()):
            ctx.register_packet(x[0], x[1], n, 0)
            ctx.register_adapter(x[2], x[3], f, 0, x[4], x[5], f, 3)
            first, (prefix,) = ctx.assemble([[(0, 0), (0, -1)]], flags)
            got = [ctx.export_cache(first, l, 0, prefix, 0) for l in range(L)]
            torch.cuda.synchronize()
            again, _ = ctx.assemble([[(0, 0), (0, -1)]], flags)
            want = [ctx.export_cache(again, l, 0, prefix, 0) for l in range(L)]
            torch.cuda.synchronize()
        for l in range(L):
            assert torch.equal(got[l][0], want[l][0]) and torch.equal(got[l][1], want[l][1])
            assert torch.equal(got[l][1], torch.cat([x[3][l], x[1][l], x[5][l], x[1][l]]))
        ctx.close()
