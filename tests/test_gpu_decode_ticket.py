"""The split tickets of decode rows in memory nothing of this process wrote:
every word larger than any launch tag (all ones, or the top bit set), random,
or zero.  The output must not depend on it, on the first use of the
workspace and on the next ones, in every form of the decode work: clusters of
4 (one row), plain splits, and the decode CTAs of a mixed launch."""
import pytest
import torch

from _cases import assert_close, device_case, host64, oracle_full
from paper_2608_15171_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q_lens,ctx_lens", [([1], [25000]), ([1] * 8, [9000 + 37 * i for i in range(8)]),
                                             ([1, 1, 40], [20000, 300, 500])], ids=["cluster", "plain", "mixed"])
def test_tickets_in_foreign_memory(q_lens, ctx_lens):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_15171_gb300 import ppas
    geo = wl.QWEN25_3B
    hq, hk, D = geo.n_q_heads, geo.n_kv_heads, geo.head_dim
    c = device_case(geo, wl.StepShape(q_lens, ctx_lens), seed=17)
    n = ppas.ppas_attention_workspace_size(q_lens, ctx_lens, hq, hk)
    want = oracle_full(c)
    first = None
    for fill in (0x00, 0xFF, 0x80, None):
        if fill is None:
            ws = torch.randint(0, 256, (n,), dtype=torch.uint8, device="cuda",
                               generator=torch.Generator("cuda").manual_seed(3))
        else:
            ws = torch.full((n,), fill, dtype=torch.uint8, device="cuda")
        for _ in range(3):
            out = torch.full((sum(q_lens), hq, D), float("nan"), dtype=torch.float32, device="cuda")
            err = torch.zeros(1, dtype=torch.int32, device="cuda")
            ppas.ppas_attention_step(c.q, c.k_cache, c.v_cache, c.num_blocks, c.tables, c.width, q_lens, ctx_lens, hq,
                                     hk, D, geo.scale, out, True, ws, n, err)
            torch.cuda.synchronize()
            assert err.item() == 0
            first = out if first is None else first
            assert torch.equal(out, first)
    assert_close(host64(first), want, "tickets")
