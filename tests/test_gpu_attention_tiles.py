"""GPU parity of verify attention at the edges of the tcgen05 form's tile
layouts: query rows around 64 (8-key groups below, page pieces above), each
page size, contexts around tiles and pages, pages outside the pool."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_20507_gb300 import binding
from paper_2607_20507_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("k,Hq,Hkv", [(10, 9, 3), (15, 4, 1), (8, 14, 2), (12, 5, 1), (12, 20, 4), (15, 32, 4)])
@pytest.mark.parametrize("ps", [16, 32, 64, 128])
def test_rows_and_pages(k, Hq, Hkv, ps):
    # 33, 64, 63, 65, 65 and 128 query rows per KV head; each request its own edge
    lens = [k + 1, 63, 64, 65, 16 * 9, 16 * 9 + 1, 128 + 31, 700]
    w = W.Workload(95, "tiles", batch=len(lens), n_draft=k, vocab=100, logit_dtype="bf16", draft_sigma=1.0,
                   temperatures=(1.0,), n_q_heads=Hq, n_kv_heads=Hkv, head_dim=128, ctx=("const", 700), page_size=ps,
                   cell=k * ps)
    inp = W.attention_inputs(w, DEV, ctx_lens=torch.tensor(lens, dtype=torch.int32))
    # pages outside the pool read as zeros, whatever their id
    bad = inp["page_table"].clone()
    bad[7, 0], bad[6, 0] = 2 ** 31 - 1, -7
    bad[5, 0] = inp["k_pages"].shape[0]
    for table in (inp["page_table"], bad):
        got = binding.cs_verify_attention(inp["q"], inp["k_pages"], inp["v_pages"], table, inp["ctx_lens"], k)
        exp = oracle.verify_attention(W.host_bits(inp["q"]), W.host_bits(inp["k_pages"]), W.host_bits(inp["v_pages"]),
                                      table.cpu().numpy(), np.asarray(lens, dtype=np.int32), k)
        got = got.float().cpu().numpy()
        assert (np.abs(got - exp) <= 2e-3 + 1e-2 * np.abs(exp)).all()


@pytest.mark.parametrize("k", [2, 9])           # the mma.sync and the tcgen05 form
@pytest.mark.parametrize("B", [1, 31, 32, 33, 64, 1025])
def test_schedule_over_batches(k, B):
    """Batches around a warp of requests and past one launch's, contexts of one
    tile to many side by side (a context may be shorter than the verify rows)."""
    Hq, Hkv, ps = 8, 2, 16
    rng = np.random.default_rng(B)
    lens = rng.choice([0, 1, k + 1, 63, 64, 65, 300, 1000 if B < 100 else 90], B).astype(np.int32)
    w = W.Workload(96, "schedule", batch=B, n_draft=k, vocab=100, logit_dtype="bf16", draft_sigma=1.0,
                   temperatures=(1.0,), n_q_heads=Hq, n_kv_heads=Hkv, head_dim=128,
                   ctx=("const", int(max(lens.max(), k + 1))), page_size=ps, cell=k * B)
    inp = W.attention_inputs(w, DEV, ctx_lens=torch.from_numpy(lens))
    got = binding.cs_verify_attention(inp["q"], inp["k_pages"], inp["v_pages"], inp["page_table"], inp["ctx_lens"], k)
    exp = oracle.verify_attention(W.host_bits(inp["q"]), W.host_bits(inp["k_pages"]), W.host_bits(inp["v_pages"]),
                                  inp["page_table"].cpu().numpy(), lens, k)
    got = got.float().cpu().numpy()
    assert (np.abs(got - exp) <= 2e-3 + 1e-2 * np.abs(exp)).all()
