"""GPU parity of the acceptance step where its launch plan changes: positions
read in phases, rows off the 16-byte grid, vocabularies of one block and of
more blocks than one CTA holds, streamed trees.  Bit-exact outside the
near-tie bands, like the other acceptance tests."""
import numpy as np
import pytest
import torch

import bench
import oracle
from paper_2607_20507_gb300 import binding
from paper_2607_20507_gb300 import workloads as W
from parity_bands import DRAW_TIE, NEAR_TIE, check_band_mismatches

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def chain(B, k, V, dtype, sigma, T, cell=0):
    w = W.Workload(92, "paths", batch=B, n_draft=k, vocab=V, logit_dtype=dtype, draft_sigma=sigma,
                   temperatures=(T,), n_q_heads=8, n_kv_heads=8, head_dim=128, ctx=("const", 64), page_size=16,
                   cell=cell)
    return W.accept_inputs(w, T, DEV)


def compare(inp, T, what, sample=24):
    """The call at its full batch against the oracle on a seeded sample of requests."""
    B = inp["target"].shape[0]
    tok, n = binding.cs_spec_accept(inp["target"], inp["draft"] if T > 0 else None, inp["draft_tokens"],
                                    inp["uniforms"], T)
    torch.cuda.synchronize()
    idx = sorted(np.random.default_rng(B).choice(B, min(B, sample), replace=False).tolist())
    sub = W.accept_subset(inp, idx)
    eo, en, am, dm = oracle.spec_accept(W.host_bits(sub["target"]), W.host_bits(sub["draft"]) if T > 0 else None,
                                        sub["draft_tokens"].cpu().numpy(), sub["uniforms"].cpu().numpy(), T,
                                        with_draw_margin=True)
    tie = (am < NEAR_TIE) | (dm < DRAW_TIE)
    tok, n = tok.cpu().numpy(), n.cpu().numpy()
    mism = np.any(tok[idx] != eo, axis=1) | (n[idx] != en)
    assert not (mism & ~tie).any(), f"{what}: requests {[idx[i] for i in np.nonzero(mism & ~tie)[0]]} differ"
    check_band_mismatches(int((mism & tie).sum()), len(idx), what)
    k = tok.shape[1] - 1
    assert ((n >= 0) & (n <= k)).all() and (tok[np.arange(B), n] >= 0).all()
    return n


# calls of 60 to 190 us at the copy bandwidth, read in two to four phases
@pytest.mark.parametrize("B,k,V,dtype,sigma,T", [
    (256, 8, 128256, "bf16", 0.7, 0.8),    # [0, 1], [2, 3], [4, 8]
    (400, 1, 128256, "bf16", 0.7, 0.8),    # [0], [1]: a phase of nothing but the position without a draft
    (256, 8, 128256, "bf16", 0.7, 0.0),
    (128, 16, 128256, "bf16", 0.1, 1.0),   # four phases, most requests pass all of them
    (128, 11, 128256, "bf16", 0.5, 1.0),   # two phases
    (160, 12, 128257, "bf16", 0.7, 0.8),   # rows at every alignment
    (96, 12, 128257, "bf16", 0.7, 0.8),    # at once: 98 us
    (96, 16, 128257, "bf16", 0.7, 0.0),
    (97, 9, 100003, "f32", 1.0, 1.0),
    (128, 3, 128256, "f32", 0.7, 0.8),     # from 60 us on: 513 KB of a row pair for a CTA of the walk
    (256, 2, 128256, "bf16", 0.7, 0.8),    # [0, 1], [2]
])
def test_positions_read_in_phases(B, k, V, dtype, sigma, T):
    n = compare(chain(B, k, V, dtype, sigma, T, cell=B + k), T, f"B={B} k={k} V={V} {dtype} T={T}")
    assert n.min() < n.max()


@pytest.mark.parametrize("B,k,kernels", [
    (256, 8, 8),   # three phases of a statistics and a test kernel, the last one's masses, the walk
    (128, 11, 6),  # two phases
    (128, 8, 2),   # at once
    (256, 2, 5),   # a first split may leave the position without a draft alone
    (400, 1, 5),   # the second phase decides no pair: no masses
])
def test_every_launch_of_a_phased_call_has_work(B, k, kernels):
    inp = chain(B, k, 128256, "bf16", 0.7, 0.8)
    call = lambda: binding.cs_spec_accept(inp["target"], inp["draft"], inp["draft_tokens"], inp["uniforms"], 0.8)  # noqa: E731
    call()
    assert bench.kernel_launches(call) == kernels


def test_phases_with_every_first_rejection_and_empty_residuals():
    # p == q: only an out-of-range token is rejected, and its residual is
    # empty, so the draw falls back to p; request b is rejected at position
    # b % 10 (9: not at all)
    B, k, V, T = 100, 9, 128256, 1.0
    inp = chain(B, k, V, "bf16", 0.5, T, cell=3)
    inp["draft"] = inp["target"][:, :k].contiguous()
    for b in range(B):
        if b % 10 < k:
            inp["draft_tokens"][b, b % 10] = V
    n = compare(inp, T, "p == q", sample=40)
    assert (n == np.arange(B) % 10).all()


@pytest.mark.parametrize("V", [1, 2, 8, 9, 511, 513, 1025, 1032, 2040, 2049, 4097, 4104])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_vocabularies_around_a_block(V, dtype):
    for T in (0.0, 0.9):
        compare(chain(33, 5, V, dtype, 0.7, T, cell=V), T, f"V={V} {dtype} T={T}", sample=33)


@pytest.mark.parametrize("dtype,V", [("f32", 1 << 20), ("f32", (1 << 20) + 5), ("bf16", 1_500_001)])
def test_vocabularies_of_many_blocks(dtype, V):
    compare(chain(3, 2, V, dtype, 0.5, 1.0, cell=5), 1.0, f"V={V} {dtype}")
    z = torch.randn(3, V, generator=torch.Generator().manual_seed(V)) * 3.0
    z = z.to(torch.float32 if dtype == "f32" else torch.bfloat16).to(DEV)
    u = torch.rand(3, generator=torch.Generator().manual_seed(V + 1)).to(DEV)
    for T in (0.0, 0.8):
        got = binding.cs_sample(z, u, T).cpu().numpy()
        exp, margin = oracle.sample(W.host_bits(z), u.cpu().numpy(), T, with_margin=True)
        assert ((got == exp) | (margin < DRAW_TIE)).all()


@pytest.mark.parametrize("V", [4194301, 4194302, 4194304])   # the last one is the largest that calls take
@pytest.mark.parametrize("first", [0, 1])
def test_largest_f32_vocabularies_at_any_alignment(V, first):
    g = torch.Generator(device=DEV).manual_seed(V + first)
    flat = torch.randn((first + 4 * V,), generator=g, device=DEV) * 3.0
    z = flat[first:first + 2 * V].view(2, V)
    u = torch.rand((2, 2), generator=g, device=DEV)
    for T in (0.0, 0.8):
        got = binding.cs_sample(z, u[:, 0].contiguous(), T).cpu().numpy()
        exp, margin = oracle.sample(W.host_bits(z), u[:, 0].cpu().numpy(), T, with_margin=True)
        assert ((got == exp) | (margin < DRAW_TIE)).all()
    if V == 4194302:
        z = flat[first:first + 3 * V].view(1, 3, V)
        draft = (z[:, :2] + 0.5 * torch.randn((1, 2, V), generator=g, device=DEV)).contiguous()
        inp = dict(target=z, draft=draft, draft_tokens=draft.argmax(dim=2).int(), uniforms=torch.rand((1, 3), generator=g, device=DEV))
        for T in (0.0, 0.8):
            compare(inp, T, f"V={V}")


@pytest.mark.parametrize("B,branching,V,dtype,T", [
    (40, (3, 2, 2, 1), 32001, "bf16", 0.7),    # streamed, rows at every alignment
    (40, (3, 2, 2, 1), 32001, "bf16", 0.0),
    (160, (2, 2, 1), 128256, "bf16", 1.0),     # streamed by clusters of four
    (3, (6, 4, 1), 32768, "f32", 0.8),         # every row read first
])
def test_streamed_trees(B, branching, V, dtype, T):
    w = W.TreeWorkload(93, "paths", batch=B, branching=branching, vocab=V, logit_dtype=dtype, draft_sigma=0.5,
                       temperatures=(T,), n_q_heads=8, n_kv_heads=8, head_dim=128, ctx=("const", 64), page_size=16)
    inp = W.tree_accept_inputs(w, T, DEV)
    draft = inp["draft"] if T > 0 else None
    tok, path, n = binding.cs_tree_accept(inp["target"], draft, inp["parents"], inp["node_tokens"],
                                          inp["uniforms"], T)
    idx = sorted(np.random.default_rng(B).choice(B, min(B, 12), replace=False).tolist())
    sub = {k: v[torch.as_tensor(idx, device=DEV)].contiguous() for k, v in inp.items()}
    exp = oracle.tree_accept(W.host_bits(sub["target"]), W.host_bits(sub["draft"]) if T > 0 else None,
                             sub["parents"].cpu().numpy(), sub["node_tokens"].cpu().numpy(),
                             sub["uniforms"].cpu().numpy(), T)
    tok, path, n = tok.cpu().numpy()[idx], path.cpu().numpy()[idx], n.cpu().numpy()[idx]
    mism = np.any(tok != exp["tokens"], axis=1) | np.any(path != exp["path"], axis=1) | (n != exp["n_accepted"])
    assert not (mism & ~((exp["margin"] < NEAR_TIE) | (exp["draw_margin"] < DRAW_TIE))).any()
