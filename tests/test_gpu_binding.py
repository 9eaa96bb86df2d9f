"""The binding's compiled marshalling: given outputs, workspaces and streams
are used, and an argument that a call does not take raises what the Python
checks raise."""
import random
import sys
import threading
import time

import pytest
import torch

import bench
from paper_2607_20507_gb300 import binding
from paper_2607_20507_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def inputs():
    w = W.Workload(94, "binding", batch=3, n_draft=3, vocab=3001, logit_dtype="bf16", draft_sigma=0.7,
                   temperatures=(0.8,), n_q_heads=16, n_kv_heads=4, head_dim=128, ctx=("uniform", 40, 400), page_size=16)
    a, c = W.attention_inputs(w, DEV), W.accept_inputs(w, 0.8, DEV)
    return ([a[k] for k in ("q", "k_pages", "v_pages", "page_table", "ctx_lens")],
            [c[k] for k in ("target", "draft", "draft_tokens", "uniforms")])


def test_given_outputs_workspace_and_stream():
    a, c = inputs()
    expect, (tok, n) = binding.cs_verify_attention(*a, 3), binding.cs_spec_accept(*c, 0.8)
    out = torch.empty_like(a[0])
    ws = torch.zeros(binding.cs_verify_attention_workspace_bytes(a[0], a[1], a[3], 3), dtype=torch.uint8, device=DEV)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    assert binding.cs_verify_attention(*a, 3, out=out, workspace=ws, stream=side.cuda_stream) is out
    t2, n2 = torch.empty_like(tok), torch.empty_like(n)
    r = binding.cs_spec_accept(*c, 0.8, out_tokens=t2, out_n_accepted=n2, stream=side.cuda_stream)
    side.synchronize()
    torch.cuda.synchronize()
    assert r[0].data_ptr() == t2.data_ptr() and r[1].data_ptr() == n2.data_ptr()
    assert torch.equal(out, expect) and torch.equal(t2, tok) and torch.equal(n2, n)
    with torch.cuda.stream(side):   # the current stream
        again = binding.cs_verify_attention(*a, 3, sm_scale=0)
    side.synchronize()
    assert torch.equal(again, expect)


def test_refusals():
    a, c = inputs()
    for i, bad in ((0, a[0].float()), (0, a[0].transpose(1, 2)), (1, a[1].cpu()), (3, a[3].long()), (4, a[4][None])):
        with pytest.raises((TypeError, ValueError)):
            binding.cs_verify_attention(*a[:i], bad, *a[i + 1:], 3)
    with pytest.raises(ValueError, match="n_draft"):
        binding.cs_verify_attention(*a, 2)
    with pytest.raises(ValueError, match="same shape"):
        binding.cs_verify_attention(a[0], a[1], a[2][:-1].contiguous(), *a[3:], 3)
    with pytest.raises(binding.CacheSpecError) as e:
        binding.cs_verify_attention(*a, 3, workspace=torch.zeros(256, dtype=torch.uint8, device=DEV))
    assert e.value.status == binding.CS_ERR_WORKSPACE
    with pytest.raises(binding.CacheSpecError) as e:
        binding.cs_spec_accept(*c, -1)
    assert e.value.status == binding.CS_ERR_INVALID_ARG
    with pytest.raises(ValueError):
        binding.cs_spec_accept(c[0], c[1][:, :2].contiguous(), *c[2:], 0.8)
    with pytest.raises(TypeError):
        binding.cs_sample(c[0][:, 0].contiguous().half(), c[3][:, 0].contiguous(), 1.0)
    with pytest.raises(TypeError):
        binding.cs_kv_commit(a[4].long(), a[4], 3)


def test_stream_of_more_than_a_handle():
    """Its low 64 bits count, as in every ctypes call (here 0: the default stream)."""
    lens, n = torch.tensor([9, 5], dtype=torch.int32, device=DEV), torch.tensor([1, 0], dtype=torch.int32, device=DEV)
    binding.cs_kv_commit(lens, n, 3, stream=1 << 70)
    assert lens.tolist() == [7, 2]
    z, u = torch.randn((2, 1000), device=DEV), torch.zeros((2,), device=DEV)
    t = binding.cs_sample(z, u, 0.0, stream=1 << 70)
    assert torch.equal(t, z.argmax(dim=1).int())


def run_threads(works):
    """Each callable in a thread of its own; the first exception is raised here."""
    errors = []

    def guarded(f):
        try:
            f()
        except BaseException as e:   # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=guarded, args=(f,)) for f in works]
    before = sys.getswitchinterval()
    sys.setswitchinterval(1e-6)
    try:
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        sys.setswitchinterval(before)
    if errors:
        raise errors[0]


def test_more_workspaces_than_one_thread_can_keep():
    """Over a hundred default workspaces of different sizes, taken by three threads at a time."""
    z = torch.randn((120, 128256), device=DEV).to(torch.bfloat16)
    u = torch.zeros((120,), device=DEV)
    top = (z == z.max(dim=1, keepdim=True).values).int().argmax(dim=1).int()   # the lowest of equal ids
    torch.cuda.synchronize()

    def work(seed):
        sizes = list(range(1, 121))
        random.Random(seed).shuffle(sizes)
        got = [(b, binding.cs_sample(z[:b], u[:b], 0.0)) for b in sizes]
        for b, t in got:
            assert torch.equal(t, top[:b]), b

    run_threads([lambda s=s: work(s) for s in range(3)])


def test_default_workspace_by_any_name_of_its_device():
    """A caller reads the status of its default calls from the workspace that they use."""
    a, c = inputs()
    d = binding.attn_dims(a[0], a[1], a[3])
    binding.cs_verify_attention(*a, 3)
    ws = [binding.verify_attention_workspace(d, 3, dev) for dev in (DEV, "cuda", torch.device(DEV), a[0].device)]
    assert len({w.data_ptr() for w in ws}) == 1
    assert torch.count_nonzero(ws[0]).item() > 0 and binding.cs_read_device_status(ws[0]) == 0


def test_two_streams_share_nothing():
    """The same calls on two streams, with nothing between them, on different inputs: as one after the other.
    The acceptance is long enough to be read in phases, whose decisions are in the workspace."""
    def case(seed):
        kw = dict(vocab=128256, logit_dtype="bf16", draft_sigma=0.7, temperatures=(0.8,), n_q_heads=16, n_kv_heads=4,
                  head_dim=128, page_size=16)
        wa = W.Workload(95, "streams", batch=40, n_draft=8, ctx=("uniform", 100, 3000), cell=seed, **kw)
        wc = W.Workload(95, "streams", batch=160, n_draft=8, ctx=("const", 64), cell=seed, **kw)
        a, c = W.attention_inputs(wa, DEV), W.accept_inputs(wc, 0.8, DEV)
        r = W.route_inputs(W.RouteWorkload(30, "streams", 300, 2000, 384), DEV, seed=seed)
        return ([a[k] for k in ("q", "k_pages", "v_pages", "page_table", "ctx_lens")],
                [c[k] for k in ("target", "draft", "draft_tokens", "uniforms")],
                (r["emb"], r["centroids"], binding.cs_route_norms(r["centroids"])))

    def calls(x):
        a, c, r = x
        return (binding.cs_verify_attention(*a, 8), *binding.cs_spec_accept(*c, 0.8),
                binding.cs_sample(c[0][:, 0].contiguous(), c[3][:, 0].contiguous(), 0.8),
                *binding.cs_route(*r, W.ROUTE_TAU))

    x = [case(s) for s in (1, 2)]
    expect = [calls(v) for v in x]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in x]
    got = [[], []]
    for _ in range(12):
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                got[i].append(calls(x[i]))
    torch.cuda.synchronize()
    for i in range(2):
        for g in got[i]:
            for u, v in zip(g, expect[i]):
                assert torch.equal(u, v)


def test_capture_adds_no_fill():
    """Captured after the same calls, with default workspaces: the calls' own kernels and nothing else."""
    a, c = inputs()
    r = W.route_inputs(W.RouteWorkload(30, "capture", 70, 300, 128), DEV, seed=2)
    route = (r["emb"], r["centroids"], binding.cs_route_norms(r["centroids"]))
    z, u = c[0][:, 0].contiguous(), c[3][:, 0].contiguous()

    def step():
        return (binding.cs_verify_attention(*a, 3), *binding.cs_spec_accept(*c, 0.8), binding.cs_sample(z, u, 0.8),
                *binding.cs_route(*route, W.ROUTE_TAU))

    expect = step()
    assert bench.kernel_launches(step) == 8   # two each
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = step()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    for x, y in zip(got, expect):
        assert torch.equal(x, y)


def test_new_workspace_is_filled_on_its_stream():
    """With the current stream busy, the zero fill of a new workspace does not come after the call that uses it."""
    a, c = inputs()
    a = [a[0][:2].contiguous(), *a[1:3], a[3][:2].contiguous(), a[4][:2].contiguous()]
    expect = binding.cs_verify_attention(*a, 3)
    d = binding.attn_dims(a[0], a[1], a[3])
    out, side = torch.empty_like(expect), torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)   # about 50 ms
    binding.cs_verify_attention(*a, 3, out=out, stream=side.cuda_stream)
    with torch.cuda.stream(side):
        ws = binding.verify_attention_workspace(d, 3, DEV)
        early = ws.clone()
        assert torch.equal(out, expect)
    torch.cuda.synchronize()
    assert torch.count_nonzero(early).item() > 0 and torch.equal(ws, early)
    assert ws.data_ptr() != binding.verify_attention_workspace(d, 3, DEV).data_ptr()


def test_other_threads_run_while_a_launch_waits():
    """The stream is busy for about a second and its queue fills up: the launching thread waits, the others do not."""
    lens, n = torch.zeros((4,), dtype=torch.int32, device=DEV), torch.zeros((4,), dtype=torch.int32, device=DEV)
    binding.cs_kv_commit(lens, n, 3)
    torch.cuda.synchronize()
    gaps, stop = [], threading.Event()

    def tick():
        t = time.perf_counter()
        while not stop.is_set():
            time.sleep(0.002)
            now = time.perf_counter()
            gaps.append(now - t)
            t = now

    ticker = threading.Thread(target=tick)
    ticker.start()
    try:
        torch.cuda._sleep(2_000_000_000)
        t0 = time.perf_counter()
        for _ in range(8192):
            binding.cs_kv_commit(lens, n, 3)
        waited = time.perf_counter() - t0
    finally:
        stop.set()
        ticker.join()
    torch.cuda.synchronize()
    assert waited > 0.3, "the queue did not fill up"
    assert max(gaps) < 0.5 * waited


def test_threads_on_one_stream_share_its_workspace():
    """Calls of one shape from four threads on the same stream, each of several kernels: as one after the other."""
    w = W.Workload(96, "threads", batch=96, n_draft=8, vocab=128256, logit_dtype="bf16", draft_sigma=0.7,
                   temperatures=(0.8,), n_q_heads=16, n_kv_heads=4, head_dim=128, ctx=("const", 64), page_size=16)
    x = []
    for seed in range(4):
        c = W.accept_inputs(w.with_(cell=seed), 0.8, DEV)
        x.append([c[k] for k in ("target", "draft", "draft_tokens", "uniforms")])
    expect = [binding.cs_spec_accept(*c, 0.8) for c in x]
    torch.cuda.synchronize()

    def work(i):
        got = [binding.cs_spec_accept(*x[i], 0.8) for _ in range(40)]
        torch.cuda.synchronize()
        for tok, n in got:
            assert torch.equal(tok, expect[i][0]) and torch.equal(n, expect[i][1])

    run_threads([lambda i=i: work(i) for i in range(4)])


class Interpreted:
    """In the marshalling module's place: takes nothing, so that binding.py's own checks run."""

    def __getattr__(self, name):
        return lambda *args: None


def both_ways(monkeypatch, call):
    """A call's result, or its exception's type, through the compiled marshalling and without it."""
    got = []
    for fast in (binding._load_fast(), Interpreted()):
        with monkeypatch.context() as m:
            m.setattr(binding, "_fast", fast)
            try:
                r = call()
                got.append([t.clone() for t in (r if isinstance(r, tuple) else (r,)) if t is not None])
            except Exception as e:   # noqa: BLE001
                got.append((type(e), getattr(e, "status", None)))
    return got


def test_marshalling_does_what_the_checks_do(monkeypatch):
    a, c = inputs()
    tw = W.TreeWorkload(97, "ways", batch=3, branching=(2, 1), vocab=3001, logit_dtype="f32", draft_sigma=0.7,
                        temperatures=(0.8,), n_q_heads=16, n_kv_heads=4, head_dim=128, ctx=("uniform", 40, 400),
                        page_size=16)
    ta, tc = W.tree_attention_inputs(tw, DEV), W.tree_accept_inputs(tw, 0.8, DEV)
    tree = [tc[k] for k in ("target", "draft", "parents", "node_tokens", "uniforms")]
    path, n = binding.cs_tree_accept(*tree, 0.8)[1:]
    r = W.route_inputs(W.RouteWorkload(30, "ways", 5, 300, 128), DEV, seed=1)
    route = (r["emb"], r["centroids"], binding.cs_route_norms(r["centroids"]))
    rows = [torch.randn((3, 4, 4, 128), device=DEV).to(torch.bfloat16) for _ in range(2)]

    def in_place(call, *written):
        """Clones of what a call writes into copies of its arguments."""
        def run():
            x = [t.clone() for t in written]
            call(*x)
            return tuple(x)
        return run

    b = binding
    good = [lambda: b.cs_verify_attention(*a, 3), lambda: b.cs_spec_accept(*c, 0.8),
            lambda: b.cs_spec_accept(c[0], None, *c[2:], 0), lambda: b.cs_tree_accept(*tree, 0.8),
            lambda: b.cs_tree_verify_attention(*[ta[k] for k in ("q", "k_pages", "v_pages", "page_table", "ctx_lens",
                                                                 "parents")]),
            lambda: b.cs_sample(c[0][:, 0].contiguous(), c[3][:, 0].contiguous(), 0.8),
            lambda: b.cs_route(*route, W.ROUTE_TAU),
            in_place(lambda k, v: b.cs_kv_append(*rows, k, v, a[3], a[4]), a[1], a[2]),
            in_place(lambda x: b.cs_kv_commit(x, n, 3), a[4]),
            in_place(lambda k, v, x: b.cs_kv_commit_tree(k, v, ta["page_table"], x, path, n), ta["k_pages"],
                     ta["v_pages"], ta["ctx_lens"])]
    for i, call in enumerate(good):
        fast, slow = both_ways(monkeypatch, call)
        assert len(fast) > 0 and len(fast) == len(slow), i
        for x, y in zip(fast, slow):
            assert isinstance(x, torch.Tensor) and x.dtype == y.dtype and torch.equal(x, y), i
    bad = [lambda: b.cs_verify_attention(a[0].float(), *a[1:], 3), lambda: b.cs_verify_attention(*a, 2),
           lambda: b.cs_verify_attention(*a, 3, sm_scale=float("nan")), lambda: b.cs_verify_attention(*a, "3"),
           lambda: b.cs_verify_attention(*a, 3, out=torch.empty(1, device=DEV)),
           lambda: b.cs_spec_accept(c[0], None, *c[2:], 0.8), lambda: b.cs_spec_accept(*c, float("inf")),
           lambda: b.cs_spec_accept(*c, 0.8, out_tokens=c[3]),
           lambda: b.cs_spec_accept(c[0], c[1].float(), *c[2:], 0.8), lambda: b.cs_spec_accept(*c, None),
           lambda: b.cs_spec_accept(*c, 0.8, workspace=torch.zeros(256, dtype=torch.uint8, device=DEV)),
           lambda: b.cs_tree_accept(*tree[:2], tree[2][:, 1:].contiguous(), *tree[3:], 0.8),
           lambda: b.cs_sample(c[0], c[3], 0.8), lambda: b.cs_sample(c[0][:, 0], c[3][:, 0], 0.8),
           lambda: b.cs_route(route[0], route[1][:, :64].contiguous(), route[2], 0.5),
           lambda: b.cs_route(*route, float("nan")),
           lambda: b.cs_kv_append(rows[0], rows[1][:2].contiguous(), a[1], a[2], a[3], a[4]),
           lambda: b.cs_kv_commit(a[4], n, 17), lambda: b.cs_kv_commit(a[4].cpu(), n, 3),
           lambda: b.cs_kv_commit_tree(ta["k_pages"], ta["v_pages"].float(), ta["page_table"], ta["ctx_lens"], path, n)]
    for i, call in enumerate(bad):
        fast, slow = both_ways(monkeypatch, call)
        assert isinstance(fast, tuple) and fast == slow, (i, fast, slow)
