"""The native call module (csrc/pycall.cpp): what it does not take goes to the ctypes path, which
raises the binding's errors; both paths give the same results."""
import weakref

import numpy as np
import pytest
import torch

from paper_2607_10661_gb300 import ptd
from paper_2607_10661_gb300 import synthetic as syn

FUNCTIONS = {"tree_attention": 11, "topk_draft": 6, "verify_greedy": 9, "kv_compact": 6, "verify_sampling": 11,
             "verify_and_compact": 11, "tree_verify_step": 4, "draft_tree_update": 15, "pool_merge": 9,
             "pool_retrieve": 10, "tree_rope_append": 12, "lm_head_topk": 8}


@pytest.fixture(scope="module")
def calls():
    import __graft_entry__

    __graft_entry__.build()
    return ptd._native()


@pytest.mark.parametrize("name", list(FUNCTIONS))
def test_native_calls_leave_other_arguments_alone(calls, name):
    """Host tensors, plain objects and wrong counts are not taken (None: nothing was enqueued)."""
    f = getattr(calls, name)
    host = torch.zeros((2, 4), dtype=torch.int32)
    for filler in (host, None, 3, [1, 2], 0.5):
        assert f(*([filler] * FUNCTIONS[name])) is None
    assert f() is None and f(*([host] * (FUNCTIONS[name] + 1))) is None


def test_native_calls_bind_without_the_private_stream_functions(calls, monkeypatch):
    """A torch without its raw stream and device functions (private names): the public ones are taken."""
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.delattr(torch._C, "_cuda_getDevice", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: type("S", (), {"cuda_stream": 4096 + device})())
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(ptd, "_calls", None)
    try:
        assert ptd._native() is calls
        stream, device = ptd._stream_getters()
        assert stream(device()) == 4099
    finally:
        monkeypatch.undo()
        ptd._calls = None
        ptd._native()


def test_native_call_keeps_its_structures(calls):
    """The ctypes structures of a call live until it returns, also where `c` is made anew at each read
    (the call is refused by the library's checks: no batch)."""
    alive = []

    class Holder:
        def __init__(self, cls):
            self.cls, self.refs = cls, []

        @property
        def c(self):
            s = self.cls()
            self.refs.append(weakref.ref(s))
            return s

    tree, cache = Holder(type("T", (ptd._Tree,), {})), Holder(type("C", (ptd._Cache,), {}))

    class FakeTensor:
        is_cuda, dtype = True, torch.int32

        def is_contiguous(self):
            return True

        def data_ptr(self):
            alive.extend(r() is not None for r in tree.refs + cache.refs)
            return 16

    args = (ptd.LIB_PATH, FakeTensor, torch.int32, torch.float32, torch.bfloat16, lambda d: 0, lambda: 0)
    try:
        calls.load(*args)
        x = FakeTensor()
        assert calls.kv_compact(tree, cache, x, x, x, 0) == -ptd.INVALID_ARG
    finally:
        ptd._calls = None
        ptd._native()
    assert len(alive) == 6 and all(alive)
    assert all(r() is None for r in tree.refs + cache.refs)   # and no longer


@pytest.mark.gpu
def test_native_and_ctypes_paths_agree(calls, monkeypatch):
    class Refuse:
        def __getattr__(self, name):
            return lambda *a: None

    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((5, 777), generator=g, device="cuda").to(torch.bfloat16)
    out = []
    for native in (True, False):
        if not native:
            monkeypatch.setattr(ptd, "_calls", Refuse())
        idx = torch.zeros((5, 3), dtype=torch.int32, device="cuda")
        val = torch.zeros((5, 3), device="cuda")
        assert ptd.topk_draft(x, 3, idx, val) == 1
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        idx2, val2 = torch.zeros_like(idx), torch.zeros_like(val)
        assert ptd.topk_draft(x, 3, idx2, val2, vocab=np.int64(500), stream=side) == 1
        torch.cuda.synchronize()
        out.append((idx, val, idx2, val2))
        with pytest.raises(TypeError):
            ptd.topk_draft(x, 3, idx.float(), val)
        with pytest.raises(ValueError):
            ptd.topk_draft(x.cpu(), 3, idx, val)
        with pytest.raises(ValueError):
            ptd.topk_draft(x[:, ::2], 3, idx, val)
        with pytest.raises(ptd.PtdError) as e:
            ptd.topk_draft(x, 17, idx, val)
        assert e.value.status == ptd.INVALID_ARG
        with torch.cuda.stream(side):   # the current stream is asked for at every call
            ptd.topk_draft(x, 3, idx2, val2)
        side.synchronize()
        assert torch.equal(idx2, idx) and torch.equal(val2, val)
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.gpu
def test_native_step_matches_ctypes_step(calls, monkeypatch):
    from paper_2607_10661_gb300.harness import DeviceWorkload

    class Refuse:
        def __getattr__(self, name):
            return lambda *a: None

    w = syn.Workload(syn.shrink(syn.CONFIGS["llama3-8b-gqa"], layers=2, ctx=(300, 300), vocab=5000), 7)
    a, b = DeviceWorkload(w), DeviceWorkload(w)
    na = a.step()
    monkeypatch.setattr(ptd, "_calls", Refuse())
    nb = b.step()
    torch.cuda.synchronize()
    assert na == nb
    for name in ("attn_out", "topk_idx", "topk_val", "accepted", "accept_len", "bonus", "new_ctx", "k", "v"):
        assert torch.equal(getattr(a, name), getattr(b, name)), name


@pytest.mark.gpu
def test_every_native_call_is_taken_and_matches_ctypes(calls, monkeypatch):
    """Each function of the module takes its plain arguments (kernels launched, not None) and gives what the
    ctypes path gives."""
    from paper_2607_10661_gb300.harness import DeviceWorkload

    taken = {}

    class Record:
        def __getattr__(self, name):
            def call(*a):
                r = getattr(calls, name)(*a)
                taken[name] = r
                return r

            return call

    class Refuse:
        def __getattr__(self, name):
            return lambda *a: None

    cfg = syn.shrink(syn.CONFIGS["llama3-8b-gqa"], layers=2, ctx=(300, 300), vocab=5000)

    def run_all():
        """Every call of the binding once; their launches and outputs."""
        g = torch.Generator(device="cuda").manual_seed(11)
        i32 = dict(dtype=torch.int32, device="cuda")
        zeros = lambda *shape: torch.zeros(shape, **i32)
        dw = DeviceWorkload(syn.Workload(cfg, 7))
        n, B, k = dw.w.n_total, cfg.batch, cfg.k
        kv = [torch.randn((2, n, cfg.hkv, cfg.d), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2)]
        pos = zeros(n)
        launches = [ptd.tree_rope_append(dw.tree, dw.cache, 0, dw.q, cfg.hq, *kv, 1e4, dw.dev_status, positions_out=pos),
                    dw.attention(), dw.topk(), dw.verify(), dw.compact()]
        out = [x.clone() for x in (pos, dw.attn_out, dw.topk_idx, dw.topk_val, dw.accepted, dw.accept_len, dw.bonus,
                                   dw.new_ctx, dw.k, dw.v)]
        launches += [dw.verify_and_compact(), dw.step()]
        out += [x.clone() for x in (dw.accepted, dw.accept_len, dw.bonus, dw.new_ctx, dw.k, dw.v, dw.attn_out)]
        u, ub = (torch.rand(m, generator=g, device="cuda") for m in (n, B))
        sampled = zeros(B, dw.w.max_nodes), zeros(B), zeros(B)
        launches.append(ptd.verify_sampling(dw.tree, dw.tokens, dw.logits, 0.8, u, ub, *sampled, dw.dev_status))
        hidden, weight = (torch.randn((m, 256), generator=g, device="cuda").to(torch.bfloat16) for m in (n, 3000))
        idx, val = zeros(n, k), torch.zeros((n, k), device="cuda")
        ws = torch.empty(ptd.lm_head_workspace_size(n, 3000), dtype=torch.uint8, device="cuda")
        launches.append(ptd.lm_head_topk(hidden, weight, k, idx, val, ws, dw.dev_status))
        forest = zeros(1), zeros(1, 128), zeros(1, 128), zeros(1, 128), zeros(1, n)
        count, parents, tokens = torch.full((1,), n, **i32), dw.parents.view(1, -1), dw.tokens.view(1, -1)
        launches.append(ptd.draft_tree_update(count, parents, tokens, dw.topk_idx, 2, 4, 6, 128, *forest, dw.dev_status))
        pool = ptd.CandidatePool(4096, "cuda")
        launches.append(pool.merge(0, *forest[:3], dw.dev_status))
        got = zeros(1), zeros(64), zeros(64)
        launches.append(pool.retrieve(forest[2][0, :1].clone(), 4, 6, 64, *got))
        torch.cuda.synchronize()
        assert int(dw.dev_status.item()) == 0
        return launches, out + [idx, val, *sampled, *forest, *got]

    monkeypatch.setattr(ptd, "_calls", Record())
    native = run_all()
    assert set(taken) == set(FUNCTIONS) and all(isinstance(r, int) and r > 0 for r in taken.values()), taken
    monkeypatch.setattr(ptd, "_calls", Refuse())
    plain = run_all()
    assert native[0] == plain[0]
    for i, (a, b) in enumerate(zip(native[1], plain[1])):
        assert torch.equal(a, b), i
