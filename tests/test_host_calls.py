"""The native host side of the short calls: what it does not handle it leaves to the general path, what it handles gives the same."""
import pytest
import torch


def _host():
    from paper_2512_21450_b200 import binding
    binding.load_library()
    return binding._host


def test_library_is_published_with_its_host_half(monkeypatch):
    from paper_2512_21450_b200 import binding

    def fails(lib):
        raise RuntimeError("no host half")
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_load_host_calls", fails)
    for _ in range(2):   # the second call must not return a library whose short calls have no host half
        with pytest.raises(RuntimeError, match="no host half"):
            binding.load_library()


@pytest.mark.parametrize("content", [None, b"", b"\x7fELF of another Python"])
def test_calls_are_general_without_a_loadable_host_half(monkeypatch, tmp_path, content):
    from paper_2512_21450_b200 import binding
    path = tmp_path / "_host_calls.so"
    if content is not None:
        path.write_bytes(content)
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_host", None)
    monkeypatch.setattr(binding, "HOST_PATH", str(path))
    with pytest.warns(RuntimeWarning, match="marshalled in Python"):
        lib = binding.load_library()
    assert binding.load_library() is lib and binding.debug_workspace(256, 256, 4096)[0] > 0
    assert not binding._handled(binding._host.token_loss(0, None), "rl_token_loss")


def test_host_half_is_named_after_what_it_was_built_for():
    import sys
    from paper_2512_21450_b200 import binding, build
    assert build.HOST_OUT == binding.HOST_PATH
    assert sys.implementation.cache_tag in build.HOST_OUT and torch.__version__ in build.HOST_OUT


def test_unusual_arguments_are_left_to_the_general_path():
    import numpy as np
    h, x, i32 = _host(), torch.zeros(8), torch.zeros(3, dtype=torch.int32)

    class Sub(torch.Tensor):
        pass
    for out in (h.token_loss(), h.token_loss(0, x),                                          # too few arguments
                h.token_loss(0, x, x, x, x, x, None, 0.2, 0.2, 0.0, 0.0, None, None),        # memory of the host
                h.token_loss(0, "x", x, x, x, x, None, 0.2, 0.2, 0.0, 0.0, None, None),
                h.token_loss(2 ** 70, x, x, x, x, x, None, 0.2, 0.2, 0.0, 0.0, None, None),
                h.token_loss(0, x.as_subclass(Sub), x, x, x, x, None, 0.2, 0.2, 0.0, 0.0, None, None),
                h.grpo_advantages(0, x, np.int64(4), 1, 1e-6, i32, 8), h.grpo_advantages(0, x, 4, 1, 1e-6, i32, None),
                h.kl_shaped_returns(0, x, x, x, None, i32, 8, 0.1, 1.0, 1, None),
                h.token_logprobs(0, None, x, x, i32, None), h.policy_loss(*range(23))):
        assert out is NotImplemented


def test_arrays_that_do_not_fit_their_call_are_refused(monkeypatch):
    """Arrays are read and written by address: a short one, one of another type or with gaps would be read or written past."""
    from paper_2512_21450_b200 import Context, binding

    class Library:
        def __getattr__(self, name):
            return lambda *args: 0
    monkeypatch.setattr(binding, "_host", _General())
    c = Context.__new__(Context)
    c.lib, c.handle, c._address, c._ws = Library(), None, 0, None
    c._bind_stream, c.ensure_workspace = lambda: None, lambda *args, **kw: None
    T, d, V = 12, 64, 300
    H, W = torch.zeros(T, d, dtype=torch.bfloat16), torch.zeros(V, d, dtype=torch.bfloat16)
    tok, x, mask, off = torch.zeros(T, dtype=torch.int32), torch.zeros(T), torch.ones(T, dtype=torch.uint8), torch.tensor([0, 5, T]).int()
    gaps = torch.zeros(T, 2)[:, 0]
    good = dict(tokens=tok, old_logp=x, ref_logp=x, adv=x, mask=mask, token_weight=x, loss=torch.zeros(1), dW=torch.zeros(V, d),
                dH=torch.zeros(T, d, dtype=torch.bfloat16))

    def loss(**kw):
        a = dict(good, **kw)
        fixed = [a.pop(k) for k in ("tokens", "old_logp", "ref_logp", "adv", "mask")]
        return c.rl_policy_loss_fwd_bwd(H, W, *fixed, 0.2, 0.2, 0.04, **a)
    # what was taken is taken: more than is needed, other shapes of as many entries, masks of any one-byte type, nothing at all
    for kw in (dict(), dict(mask=mask.bool()), dict(mask=None, token_weight=None), dict(adv=torch.zeros(T + 3)), dict(old_logp=x.view(3, 4)),
               dict(dW=torch.zeros(V * d), dH=torch.zeros(T + 4, d, dtype=torch.bfloat16)), dict(loss=None, dW=None, dH=None),
               dict(dH=torch.zeros(T, d), dH_fp32=True)):
        loss(**kw)
    for kw in (dict(dH=torch.zeros(T, d, dtype=torch.bfloat16), dH_fp32=True), dict(dH=torch.zeros(T, d)), dict(dH=torch.zeros(T - 1, d).bfloat16()),
               dict(dH=torch.zeros(d, T).bfloat16().t()), dict(dW=torch.zeros(V, d).bfloat16()), dict(dW=torch.zeros(V - 1, d)),
               dict(dW=torch.zeros(d, V).t()), dict(loss=torch.zeros(1).double()), dict(adv=x.double()), dict(adv=x[:-1]), dict(adv=gaps),
               dict(old_logp=gaps), dict(ref_logp=x[:-1]), dict(token_weight=x.double()), dict(token_weight=x[:1].expand(T)),
               dict(mask=mask.int()), dict(mask=mask[:-1]), dict(tokens=tok[:-1]), dict(tokens=tok.long())):
        with pytest.raises(AssertionError):
            loss(**kw)
    c.rl_token_logprobs(H, W, tok, mask.bool())
    c.rl_kl_shaped_returns(x[:2], x, x, mask.bool(), off, T, 0.1)
    for bad in (mask.float(), mask[:-1], torch.ones(T, 2, dtype=torch.uint8)[:, 0]):
        with pytest.raises(AssertionError):
            c.rl_token_logprobs(H, W, tok, bad)
        with pytest.raises(AssertionError):
            c.rl_kl_shaped_returns(x[:2], x, x, bad, off, T, 0.1)
    with pytest.raises(AssertionError):
        c.rl_kl_shaped_returns(x[:1], x, x, mask, off, T, 0.1)


_CALLS = ("grpo_advantages", "kl_shaped_returns", "token_loss", "token_logprobs", "policy_loss")


class _General:
    """Leaves every call to the general path."""

    def __getattr__(self, name):
        return lambda *args: NotImplemented


class _Recorder:
    """Passes calls on and notes which of them were handled."""

    def __init__(self, host):
        self.host, self.seen = host, []

    def __getattr__(self, name):
        def call(*args):
            out = getattr(self.host, name)(*args)
            self.seen.append((name, out is not NotImplemented))
            return out
        return call


@pytest.mark.gpu
@pytest.mark.parametrize("opt", [{}, dict(ent_coef=1e-2, agg_mode=1), dict(sequence_level=True), dict(accumulate_dW=True, agg_mode=2),
                                 dict(weight=True), dict(count=True, dH_fp32=True), dict(beta=0.0), dict(strided=True)])
def test_native_and_general_paths_agree(monkeypatch, opt):
    from paper_2512_21450_b200 import Context, binding
    g = torch.Generator(device="cuda").manual_seed(5)
    n_seq, L, d, V = 6, 20, 192, 900
    T = n_seq * L
    wide = torch.randn(T, d + 64, generator=g, device="cuda", dtype=torch.bfloat16)
    H = wide[:, :d] if opt.get("strided") else wide[:, :d].contiguous()
    W = torch.randn(V, d, generator=g, device="cuda", dtype=torch.bfloat16)
    tok = torch.randint(0, V, (T,), generator=g, device="cuda", dtype=torch.int32)
    mask = (torch.rand(T, generator=g, device="cuda") < 0.8).to(torch.uint8)
    logp = -torch.rand(T, generator=g, device="cuda") * 9
    old, ref, ent = logp + 0.05, logp - 0.1, -logp
    rewards = torch.rand(n_seq, generator=g, device="cuda")
    off = torch.arange(0, T + 1, L, dtype=torch.int32, device="cuda")
    weight = torch.rand(T, generator=g, device="cuda") if opt.get("weight") else None
    count = torch.tensor([100], device="cuda") if opt.get("count") else None
    beta = opt.get("beta", 0.04)
    out = []
    for native in (True, False):
        recorder = _Recorder(_host()) if native else _General()
        monkeypatch.setattr(binding, "_host", recorder)
        c = Context(0)
        try:
            got = {}
            for _ in range(2):   # the first call makes the workspace
                got["adv_seq"], adv = c.rl_grpo_advantages(rewards, 3, seq_offsets=off, T=T)
                got["adv"] = adv
                got["shaped"], got["returns"] = c.rl_kl_shaped_returns(got["adv_seq"], logp, ref, mask, off, T, 0.02)
                tl = c.rl_token_loss(logp, ent, old, ref if beta else None, adv, mask, 0.2, 0.3, beta, ent_coef=1e-2,
                                     token_weight=weight, token_count=count)
                got.update({"t_" + k: v for k, v in tl.items()})
                got["score"], got["score_ent"], got["score_lse"] = c.rl_token_logprobs(H, W, tok, mask)
                dH = torch.zeros(T, d, device="cuda", dtype=torch.float32 if opt.get("dH_fp32") else torch.bfloat16)
                dW = torch.ones(V, d, device="cuda")
                kw = {k: v for k, v in opt.items() if k in ("ent_coef", "agg_mode", "sequence_level", "accumulate_dW", "dH_fp32")}
                got.update(c.rl_policy_loss_fwd_bwd(H, W, tok, old, ref if beta else None, adv, mask, 0.2, 0.3, beta, dW=dW, dH=dH,
                                                    loss=torch.zeros(1, device="cuda"), seq_offsets=off, token_weight=weight,
                                                    token_count=count, **kw))
                if native:
                    handled, recorder.seen = recorder.seen, []
            if native:   # each of the five once, and none was left to the general path
                assert sorted(handled) == [(name, True) for name in sorted(_CALLS)]
            # what the library refuses is refused alike
            with pytest.raises(binding.RLHeadError, match="rl_token_loss"):
                c.rl_token_loss(logp, ent, old, None, adv, mask, 0.2, 0.3, 0.04)
            with pytest.raises(binding.RLHeadError, match="rl_grpo_advantages_ex"):
                c.rl_grpo_advantages(rewards, 4, seq_offsets=off, T=T)
            for bad in (2, -1):
                with pytest.raises(binding.RLHeadError, match="rl_policy_loss_fwd_bwd_ex"):
                    c.rl_policy_loss_fwd_bwd(H, W, tok, old, ref, adv, mask, 0.2, 0.3, 0.04, dW=dW, dH=torch.zeros(T, d, device="cuda"),
                                             loss=torch.zeros(1, device="cuda"), dH_fp32=bad)
            with pytest.raises(AssertionError):
                c.rl_token_loss(logp, ent[:-1], old, ref, adv, mask, 0.2, 0.3, 0.04)
            with pytest.raises(AssertionError):
                c.rl_token_logprobs(H, W, tok.long(), mask)
            torch.cuda.synchronize()
            out.append(got)
        finally:
            c.close()
    assert out[0].keys() == out[1].keys()
    for k in out[0]:
        assert out[0][k].dtype == out[1][k].dtype and out[0][k].shape == out[1][k].shape and torch.equal(out[0][k], out[1][k]), k


@pytest.mark.gpu
def test_one_unusual_argument_leaves_the_call_to_the_general_path():
    """Each from a call that is handled, by changing one argument."""
    import numpy as np
    from paper_2512_21450_b200 import Context

    class Sub(torch.Tensor):
        pass
    T, d, V, n = 60, 64, 300, 6
    x = -torch.rand(T, device="cuda") - 1
    gaps = torch.zeros(T, 2, device="cuda")[:, 0]
    H, W = torch.randn(T, d, device="cuda").bfloat16(), torch.randn(V, d, device="cuda").bfloat16()
    tok, mask = torch.zeros(T, dtype=torch.int32, device="cuda"), torch.ones(T, dtype=torch.uint8, device="cuda")
    off, rewards = torch.arange(0, T + 1, 10, dtype=torch.int32, device="cuda"), torch.rand(n, device="cuda")
    count = torch.tensor([T], device="cuda")
    dH, dW, loss = torch.zeros(T, d, device="cuda", dtype=torch.bfloat16), torch.zeros(V, d, device="cuda"), torch.zeros(1, device="cuda")
    c = Context(0)
    try:
        c.ensure_workspace(T, d, V)
        c._bind_stream()
        a, ws = c._address, c._ws
        good = dict(grpo_advantages=[a, rewards, 3, 1, 1e-6, off, T],
                    kl_shaped_returns=[a, rewards, x, x, mask, off, T, 0.1, 1.0, 1, None],
                    token_loss=[a, x, x, x, x, x, mask, 0.2, 0.2, 0.04, 0.01, x, count],
                    token_logprobs=[a, ws, H, W, tok, mask],
                    policy_loss=[a, ws, H, W, tok, x, x, x, mask, 0.2, 0.2, 0.04, 0.01, x, False, dW, dH, loss, 1, False, off, False, count])
        bad = dict(
            grpo_advantages=[(0, 2 ** 70), (1, rewards.double()), (1, rewards.cpu()), (1, rewards[::2]), (1, None), (2, np.int64(3)),
                             (2, 2 ** 40), (3, 1.0), (4, np.float64(1e-6)), (5, off.long()), (6, None), (6, -1)],
            kl_shaped_returns=[(1, rewards.double()), (1, rewards[:5]), (2, x[:-1]), (3, gaps), (4, mask.int()), (4, mask[:-1]), (5, off.long()),
                               (6, None), (6, -1), (7, "0.1"), (9, None), (10, x.double())],
            token_loss=[(1, "x"), (1, x.as_subclass(Sub)), (1, x.double()), (1, gaps), (2, x[:-1]), (3, x.cpu()), (6, mask.bool()),
                        (6, mask[:-1]), (7, np.float32(0.2)), (7, None), (8, 10 ** 400), (11, x.double()), (12, count.int())],
            token_logprobs=[(1, None), (1, ws[:16]), (2, H.float()), (2, H.t().contiguous().t()), (2, H[:0]), (2, H[0]), (3, W.cpu()),
                            (4, tok.long()), (4, tok[:-1]), (5, mask[:-1]), (5, mask.int())],
            policy_loss=[(1, ws[:16]), (2, H[:0]), (4, tok[:-1]), (5, None), (5, x.double()), (6, gaps), (7, x[:-1]), (8, mask[:-1]), (9, "0.2"),
                         (13, x.double()), (14, "no"), (15, dW[:-1]), (15, dW.bfloat16()), (15, None), (16, dH.float()), (16, dH[:-1]),
                         (16, dH.t().contiguous().t()), (17, loss.double()), (18, 1.5), (19, None), (20, off.long()), (21, True),
                         (22, count.int()), (22, count.repeat(2))])
        for name in _CALLS:
            call = getattr(_host(), name)
            assert type(call(*good[name])) is tuple, name
            assert call(*good[name][:-1]) is NotImplemented, name
            for i, value in bad[name]:
                assert call(*[value if k == i else v for k, v in enumerate(good[name])]) is NotImplemented, (name, i, value)
        torch.cuda.synchronize()
        assert c.last_device_status()[0] == 0
    finally:
        c.close()


# A device allocator that counts its calls, and those made by a thread that holds the interpreter's lock
_PROBE = """
#include <Python.h>
#include <cuda_runtime_api.h>
extern "C" {
int calls = 0, held = 0;
void* probe_alloc(ssize_t n, int, cudaStream_t) {
  void* p = nullptr;
  ++calls;
  held += PyGILState_Check();
  cudaMalloc(&p, n);
  return p;
}
void probe_free(void* p, ssize_t, int, cudaStream_t) { cudaFree(p); }
}
"""


@pytest.mark.gpu
def test_other_threads_run_while_outputs_are_allocated(tmp_path):
    """An allocation may wait for the GPU, and the GPU for what another thread is about to launch."""
    import ctypes
    import os
    import subprocess
    import sysconfig
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.build import nvcc_path
    src, so = tmp_path / "probe.cpp", str(tmp_path / "probe.so")
    src.write_text(_PROBE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc_path())), "include")
    subprocess.run(["g++", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-I", cuda, "-o", so, str(src)], check=True)
    T, d, V = 5000, 64, 300
    x = -torch.rand(T, device="cuda") - 1
    H = torch.randn(T, d, device="cuda").bfloat16()
    W = torch.randn(V, d, device="cuda").bfloat16()
    tok, mask = torch.zeros(T, dtype=torch.int32, device="cuda"), torch.ones(T, dtype=torch.uint8, device="cuda")
    off = torch.arange(0, T + 1, 1000, dtype=torch.int32, device="cuda")
    rewards = torch.rand(5, device="cuda")
    dH, dW, loss = torch.zeros(T, d, device="cuda", dtype=torch.bfloat16), torch.zeros(V, d, device="cuda"), torch.zeros(1, device="cuda")
    c = Context(0)
    try:
        c.ensure_workspace(T, d, V)
        c._bind_stream()
        h, probe = _host(), ctypes.CDLL(so)
        allocator = torch.cuda.memory.CUDAPluggableAllocator(so, "probe_alloc", "probe_free").allocator()
        calls, held = (ctypes.c_int.in_dll(probe, name) for name in ("calls", "held"))
        for call in (lambda: h.grpo_advantages(c._address, rewards, 5, 1, 1e-6, off, T),
                     lambda: h.kl_shaped_returns(c._address, rewards, x, x, mask, off, T, 0.1, 1.0, 1, None),
                     lambda: h.token_loss(c._address, x, x, x, x, x, mask, 0.2, 0.2, 0.04, 0.0, None, None),
                     lambda: h.token_logprobs(c._address, c._ws, H, W, tok, mask),
                     lambda: h.policy_loss(c._address, c._ws, H, W, tok, x, x, x, mask, 0.2, 0.2, 0.04, 0.0, None, False, dW, dH, loss,
                                           0, False, None, False, None)):
            before = calls.value
            pool = torch.cuda.MemPool(allocator)
            with torch.cuda.use_mem_pool(pool):
                out = call()
            assert type(out) is tuple and calls.value > before
            torch.cuda.synchronize()
            del out, pool
            torch.cuda.empty_cache()   # what the pool held goes back while the allocator is there
        assert held.value == 0
    finally:
        c.close()
