"""The native marshalling of the frequent calls (host_calls.cpp): what it takes it does as the general Python way does, and what is
not plain it leaves to that way, which has the checks and the errors."""
import os
import subprocess
import types

import pytest
import torch
from torch.overrides import TorchFunctionMode

from paper_2604_16498_b200 import binding, build

NOT_PLAIN = -1


def _calls():
    binding.load()
    assert binding._host_calls is not None
    return binding._host_calls


class _Sub(torch.Tensor):
    pass


class _Mode(TorchFunctionMode):
    def __torch_function__(self, func, types, args=(), kwargs=None):
        return func(*args, **(kwargs or {}))


def test_tensors_in_host_memory_go_the_general_way_and_are_refused_there():
    c = _calls()
    q, x = torch.zeros(1, 2, 8, 64, dtype=torch.bfloat16), torch.zeros(8, 8, dtype=torch.bfloat16)
    assert c.attn(0, q, q, q, 0, None, None, q) == NOT_PLAIN
    assert c.linear(0, x, x, None, None, 0, 0, x) == NOT_PLAIN
    assert c.swiglu(x, x, x, 0, x) == NOT_PLAIN
    for bad in ((), (0, q), (0, q, q, q, 0, None, None, None), (0, None, 1, "", 0, None, None, q), (7, q, q, q, 0, None, None, q)):
        assert c.attn(*bad) == NOT_PLAIN
    with pytest.raises(ValueError):
        binding.attn_fused(q, q, q, out=q)
    with pytest.raises(ValueError):
        binding.linear_act(x, x, out=x)


def test_bind_wants_nine_addresses():
    c = _calls()
    for bad in ((), (1,) * 8, (0,) * 9, ("x",) * 9):
        with pytest.raises((TypeError, ValueError)):
            c.bind(*bad)


@pytest.mark.parametrize("built_for", [None, "torch 2.10.0 abc python .cpython-312-x86_64-linux-gnu.so"])
def test_a_module_built_for_another_torch_is_not_used(monkeypatch, built_for):
    lib = binding.load()
    fake = types.SimpleNamespace(bind=lambda *a: pytest.fail("bound"), **({} if built_for is None else {"built_for": built_for}))
    monkeypatch.setattr("paper_2604_16498_b200.host_calls", fake, raising=False)
    monkeypatch.setattr(binding, "_host_calls", None)
    binding._bind_host_calls(lib)
    assert binding._host_calls is None


def _fake_tree(monkeypatch, tmp_path):
    for name, path in (("HERE", ""), ("CSRC", "csrc"), ("INCLUDE", "include"), ("LIB", "libforge.so"), ("HOST_CALLS", "host_calls.x.so"), ("OBJ_DIR", "obj")):
        monkeypatch.setattr(build, name, str(tmp_path / path))
    for name in ("csrc/a.cu", "csrc/host_calls.cpp", "include/forge.h"):
        (tmp_path / name).parent.mkdir(exist_ok=True)
        (tmp_path / name).write_text("")
        os.utime(tmp_path / name, (1e9, 1e9))
    ran = []

    def run(cmd, **kw):
        ran.append(os.path.basename(cmd[0]))
        if "-o" in cmd and not (ran[-1] == "g++" and run.gxx_fails):
            with open(cmd[cmd.index("-o") + 1], "w") as f:
                f.write(" ".join(cmd))
        return subprocess.CompletedProcess(cmd, int(ran[-1] == "g++" and run.gxx_fails), "", "no headers")
    run.gxx_fails = False
    monkeypatch.setattr(build.subprocess, "run", run)
    return ran, run


def test_the_library_is_built_where_the_module_cannot_be(monkeypatch, tmp_path, capsys):
    ran, run = _fake_tree(monkeypatch, tmp_path)
    run.gxx_fails = True
    (tmp_path / "host_calls.x.so").write_text("of another torch")
    os.utime(tmp_path / "host_calls.x.so", (2e9, 2e9))
    assert build.build() == str(tmp_path / "libforge.so") and (tmp_path / "libforge.so").exists()
    assert not (tmp_path / "host_calls.x.so").exists() and "no headers" in capsys.readouterr().err


def test_each_part_is_rebuilt_for_its_own_reasons(monkeypatch, tmp_path):
    ran, run = _fake_tree(monkeypatch, tmp_path)
    build.build()
    assert sorted(ran) == ["g++", "nvcc", "nvcc"]  # one source, the link
    ran.clear()
    build.build()
    assert ran == []
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    build.build()
    assert ran == ["g++"]
    ran.clear()
    os.utime(tmp_path / "csrc/host_calls.cpp", (3e9, 3e9))
    build.build()
    assert ran == ["g++"]
    ran.clear()
    os.utime(tmp_path / "csrc/a.cu", (3e9, 3e9))
    os.utime(tmp_path / "host_calls.x.so", (4e9, 4e9))
    build.build()
    assert ran == ["nvcc", "nvcc"]


def _attn_args(D=64, dtype=torch.bfloat16):
    g = torch.Generator(device="cuda").manual_seed(5)
    mk = lambda h, s: torch.randn((2, h, s, D), generator=g, device="cuda").to(dtype)
    q, k, v = mk(4, 40), mk(2, 70), mk(2, 70)
    return q, k, v, torch.full_like(q, float("nan"))


def _general(monkeypatch, fn, *a, **kw):
    with monkeypatch.context() as m:
        m.setattr(binding, "_host_calls", None)
        return fn(*a, **kw)


@pytest.mark.gpu
@pytest.mark.parametrize("fn,dtype", [("attn_fused", torch.bfloat16), ("attn_fused_f16", torch.float16), ("attn_fused_f32", torch.float32)])
def test_attention_equals_the_general_way(monkeypatch, fn, dtype):
    q, k, v, out = _attn_args(dtype=dtype)
    lens = torch.tensor([70, 33], dtype=torch.int32, device="cuda")
    for mask, ln, scale in ((0, None, None), (1, None, 0.3), (3, lens, None)):
        ty = ("attn_fused", "attn_fused_f16", "attn_fused_f32").index(fn)
        assert _calls().attn(ty, q, k, v, mask, ln, scale, out) == binding.OK
        want = _general(monkeypatch, getattr(binding, fn), q, k, v, mask, ln, scale)
        assert torch.equal(out, want)
        out.fill_(float("nan"))
        assert getattr(binding, fn)(q, k, v, mask, ln, scale, out=out) is out and torch.equal(out, want)
    binding.check_status()


@pytest.mark.gpu
def test_decode_and_linears_equal_the_general_way(monkeypatch):
    _calls()
    g = torch.Generator(device="cuda").manual_seed(6)
    for dt in (torch.bfloat16, torch.float16):
        r = lambda *s: torch.randn(s, generator=g, device="cuda").to(dt)
        q, k, v, lens = r(3, 8, 64), r(3, 2, 100, 64), r(3, 2, 100, 64), torch.tensor([100, 1, 50], dtype=torch.int32, device="cuda")
        ws = torch.empty(binding.attn_decode_workspace_bytes(3, 8, 64, 4), dtype=torch.uint8, device="cuda")
        binding.attn_decode_workspace_init(ws)
        out = torch.full_like(q, float("nan"))
        assert _calls().decode(int(dt == torch.float16), q, k, v, lens, 4, None, out, ws) == binding.OK
        assert torch.equal(out, _general(monkeypatch, binding.attn_decode_splitkv, q, k, v, lens, 4))
        x, b, res = r(20, 64), r(48), r(20, 48)
        for layout, w in ((binding.W_KN, r(64, 48)), (binding.W_NK, r(48, 64))):
            for bb, rr in ((None, None), (b, res)):
                y = torch.full_like(res, float("nan"))
                assert _calls().linear(int(dt == torch.float16), x, w, bb, rr, binding.ACT_SILU, layout, y) == binding.OK
                assert torch.equal(y, _general(monkeypatch, binding.linear_act, x, w, bb, rr, binding.ACT_SILU, layout))
    x, w = torch.randn((20, 64), generator=g, device="cuda").half(), torch.randint(-127, 128, (48, 64), generator=g, device="cuda").to(torch.int8)
    sc, y = torch.rand(48, generator=g, device="cuda"), torch.empty((20, 48), dtype=torch.float16, device="cuda")
    assert _calls().linear_w8(x, w, sc, None, None, binding.ACT_RELU, y) == binding.OK
    assert torch.equal(y, _general(monkeypatch, binding.linear_act_w8a16, x, w, sc, None, None, binding.ACT_RELU))
    x, wg, wu = (torch.randn(s, generator=g, device="cuda").bfloat16() for s in ((20, 64), (64, 48), (64, 48)))
    y = torch.empty((20, 48), dtype=torch.bfloat16, device="cuda")
    assert _calls().swiglu(x, wg, wu, binding.W_KN, y) == binding.OK
    assert torch.equal(y, _general(monkeypatch, binding.linear_swiglu, x, wg, wu, binding.W_KN))
    binding.check_status()


@pytest.mark.gpu
def test_whatever_is_not_plain_is_left_to_the_general_way():
    c = _calls()
    q, k, v, out = _attn_args()
    lens = torch.tensor([70, 33], dtype=torch.int32, device="cuda")
    assert c.attn(0, q, k, v, 0, None, None, out) == binding.OK
    turned = q.transpose(1, 2).contiguous().transpose(1, 2)
    for bad in ((1, q, k, v, 0, None, None, out), (0, turned, k, v, 0, None, None, out), (0, q, k, v, 0, None, None, turned),
                (0, q.as_subclass(_Sub), k, v, 0, None, None, out), (0, q, k[:1], v[:1], 0, None, None, out),
                (0, q, k, v[:, :, :69], 0, None, None, out), (0, q, k, v, 0, None, None, out[:, :3]), (0, q[0], k, v, 0, None, None, out),
                (0, q, k, v, 2, lens[:1], None, out), (0, q, k, v, 2, lens.long(), None, out), (0, q, k, v, True, None, None, out),
                (0, q, k, v, 1 << 40, None, None, out), (0, q, k, v, 0, None, 1, out), (0, q, k, v, 0, None, None, None)):
        assert c.attn(*bad) == NOT_PLAIN
    with _Mode():
        assert c.attn(0, q, k, v, 0, None, None, out) == NOT_PLAIN
    seen = []
    torch.vmap(lambda t: seen.append(c.attn(0, t, k, v, 0, None, None, out)) or t)(q.unsqueeze(0))
    assert seen == [NOT_PLAIN]
    # refused by the library: its status
    assert c.attn(0, q, k, v, 9, None, None, out) == binding.ERR_INVALID_ARG
    with pytest.raises(binding.ForgeError):
        binding.attn_fused(q, k, v, 9, out=out)
