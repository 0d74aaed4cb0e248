"""The CPython extension behind the binding: it takes plain calls only, and what it takes gives the bytes of the ctypes route."""
import runpy
import types

import pytest
import torch


@pytest.fixture(scope="module")
def B():
    from paper_2605_26266_b200 import build
    build.build_library()
    from paper_2605_26266_b200 import binding
    return binding


def test_the_extension_is_the_one_that_runs_and_takes_plain_calls_only(B):
    from paper_2605_26266_b200 import _py_call
    assert B._append_call is _py_call.append and B._attn_call is _py_call.attn
    x = torch.zeros(1, 2, 16, 128, dtype=torch.bfloat16)                               # on the CPU
    for args in [(0, 0, x, x, 0), (0, 0, None, x, 0), ("0", 0, x, x, 0), (0, 0.0, x, x, 0), (0, 0, x, x), (1 << 90, 0, x, x[0], None)]:
        assert _py_call.append(*args) == B._NOT_PLAIN
    attn = [0, 0, 0, x, x, x, x, 0.1, 1, None, None, None, None, 0]
    for i, v in [(0, None), (3, x), (4, "k"), (7, 1), (8, 1.0), (9, 5), (12, b""), (13, None)]:
        assert _py_call.attn(*(attn[:i] + [v] + attn[i + 1:])) == B._NOT_PLAIN
    with pytest.raises(TypeError):
        _py_call.bind(1, 2)
    cache = B.Cache(1, 2, 128, 2, 64, 128, device="cpu")
    for k, v in [(x, x), (x.float(), x), (x[:, :, :8], x)]:
        with pytest.raises(AssertionError):
            B.kvq_quantize_append(cache, k, v)
        with pytest.raises(AssertionError):
            B.kvq_attn_corrected(cache, x, k, v, 0.1, out=x)
    assert cache.length == 0 and cache.workspace is None


@pytest.mark.parametrize("built_for", [None, "torch 1.0 python 0x30c03f0"])
def test_an_extension_of_another_torch_or_python_is_not_used(B, monkeypatch, built_for):
    """It would load and read tensors by the layout it was compiled with."""
    import paper_2605_26266_b200 as package

    def used(*_):
        raise AssertionError("used")
    other = types.ModuleType("_py_call")
    other.bind = other.append = other.attn = used
    if built_for:
        other.built_for = built_for
    monkeypatch.setattr(package, "_py_call", other, raising=False)
    again = runpy.run_path(B.__file__, run_name=B.__name__)                    # the module once more, beside the one that is loaded
    assert again["_append_call"]() == again["_attn_call"]() == B._NOT_PLAIN


@pytest.mark.parametrize("how", ["no compiler", "no Python.h"])
def test_the_library_is_built_without_the_extension(B, monkeypatch, tmp_path, how):
    """The library is complete without it, and the binding has its ctypes route; a file of former sources is not left behind."""
    from paper_2605_26266_b200 import build
    run = build.subprocess.run

    def without_gxx(cmd, **kw):
        if cmd[0] != "g++":
            return run(cmd, **kw)
        if how == "no compiler":
            raise FileNotFoundError("g++")
        return build.subprocess.CompletedProcess(cmd, 1, "", "Python.h: No such file or directory")
    former = tmp_path / "_py_call.so"
    former.write_bytes(b"former")
    monkeypatch.setattr(build, "PY_CALL", str(former))
    monkeypatch.setattr(build.subprocess, "run", without_gxx)
    with pytest.warns(UserWarning, match="ctypes"):
        assert build.build_library() == build.LIB
    assert not former.exists()


def test_a_call_that_fails_is_not_issued_again(B, monkeypatch):
    """A status of the native call is raised as it is: some of its kernels may have been launched, and the second call's could
    succeed."""
    class OnDevice:                                              # as much of a tensor as the route up to the status looks at
        is_cuda, dtype, device, shape = True, torch.bfloat16, "cuda:0", (1, 2, 16, 128)
        stride, data_ptr = (lambda self: (4096, 2048, 128, 1)), (lambda self: 4096)
    issued = []

    def native(*args):
        issued.append(args)
        return B.KVQ_ERR_CUDA

    def through_ctypes(*args):
        issued.append(args)
        return B.KVQ_OK
    monkeypatch.setattr(B, "_attn_call", native)
    monkeypatch.setattr(B, "_attn_corrected", through_ctypes)
    monkeypatch.setattr(B, "_stream", lambda: 0)
    cache, x = B.Cache(1, 2, 128, 2, 64, 128, device="cpu"), OnDevice()
    cache.workspace = torch.empty(1 << 20, dtype=torch.uint8)
    with pytest.raises(B.KvqError, match="kvq_attn_corrected") as e:
        B.kvq_attn_corrected(cache, x, x, x, 0.1, cache_len=64, out=x)
    assert e.value.status == B.KVQ_ERR_CUDA and len(issued) == 1
    with pytest.raises(B.KvqError, match="kvq_attn_workspace_bytes"):        # refused before that: named as ever
        B.kvq_attn_corrected(cache, x, x, x, 0.1, flags=1 << 20, cache_len=64, out=x)
    assert len(issued) == 2


@pytest.mark.gpu
@pytest.mark.parametrize("d,m,layout", [(128, 40, "dense"), (128, 300, "interleaved"), (64, 40, "padded"), (64, 700, "dense")])
def test_both_routes_give_the_same_bytes(B, d, m, layout, monkeypatch):
    g = torch.Generator(device="cuda").manual_seed(5)

    def tensor(t):
        x = torch.randn(2, 3, t, d, device="cuda", generator=g).bfloat16()
        if layout == "interleaved":
            return x.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
        if layout == "padded":
            return torch.nn.functional.pad(x, (0, 24))[..., :d]
        return x
    pk, pv, q, k, v = tensor(500), tensor(500), tensor(m), tensor(m), tensor(m)
    results = []
    for native in (True, False):
        if not native:
            monkeypatch.setattr(B, "_append_call", lambda *_: B._NOT_PLAIN)
            monkeypatch.setattr(B, "_attn_call", lambda *_: B._NOT_PLAIN)
        cache = B.Cache(2, 3, d, 2, 64, 640)
        assert B.kvq_quantize_append(cache, pk, pv) == 500 and B.kvq_quantize_append(cache, pk[:, :, :16], pv[:, :, :16]) == 516
        lse = torch.zeros(2, 3, m, device="cuda")
        mass, status = torch.zeros_like(lse), torch.zeros(1, dtype=torch.int32, device="cuda")
        given = torch.empty_like(q)
        assert B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, out=given, lse=lse, cached_mass=mass, status_word=status) is given
        made = B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, cache_begin=16, cache_len=400)
        assert made.is_contiguous()
        with pytest.raises(B.KvqError) as e:
            B.kvq_attn_corrected(cache, q, k, v, d ** -0.5, cache_begin=8, out=given)
        assert e.value.status == B.KVQ_ERR_ALIGNMENT
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        results.append([t.clone() for t in (*cache.buffers, given.view(torch.int16), lse, mass, made.view(torch.int16))])
    assert all(torch.equal(a, b) for a, b in zip(*results))
