"""The Python entry of the per-step calls (csrc/novakv_calls.c): what it refuses, and what it takes as before.  Arguments are
formed before the library is called, and the library refuses a null context before it touches a device, so this runs anywhere;
what needs a context is marked for the GPU."""
import sysconfig
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2608_04074_b200 import binding, build

torch = pytest.importorskip("torch")

EINVAL = 1
# name, arguments; L layer, T tensor whose shape, type or size is read, P pointer only, N integer, F scale, O pointer or None
CALLS = {
    "novakv_encode_append": "LOPPPTPTP",
    "novakv_encode_append_scaled": "LOPPPTPPTP",
    "novakv_encode_append_deployed": "LOPPPTPPPTP",
    "novakv_decode_attention": "LTTPTPTTF",
    "novakv_decode_attention_scaled": "LTTPPTPTTF",
    "novakv_decode_attention_sink": "LTTPOPTPTTF",
    "novakv_decode_attention_banded": "LTTPOOTPTPNPTTF",
    "novakv_decode_attention_deployed": "LTTPPPOTPOONOTTF",
    "novakv_band_append": "LTPTPNNNPPTPOOTPT",
    "novakv_bf16_decode_attention": "TTPTPTTFN",
    "novakv_step_host": "LOPPPTTPTPPTTF",
    "novakv_step_host_async": "LOPPPTTPTPPTTF",
}


@pytest.fixture(scope="module")
def calls():
    build.build_cuda()
    assert build.LIB_CALLS.exists()
    from paper_2608_04074_b200 import _novakv_calls
    _novakv_calls.setup(lambda device: 0, lambda: 0, torch.float32)
    yield _novakv_calls.bind(binding.load_library()._handle)
    if torch.cuda.is_available():                        # (contexts of other tests ask the same functions)
        _novakv_calls.setup(torch._C._cuda_getCurrentRawStream, torch._C._cuda_getDevice, torch.float32)


def _args(kinds):
    t = torch.zeros((2, 3, 4), dtype=torch.bfloat16)
    return [{"L": 0, "N": 64, "F": 0.5}.get(k, t) for k in kinds]


def test_extension_is_named_after_its_interpreter():
    """Another Python minor version must not find it (it would run with this one's inlined object layout)."""
    assert build.LIB_CALLS.name == "_novakv_calls" + sysconfig.get_config_var("EXT_SUFFIX") != "_novakv_calls.so"


def test_library_is_built_where_the_extension_cannot_be(monkeypatch, tmp_path):
    monkeypatch.setattr(build.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    monkeypatch.setattr(build, "LIB_CALLS", tmp_path / "calls.so")
    with pytest.warns(UserWarning, match="Python entry"):
        assert build.build_cuda() == build.LIB_CUDA
    with pytest.raises(RuntimeError):
        build.build_calls()


def test_every_call_is_bound(calls):
    assert set(calls) == set(CALLS)


@pytest.mark.parametrize("name", CALLS)
def test_null_context_and_argument_count(calls, name):
    args = _args(CALLS[name])
    for handle in (0, None):
        assert calls[name](handle, *args) == EINVAL
    for wrong in (args[:-1], args + [0]):
        with pytest.raises(TypeError, match="positional"):
            calls[name](0, *wrong)
    with pytest.raises(TypeError):
        calls[name](0, *args[:-1], last=args[-1])


@pytest.mark.parametrize("name", [n for n in CALLS if CALLS[n][0] == "L"])
@pytest.mark.parametrize("layer", [1.5, 0.0, "0", None, np.float32(0)])
def test_layer_that_is_no_integer_is_refused(calls, name, layer):
    with pytest.raises(TypeError):
        calls[name](0, layer, *_args(CALLS[name])[1:])


def test_integers_of_any_kind_are_layers(calls):
    for layer in (0, True, np.int32(0), np.int64(0), torch.tensor(0)):
        assert calls["novakv_decode_attention"](0, layer, *_args(CALLS["novakv_decode_attention"])[1:]) == EINVAL


@pytest.mark.parametrize("name,i", [(n, i) for n in CALLS for i, k in enumerate(CALLS[n]) if k == "T"])
@pytest.mark.parametrize("bad", [None, 7, SimpleNamespace(data_ptr=lambda: 0)])
def test_tensor_that_is_none_or_no_tensor_is_refused(calls, name, i, bad):
    args = _args(CALLS[name])
    args[i] = bad
    with pytest.raises(AttributeError):
        calls[name](0, *args)


@pytest.mark.parametrize("name,i", [(n, i) for n in CALLS for i, k in enumerate(CALLS[n]) if k in "PO"])
def test_pointer_arguments(calls, name, i):
    """None is a null pointer (the library judges it); what has no address is refused."""
    args = _args(CALLS[name])
    args[i] = None
    assert calls[name](0, *args) == EINVAL
    for bad in (7, np.zeros(4)):
        args[i] = bad
        with pytest.raises(AttributeError):
            calls[name](0, *args)


@pytest.mark.parametrize("bad", ["x", None, [1.0]])
def test_scale_that_is_no_number_is_refused(calls, bad):
    args = _args(CALLS["novakv_decode_attention"])
    args[-1] = bad
    with pytest.raises(TypeError):
        calls["novakv_decode_attention"](0, *args)
    args[-1] = np.float32(0.5)
    assert calls["novakv_decode_attention"](0, *args) == EINVAL


def test_errors_of_the_stream_query_are_passed_on(calls):
    from paper_2608_04074_b200 import _novakv_calls

    def broken(*_):
        raise RuntimeError("no device")
    try:
        for stream, device in ((broken, lambda: 0), (lambda device: 0, broken), (lambda device: "s", lambda: 0)):
            _novakv_calls.setup(stream, device, torch.float32)
            with pytest.raises((RuntimeError, TypeError)):
                calls["novakv_decode_attention"](0, *_args(CALLS["novakv_decode_attention"]))
    finally:
        _novakv_calls.setup(lambda device: 0, lambda: 0, torch.float32)


# ------------------------------------------------------------------------------------------------ with a context
@pytest.fixture(scope="module")
def loaded():
    from gpu_common import Case
    from paper_2608_04074_b200 import workloads
    from paper_2608_04074_b200.runtime import PagedCache
    case = Case(workloads.tiny())
    cache = PagedCache(case.ctx, np.array([700, 90], np.int32), seed=3)
    gen = torch.Generator(device="cuda").manual_seed(5)
    for pool in (cache.k_pages, cache.v_pages):
        pool.copy_(torch.randint(0, 256, pool.shape, generator=gen, dtype=torch.uint8, device="cuda"))
    q = torch.randn((2, case.ctx.n_q_heads, case.ctx.head_dim), generator=gen, device="cuda").to(torch.bfloat16)
    return case, cache, q


@pytest.mark.gpu
def test_closed_context_is_refused(loaded):
    from paper_2608_04074_b200.binding import Context, NovaKVError
    case, cache, q = loaded
    closed = Context(case.ctx.n_q_heads, case.ctx.n_kv_heads, case.ctx.head_dim)
    closed.close()
    out = torch.full(q.shape, 5.0, device="cuda")
    with pytest.raises(NovaKVError, match="invalid argument"):
        closed.novakv_decode_attention(0, q, cache.k_pages, cache.v_pages, cache.page_table, cache.seq_lens, out, cache.workspace)
    assert (out == 5.0).all()


@pytest.mark.gpu
@pytest.mark.parametrize("missing", ["q", "k_pages", "v_pages", "page_table", "seq_lens", "out", "workspace"])
def test_required_tensor_left_out(loaded, missing):
    case, cache, q = loaded
    args = dict(q=q, k_pages=cache.k_pages, v_pages=cache.v_pages, page_table=cache.page_table, seq_lens=cache.seq_lens,
                out=torch.empty(q.shape, device="cuda"), workspace=cache.workspace)
    args[missing] = None
    before = case.ctx.novakv_launch_count()
    with pytest.raises((AttributeError, binding.NovaKVError)):
        case.ctx.novakv_decode_attention(0, **args)
    assert case.ctx.novakv_launch_count() == before


@pytest.mark.gpu
def test_call_goes_to_the_current_stream(loaded):
    """On a side stream, behind work that takes a while there: the call has to wait for it, and the default stream not for
    the call."""
    case, cache, q = loaded
    expected = cache.decode(0, q)
    other = cache.decode(0, -q)
    assert not torch.equal(expected, other)
    torch.cuda.synchronize()
    side, late, out = torch.cuda.Stream(), torch.empty_like(q), torch.zeros_like(expected)
    late.copy_(-q)
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)                    # some 10 ms
        late.copy_(q)
        cache.decode(0, late, out=out)
        done.record()
    torch.cuda.current_stream().synchronize()
    assert not done.query()
    side.synchronize()
    assert torch.equal(out, expected)
