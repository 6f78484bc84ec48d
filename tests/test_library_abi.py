"""CPU-side checks of the boundary: the library builds/loads, exports every symbol
the header declares, rejects bad arguments before touching a device, and its pure
host helpers reproduce the paper's printed numbers."""
import ctypes
import importlib.util
import os
import re
import sys
import types

import pytest
import torch

from paper_2604_18103_b200 import build as dash_build
from paper_2604_18103_b200 import dash

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GOLD = os.path.join(ROOT, "tests", "golden", "theory_speedup_vs_len.txt")


@pytest.fixture(scope="module")
def lib():
    dash_build.build()
    return dash.lib()


def _declared(header):
    hdr = open(os.path.join(ROOT, "include", header)).read()
    hdr = re.sub(r"/\*.*?\*/", "", hdr, flags=re.S)
    return set(re.findall(r"\b(dash_[a-z_0-9]+)\s*\(", hdr))


def test_every_declared_symbol_is_exported(lib):
    assert sorted(os.listdir(os.path.join(ROOT, "include"))) == ["dash.h", "dash_testing.h"]
    assert _declared("dash.h") == set(dash.EXPORTS)
    assert _declared("dash_testing.h") == set(dash.TEST_HOOKS)
    for name in dash.EXPORTS + dash.TEST_HOOKS:
        assert hasattr(lib, name), name


def test_keep_count_and_flops_helpers_match_paper_table(lib):
    for line in open(GOLD):
        if line.startswith("#") or not line.strip():
            continue
        n, n_hat, r_pct, s = line.split()
        n, n_hat = int(n), int(n_hat)
        assert dash.dash_keep_count(n, 0.667, 64, 32, 1) == n_hat
        sp = dash.dash_flops_speedup(n, n_hat, 28, 11, 3584, 18944)
        assert round(sp, 2) == pytest.approx(float(s), abs=0.0051)
        assert round(100 * (1 - 1 / sp), 2) == pytest.approx(float(r_pct), abs=0.0051)
    assert dash.dash_keep_count(8192, 0.4) == 4915
    assert dash.dash_keep_count(131072, 0.8) == 26214
    assert dash.dash_keep_count(10, 1.0) == -1 and dash.dash_keep_count(-1, 0.5) == -1
    assert dash.dash_flops_per_layer(2, 3, 5) == 4 * 2 * 9 + 2 * 4 * 3 + 2 * 2 * 3 * 5


def test_invalid_arguments_are_rejected_before_any_launch(lib):
    nul = ctypes.c_void_p(0)
    fake = ctypes.c_void_p(4096)            # never dereferenced: validation fails first
    # d not a multiple of 8
    assert lib.dash_delta_norm(fake, fake, 4, 12, 12, 12, dash.BF16, 0, 0.0, fake, nul, 0, nul, None, nul, nul) == 1
    # null U
    assert lib.dash_delta_norm(nul, fake, 4, 16, 16, 16, dash.BF16, 0, 0.0, fake, nul, 0, nul, None, nul, nul) == 1
    # misaligned pointer
    assert lib.dash_delta_norm(ctypes.c_void_p(4100), fake, 4, 16, 16, 16, dash.BF16, 0, 0.0, fake, nul, 0, nul, None, nul, nul) == 1
    # select without sequence boundaries / keep-count without counts
    assert lib.dash_select(fake, 8, nul, 1, 0, 0.0, nul, 0, 0, fake, nul) == 1
    assert lib.dash_select(fake, 8, fake, 1, 1, 0.0, nul, 0, 0, fake, nul) == 1
    # compaction: missing / too-small workspace
    assert lib.dash_compact(fake, 8, fake, 1, None, 0, nul, nul, nul, nul, nul, fake, nul, nul, 0, nul) == 3
    assert lib.dash_compact(fake, 1 << 20, fake, 1, None, 0, nul, nul, nul, nul, nul, fake, nul, fake, 512, nul) == 3
    # scatter: bad `which`
    assert lib.dash_scatter(fake, 8, 64, 64, nul, nul, 3, nul, fake, 64, nul) == 1
    # attention: head_dim 96 unsupported, non-causal unsupported, Hq % Hkv
    args = lambda Hq, Hkv, D, causal: (fake, fake, fake, fake, nul, Hq * D, Hkv * D, Hkv * D, Hq * D, fake, 1, 256, 256,
                                       Hq, Hkv, D, 0.1, causal, dash.BF16, nul, 0, nul)
    assert lib.dash_varlen_attention(*args(4, 2, 96, 1)) == 2
    assert lib.dash_varlen_attention(*args(4, 2, 128, 0)) == 2
    assert lib.dash_varlen_attention(*args(4, 3, 128, 1)) == 1
    assert lib.dash_status_string(3).decode().startswith("workspace")
    assert dash.dash_workspace_bytes(dash.WS_COMPACT, 131072) >= 131072 // 32 * 8


def _cfgs(sh, dt):
    c = dash.LayerCfg(d=sh[0], Hq=sh[1], Hkv=sh[2], D=sh[3], dt=dt, Wqkv=4096, Wo=4096, rms_weight=4096, rms_eps=1e-6, rope_base=1e4, scatter_which=2)
    return c, dash.BlockCfg(attn=c, m=sh[4], Wgu=4096, Wd=4096, rms2_weight=4096)


def _totals(lib, layer, block, n, S=1):
    a, b = dash.LayerWsLayout(), dash.BlockWsLayout()
    assert lib.dash_layer_workspace(ctypes.byref(layer), n, S, ctypes.byref(a)) == 0
    assert lib.dash_block_workspace(ctypes.byref(block), n, S, ctypes.byref(b)) == 0
    return a.total, b.total


@pytest.mark.parametrize("dt", [dash.BF16, dash.F32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("shape", [(3584, 28, 4, 128, 18944), (512, 8, 2, 128, 1024), (8192, 4, 2, 64, 256)], ids=["7b", "mini", "deep"])
def test_step_workspace_holds_what_the_step_can_use(lib, shape, dt):
    """A step asks for its tensors and, where it cuts a projection along K, for the partial tiles (2 x 256 KB per pair of CTAs), else for none;
    and a workspace of n rows serves every step of fewer rows."""
    d, Hq, Hkv, D, m = shape
    layer, block = _cfgs(shape, dt)
    nq, hd, es = (Hq + 2 * Hkv) * D, Hq * D, 2 if dt == dash.BF16 else 4

    def needs(n, ffn):
        b = n * (3 * d + nq + hd) * es + n * (D // 2) * 8 + n * -(-d // 128) * 16 + 8 * n      # activations, rotary table, per-row sums and factors
        b += n * (3 * m + d) * es if ffn else 0
        if dt == dash.F32:                                                                     # bf16 copies of what is multiplied
            b += (n * max(d, hd) + d * nq + hd * d + n * nq) * 2 + ((n * max(m, d) + d * 2 * m) * 2 if ffn else 0)
            return b
        projections = [(nq, d), (d, hd)] + ([(2 * m, d), (d, m)] if ffn else [])
        return b + max(lib.dash_testing_gemm_groups(n, N, K) for N, K in projections) * -(-n // 256) * 2 * 256 * 1024

    for n in (1, 2, 100, 256, 257, 701, 2368, 5376, 5377, 8192, 18944, 18945, 32768):
        for ffn, total in enumerate(_totals(lib, layer, block, n)):
            most = max(needs(r, ffn) for r in [n, *range(256, min(n, 75 * 256), 256)])
            assert most <= total <= most + 80 * n + 40000, (n, ffn)                            # lists, look-back words, alignment


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_stream_handle_without_torchs_private_functions(monkeypatch, missing):
    """A torch that lacks one of the two private functions behind the short way to the current stream's handle: the public way."""
    monkeypatch.delattr(torch._C, missing, raising=False)
    spec = importlib.util.spec_from_file_location("dash_on_another_torch", dash.__file__)
    other = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(other)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=7))
    assert other._stream() == 7


@pytest.mark.parametrize("D", [64, 128])
def test_an_sm_takes_as_many_decode_ctas_as_its_tensor_memory_holds(lib, D):
    """Two, 256 of the SM's 512 columns each; a third CTA (228 KB of shared memory per SM, 1 KB of it the system's per CTA) would hold its share of the
    caches' blocks back until one of the two has left."""
    assert 228 * 1024 // (lib.dash_testing_decode_smem_bytes(D) + 1024) == 2


class _Tensor:
    """What the binding's C part asks of a tensor."""

    def __init__(self, shape, ptr=4096, dtype=torch.bfloat16, is_cuda=True):
        self.shape, self.ptr, self.dtype, self.is_cuda = shape, ptr, dtype, is_cuda

    def data_ptr(self):
        if self.ptr is None:
            raise RuntimeError("no storage")
        return self.ptr

    def stride(self, dim):
        return 96 if len(self.shape) < 3 else self.shape[1] * self.shape[2]

    def numel(self):
        return 256


def test_the_bindings_c_part_checks_and_raises_as_the_python_one(lib):
    """Decoding goes through csrc/pycall.c: host tensors, wrong dimensions and types and a tensor without storage raise what the checks in Python
    raise; what is left is refused by the library (head dimension 96: unsupported, misaligned cache: invalid, no room: workspace)."""
    t, k = _Tensor((1, 28, 128)), _Tensor((10, 4, 128))

    def call(q=t, K=k, V=k, cu=t, scale=None, out=t, ws=t):
        return dash._pycall.decode(q, K, V, cu, scale, out, None, ws, 0)

    with pytest.raises(ValueError, match="device tensor expected"):
        call(V=_Tensor((10, 4, 128), is_cuda=False))
    with pytest.raises(ValueError):
        call(q=_Tensor((28, 128)))
    with pytest.raises(TypeError, match="unsupported dtype"):
        call(q=_Tensor((1, 28, 128), dtype=torch.float16))
    with pytest.raises(TypeError):
        call(scale="large")
    with pytest.raises(RuntimeError, match="no storage"):
        call(K=_Tensor((10, 4, 128), ptr=None))
    with pytest.raises(AttributeError):
        call(ws=3)
    with pytest.raises(ValueError, match="device tensor expected"):
        dash.dash_decode_attention(torch.zeros(1, 28, 128).bfloat16(), torch.zeros(10, 4, 128).bfloat16(), torch.zeros(10, 4, 128).bfloat16(), torch.zeros(2, dtype=torch.int32))
    assert call(q=_Tensor((1, 28, 96)), K=_Tensor((10, 4, 96)), V=_Tensor((10, 4, 96))) == 2
    assert call(q=_Tensor((1, 28, 128), dtype=torch.float32)) == 2
    assert call(K=_Tensor((10, 4, 128), ptr=4100)) == 1 and call(scale=-1.0) == 1 and call(scale=0.1) == 3


def test_a_thread_that_finds_the_library_loaded_can_decode(lib):
    """Between any two bytecodes of the first lib() another thread may run: as soon as that one would find the library loaded, a decoding call reaches its
    checks."""
    spec = importlib.util.spec_from_file_location("paper_2604_18103_b200.dash_again", dash.__file__)
    again = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(again)
    host = [torch.zeros(1, 28, 128).bfloat16(), torch.zeros(10, 4, 128).bfloat16()]
    seen, busy = [], []

    def other_thread(code, offset):
        if again._lib is not None and not busy:
            busy.append(True)
            try:
                again.dash_decode_attention(host[0], host[1], host[1], torch.zeros(2, dtype=torch.int32), out=host[0], ws=torch.zeros(256, dtype=torch.uint8))
            except Exception as e:
                seen.append(type(e))
            busy.pop()

    again._stream = lambda: 0
    m = sys.monitoring
    m.use_tool_id(m.DEBUGGER_ID, "every bytecode")
    m.register_callback(m.DEBUGGER_ID, m.events.INSTRUCTION, other_thread)
    m.set_local_events(m.DEBUGGER_ID, again.lib.__code__, m.events.INSTRUCTION)
    try:
        again.lib()
    finally:
        m.set_local_events(m.DEBUGGER_ID, again.lib.__code__, 0)
        m.free_tool_id(m.DEBUGGER_ID)
    assert seen and set(seen) == {ValueError}, seen


def test_without_its_c_part_the_library_builds_loads_and_decodes_through_ctypes(lib, monkeypatch, tmp_path, capfd):
    """No C compiler, or a tree built under another Python (the C part's name carries the interpreter's tag): every entry point is there, a decoding
    call raises and is refused as with it."""
    monkeypatch.setattr(dash_build, "PYCALL", str(tmp_path / os.path.basename(dash_build.PYCALL)))
    with open(dash_build.PYCALL, "w") as f:
        f.write("of an older source")
    with monkeypatch.context() as m:
        m.setenv("PATH", str(tmp_path))
        assert dash_build.build_pycall(force=True) is None and not os.path.exists(dash_build.PYCALL) and "ctypes" in capfd.readouterr().err
    assert dash_build.build_pycall() == dash_build.PYCALL and os.path.exists(dash_build.PYCALL)
    spec = importlib.util.spec_from_file_location("paper_2604_18103_b200.dash_without", dash.__file__)
    without = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(without)
    without.PYCALL_PATH, without._stream = str(tmp_path / "none.so"), lambda: 0
    assert without.lib().dash_keep_count(8192, 0.4, 0, 0, 0) == 4915 and without._pycall is False
    t, k = _Tensor((1, 28, 128)), _Tensor((10, 4, 128))

    def refused(error, q=t, K=k, V=k, scale=None, out=t, ws=t):
        for module in (dash, without):
            with monkeypatch.context() as m:
                m.setattr(module, "_stream", lambda: 0)
                with pytest.raises(error) as e:
                    module.dash_decode_attention(q, K, V, t, scale=scale, out=out, ws=ws)
            yield getattr(e.value, "status", None)

    assert list(refused(ValueError, V=_Tensor((10, 4, 128), is_cuda=False))) == [None] * 2
    assert list(refused(ValueError, q=_Tensor((28, 128)))) == [None] * 2
    assert list(refused(TypeError, q=_Tensor((1, 28, 128), dtype=torch.float16))) == [None] * 2
    for want, kw in ((2, dict(q=_Tensor((1, 28, 96)), K=_Tensor((10, 4, 96)), V=_Tensor((10, 4, 96)))), (1, dict(K=_Tensor((10, 4, 128), ptr=4100))),
                     (1, dict(scale=-1.0)), (3, dict(scale=0.1))):
        assert list(refused(RuntimeError, **kw)) == [want] * 2


def test_decode_takes_for_a_scale_what_float_takes(lib, monkeypatch):
    """As the other attention entry points do: -1 in any form is read and refused by the library, text that is no number is a ValueError."""
    monkeypatch.setattr(dash, "_stream", lambda: 0)
    t, k = _Tensor((1, 28, 128)), _Tensor((10, 4, 128))
    for scale in (-1, -1.0, "-1.0", torch.tensor(-1.0)):
        with pytest.raises(dash.DashError) as e:
            dash.dash_decode_attention(t, k, k, t, scale=scale, out=t, ws=t)
        assert e.value.status == 1
    with pytest.raises(ValueError):
        dash.dash_decode_attention(t, k, k, t, scale="large", out=t, ws=t)
