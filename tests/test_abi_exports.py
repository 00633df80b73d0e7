"""The C-ABI library builds for sm_100a, loads without a GPU, and exports every entry point the
public header declares (no compute calls here)."""
import ctypes
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def libpath():
    from paper_2503_07518_b200 import build
    return build.build()


def declared_functions():
    src = open(os.path.join(ROOT, "include", "tokenbutler.h")).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return sorted(set(re.findall(r"\b(tb_[a-z_]+)\s*\(", src)))


def test_header_declares_the_path_entry_points():
    names = declared_functions()
    for must in ("tb_append_kv", "tb_project_keys", "tb_score_tokens", "tb_select_topk", "tb_sparse_decode_attention"):
        assert must in names


def test_library_exports_every_declared_symbol(libpath):
    lib = ctypes.CDLL(libpath)
    for name in declared_functions():
        assert hasattr(lib, name), name


def test_binding_lists_the_same_names(libpath):
    from paper_2503_07518_b200 import binding
    assert sorted(binding.EXPORTS) == declared_functions()


def test_host_validation_needs_no_gpu(libpath):
    from paper_2503_07518_b200 import binding as b
    L = b.lib()
    cfg = b.tb_config(2, 8, 8, 128, 32, b.TB_BF16, 1, 1024, 64, 1, 0, 0)
    sizes = [ctypes.c_size_t() for _ in range(4)]
    assert L.tb_query_sizes(ctypes.byref(cfg), *[ctypes.byref(s) for s in sizes]) == b.TB_OK
    assert sizes[0].value == 2 * 1 * 8 * 1024 * 2 * 128 * 2            # interleaved K|V rows
    assert sizes[1].value == 2 * 1 * 8 * 1024 * 32 * 2                  # projected keys
    bad = b.tb_config(2, 8, 8, 96, 32, b.TB_BF16, 1, 1024, 64, 1, 0, 0)
    assert L.tb_query_sizes(ctypes.byref(bad), *[ctypes.byref(s) for s in sizes]) == b.TB_ERR_UNSUPPORTED
    bad = b.tb_config(2, 9, 8, 128, 32, b.TB_BF16, 1, 1024, 64, 1, 0, 0)
    assert L.tb_query_sizes(ctypes.byref(bad), *[ctypes.byref(s) for s in sizes]) == b.TB_ERR_INVALID_ARG
    assert L.tb_status_string(b.TB_ERR_UNPROJECTED) == b"candidate keys not projected"


def test_predictor_host_validation_needs_no_gpu(libpath):
    from paper_2503_07518_b200 import binding as b
    L = b.lib()
    one = ctypes.c_void_p(16)                           # any aligned non-null address: never dereferenced on these paths
    ok = dict(dtype=b.TB_BF16, model_dim=4096, hidden_dim=512, n_q_heads=32, n_slots=4, imp_dim=32, activation=b.TB_ACT_GELU,
              ln_eps=1e-5, ln_weight=16, ln_bias=16, w1=16, w2=16)

    def call(n_tokens=1, hidden=one, **over):
        p = b.tb_predictor(**{**ok, **over})
        return L.tb_predict_importance_queries(ctypes.byref(p), hidden, n_tokens, one, one, None)

    assert call(w1=None) == b.TB_ERR_INVALID_ARG
    assert call(hidden=None) == b.TB_ERR_INVALID_ARG
    assert call(n_tokens=0) == b.TB_ERR_INVALID_ARG
    assert call(activation=7) == b.TB_ERR_INVALID_ARG
    assert call(ln_weight=24) == b.TB_ERR_INVALID_ARG      # not 16-byte aligned
    assert call(model_dim=4100) == b.TB_ERR_UNSUPPORTED    # rows are read 16 bytes at a time
    assert call(n_tokens=65) == b.TB_ERR_CAPACITY


def test_extension_module_unpacks_like_ctypes(libpath):
    from paper_2503_07518_b200 import binding as b
    b.lib()
    p, s = b.select_params(4), type("Stream", (), {"cuda_stream": 0})()
    # a null context reaches the entry point and is refused there; what cannot be unpacked raises before the call
    assert b._calls.select_topk(None, 0, 1, (0,), 1, None, p, None, None, s) == b.TB_ERR_INVALID_ARG
    assert b._calls.append_kv(None, 0, 1, None, list(range(100)), None, None, s) == b.TB_ERR_INVALID_ARG
    for bad in ((None, 0, 1, None, 1, None, object(), None, None, s), (None, 0, 1, ["x"], 1, None, p, None, None, s),
                (None, "0", 1, None, 1, None, p, None, None, s), (None, 0, 1, None, 1, None, p, None, None)):
        with pytest.raises((TypeError, ValueError)):
            b._calls.select_topk(*bad)


@pytest.mark.parametrize("call", [
    "append_kv(None, 0, 1, None, [1], sparse, None, s)",
    "select_topk(None, 0, 1, None, 1, sparse, p, None, None, s)",
    "project_keys(None, 0, 1, None, [0], [1], 1, None)",                       # the current stream of no device
    "predict_importance_queries(0, 1, 1, 16, 0, 1e-5, sparse, None, m, None, m, None, None, s)",
    "predict_importance_queries(0, 1, 1, 16, 0, 1e-5, None, None, m, None, m[0], None, None, s)",   # no second size
])
def test_what_torch_throws_is_a_python_exception(libpath, call):
    import subprocess
    code = ("import torch\nfrom paper_2503_07518_b200 import binding as b\nb.lib()\n"
            "sparse, m = torch.eye(3).to_sparse(), torch.zeros(4, 8)\n"
            "p, s = b.select_params(4), type('Stream', (), {'cuda_stream': 0})()\n"
            "try:\n    b._calls.%s\nexcept Exception as e:\n    print('raised', type(e).__name__)" % call)
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, CUDA_VISIBLE_DEVICES=""), capture_output=True, text=True)
    assert r.returncode == 0 and "raised" in r.stdout, (r.returncode, r.stdout, r.stderr[-300:])


def test_predictor_binding_takes_what_has_a_shape(libpath):
    """Sizes are read from the leading dimensions of tensors of any rank, and of other objects with a shape and a data_ptr()."""
    import torch
    from paper_2503_07518_b200 import binding as b

    class Where:
        def __init__(self, t):
            self.shape, self.data_ptr = t.shape, t.data_ptr

    t = torch.zeros(64, 64)
    s = type("Stream", (), {"cuda_stream": 0})()
    call = lambda hidden, w1: b.predict_importance_queries(hidden, t, t, w1, t, b.TB_F32, 1, 1, 16, t, t, ln_eps=-1.0, stream=s)  # noqa: E731
    for hidden, w1 in ((t, t), (t.view(64, 64, 1), t.view(64, 8, 8)), (t, t.view(-1)), (Where(t), Where(t))):
        assert call(hidden, w1) == b.TB_ERR_INVALID_ARG            # the library's answer to a negative epsilon
    for hidden in (t.view(-1), None, 3):
        with pytest.raises((IndexError, AttributeError, TypeError)):
            call(hidden, t)


def test_a_module_built_for_another_torch_is_not_loaded(libpath, monkeypatch):
    """It is rebuilt by the build and refused by the binding: its symbols are those of the torch and Python it was built for."""
    from paper_2503_07518_b200 import binding as b
    from paper_2503_07518_b200 import build
    import importlib.metadata
    assert build.calls_match() and not build._stale()
    real = importlib.metadata.version
    monkeypatch.setattr(importlib.metadata, "version", lambda name: real(name) + "1" if name == "torch" else real(name))
    assert build._stale()
    monkeypatch.setattr(b, "_lib", None)
    with pytest.raises(RuntimeError, match="built for torch"):
        b.lib()
