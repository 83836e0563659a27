"""The C-ABI library: it loads, exports every symbol the header declares, and
rejects bad arguments on the host before touching a device (no GPU needed)."""
import ctypes
import os
import re

import pytest

import paper_2604_13349_b200 as P
from paper_2604_13349_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load()


def declared_functions():
    text = open(os.path.join(ROOT, "include", "obf.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    text = re.sub(r"^\s*#.*$", "", text, flags=re.M)            # preprocessor lines declare nothing
    return sorted(set(re.findall(r"\b(\w+)\s*\([^;{}]*\)\s*;", text)))


def test_header_functions_are_all_exported(lib):
    names = declared_functions()
    assert set(binding.EXPORTS) == set(names)
    for n in names:
        assert getattr(lib, n) is not None


def test_struct_sizes_match_the_header():
    assert ctypes.sizeof(binding.ObfParams) == 36
    assert ctypes.sizeof(binding.ObfDiag) == 60
    assert ctypes.sizeof(binding.ObfCache) == 128


def test_status_strings(lib):
    seen = {P.obf_status_string(c) for c in range(6)}
    assert len(seen) == 6 and "ok" in seen
    assert P.obf_status_string(99) == "unknown status"


def _params(**kw):
    base = dict(layers=1, kv_heads=2, q_heads=8, head_dim=64, n_obs=16, rank=1, dtype=P.OBF_F32)
    base.update(kw)
    return P.make_params(**base)


def _cache(T=256, budget=32, ptr=0x1000):
    return P.make_cache(ptr, ptr, ptr, T, budget, ptr, ptr, ptr)


def test_workspace_size_grows_with_the_problem(lib):
    a = P.obf_workspace_bytes(_params(), [_cache()])
    b = P.obf_workspace_bytes(_params(), [_cache(T=512)])
    c = P.obf_workspace_bytes(_params(rank=0), [_cache()])
    d = P.obf_workspace_bytes(_params(), [_cache(), _cache(T=100, budget=7)])
    assert b > a > c > 0 and d > a
    assert a % 256 == 0


@pytest.mark.parametrize("kw,code", [
    (dict(head_dim=96), binding.OBF_ERR_UNSUPPORTED),
    (dict(dtype=7), binding.OBF_ERR_UNSUPPORTED),
    (dict(q_heads=7), binding.OBF_ERR_INVALID_ARG),
    (dict(rank=-1), binding.OBF_ERR_INVALID_ARG),
    (dict(rank=65), binding.OBF_ERR_INVALID_ARG),
    (dict(layers=0), binding.OBF_ERR_INVALID_ARG),
    (dict(n_obs=0), binding.OBF_ERR_INVALID_ARG),
    (dict(eps=-1.0), binding.OBF_ERR_INVALID_ARG),
])
def test_bad_params_are_rejected_on_the_host(lib, kw, code):
    with pytest.raises(P.ObfError) as e:
        P.obf_workspace_bytes(_params(**kw), [_cache()])
    assert e.value.code == code


@pytest.mark.parametrize("cache,code", [
    (dict(T=0), binding.OBF_ERR_INVALID_ARG),
    (dict(budget=0), binding.OBF_ERR_INVALID_ARG),
    (dict(T=(1 << 20) + 1), binding.OBF_ERR_INVALID_ARG),
])
def test_bad_cache_shapes_are_rejected_on_the_host(lib, cache, code):
    with pytest.raises(P.ObfError) as e:
        P.obf_workspace_bytes(_params(), [_cache(**cache)])
    assert e.value.code == code


def test_compress_rejects_before_any_launch(lib):
    # None of these calls reaches the CUDA runtime: validation comes first.
    p = _params()
    pp, arr = ctypes.byref(p), (binding.ObfCache * 1)(_cache())
    assert lib.obf_compress(pp, arr, 0, 0x100, 1 << 30, None) == binding.OBF_ERR_INVALID_ARG
    assert lib.obf_compress(pp, arr, 33, 0x100, 1 << 30, None) == binding.OBF_ERR_UNSUPPORTED
    assert lib.obf_compress(None, arr, 1, 0x100, 1 << 30, None) == binding.OBF_ERR_INVALID_ARG
    assert lib.obf_compress(pp, arr, 1, None, 1 << 30, None) == binding.OBF_ERR_WORKSPACE
    assert lib.obf_compress(pp, arr, 1, 0x101, 1 << 30, None) == binding.OBF_ERR_WORKSPACE     # misaligned
    assert lib.obf_compress(pp, arr, 1, 0x100, 16, None) == binding.OBF_ERR_WORKSPACE          # too small
    null_k = (binding.ObfCache * 1)(P.make_cache(None, 0x1000, 0x1000, 256, 32, 0x1000, 0x1000, 0x1000))
    assert lib.obf_compress(pp, null_k, 1, 0x100, 1 << 30, None) == binding.OBF_ERR_INVALID_ARG
    odd = (binding.ObfCache * 1)(P.make_cache(0x1004, 0x1000, 0x1000, 256, 32, 0x1000, 0x1000, 0x1000))
    assert lib.evict_only(pp, odd, 1, 0x100, 1 << 30, None) == binding.OBF_ERR_INVALID_ARG
    assert lib.obf_compress_host(pp, arr, 1, None, 0, None) == binding.OBF_ERR_WORKSPACE
    assert lib.obf_last_launch_count() == 0


@pytest.mark.parametrize("dtype", [P.OBF_F32, P.OBF_BF16])
@pytest.mark.parametrize("T", [300, 4000])
def test_a_workspace_smaller_than_reported_is_refused(lib, dtype, T):
    # also where the shape-generic kernels could make do with less
    params, caches = _params(dtype=dtype, flags=binding.OBF_FLAG_GENERIC_PATH), [_cache(T=T)]
    need = P.obf_workspace_bytes(params, caches)
    for call in (P.obf_compress, P.evict_only):
        if call is P.evict_only:
            params.rank = 0
            need = P.obf_workspace_bytes(params, caches)
        assert call(params, caches, 0x1000, need - 1, stream=0, check=False) == binding.OBF_ERR_WORKSPACE


@pytest.mark.parametrize("dtype", [P.OBF_F32, P.OBF_BF16])
def test_the_host_arena_holds_the_workspace_of_every_slab_of_layers(lib, dtype):
    # the host-staged call works on four slabs of layers; a slab's heads can be split more finely than the whole call's
    e = 4 if dtype == P.OBF_F32 else 2

    def up(x):
        return (x + 255) // 256 * 256

    for kv_heads, d, n_obs in ((8, 64, 8), (8, 128, 16), (3, 128, 48), (1, 64, 40)):
        for layers in list(range(1, 41)) + [99]:
            for T in (129, 400, 1024, 3000):
                params = _params(layers=layers, kv_heads=kv_heads, q_heads=4 * kv_heads, head_dim=d, n_obs=n_obs, rank=2, dtype=dtype)
                cache = _cache(T=T, budget=20)
                rows = layers * kv_heads
                data = (2 * up(rows * T * d * e) + up(rows * 4 * n_obs * d * e) + 2 * up(rows * 20 * d * e) + up(rows * 20 * 4)
                        + up(rows * binding.DIAG_BYTES) + up(rows * d * 4))
                room = P.obf_host_arena_bytes(params, [cache]) - data
                n = min(layers, 4)
                for sl in range(n):
                    params.layers = layers * (sl + 1) // n - layers * sl // n
                    assert P.obf_workspace_bytes(params, [cache]) <= room, (kv_heads, d, layers, T, sl)


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(build, "LIB_PATH", str(tmp_path / "nope.so"))
    with pytest.raises(RuntimeError, match="no CPU fallback"):
        binding.load()
