"""CPU-only checks of the C-ABI boundary: the library loads, exports every symbol the header
declares, and its host-side validation returns status codes (no kernel is launched)."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "include", "wersa.h")


@pytest.fixture(scope="module")
def lib():
    from paper_2507_08637_b200 import build
    path = build.build()
    return ctypes.CDLL(path)


def declared_symbols():
    text = open(HEADER).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(wersa_[a-z_0-9]+)\s*\(", text)))


def test_header_declares_the_four_core_entry_points():
    syms = declared_symbols()
    for name in ("wersa_create", "wersa_forward", "wersa_backward", "wersa_destroy"):
        assert name in syms


def test_library_exports_every_declared_symbol(lib):
    for name in declared_symbols():
        assert hasattr(lib, name), name


def _cfg(**kw):
    from paper_2507_08637_b200 import make_config
    base = dict(batch=1, heads=8, seq_len=131072, head_dim=64, levels=8, features=256)
    base.update(kw)
    return make_config(**base)


def test_workspace_bytes_and_validation():
    import paper_2507_08637_b200 as w
    full = w.wersa_workspace_bytes(_cfg())
    fwd_only = w.wersa_workspace_bytes(_cfg(flags=w.WERSA_FLAG_FORWARD_ONLY))
    assert full % 256 == 0 and 0 < fwd_only < full
    # invalid or unsupported configurations give 0
    for bad in (dict(batch=0), dict(heads=-1), dict(seq_len=1), dict(head_dim=128), dict(head_dim=20), dict(levels=0),
                dict(levels=9), dict(features=100), dict(features=1280), dict(features=512, dtype="f32"),
                dict(features=512, flags=w.WERSA_FLAG_SIMT_ONLY), dict(seq_len=100, levels=8), dict(eps=-1.0),
                dict(bw_floor=0.0)):
        assert w.wersa_workspace_bytes(_cfg(**bad)) == 0, bad
    # narrower heads run zero-padded (more workspace); feature maps up to 1024 run in groups of 256 (bf16)
    assert w.wersa_workspace_bytes(_cfg(head_dim=32)) > full
    assert w.wersa_workspace_bytes(_cfg(head_dim=16, dtype="f32", features=64)) > 0
    assert w.wersa_workspace_bytes(_cfg(features=1024)) > fwd_only
    assert w.wersa_workspace_bytes(_cfg(features=512, head_dim=32)) > 0
    # 2^L may reach the next power of two above n (zero padding of the wavelet transform)
    assert w.wersa_workspace_bytes(_cfg(seq_len=200, levels=8)) > 0


def test_workspace_of_fp32_on_the_tensor_cores():
    """Operands as planes against the FFMA kernels' workspace: 18 bytes an element of a tensor against 8 for a forward, 32
    against 16 with a backward, by the head's own width where the FFMA kernels' is 64 columns always, and a 20th for the
    per-token and per-slab arrays; the FFMA kernels' own where the planes would take more than 64 GiB."""
    import paper_2507_08637_b200 as w

    def nbytes(flags, **shape):
        return w.wersa_workspace_bytes(_cfg(dtype="f32", grad_dtype="f32", flags=flags, levels=4, **shape))

    for shape in (dict(batch=2, heads=8, seq_len=4096), dict(batch=1, heads=8, seq_len=30000)):
        for features in (128, 256):
            for d in (8, 16, 32, 64):
                kw = dict(shape, features=features, head_dim=d)
                fwd, ffma_fwd = (nbytes(f | w.WERSA_FLAG_FORWARD_ONLY, **kw) for f in (0, w.WERSA_FLAG_SIMT_ONLY))
                train, ffma_train = nbytes(0, **kw), nbytes(w.WERSA_FLAG_SIMT_ONLY, **kw)
                tensor = shape["batch"] * shape["heads"] * shape["seq_len"] * 64
                assert fwd <= ffma_fwd + (18 * d / 64 - 8 + 0.9) * tensor, (kw, fwd, ffma_fwd)
                assert train <= ffma_train + (32 * d / 64 - 16 + 1.6) * tensor, (kw, train, ffma_train)
    for flags in (0, w.WERSA_FLAG_FORWARD_ONLY):
        kw = dict(batch=64, heads=64, seq_len=32768, features=256)
        assert nbytes(flags, **kw) == nbytes(flags | w.WERSA_FLAG_SIMT_ONLY, **kw)


def test_create_rejects_bad_arguments_without_a_device(lib):
    import paper_2507_08637_b200 as w
    lib.wersa_create.restype = ctypes.c_int
    lib.wersa_create.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p]
    handle = ctypes.c_void_p()
    cfg = _cfg()
    need = w.wersa_workspace_bytes(cfg)
    assert lib.wersa_create(None, None, 0, ctypes.byref(handle)) == 1
    assert lib.wersa_create(ctypes.byref(cfg), None, need, ctypes.byref(handle)) == 3
    assert lib.wersa_create(ctypes.byref(cfg), ctypes.c_void_p(256), need - 1, ctypes.byref(handle)) == 3
    assert lib.wersa_create(ctypes.byref(cfg), ctypes.c_void_p(257), need, ctypes.byref(handle)) == 3
    bad = _cfg(features=100)
    assert lib.wersa_create(ctypes.byref(bad), ctypes.c_void_p(256), 1 << 40, ctypes.byref(handle)) == 2
    bad = _cfg(levels=0)
    assert lib.wersa_create(ctypes.byref(bad), ctypes.c_void_p(256), 1 << 40, ctypes.byref(handle)) == 1
    assert handle.value is None
    # a context is host memory only: creating and destroying one touches no device
    assert lib.wersa_create(ctypes.byref(cfg), ctypes.c_void_p(256), need, ctypes.byref(handle)) == 0
    lib.wersa_launch_count.argtypes = [ctypes.c_void_p, ctypes.c_int]
    assert lib.wersa_launch_count(handle, 0) == 0
    lib.wersa_forward.restype = ctypes.c_int
    lib.wersa_forward.argtypes = [ctypes.c_void_p] * 11
    assert lib.wersa_forward(handle, None, None, None, None, None, None, None, None, None, None) == 1
    lib.wersa_forward_host.restype = ctypes.c_int
    lib.wersa_forward_host.argtypes = [ctypes.c_void_p] * 15
    assert lib.wersa_forward_host(handle, *([None] * 14)) == 1
    assert lib.wersa_forward_host(None, *([ctypes.c_void_p(256)] * 14)) == 1
    lib.wersa_destroy.argtypes = [ctypes.c_void_p]
    assert lib.wersa_destroy(handle) == 0
    assert lib.wersa_destroy(None) == 0


def test_status_strings(lib):
    lib.wersa_status_string.restype = ctypes.c_char_p
    seen = {lib.wersa_status_string(i) for i in range(7)}
    assert len(seen) == 7 and all(s for s in seen)


def test_plan_does_not_depend_on_what_its_memory_held(lib):
    """Every part of a plan is decided when it is made, also what wersa_create decides again where there is a device: made over
    memory of two fills, it differs nowhere but behind its end."""
    make_plan = lib._ZN5wersa9make_planERK12wersa_configPNS_4PlanE   # wersa::make_plan(const wersa_config&, Plan*)
    size = 4096
    for kw in (dict(), dict(features=64), dict(features=1024), dict(dtype="f32"), dict(dtype="f32", features=64, seq_len=500)):
        plans = []
        for fill in (0x55, 0xAA):
            plan = ctypes.create_string_buffer(bytes([fill]) * size, size)
            assert make_plan(ctypes.byref(_cfg(**kw)), plan) == 0
            plans.append(plan.raw)
        first = next(i for i in range(size) if plans[0][i] != plans[1][i])
        assert all(plans[0][i] != plans[1][i] for i in range(first, size)), kw


@pytest.mark.parametrize("slabs,n,dtype", [(1, 16000, "bf16"), (1, 4000, "f32"), (8, 16384, "bf16"), (40, 2500, "bf16"), (8, 131072, "bf16")])
def test_static_gate_cuts_a_slab_as_documented(lib, slabs, n, dtype):
    """The mean pool of wersa_gate_static is no cluster, whatever contexts of the shape take: about four row chunks per
    multiprocessor over all slabs, of 128 rows and more, in its scratch one after the other."""
    make_plan = lib._ZN5wersa9make_planERK12wersa_configPNS_4PlanE   # wersa::make_plan(const wersa_config&, Plan*)
    needed = lib._ZN5wersa28static_scratch_floats_neededERKNS_4PlanE   # wersa::static_scratch_floats_needed(const Plan&)
    needed.restype = ctypes.c_size_t
    plan = ctypes.create_string_buffer(4096)
    assert make_plan(ctypes.byref(_cfg(batch=1, heads=slabs, seq_len=n, head_dim=64, levels=3, features=256, dtype=dtype)), plan) == 0
    chunks = min(-(-592 // slabs), -(-n // 128))
    rows = -(-(-(-n // chunks)) // 32) * 32
    assert needed(plan) == slabs * (64 * -(-n // rows) + 4)


def test_static_gate_makes_no_tile_plan():
    """wersa_gate_static needs none of the choices that fp32 contexts search for: refusing a problem that does not fit its
    array takes an fp32 call the time it takes a bf16 one (least of 20 batches of 200 calls)."""
    import time
    import paper_2507_08637_b200 as w
    from paper_2507_08637_b200 import binding
    lib, at = binding._lib(), ctypes.c_void_p(256)
    least = {}
    for dtype, features in (("f32", 64), ("bf16", 128)):
        cfg = _cfg(batch=8000, heads=1, seq_len=20000, levels=3, features=features, dtype=dtype)   # 16000 counters: too many
        args = (ctypes.byref(cfg), at, None, None, at, at, at, None)
        assert lib.wersa_gate_static(*args) == 7
        times = []
        for _ in range(20):
            t0 = time.perf_counter()
            for _ in range(200):
                lib.wersa_gate_static(*args)
            times.append((time.perf_counter() - t0) / 200)
        least[dtype] = min(times)
    assert least["f32"] <= least["bf16"] + 1e-6, least


def test_current_stream_without_torch_internals(monkeypatch):
    """The current stream's handle comes from torch's public interface where the internal calls are missing."""
    import types
    import torch
    from paper_2507_08637_b200 import binding
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=4321))
    for name in ("_raw_stream", "_current_device"):
        with monkeypatch.context() as m:
            m.setattr(binding, name, None)
            assert binding._stream_ptr(None) == 4321
    monkeypatch.setattr(binding, "_current_device", lambda: 3)
    monkeypatch.setattr(binding, "_raw_stream", lambda device: 100 + device)
    assert binding._stream_ptr(None) == 103
    assert binding._stream_ptr(types.SimpleNamespace(cuda_stream=7)) == 7
