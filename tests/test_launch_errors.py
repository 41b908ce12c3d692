"""Every launch that fails is reported by the call that made it: the library's host code on a CUDA runtime without a device, whose
launches fail one at a time."""
import ctypes
import glob
import os
import subprocess

import pytest
import torch

from paper_2608_04405_b200 import binding as B
from paper_2608_04405_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
N = 512
WORK = [("bf16", 64, 2, {}), ("bf16", 128, 16, {}), ("bf16", 256, 2, {}), ("f32", 64, 2, {}), ("f32", 128, 16, {}),
        ("bf16", 64, 2, {"small": True}), ("f32", 32, 2, {"small": True}), ("bf16", 64, 2, {"fit_power_iters": 1}),
        ("bf16", 128, 2, {"eas_ppm": 20000}), ("bf16", 128, 2, {"score_mode": 1})]


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    build.build_library()
    so = str(tmp_path_factory.mktemp("fake") / "libbpc_fake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.NVCC)), "include")
    subprocess.run(["g++", "-shared", "-fPIC", "-I" + cuda, "-Wl,-Bsymbolic", "-o", so, os.path.join(HERE, "fake_cudart.cpp"),
                    *glob.glob(os.path.join(build.OBJ, "*.o"))], check=True)
    return so


@pytest.fixture
def lib(fake, monkeypatch):
    monkeypatch.setattr(B, "LIB_PATH", fake)
    monkeypatch.setattr(B, "lib", B._load())
    monkeypatch.setattr(B, "_stream", lambda: 0)
    B.lib.contexts = []
    yield B.lib
    for ctx in B.lib.contexts:
        ctx.close()


def _calls(dtype, bits, units, small=False, **options):
    """The context, memory that the calls are given, and a user's calls in order, each by name."""
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    ctx = B.Context(B.make_config(units, 2, 1, N, bits, dt, **options))
    B.lib.contexts.append(ctx)
    ctx.set_seq_lens([N - 2] * units)
    aligned = torch.zeros(16 << 20, dtype=torch.uint8)
    ptr = aligned.data_ptr() + 63 & ~63
    raw = B.lib
    h, cfg = ctx._h, ctx.cfg
    ws = B.lib.bpc_fit_workspace_min_bytes(ctypes.byref(cfg)) if small else ctx.fit_workspace_bytes()
    calls = [("set_projection", lambda: raw.bpc_set_projection(h, ptr, None)),
             ("fit", lambda: raw.bpc_fit(h, ptr, ptr, ptr, ws, None)),
             ("encode", lambda: raw.bpc_encode_keys(h, ptr, ptr, None)),
             ("append", lambda: raw.bpc_append(h, ptr, ptr, ptr, ptr, ptr, None)),
             ("decode", lambda: raw.bpc_decode_attn(h, ptr, ptr, ptr, ptr, 20000, 0, ptr, None, None)),
             ("step", lambda: raw.bpc_append_decode_attn(h, ptr, ptr, ptr, ptr, ptr, ptr, 20000, 0, ptr, None, None)),
             ("exact", lambda: raw.bpc_exact_topk(h, ptr, ptr, 20000, 0, ptr, ptr, ptr, None))]
    if options.get("eas_ppm"):
        calls.insert(3, ("build_eas", lambda: raw.bpc_build_eas(h, None)))
    return ctx, aligned, calls


@pytest.mark.parametrize("dtype,bits,units,options", WORK)
def test_a_failed_launch_fails_its_call(lib, dtype, bits, units, options):
    ctx, memory, calls = _calls(dtype, bits, units, **options)
    for name, call in calls:
        lib.fake_fail_at(-1)
        assert call() == B.BPC_OK, name
        launches = lib.fake_launches()
        assert launches >= 1, name
        for k in sorted({*range(min(launches, 24)), *range(max(launches - 24, 0), launches)}):
            ctx.set_seq_lens([N - 2] * units)
            lib.fake_fail_at(k)
            assert B.STATUS_NAMES[call()] == "BPC_ERR_CUDA", (name, k, launches)
            assert lib.fake_pending_error() == 0, (name, k)   # (nothing is left for a later call to find)


@pytest.mark.parametrize("dtype,units", [("bf16", 2), ("bf16", 16), ("f32", 2), ("f32", 16)])
def test_a_failed_fit_leaves_no_projection(lib, dtype, units):
    lib.fake_fail_at(-1)
    ctx, memory, calls = _calls(dtype, 64, units)
    assert dict(calls)["fit"]() == B.BPC_OK
    for k in range(lib.fake_launches()):
        lib.fake_fail_at(-1)
        ctx, memory, calls = _calls(dtype, 64, units)
        calls = dict(calls)
        lib.fake_fail_at(k)
        assert B.STATUS_NAMES[calls["fit"]()] == "BPC_ERR_CUDA", k
        assert B.STATUS_NAMES[calls["encode"]()] == "BPC_ERR_NOT_FITTED", k
