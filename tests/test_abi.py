"""The C-ABI library loads, exports every symbol the header declares, and rejects bad arguments on the host
(no GPU needed: nothing here launches a kernel)."""
import ctypes
import os
import re
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def binding():
    from paper_2507_05228_b200 import build
    build.build_library()
    from paper_2507_05228_b200 import binding as b
    return b


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "cascade.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(cascade_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(binding):
    names = _declared_functions()
    assert {"cascade_shard_plan", "cascade_attn_partials", "cascade_merge", "cascade_attn_sharded"} <= set(names)
    L = binding.lib()
    for n in names:
        assert hasattr(L, n), n
    assert set(binding.EXPORTS) == set(names)
    assert binding.cascade_version() >= 100


def test_library_does_not_import_or_link_the_oracle():
    pkg = os.path.join(ROOT, "paper_2507_05228_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                src = open(os.path.join(dirpath, f)).read()
                assert "oracle" not in src.lower() or f == "workloads.py", f
    src = open(os.path.join(pkg, "workloads.py")).read()
    assert "import oracle" not in src and "from oracle" not in src


def test_host_side_argument_checks(binding):
    L = binding.lib()
    out = ctypes.c_void_p()
    good = np.zeros(8, np.int32)
    p = good.ctypes.data_as(ctypes.c_void_p)
    assert L.cascade_shard_plan_host(1, 8, 8, None, p, 1, 1, 0, 1, ctypes.byref(out)) == 1
    assert L.cascade_shard_plan_host(1, 0, 8, p, p, 1, 1, 0, 1, ctypes.byref(out)) == 1
    bad = np.array([0, 1, 2, 5, 0, 1, 2, 0], np.int32)
    assert L.cascade_shard_plan_host(1, 8, 8, bad.ctypes.data_as(ctypes.c_void_p), p, 3, 1, 0, 1,
                                     ctypes.byref(out)) == 2
    assert b"q_shard_of[3] = 5" in L.cascade_last_error()
    neg = np.array([0, -1], np.int32)
    assert L.cascade_shard_plan_host(1, 2, 2, neg.ctypes.data_as(ctypes.c_void_p), p, 1, 1, 0, 1,
                                     ctypes.byref(out)) == 2
    # merge: null pointers / unsupported shapes are refused before any CUDA call
    S = binding.Strides(0, 0, 0)
    assert L.cascade_merge(1, 1, 2, 4, 2, 128, None, None, None, None, 0, None, S, None, None) == 1
    assert L.cascade_merge(1, 1, 2, 4, 2, 96, 256, 256, 256, None, 0, 256, S, None, None) == 3
    assert L.cascade_merge(7, 1, 2, 4, 2, 128, 256, 256, 256, None, 0, 256, S, None, None) == 3
    assert L.cascade_merge(1, 1, 2, 4, 2, 128, 264, 256, 256, None, 0, 256, S, None, None) == 1  # misaligned
    # a host-only plan is readable but cannot be used by the attention calls
    plan = binding.cascade_shard_plan_host(good, good, 1, 1)
    assert plan.get("q_idx").tolist() == [list(range(8))]
    S4 = binding.Strides(1024, 128, 128)
    rc = L.cascade_attn_partials(plan.handle, 1, 1, 1, 1, 128, 1.0, 256, S4, 256, S4, 256, S4, 256, 256, 256,
                                 None, 0, None)
    assert rc == 1 and b"cascade_shard_plan_host" in L.cascade_last_error()
    # the host-buffer call refuses null pointers and a host-only plan before touching CUDA; its workspace size is
    # staging for q, k, v, o plus one head group's scratch
    hb = np.zeros(16, np.uint8).ctypes.data_as(ctypes.c_void_p)
    assert L.cascade_attn_sharded_host(plan.handle, 1, 1, 4, 2, 128, 1.0, None, hb, hb, hb, hb, 0, None) == 1
    assert L.cascade_attn_sharded_host(plan.handle, 1, 1, 4, 2, 128, 1.0, hb, hb, hb, hb, hb, 0, None) == 1
    assert b"cascade_shard_plan_host" in L.cascade_last_error()
    nbytes = ctypes.c_size_t()
    assert L.cascade_workspace_bytes(plan.handle, 2, 1, 1, 4, 2, 128, ctypes.byref(nbytes)) == 0
    q_b, kv_b = 8 * 4 * 128 * 2, 8 * 2 * 128 * 2
    assert nbytes.value >= 2 * q_b + 2 * kv_b and nbytes.value % 256 == 0
    assert L.cascade_workspace_bytes(plan.handle, 0, 1, 1, 4, 3, 128, ctypes.byref(nbytes)) == 1
    assert L.cascade_workspace_bytes(plan.handle, 9, 1, 1, 4, 2, 128, ctypes.byref(nbytes)) == 1
    plan.destroy()


def test_workspace_of_the_tensor_core_route_is_two_copies(binding):
    """A copy of K and one of V, each rounded up to 256 bytes, for every call: programs size it by this documented sum."""
    plan = binding.cascade_shard_plan_host(np.zeros(77, np.int32), np.zeros(77, np.int32), 1, 1)
    for B, H, Hkv in ((1, 4, 4), (3, 6, 2)):
        for d in (64, 128):
            copies = 2 * ((B * Hkv * 77 * d * 2 + 255) // 256 * 256)
            for call in (binding.CALL_PARTIALS, binding.CALL_SHARDED):
                assert binding.cascade_workspace_bytes(plan, call, binding.BF16, B, H, Hkv, d) == copies
    plan.destroy()


def test_workspace_of_split_fp32_operands_is_asked_for_where_they_are_used(binding):
    """fp32, heads of 64: three bf16 copies of K and of V and their flags, or nothing where the ALU kernels are taken."""
    def need(n_q, n_kv, B, H, off, causal, call):
        plan = binding.cascade_shard_plan_host(np.arange(n_q, dtype=np.int32) % 4, np.arange(n_kv, dtype=np.int32) % 4, 4, 4, off, causal)
        n = binding.cascade_workspace_bytes(plan, call, binding.F32, B, H, H, 64)
        plan.destroy()
        return n

    def copies(n_kv, mats):
        return 2 * (-(-3 * mats * n_kv * 128 // 256) * 256) + -(-2 * mats * -(-n_kv // 64) // 256) * 256

    sharded, partials, host = binding.CALL_SHARDED, binding.CALL_PARTIALS, binding.CALL_SHARDED_HOST
    for call in (sharded, partials):
        assert need(512, 512, 16, 16, 0, False, call) == copies(512, 256)
        assert need(33, 33, 1, 8, 0, False, call) == 0
        # a block of queries that is moved along a cache: the same wherever it stands, as scratch is taken once
        assert need(256, 8192, 4, 16, 0, True, call) == need(256, 8192, 4, 16, 7936, True, call) == copies(8192, 64)
    staging = lambda n, B, H: 4 * (B * n * H * 64 * 4)  # (multiples of 256)
    assert need(256, 256, 1, 8, 0, True, host) == staging(256, 1, 8)
    assert need(512, 512, 16, 16, 0, False, host) == staging(512, 16, 16) + copies(512, 16 * 4)  # four heads at a time


def test_tensors_without_storage_raise(binding):
    """torch.func.vmap hands out tensors that throw when asked for their data pointer.  In a child process: an exception that
    leaves the interpreter lock released takes the interpreter down with it."""
    code = """
import numpy as np, torch
from paper_2507_05228_b200 import binding as cb
plan = cb.cascade_shard_plan_host(np.zeros(4, np.int32), np.zeros(4, np.int32), 1, 1)
one = cb.cascade_shard_plan_host(np.zeros(1, np.int32), np.zeros(4, np.int32), 1, 1)
table = torch.zeros(8, 64, 2)
calls = {
    "sharded": lambda x: cb.cascade_attn_sharded(plan, x, x, x, 1.0, want_lse=False)[0],
    "rope": lambda x: cb.cascade_attn_sharded_rope(plan, x, x, x, 1.0, table, want_lse=False)[0],
    "partials": lambda x: cb.cascade_attn_partials(plan, x, x, x, 1.0)[0],
    "merge": lambda x: cb.cascade_merge(x[None], x[None, ..., 0], x[None, ..., 0], want_lse=False)[0],
    "step": lambda x: cb.cascade_decode_step_rope(one, x[:, :1], x[:, :1], x[:, :1], x, x, 0, 1.0, table, want_lse=False)[0],
    "static": lambda x: cb.cascade_attn_decode_static(one, x[:, :1], x, x, 1.0, want_lse=False)[0],
}
for name, call in calls.items():
    try:
        torch.func.vmap(call)(torch.zeros(3, 1, 4, 2, 128, dtype=torch.bfloat16))
    except RuntimeError as e:
        assert "data pointer" in str(e), (name, e)
    else:
        raise AssertionError(name)
print("all raised")
"""
    run = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert run.returncode == 0 and "all raised" in run.stdout, (run.returncode, run.stderr[-2000:])
