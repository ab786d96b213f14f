"""The call module's behaviour at its edges.  What could take the test process down runs in a child process."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest
import torch

from paper_2605_13915_b200 import binding

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _child(code):
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


def test_exceptions_of_the_tensor_library_become_python_exceptions():
    """An exception of the tensor library (here from asking for a stream without a driver, or for the address of a tensor without
    storage) is raised in Python; one that left the C++ code would end the process."""
    out = _child("""
        import torch
        from torch._subclasses.fake_tensor import FakeTensorMode
        from paper_2605_13915_b200 import binding
        calls = binding._calls()
        with FakeTensorMode():
            t = lambda *s, dtype=torch.int8: torch.empty(*s, dtype=dtype, device="cuda")
            x, w, s, y = t(16, 64, dtype=torch.bfloat16), t(32, 64), t(32, dtype=torch.float32), t(16, 32, dtype=torch.bfloat16)
            ws = t(4096, dtype=torch.uint8)
            q = t(1, 4, 64, dtype=torch.bfloat16)
            k, ks, cu = t(8, 1, 64), t(8, 1, dtype=torch.float32), t(2, dtype=torch.int32)
            w3, s2 = t(1, 32, 64), t(1, 32, dtype=torch.float32)
            for name, args in (("gemm_w8a16", (x, w, s, ws, y, None, 0)), ("gemm_w4a16", (x, w, s, 1, ws, y)),
                               ("grouped_gemm_w8a16", (x, w3, s2, [16], ws, y)),
                               ("grouped_gemm_w4a16", (x, t(1, 32, 32), s2, [16], 1, ws, y)),
                               ("attn_decode_int8kv", (q, k, k, ks, ks, cu, 8, 0.1, 64, ws, q, None)),
                               ("attn_decode_int8kv_spec", (q[None], k, k, ks, ks, cu, 8, 0.1, 64, ws, q[None], None)),
                               ("attn_decode_int8kv_paged", (q, k, k, ks, ks, cu[None], cu, 8, 8, 0.1, 64, ws, q, None))):
                try:
                    print("refused" if getattr(calls, name)(*args) != binding.MSD_OK else "launched", name)
                except RuntimeError as e:
                    print("raised", name)
        """)
    # (with a driver a fake tensor's address is null, which the library refuses; without one, asking for the stream throws)
    assert out.count("raised") + out.count("refused") == 7 and "launched" not in out


def test_workspace_that_ends_before_its_first_boundary_is_empty():
    """The wrappers that go through ctypes: what lies before the first 1024-byte boundary is no workspace, and none is left of a
    tensor that ends there (the difference, as an unsigned size, would pass for any amount)."""
    buf = torch.zeros(4096, dtype=torch.uint8)
    off = -buf.data_ptr() % 1024
    assert binding._ws_ptr(buf[off + 1:off + 2])[1] == 0
    assert binding._ws_ptr(buf[off:off + 2048])[1] == 2048
    assert binding._ws_ptr(buf[off:off + 2048].view(torch.int32))[1] == 2048      # bytes, whatever the elements
    assert binding._ws_ptr(buf[off + 1000:off + 2048])[1] == 1024



def test_module_built_for_another_torch_is_stale(monkeypatch):
    from paper_2605_13915_b200 import build
    binding.lib()
    assert not build.needs_build()
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".post1")
    assert build.needs_build()


@pytest.mark.gpu
def test_workspace_and_outputs_are_checked():
    """Workspaces that are too small are refused however they lie; outputs and workspaces that the kernels cannot write are refused
    before a launch."""
    dev = "cuda"
    x, w, s = torch.ones(16, 64, dtype=torch.bfloat16, device=dev), torch.ones(64, 64, dtype=torch.int8, device=dev), torch.ones(64, device=dev)
    y = torch.empty(16, 64, dtype=torch.bfloat16, device=dev)
    need = binding.gemm_w8a16_workspace_bytes(16, 64, 64)
    buf = torch.zeros(need + 4096, dtype=torch.uint8, device=dev)
    off = -buf.data_ptr() % 1024
    for ws in (buf[off + 1:off + 2], buf[off + 1:off + 2 + need], buf[off:off + need - 1]):
        with pytest.raises(binding.MsdError) as e:
            binding.gemm_w8a16(x, w, s, ws=ws, out=y)
        assert e.value.code == 5                                     # MSD_ERR_WORKSPACE_TOO_SMALL
    good = buf[off:off + need]
    assert torch.equal(binding.gemm_w8a16(x, w, s, ws=good, out=y), torch.full_like(y, 64.0))
    wide = torch.empty(16, 128, dtype=torch.bfloat16, device=dev)
    for bad in (dict(ws=good, out=y.cpu()), dict(ws=good.cpu(), out=y), dict(ws=good, out=wide[:, :64]), dict(ws=good, out=y.T)):
        with pytest.raises(ValueError):
            binding.gemm_w8a16(x, w, s, **bad)
    for bad in (y.to_sparse(), torch.empty(16, 64, dtype=torch.bfloat16, device="meta")):
        with pytest.raises((RuntimeError, ValueError)):
            binding.gemm_w8a16(x, w, s, ws=good, out=bad)
    torch.cuda.synchronize()
    binding.last_device_status()


@pytest.mark.gpu
def test_other_python_threads_run_during_a_call(tmp_path):
    """A launch waits where the stream's queue is full; the interpreter's other threads must not wait with it.  A stand-in for the
    library's function that sleeps takes its place in the child, so that nothing is launched."""
    (tmp_path / "slow.c").write_text("#include <unistd.h>\nint msd_gemm_w8a16_ex() { usleep(1500000); return 0; }\n")
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(tmp_path / "slow.so"), str(tmp_path / "slow.c")], check=True)
    out = _child(f"""
        import ctypes, threading, time
        ctypes.CDLL({str(tmp_path / "slow.so")!r}, mode=ctypes.RTLD_GLOBAL)
        import torch
        from paper_2605_13915_b200 import binding
        calls = binding._calls()
        t = lambda *s, dtype=torch.int8: torch.zeros(*s, dtype=dtype, device="cuda")
        args = (t(16, 64, dtype=torch.bfloat16), t(32, 64), t(32, dtype=torch.float32), t(4096), t(16, 32, dtype=torch.bfloat16), None, 0)
        torch.cuda.synchronize()
        spent = []
        def call():
            t0 = time.monotonic()
            calls.gemm_w8a16(*args)
            spent.append(time.monotonic() - t0)
        thread = threading.Thread(target=call)
        t0 = time.monotonic()
        thread.start()
        time.sleep(0.2)
        print("others", time.monotonic() - t0)
        thread.join()
        print("call", spent[0])
        """)
    took = dict(line.split() for line in out.splitlines())
    assert float(took["call"]) >= 1.4 and float(took["others"]) < 1.0


@pytest.mark.gpu
def test_argument_forms():
    """Rows per expert as anything that int() takes; a missing scale or length array is the library's null pointer, a page size it
    does not know its MSD_ERR_UNSUPPORTED."""
    dev = "cuda"
    x, w, s = torch.ones(5, 64, dtype=torch.bfloat16, device=dev), torch.ones(2, 64, 64, dtype=torch.int8, device=dev), torch.ones(2, 64, device=dev)
    want = torch.full((5, 64), 64.0, dtype=torch.bfloat16, device=dev)
    for sizes in ([2, 3], (2.0, 3.0), np.array([2, 3]), np.array([2.0, 3.0], np.float32), torch.tensor([2, 3]), torch.tensor([2.0, 3.0]),
                  ["2", "3"]):
        assert torch.equal(binding.grouped_gemm_w8a16(x, w, s, sizes), want)
    with pytest.raises(ValueError):
        binding.grouped_gemm_w8a16(x, w, s, ["two", 3])
    with pytest.raises(AssertionError):
        binding.grouped_gemm_w8a16(x, w, s, [2, 2])

    def code(fn, *args, **kw):
        with pytest.raises(binding.MsdError) as e:
            fn(*args, **kw)
        return e.value.code
    assert code(binding.gemm_w8a16, x, w[0], None) == 1
    q, k, ks = torch.ones(1, 4, 64, dtype=torch.bfloat16, device=dev), torch.ones(16, 1, 64, dtype=torch.int8, device=dev), torch.ones(16, 1, device=dev)
    cu, table, lens = (torch.tensor(v, dtype=torch.int32, device=dev) for v in ([0, 16], [[0, 1]], [16]))
    assert code(binding.attn_decode_int8kv, q, k, k, None, ks, cu, 16, 0.125) == 1
    assert code(binding.attn_decode_int8kv, q, k, k, ks, ks, None, 16, 0.125) == 1
    assert code(binding.attn_decode_int8kv_paged, q, k, k, ks, ks, table, None, 8, 16, 0.125) == 1
    for page in (-8, 0, 24):
        assert code(binding.attn_decode_int8kv_paged, q, k, k, ks, ks, table, lens, page, 16, 0.125) == 4
    split = binding.attn_decode_int8kv(q, k.view(16, 1, 4, 16), k, ks, ks, cu, 16, 0.125)       # rows in pieces: the same bytes
    assert torch.equal(split, binding.attn_decode_int8kv(q, k, k, ks, ks, cu, 16, 0.125))
    torch.cuda.synchronize()
    binding.last_device_status()
